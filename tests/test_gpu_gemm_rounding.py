"""FP64 contractions of the sliced route are rounded once, to nearest, and are odd in
each operand: 600 x 600 x 64 (its smallest work), of whose products n are nonzero.

Elements in [1/2, 1) are held exactly, so an element of C is off by half an ulp and the
dropped digit products, 2^-60.4 each.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M = N = 600
K = 64


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    from paper_2205_11990_gb300 import vpmps
    c = vpmps.Context()
    yield c
    c.close()


def gemm(ctx, A, B):
    import torch
    return ctx.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()).cpu().numpy()


@pytest.mark.parametrize("n", [1, 3, 5, 8, 11, 16, 60])
def test_half_an_ulp_and_no_bias(ctx, n):
    rng = np.random.default_rng(n)
    a = rng.integers(2 ** 52, 2 ** 53, size=(M, n))
    b = rng.integers(2 ** 52, 2 ** 53, size=(n, N))
    A, B = np.zeros((M, K)), np.zeros((K, N))
    A[:, :n], B[:n] = np.ldexp(a.astype(np.float64), -53), np.ldexp(b.astype(np.float64), -53)
    rows = np.arange(0, M, 15)
    C = gemm(ctx, A, B)[rows]
    exact = a[rows].astype(object) @ b.astype(object)  # times 2^-106
    got = np.ldexp(C, 55).astype(np.int64).astype(object) * 2 ** 51  # an ulp is 2^-55 or more
    err = ((got - exact) / 2.0 ** 106).astype(np.float64)
    ulp = np.spacing(C)
    assert np.all(np.abs(err) <= 0.5 * ulp + n * 2.0 ** -60.4)
    if n > 1:  # 24000 errors of variance 1/12 ulp: five standard deviations of their mean, and the drop
        assert abs(np.mean(err / ulp)) <= 5 * (1 / 12 / err.size) ** 0.5 + 2.0 ** -6


@pytest.mark.parametrize("shape", [(600, 600, 64), (341, 500, 503), (70, 2600, 511)])
def test_odd_in_each_operand(ctx, shape):
    m, n, k = shape
    rng = np.random.default_rng(k)
    A, B = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    C = gemm(ctx, A, B)
    assert np.array_equal(gemm(ctx, -A, B), -C)
    assert np.array_equal(gemm(ctx, A, -B), -C)
