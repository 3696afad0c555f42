"""FP64 contractions on the FMA pipe (vp_gemm below the sliced route's size): the
16, 32 and 64 tiles at their edges, one to eight K slices with remainders.

Each element is K fused multiply-adds in some order, partial sums and the factor
alpha: |C - alpha A B| <= (K + 16) 2^-53 |alpha| (|A| |B|) to first order, and an
element of integers below 2^53 is exact.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 1, 4096), (8, 8, 16), (15, 17, 31), (16, 16, 63), (16, 16, 64), (17, 15, 129), (33, 31, 257),
          (56, 30, 128), (64, 64, 500), (129, 127, 255), (200, 3, 700), (3, 700, 200), (513, 4, 2), (700, 700, 33),
          (1025, 515, 17), (240, 240, 240), (70000, 5, 3)]


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    from paper_2205_11990_gb300 import vpmps
    c = vpmps.Context()
    yield c
    c.close()


def dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("shape", SHAPES)
def test_against_extended_precision(ctx, shape):
    M, N, K = shape
    rng = np.random.default_rng(sum(shape))
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    C = ctx.gemm(dev(A), dev(B), alpha=0.75).cpu().numpy()
    rows = np.unique(np.r_[rng.choice(M, min(M, 40), replace=False), M - 1])
    ref = 0.75 * (A[rows].astype(np.longdouble) @ B.astype(np.longdouble))
    bound = (K + 16) * 2.0 ** -53 * (np.abs(A[rows]) @ np.abs(B))
    assert np.all(np.abs(C[rows] - ref) <= bound)


@pytest.mark.parametrize("shape", SHAPES)
def test_integers_exact(ctx, shape):
    M, N, K = shape
    rng = np.random.default_rng(1 + sum(shape))
    A = rng.integers(-2 ** 18, 2 ** 18, size=(M, K))
    B = rng.integers(-2 ** 18, 2 ** 18, size=(K, N))
    C = ctx.gemm(dev(A.astype(np.float64)), dev(B.astype(np.float64)), alpha=-0.5).cpu().numpy()
    assert np.array_equal(C * -2.0, (A @ B).astype(np.float64))
