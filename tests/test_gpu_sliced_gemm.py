"""FP64 contractions sliced over the tensor cores (the route of large vp_gemm
calls in FP64), at the edges of its tiles (128 x 48, K stages of 64, K slices of
at most 512), in both tile orientations and with non-finite operands.

Error bound, per element of C = A B with row scale a_i = max_k |A_ik| and column
scale b_j = max_k |B_kj|: an element is held to 2^-56 of a power of two below
2 a_i (or 2 b_j), and digit products below 2^-61 of the two scales are dropped, so
|C - AB| <= K a_i b_j (2 * 2^-54 + 4 * 2^-61) + 2^-53 |C| per K slice, plus the
rounding of the at most 32 slices' sum: K a_i b_j 2^-52.5 covers all of it with
|C| <= K a_i b_j / 8 for these random operands.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# M, N, K with M N K >= 2e7 (the route's smallest work) and around it
SHAPES = [(1024, 400, 64), (641, 497, 65), (128, 48, 3300), (129, 49, 3300), (127, 2400, 127), (512, 96, 513),
          (16, 2600, 512), (2600, 17, 511), (300, 290, 1025), (385, 145, 577)]


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
def test_random_against_extended_precision(ctx, shape):
    M, N, K = shape
    rng = np.random.default_rng(sum(shape))
    A = rng.standard_normal((M, K)) * np.logspace(0, -9, M)[:, None]
    B = rng.standard_normal((K, N))
    for s in (np.ones(K), np.exp2(rng.integers(-40, 41, size=K))):  # a power of two moved from B's rows to A's columns
        C = ctx.gemm(dev(A * s), dev(B / s[:, None])).cpu().numpy()
        rows, cols = rng.choice(M, min(M, 12), replace=False), rng.choice(N, min(N, 24), replace=False)
        rows[0], cols[0] = M - 1, N - 1
        ref = A[rows].astype(np.longdouble) @ B[:, cols].astype(np.longdouble)
        bound = K * np.max(np.abs(A[rows]), axis=1)[:, None] * np.max(np.abs(B[:, cols]), axis=0)[None, :] * 2.0 ** -52.5
        assert np.all(np.abs(C[np.ix_(rows, cols)] - ref) <= bound)


@pytest.mark.parametrize("shape", SHAPES)
def test_wide_integers_exact(ctx, shape):
    """Integers of 20 bits: every product and sum is an integer below 2^53."""
    M, N, K = shape
    rng = np.random.default_rng(1 + sum(shape))
    A = rng.integers(-2 ** 20, 2 ** 20, size=(M, K))
    B = rng.integers(-2 ** 20, 2 ** 20, size=(K, N))
    C = ctx.gemm(dev(A.astype(np.float64)), dev(B.astype(np.float64)), alpha=-0.25).cpu().numpy()
    assert np.array_equal(C * -4.0, (A @ B).astype(np.float64))


def test_nonfinite_and_subnormal_operands(ctx):
    rng = np.random.default_rng(5)
    M, N, K = 400, 200, 300
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    A[3, 7], A[250, 11], B[9, 60], B[7, 199] = np.inf, np.nan, -np.inf, 0.0
    C = ctx.gemm(dev(A), dev(B)).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = A @ B
    assert np.array_equal(np.isnan(C), np.isnan(ref))
    fin = np.isfinite(ref)
    assert np.array_equal(C[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)])
    assert np.max(np.abs(C[fin] - ref[fin])) < 300 * 25 * 2.0 ** -52
    A, B = rng.standard_normal((M, K)) * 1e-310, rng.standard_normal((K, N)) * 1e300
    C, ref = ctx.gemm(dev(A), dev(B)).cpu().numpy(), A @ B
    assert np.max(np.abs(C - ref)) < 300 * 25 * 2.0 ** -52 * 1e-10
    A, B = rng.standard_normal((M, K)) * 1e-200, rng.standard_normal((K, N)) * 1e-120
    C, ref = ctx.gemm(dev(A), dev(B)).cpu().numpy(), A @ B
    assert np.max(np.abs(C - ref)) <= 300 * 2.0 ** -1074  # subnormal results: an ulp per term
