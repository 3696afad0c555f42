"""FP64 contractions large enough for the sliced route, on operands whose rows and
columns hold elements of very different sizes: every element of the result keeps the
bound of an FP64 sum, whatever else its row and column hold.

The kernel leaves an element (per K slice of at most 512) off by no more than an FP64
sum of its products may be, K 2^-53 (|A| |B|)_ij, rounds it once, and adds the slices;
numpy's own sum is within K 2^-53 (|A| |B|)_ij as well: the two differ by at most
(2 K + 16) 2^-53 (|A| |B|)_ij to first order.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    from paper_2205_11990_gb300 import vpmps
    c = vpmps.Context()
    yield c
    c.close()


def check(ctx, A, B, alpha=1.0):
    import torch
    K = A.shape[1]
    C = ctx.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(np.ascontiguousarray(B)).cuda(), alpha=alpha).cpu().numpy()
    bound = (2 * K + 16) * 2.0 ** -53 * abs(alpha) * (np.abs(A) @ np.abs(B))
    assert np.all(np.abs(C - alpha * (A @ B)) <= bound)


def normals(shape, seed):
    M, N, K = shape
    rng = np.random.default_rng(seed)
    return rng, rng.standard_normal((M, K)), rng.standard_normal((K, N))


@pytest.mark.parametrize("big", [1.0, 1e8, 1e12, 1e16, 1e20, 1e40])
def test_one_large_entry(ctx, big):
    for side in range(2):
        _, A, B = normals((300, 300, 300), 3)
        (A if side == 0 else B)[0, 0] = big
        check(ctx, A, B)


# both tile orientations (128 x 48), more than one K slice, ragged edges
SHAPES = [(300, 290, 300), (641, 497, 65), (129, 49, 3300), (2600, 17, 511), (17, 2600, 511), (385, 145, 1090)]


@pytest.mark.parametrize("shape", SHAPES)
def test_large_entries_against_zeros(ctx, shape):
    """Large columns of A meet rows of B that are zero but for one entry."""
    rng, A, B = normals(shape, sum(shape))
    k = shape[2] // 3
    A[:, k] *= 1e20
    B[k, :] = 0.0
    B[k, shape[1] // 2] = 1e-20
    check(ctx, A, B, alpha=-0.75)


@pytest.mark.parametrize("shape", SHAPES)
def test_every_element_of_its_own_size(ctx, shape):
    rng, A, B = normals(shape, 1 + sum(shape))
    A *= np.exp2(rng.integers(-70, 71, size=A.shape))
    B *= np.exp2(rng.integers(-70, 71, size=B.shape))
    check(ctx, A, B)


@pytest.mark.parametrize("shape", SHAPES)
def test_graded_and_sparse(ctx, shape):
    M, N, K = shape
    rng, A, B = normals(shape, 2 + sum(shape))
    A *= np.exp2(-np.arange(K) * 60.0 / K)[None, :]
    B *= np.exp2(np.arange(K) * 90.0 / K)[:, None]
    check(ctx, A, B)
    A[rng.random(A.shape) < 0.97] = 0.0
    check(ctx, A, B)
    A[:, :K // 2] *= 1e30  # large halves that meet no element
    B[:K // 2, :] = 0.0
    check(ctx, A, B)


def test_subnormal_rows(ctx):
    _, A, B = normals((300, 290, 300), 9)
    A[::3] *= 1e-310
    B *= 1e300
    import torch
    C = ctx.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()).cpu().numpy()
    assert np.all(np.abs(C - A @ B) <= (2 * 300 + 16) * 2.0 ** -53 * (np.abs(A) @ np.abs(B)))


def test_scaled_bonds_keep_their_state(ctx):
    """The sweeps' products (R times the next core, 256 x 512 x 256) on a state whose bonds
    are scaled by powers of two, index by index: scaling is exact, so the compressed state is
    the one of the plain cores to the sweeps' own accuracy: 35 factors, each with
    orthonormality to 1e-13 sqrt(256) = 1.6e-12 at worst, below 1e-10 of the norm together
    (digits lost to the scales would be 2^40 2^-56 of it and more)."""
    rng = np.random.default_rng(4)
    n, q = 18, 256
    bonds = [min(2 ** k, 2 ** (n - k), q) for k in range(n + 1)]
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) for k in range(n)]
    scaled = [c.copy() for c in cores]
    for k in range(1, n):
        s = np.exp2(rng.integers(-40, 41, size=bonds[k]))
        scaled[k - 1] *= s
        scaled[k] /= s[:, None, None]
    out = []
    for cs in (cores, scaled):
        m = ctx.mps_from_cores(cs)
        ctx.compress(m, q, 1e-13)
        x = np.ones((1, 1))
        for c in m.cores():
            x = (x @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
        out.append(x.reshape(-1))
    assert np.linalg.norm(out[1] - out[0]) <= 1e-10 * np.linalg.norm(out[0])
