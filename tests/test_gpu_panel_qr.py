"""The panel QR of the sweeps at the edges of its plans, through mps_compress.

An MPS whose bonds double up to the middle gives the QR sweep a factor of
2 r_{k-1} x r_k at every site; the last bonds are small, so that the SVD sweep is
cheap and the dense vector short.  Nothing is truncated beyond tol = 1e-12 per
bond, so the dense vector stays: the bound is (n - 1) tol for the cuts plus, per
site, 200 roundings of 2^-47 of the double-word arithmetic.
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


def dense(cores):
    v = np.ones((1, 1))
    for c in cores:
        v = (v @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
    return v.reshape(-1)


BONDS = [
    [1, 2, 4, 8, 16, 32, 64, 33, 5, 3, 1],                      # one block, whole panels, 32 / 64 rows
    [1, 2, 3, 6, 11, 21, 41, 65, 66, 30, 7, 2, 1],              # last panels of 1, 2, 3 columns, past 64 rows
    [1, 2, 4, 7, 14, 27, 54, 107, 129, 130, 6, 3, 1],           # past 128 rows: two rows a thread
    [1, 2, 4, 8, 16, 32, 64, 100, 190, 257, 300, 5, 1],         # past 256 and 512 rows in a cluster
    [1, 2, 4, 5, 9, 17, 33, 50, 99, 150, 299, 7, 1],            # more columns than rows (n <= 2 m)
    [1, 2, 4, 8, 16, 32, 64, 128, 256, 512, 1024, 5, 3, 1],     # the grid (1024 x 1024), 2048 rows
    [1, 2, 4, 8, 15, 29, 57, 113, 225, 449, 897, 1793, 3, 1],   # ragged; the most rows of a panel thread
]


@pytest.mark.parametrize("bonds", BONDS)
@pytest.mark.parametrize("kind", ["random", "graded", "deficient"])
def test_compression_keeps_the_vector(ctx, bonds, kind):
    rng = np.random.default_rng(len(bonds) + bonds[-4] + len(kind))
    cores = []
    for k in range(len(bonds) - 1):
        c = rng.standard_normal((bonds[k], 2, bonds[k + 1])) / np.sqrt(2 * bonds[k])
        if kind == "graded":
            c = c * np.logspace(0, -9, bonds[k + 1])
        if kind == "deficient" and bonds[k + 1] > 3:  # half the columns repeat the others
            h = bonds[k + 1] // 2
            c[:, :, bonds[k + 1] - h:] = c[:, :, :h]
        cores.append(c)
    ref = dense(cores)
    m = ctx.mps_from_cores(cores)
    ctx.compress(m, 1 << 20, 1e-12)
    err = np.linalg.norm(m.to_dense() - ref) / np.linalg.norm(ref)
    assert err < len(bonds) * (1e-12 + 200 * 2.0 ** -47), err


def test_column_far_below_its_scale(ctx):
    """A residual 1e-28 of its column: squares would leave the FP32 range without
    the rescaling, and the reflector its orthogonality."""
    tiny = 1e-28
    c1 = np.array([[1.0, 1.0], [0.0, tiny], [0.0, 2 * tiny], [0.0, -tiny]]).reshape(2, 2, 2)
    c0 = np.eye(2).reshape(1, 2, 2)
    c2 = np.array([[1.0, 2.0], [-1.0, -2.0]]).reshape(2, 2, 1)  # cancels the first column exactly
    ref = dense([c0, c1, c2])
    assert 0 < np.max(np.abs(ref)) < 1e-26
    m = ctx.mps_from_cores([c0, c1, c2])
    ctx.compress(m, 8, 1e-12)
    assert np.linalg.norm(m.to_dense() - ref) < 1e-11 * np.linalg.norm(ref)


def test_zero_columns(ctx):
    c = [np.zeros((1, 2, 6)), np.zeros((6, 2, 5)), np.ones((5, 2, 1))]
    c[0][0, 1, 2] = 3.0
    c[1][2, 0, 4] = -2.0
    m = ctx.mps_from_cores(c)
    ctx.compress(m, 8, 1e-12)
    assert np.allclose(m.to_dense(), dense(c), rtol=0, atol=1e-13)
