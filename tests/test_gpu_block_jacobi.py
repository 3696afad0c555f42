"""The block Jacobi SVD at the edges of its plans (blocks of odd and even size, one
CTA to a whole cluster, the FP64 kernels beyond), through mps_compress.

Random MPS whose middle bond q is the number of rows of the Jacobi factor.  With
tol = 1e-12 nothing but rounding is cut: the dense vector stays within (n - 1) tol
plus 200 roundings of 2^-47 per site, and every core after the first has orthonormal
rows to the kernel's rotation threshold 4e-13 sqrt(q), doubled, plus as many
roundings.
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


@pytest.mark.parametrize("q", [2, 3, 5, 12, 13, 24, 25, 31, 47, 49, 96, 97, 121, 193, 255, 450])
@pytest.mark.parametrize("grade", [0.0, 9.0])
def test_rows_orthonormal_and_vector_kept(ctx, q, grade):
    rng = np.random.default_rng(q + int(grade))
    half = max(2, int(np.ceil(np.log2(q))))
    bonds = [min(2 ** k, q) for k in range(half + 1)]
    bonds = bonds + bonds[-2::-1]
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) / np.sqrt(2 * bonds[k]) for k in range(len(bonds) - 1)]
    cores[half - 1] = cores[half - 1] * np.logspace(0, -grade, q)
    ref = dense(cores)
    m = ctx.mps_from_cores(cores)
    ctx.compress(m, 1 << 20, 1e-12)
    rounding = 200 * 2.0 ** -47
    err = np.linalg.norm(m.to_dense() - ref) / np.linalg.norm(ref)
    assert err < len(bonds) * (1e-12 + rounding), err
    for c in m.cores()[1:]:
        a = c.reshape(c.shape[0], -1)
        assert np.max(np.abs(a @ a.T - np.eye(a.shape[0]))) < 8e-13 * np.sqrt(max(a.shape)) + rounding


def test_cut_in_the_middle_of_the_spectrum(ctx):
    """chi below every bond: the result equals successive LAPACK SVDs of the unfoldings."""
    rng = np.random.default_rng(3)
    n, chi = 12, 19
    x = rng.standard_normal((64, 64)) @ np.diag(np.logspace(0, -7, 64)) @ rng.standard_normal((64, 64))
    left, right, r = x.reshape(-1) / np.linalg.norm(x), [], 1
    cores, v, rr = [], left.reshape(1, -1), 1
    for k in range(n - 1):  # exact left-canonical cores of x
        u, s, vt = np.linalg.svd(v.reshape(2 * rr, -1), full_matrices=False)
        cores.append(u.reshape(rr, 2, -1))
        v, rr = s[:, None] * vt, s.size
    cores.append(v.reshape(rr, 2, 1))
    for k in range(n - 1, 0, -1):
        u, s, vt = np.linalg.svd(left.reshape(-1, 2 * r), full_matrices=False)
        keep = min(chi, s.size)
        right.append(vt[:keep].reshape(keep, 2, r))
        left, r = u[:, :keep] * s[:keep], keep
    ref = dense([left.reshape(1, 2, r)] + right[::-1])
    m = ctx.mps_from_cores(cores)
    ctx.compress(m, chi, 1e-13)
    assert np.linalg.norm(m.to_dense() - ref) < 1e-10 * np.linalg.norm(ref)
