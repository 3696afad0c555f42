"""The formation of Q from its reflectors at the edges of its plans (32 to 4096 rows
in registers, more in memory; panels of four reflectors with a remainder), through
mps_compress.

Bonds double up to r, then drop to b: the QR sweep forms a Q of 2 r rows and b
columns there and square ones before it.  Nothing is cut beyond tol = 1e-12 per
bond, so the dense vector stays, within (n - 1) tol plus, per site, 200 roundings of
2^-47 of the double-word arithmetic, and every core after the first has orthonormal
rows to twice the Jacobi kernel's threshold 4e-13 sqrt(columns) plus as many.
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


@pytest.mark.parametrize("r,b", [(3, 1), (15, 3), (16, 4), (17, 5), (31, 6), (33, 7), (63, 9), (65, 2), (127, 13), (129, 130),
                                 (255, 31), (257, 3), (511, 6), (513, 5), (1023, 3), (1025, 2), (2049, 3)])
def test_vector_kept_and_rows_orthonormal(ctx, r, b):
    rng = np.random.default_rng(r + b)
    bonds = [1]
    while bonds[-1] < r:
        bonds.append(min(2 * bonds[-1], r))
    bonds += [b]
    while bonds[-1] > 1:
        bonds.append((bonds[-1] + 1) // 2)
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) / np.sqrt(2 * bonds[k]) for k in range(len(bonds) - 1)]
    ref = dense(cores)
    m = ctx.mps_from_cores(cores)
    ctx.compress(m, 1 << 20, 1e-12)
    rounding = 200 * 2.0 ** -47
    err = np.linalg.norm(m.to_dense() - ref) / np.linalg.norm(ref)
    assert err < len(bonds) * (1e-12 + rounding), err
    for c in m.cores()[1:]:
        a = c.reshape(c.shape[0], -1)
        assert np.max(np.abs(a @ a.T - np.eye(a.shape[0]))) < 8e-13 * np.sqrt(max(a.shape)) + rounding
