"""Factors much wider than tall (the first sites of a QR sweep whose bonds are larger
than 2^k), in one block, in a cluster and beyond, through mps_compress.

Nothing but rounding is cut at tol = 1e-12: the dense vector stays within (sites)
(tol + 200 roundings of 2^-47) of its norm.
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


# sites k = 1 .. deep: 2^k x n factors
@pytest.mark.parametrize("n,deep", [(13, 2), (129, 5), (257, 6), (600, 8), (1201, 4), (2100, 8), (5000, 1)])
def test_first_sites(ctx, n, deep):
    rng = np.random.default_rng(n)
    bonds = [1] + [n] * deep + [5, 3, 2, 1]
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) / np.sqrt(2 * bonds[k]) for k in range(len(bonds) - 1)]
    ref = dense(cores)
    m = ctx.mps_from_cores(cores)
    ctx.compress(m, 1 << 20, 1e-12)
    err = np.linalg.norm(m.to_dense() - ref) / np.linalg.norm(ref)
    assert err < len(bonds) * (1e-12 + 200 * 2.0 ** -47), err
