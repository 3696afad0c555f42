"""Factors that read their matrix where it lies (a core row-major or transposed, its
columns in norm order, or the transpose of a triangle), through mps_compress: odd
tall and wide sites, norms in rising order, scales far from one, values not finite.

Nothing but rounding is cut at tol = 1e-12: (sites) (tol + 200 roundings of 2^-47)
bounds the dense vector's error, relative to its norm.
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


BONDS = [(1, 2, 3, 5, 2, 1), (1, 2, 4, 7, 13, 8, 4, 2, 1), (1, 2, 4, 8, 16, 31, 33, 17, 9, 3, 2, 1),
         (1, 2, 4, 8, 16, 32, 64, 65, 63, 64, 32, 16, 8, 4, 2, 1), (1, 300, 5, 300, 1), (1, 2, 200, 200, 2, 1)]


@pytest.mark.parametrize("bonds", BONDS, ids=lambda b: "-".join(map(str, b)))
@pytest.mark.parametrize("scale", [0, 100, -100])
def test_sites_of_every_shape(ctx, bonds, scale):
    rng = np.random.default_rng(len(bonds) + scale + 100)
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) / np.sqrt(2 * bonds[k]) for k in range(len(bonds) - 1)]
    cores = [c * np.logspace(-4, 0, c.shape[0])[:, None, None] * np.logspace(-3, 0, c.shape[2]) for c in cores]
    cores[len(cores) // 2] *= 2.0 ** scale
    ref = dense(cores)
    m = ctx.mps_from_cores(cores)
    ctx.compress(m, 1 << 20, 1e-12)
    err = np.linalg.norm(m.to_dense() - ref) / np.linalg.norm(ref)
    assert err < len(bonds) * (1e-12 + 200 * 2.0 ** -47), err


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("site", [0, 3, 6])
def test_not_finite_is_an_error(ctx, bad, site):
    from paper_2205_11990_gb300 import vpmps
    rng = np.random.default_rng(site)
    bonds = (1, 2, 4, 8, 8, 4, 2, 1)
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) for k in range(len(bonds) - 1)]
    cores[site][0, 1, 0] = bad
    m = ctx.mps_from_cores(cores)
    with pytest.raises(vpmps.VpError):
        ctx.compress(m, 1 << 20, 1e-12)
