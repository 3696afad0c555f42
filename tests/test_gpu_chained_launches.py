"""Kernels started behind the one before them (a lone chain) and plain launches
(members of a group) read what the kernel before them wrote: the same compressions
give the same bits over many runs and on both routes.
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


@pytest.mark.parametrize("q", [2, 6, 17, 40, 96])
def test_same_bits_every_time(ctx, q):
    rng = np.random.default_rng(q)
    bonds = [1]
    while bonds[-1] < q:
        bonds.append(min(2 * bonds[-1], q))
    bonds += bonds[-2::-1]
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) for k in range(len(bonds) - 1)]
    first = None
    for _ in range(25):
        m = ctx.mps_from_cores(cores)
        ctx.compress(m, max(2, q // 2), 1e-12)
        out = np.concatenate([c.reshape(-1) for c in m.cores()])
        first = out if first is None else first
        assert np.array_equal(out, first)
