"""Kernels started behind the one before them read what that one wrote: two states of
the same sizes (some bonds may differ) in turn on one context, so that a workspace read
too early holds the other state's values, against references from routes without such launches (the
members of a group) or without earlier contents (a new context each).
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vp():
    import __graft_entry__ as g
    g.build()
    from paper_2205_11990_gb300 import vpmps
    return vpmps


def grids(lay, count):
    """Maxwellians with seeded broadband perturbations: every bond at its cap."""
    x, v = np.meshgrid(lay.x(), lay.v(), indexing="ij")
    out = []
    for seed in range(count):
        rng = np.random.default_rng(seed)
        f = np.exp(-v * v / 2)
        for m in range(1, 13):
            f = f + 0.02 * np.cos(m * 0.5 * x + rng.uniform(0, 6)) * np.exp(-((v - rng.uniform(-2, 2)) ** 2) * rng.uniform(0.5, 2))
        out.append(np.ascontiguousarray(f))
    return out


@pytest.mark.parametrize("bits,chi", [(5, 8), (7, 24)])
@pytest.mark.parametrize("streams", [1, 2])
def test_steps_in_turn_equal_the_group(vp, bits, chi, streams):
    from paper_2205_11990_gb300 import inputs as I
    ctx = vp.Context()
    lay = I.Layout(bits, bits, 0.0, 4 * math.pi, -6.0, 6.0, I.SEQ)
    fs = grids(lay, 2)

    def sims(streams):
        return [ctx.sim(lay, ctx.mps_from_grid(lay, f, chi, 1e-10), 0.01, chi, streams=streams) for f in fs]

    grp, members, lone = ctx.group(2), sims(1), sims(streams)
    for s in members:
        grp.add(s)
    for _ in range(4):
        recs, status = grp.step()
        assert status == [0, 0]
        for s, m, r in zip(lone, members, recs):
            assert s.step(1)[0] == r
            assert np.array_equal(s.state().to_grid(lay), m.state().to_grid(lay))
    ctx.close()


@pytest.mark.parametrize("q", [2, 6, 17, 40, 96])
def test_compressions_in_turn_equal_a_new_context(vp, q):
    bonds = [1]
    while bonds[-1] < q:
        bonds.append(min(2 * bonds[-1], q))
    bonds += bonds[-2::-1]

    def compressed(ctx, seed):
        rng = np.random.default_rng(seed)
        m = ctx.mps_from_cores([rng.standard_normal((bonds[k], 2, bonds[k + 1])) for k in range(len(bonds) - 1)])
        ctx.compress(m, max(2, q // 2), 1e-12)
        return np.concatenate([c.reshape(-1) for c in m.cores()])

    refs = []
    for seed in range(2):
        fresh = vp.Context()
        refs.append(compressed(fresh, seed))
        fresh.close()
    ctx = vp.Context()
    for _ in range(8):
        for seed in range(2):
            assert np.array_equal(compressed(ctx, seed), refs[seed])
    ctx.close()
