"""A caller's allocator need not align its blocks to more than the eight bytes of a
double: every result keeps its bits with blocks that start 8 bytes past a 16-byte
boundary.  (Q's formation copies its panels 16 bytes at a time.)
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def contexts():
    """A context on torch's allocator, then one whose blocks are off by eight bytes."""
    import torch

    import __graft_entry__ as g
    g.build()
    from paper_2205_11990_gb300 import vpmps
    ctx = vpmps.Context()
    yield ctx
    ctx.close()
    alloc, delete, moved = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete, set()

    def alloc8(nbytes, *args):
        p = alloc(nbytes + 16, *args) + 8
        moved.add(p)
        return p

    def delete8(p):
        if p in moved:
            moved.remove(p)
            p -= 8
        delete(p)

    with pytest.MonkeyPatch.context() as mp:
        mp.setattr(torch.cuda, "caching_allocator_alloc", alloc8)
        mp.setattr(torch.cuda, "caching_allocator_delete", delete8)
        ctx = vpmps.Context()
        yield ctx
        ctx.close()
        assert not moved


@pytest.mark.parametrize("q", [2, 17, 40, 96, 200, 520])
def test_compression_keeps_its_bits(q):
    rng = np.random.default_rng(q)
    bonds = [1]
    while bonds[-1] < q:
        bonds.append(min(2 * bonds[-1], q))
    bonds += bonds[-2::-1]
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) for k in range(len(bonds) - 1)]
    out = []
    for ctx in contexts():
        m = ctx.mps_from_cores(cores)
        ctx.compress(m, max(2, q // 2), 1e-12)
        out.append(np.concatenate([c.reshape(-1) for c in m.cores()]))
    assert np.array_equal(out[0], out[1])


def test_run_keeps_its_bits():
    from paper_2205_11990_gb300 import inputs as I
    lay = I.Layout(6, 5, 0.0, 4 * math.pi, -6.0, 6.0, I.SEQ)
    f0 = I.landau(lay, 0.05, 0.5)
    out = [ctx.run(lay, f0, 0.02, 2, 16)[0] for ctx in contexts()]
    assert np.array_equal(np.asarray(out[0]), np.asarray(out[1]))


def test_large_product_keeps_its_bits():
    import torch
    A = torch.randn(400, 300, dtype=torch.float64, device="cuda")
    B = torch.randn(300, 500, dtype=torch.float64, device="cuda")
    out = [ctx.gemm(A, B).cpu().numpy() for ctx in contexts()]
    assert np.array_equal(out[0], out[1])
