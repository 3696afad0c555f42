"""FP64 contractions with millions of columns: every one of up to 64 x 65535 = 4194240 is
taken on every route (tiles of 16, 32 and 64 on the FMA pipe, the sliced products), one
more is refused.
"""
import pytest

pytestmark = pytest.mark.gpu

LIMIT = 64 * 65535


@pytest.fixture(scope="module")
def vp():
    import __graft_entry__ as g
    g.build()
    from paper_2205_11990_gb300 import vpmps
    return vpmps


@pytest.mark.parametrize("shape", [(2, 2 ** 21, 2), (2, LIMIT, 2), (1, LIMIT, 1), (17, 2097121, 8), (64, 2 ** 21, 8),
                                   (100, 1048561, 5), (100, 3200000, 64), (128, 3200000, 64)])
def test_wide_integers_exact(vp, shape):
    import torch
    M, N, K = shape
    ctx = vp.Context()
    g = torch.Generator(device="cuda").manual_seed(N)
    A = torch.randint(-1024, 1024, (M, K), device="cuda", generator=g, dtype=torch.int64).double()
    B = torch.randint(-1024, 1024, (K, N), device="cuda", generator=g, dtype=torch.int64).double()
    C = ctx.gemm(A, B)
    ref = torch.zeros(M, N, dtype=torch.float64, device="cuda")  # integers below 2^27: exact in any order
    for k in range(K):
        ref.addcmul_(A[:, k:k + 1], B[k:k + 1])
    assert torch.equal(C, ref)
    ctx.close()


def test_too_wide_is_refused(vp):
    import torch
    ctx = vp.Context()
    with pytest.raises(vp.VpError, match="N too large"):
        ctx.gemm(torch.ones(1, 1, dtype=torch.float64, device="cuda"), torch.ones(1, LIMIT + 1, dtype=torch.float64, device="cuda"))
    ctx.close()
