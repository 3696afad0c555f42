"""Scratch of the sliced FP64 contractions: the digits (16 bytes an element, at most 1 GiB
an operand at a time) and, per element, one byte of magnitude; no copies of the product.
Without that memory the product is formed on the FMA pipe.

Errors: the slices of K are summed one after the other or over a cluster of CTAs, within
the bound of an FP64 sum; numpy's sum is within the same (test_gpu_gemm_elementwise.py).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vp():
    import __graft_entry__ as g
    g.build()
    from paper_2205_11990_gb300 import vpmps
    return vpmps


def operands(M, N, K, seed=0):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g),
            torch.randn(K, N, dtype=torch.float64, device="cuda", generator=g))


def check(A, B, C):
    import torch
    M, K = A.shape
    rows = torch.unique(torch.cat([torch.arange(0, M, max(1, M // 24)), torch.tensor([M - 1])]))
    a, b, c = A[rows.cuda()].cpu().numpy(), B.cpu().numpy(), C[rows.cuda()].cpu().numpy()
    assert np.all(np.abs(c - a @ b) <= (2 * K + 16) * 2.0 ** -53 * (np.abs(a) @ np.abs(b)))


# several K slices a CTA, a cluster of CTAs, both; swapped tiles; more than a band of digits
# in A, in B, in both (from K x rows = 2^26 on); the FMA pipe from K = 2^19 on
SHAPES = [(900, 1100, 2100), (260, 200, 5000), (48, 128, 9000), (128, 600, 6147), (40000, 64, 2048), (64, 40000, 2048),
          (200, 130, 300000), (48, 40, 600000)]


@pytest.mark.parametrize("shape", SHAPES)
def test_slices_and_bands(vp, shape):
    ctx = vp.Context()
    A, B = operands(*shape)
    check(A, B, ctx.gemm(A, B))
    ctx.close()


def test_no_copies_of_the_product(vp):
    import torch
    ctx = vp.Context()
    M, N, K = 8192, 4096, 4096  # eight K slices
    A, B = operands(M, N, K)
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated()
    C = ctx.gemm(A, B)
    used = torch.cuda.max_memory_allocated() - before - C.numel() * 8
    # digits and magnitudes of both, rounded up to tiles, with a quarter to spare in reserve
    assert used <= 1.25 * 1.03 * 17 * K * (M + N) + 2 ** 24
    check(A, B, C)
    ctx.close()


def test_without_memory_the_fma_pipe(vp):
    ctx = vp.Context()
    A, B = operands(400, 300, 500)
    ctx.set_alloc_budget(0)
    C0 = ctx.gemm(A, B)
    check(A, B, C0)
    ctx.set_alloc_budget(1)  # one operand's digits
    check(A, B, ctx.gemm(A, B))
    ctx.set_alloc_budget(None)
    check(A, B, ctx.gemm(A, B))
    ctx.close()


def test_several_slices_with_elements_formed_again(vp):
    """4096 x 4096 x 1100: three slices one after the other in a CTA, entries of every size
    in a tenth of the rows and columns, a NaN and an Inf in others."""
    import torch
    ctx = vp.Context()
    A, B = operands(4096, 4096, 1100, 3)
    rng = np.random.default_rng(3)
    rows, cols = torch.from_numpy(rng.choice(4096, 400, False)).cuda(), torch.from_numpy(rng.choice(4096, 400, False)).cuda()
    A[rows] *= torch.exp2(torch.from_numpy(rng.integers(-70, 71, (400, 1100))).cuda().double())
    B[:, cols] *= torch.exp2(torch.from_numpy(rng.integers(-70, 71, (1100, 400))).cuda().double())
    A[7, 600], B[1099, 9] = float("nan"), float("inf")
    C = ctx.gemm(A, B, alpha=-0.5).cpu().numpy()
    a, b = A.cpu().numpy(), B.cpu().numpy()
    assert np.all(np.isnan(C[7])) and not np.any(np.isfinite(C[:, 9]))
    keep, kept = np.arange(4096) != 7, np.arange(4096) != 9
    a, b, C = a[keep], b[:, kept], C[keep][:, kept]
    assert np.all(np.abs(C + 0.5 * (a @ b)) <= 0.5 * (2 * 1100 + 16) * 2.0 ** -53 * (np.abs(a) @ np.abs(b)))
    ctx.close()
