"""Operands graded against each other in segments scattered over rows and the sum: while the splitting pass
looks through the FP32 operands, some warps find the word that ends the search and others raise it.

Tolerance: 3 * 2^-22 of |a b| for the split plus the truncating FP32 accumulation of at most ~48 * 2^-23 of
a chunk's partial sums: 4e-6 of sum |a b| componentwise. The same call twice: the same bits."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("share", [1e-3, 0.05, 0.5])
@pytest.mark.parametrize("M,N,K", [(2304, 2304, 4096), (2100, 2301, 4101)])
def test_scattered_segments(M, N, K, share):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    g = torch.Generator(device="cuda").manual_seed(11)
    ld, nseg = (K + 3) // 4 * 4, (K + 255) // 256
    A, B = (torch.randn(r, ld, device="cuda", generator=g) for r in (M, N))
    f = torch.exp2(-(torch.arange(ld, device="cuda") % 256).float() / 8)
    seg = torch.arange(ld, device="cuda") // 256
    pick = [torch.rand(r, nseg, device="cuda", generator=g) < share for r in (M, N)]
    A = torch.where(pick[0][:, seg], A * f, A)
    B = torch.where(pick[1][:, seg], B / f, B)
    C = [torch.full((M, N), float("nan"), device="cuda") for _ in range(2)]
    for c in C:
        fp.fpeps_gemm_f32(fp.PRECISIONS["tf32x3"], A, B, c, K=K)
    a, b = A[:, :K].double(), B[:, :K].double()
    assert ((C[0].double() - a @ b.T).abs() / (a.abs() @ b.abs().T)).max().item() < 4e-6
    assert torch.equal(C[0], C[1])
