"""The scales of a tensor-core product on planes (the large sizes) belong to one row of A and one row of B each: with powers
of two on the rows of both operands the product is that of the bare operands times the same powers, bit
for bit (every value stays a normal number). A stale or foreign scale moves a column by a factor."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(2304, 2304, 4096), (2100, 2301, 4101), (500, 9936, 12000), (300, 30000, 8192),
                                   (1000, 2000, 500), (256, 4000, 3000), (100, 5000, 3000), (128, 128, 32)])
def test_powers_of_two_on_rows_come_out_exactly(M, N, K):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    g = torch.Generator(device="cuda").manual_seed(M)
    ld = (K + 3) // 4 * 4
    A = torch.randn(M, ld, device="cuda", generator=g)
    B = torch.randn(N, ld, device="cuda", generator=g)
    a = torch.exp2((torch.arange(M, device="cuda") % 41 - 20).float())[:, None]
    b = torch.exp2((torch.arange(N, device="cuda") * 7 % 31 - 15).float())[:, None]
    C0 = torch.empty(M, N, device="cuda")
    fp.fpeps_gemm_f32(fp.TF32X3, A, B, C0, K=K)
    ref = C0 * a * b.T
    for _ in range(3):
        C = torch.full((M, N), float("nan"), device="cuda")
        fp.fpeps_gemm_f32(fp.TF32X3, A * a, B * b, C, K=K)
        assert torch.equal(C, ref)
