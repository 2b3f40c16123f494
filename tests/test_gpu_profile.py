"""Kernel-class records: the FP64 products inside the small SVD belong to its own record (class 4) and are
not counted a second time as CUDA-core products (class 1)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [12, 60, 160])
def test_svd_is_one_record(k):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    M = torch.linalg.qr(torch.randn(k, k, dtype=torch.float64, device="cuda"))[1].T.contiguous()
    fp.fpeps_profile(True)
    try:
        fp.fpeps_svd_f64(M)
        fp.fpeps_gemm_f32(fp.F32, *(torch.ones(64, 64, device="cuda") for _ in range(3)))
        torch.cuda.synchronize()
        read = {i: fp.fpeps_profile_read(i) for i in (1, 4)}
    finally:
        fp.fpeps_profile(False)
    assert read[4]["launches"] == 1 and read[4]["ms"] > 0
    assert read[1]["launches"] == 1 and read[1]["flops"] == 2 * 64 ** 3
