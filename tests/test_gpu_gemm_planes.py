"""The tensor-core GEMM on FP16 planes (large products): ragged edges in every direction, tiles cut
over the CTA pairs, sums longer than one panel, rows whose scales lie near the ends of FP32, and
non-finite input; and the output map of a site map through the adjoint identity.

Tolerances: every product carries at most 3 * 2^-22 of |a b| from the split, and the FP32 accumulation
of the tensor cores (truncating, chunks of 256 terms) at most ~48 * 2^-23 of a chunk's partial sums,
so componentwise 4e-6 of sum |a b| bounds both."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(2100, 2301, 4101, 3), (2304, 2304, 4096, 0), (300, 30000, 30000, 0), (600, 12000, 20000, 0), (5000, 1540, 4000, 4),
         (129, 9000, 9001, 3)]


@pytest.fixture(scope="module")
def fp():
    import torch
    from paper_2511_01039_gb300 import fpeps
    torch.cuda.set_device(0)
    return fpeps


def _err(C, A, B):
    worst = 0.0
    for c, b in zip(C.split(2048, 1), B.split(2048)):
        ref, mag = A.double() @ b.double().T, A.double().abs() @ b.double().abs().T
        worst = max(worst, ((c.double() - ref).abs() / mag).max().item())
    return worst


@pytest.mark.parametrize("mode", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("M,N,K,pad", SIZES)
def test_large_products_against_fp64(fp, M, N, K, pad, mode):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.randn(M, K + pad, device="cuda", generator=g)
    B = torch.randn(N, K + pad, device="cuda", generator=g)
    C = torch.full((M, N), float("nan"), device="cuda")
    fp.fpeps_gemm_f32(fp.PRECISIONS[mode], A, B, C, K=K)
    assert _err(C, A[:, :K], B[:, :K]) < 4e-6


@pytest.mark.parametrize("ea,eb", [(-100, 100), (100, -100), (-60, -50), (60, 50), (-110, 20)])
def test_scales_near_the_ends_of_fp32(fp, ea, eb):
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn(2000, 4000, device="cuda", generator=g)
    B = torch.randn(2000, 4000, device="cuda", generator=g)
    C = torch.empty(2000, 2000, device="cuda")
    fp.fpeps_gemm_f32(fp.TF32X3, A * 2.0 ** ea, B * 2.0 ** eb, C)
    assert _err(C.double() * 2.0 ** -(ea + eb), A, B) < 4e-6


def test_non_finite_rows_stay_non_finite_and_apart(fp):
    import torch
    A = torch.ones(2000, 4000, device="cuda")
    B = torch.ones(2000, 4000, device="cuda")
    A[7, 3], A[300, 3999], B[1999, 256] = float("nan"), float("inf"), float("-inf")
    C = torch.empty(2000, 2000, device="cuda")
    fp.fpeps_gemm_f32(fp.TF32X3, A, B, C)
    bad = ~torch.isfinite(C)
    assert bad[7].all() and bad[300].all() and bad[:, 1999].all()
    bad[7] = bad[300] = False
    bad[:, 1999] = False
    assert not bad.any()


def test_site_map_adjoint_at_large_size(fp):
    """<Theta x, y> = <x, Theta^T y>: both products of either map run on planes at this size, with the
    bundle-split output maps of the path."""
    import torch
    from paper_2511_01039_gb300 import workloads as WL
    from synth import lattice as L
    D, w, chi, k = 6, 4, 500, 30
    b = D * w * D
    peps = L.random_peps(3, 3, D, 4, seed=2)
    pepo = L.fsm_pepo(L.random_hamiltonian(3, 3, 4, w - 2, 2))
    env = fp.Env(peps, pepo, D=D, p=4, w=w, chi=chi, prec="tf32x3", seed=1)
    g = np.random.default_rng(3)
    bnd = [g.standard_normal(s, dtype=np.float32) for s in ((1, b, chi), (chi, b, chi), (chi, b, 1))]
    fp.fpeps_import_boundary(env.h, WL.boundary_blob(bnd, 1, 1, 4), 1, 1)
    fp.fpeps_absorb_row(env.h, 1, 1)
    e = g.standard_normal((chi, chi, b), dtype=np.float32)
    x = g.standard_normal((k, chi, b), dtype=np.float32)
    y = g.standard_normal((k, chi, b), dtype=np.float32)
    fx = env.apply_theta_op(0, 1, e, x, (chi, b)).astype(np.float64)
    ty = env.apply_theta_op(1, 1, e, y, (chi, b)).astype(np.float64)
    env.close()
    for i in range(k):
        lhs, rhs = np.vdot(fx[i], y[i]), np.vdot(x[i], ty[i])
        assert abs(lhs - rhs) < 1e-5 * np.linalg.norm(fx[i]) * np.linalg.norm(y[i])
    torch.cuda.synchronize()
