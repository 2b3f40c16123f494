"""CUDA-core GEMMs at the edges of their tiles (16, 32, 64 and 128 rows) and of the K split over
a cluster: sums of one k-tile, one term more, and long sums of few outputs, against an FP64
evaluation. FP32 tolerance: sqrt(K) 2^-24 random-walk rounding of sum |a b|, times 8."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,pad", [(1, 1, 1, 0), (1, 1, 36865, 0), (17, 15, 64, 1), (33, 31, 20001, 3), (65, 64, 129, 0),
                                       (256, 288, 9000, 0), (129, 97, 16, 4), (5000, 266, 266, 2), (20000, 65, 130, 4),
                                       (3000, 3000, 17, 0)])
def test_gemm_f32_tiles_and_splits(M, N, K, pad):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K + pad, device="cuda", generator=g)
    B = torch.randn(N, K + pad, device="cuda", generator=g)
    C = torch.full((M, N), float("nan"), device="cuda")
    fp.fpeps_gemm_f32(fp.F32, A, B, C, K=K)
    a, b = A[:, :K].double(), B[:, :K].double()
    err = ((C.double() - a @ b.T).abs() / (a.abs() @ b.abs().T)).max().item()
    assert err < 8 * K ** 0.5 * 2.0 ** -24, err


@pytest.mark.parametrize("chi,k", [(3, 1), (17, 5), (40, 3)])
@pytest.mark.parametrize("op", [0, 1, 2, 3])
def test_site_maps_f64_on_ragged_sizes(op, chi, k):
    """The FP64 GEMMs of a site map (few vectors, long sums) keep FP64 accuracy: the map is linear,
    so applying it to x and to x / 3 must agree to rounding, and the adjoint identity
    <map x, y> = <x, map^T y> must hold."""
    from paper_2511_01039_gb300 import fpeps as fp
    from paper_2511_01039_gb300 import workloads as WL
    from synth import lattice as L
    D, w = 3, 3
    peps = L.random_peps(3, 3, D, 4, seed=chi)
    pepo = L.fsm_pepo(L.random_hamiltonian(3, 3, 4, w - 2, chi))
    b = D * w * D
    env = fp.Env(peps, pepo, D=D, p=4, w=w, chi=chi, prec="f64", seed=1)
    bnd = L.random_boundary([1, chi, chi, 1], [b] * 3, seed=chi)
    fp.fpeps_import_boundary(env.h, WL.boundary_blob(bnd, 1, 1, 8), 1, 1)
    fp.fpeps_absorb_row(env.h, 1, 1)
    g = np.random.default_rng(chi + op)
    e = g.standard_normal((chi, chi, b))
    ins = {0: (chi, b), 1: (chi, b), 2: (b, chi), 3: (chi, b)}
    outs = {0: (chi, b), 1: (chi, b), 2: (chi, b), 3: (b, chi)}
    x = g.standard_normal((k,) + ins[op])
    y = g.standard_normal((k,) + outs[op])
    fx = env.apply_theta_op(op, 1, e, x, outs[op])
    f3 = env.apply_theta_op(op, 1, e, x / 3.0, outs[op])
    ty = env.apply_theta_op(op ^ 1, 1, e, y, ins[op])
    env.close()
    assert np.abs(fx - 3.0 * f3).max() < 1e-12 * np.abs(fx).max()
    lhs, rhs = np.vdot(fx, y), np.vdot(x, ty)
    assert abs(lhs - rhs) < 1e-12 * np.linalg.norm(fx) * np.linalg.norm(y)
