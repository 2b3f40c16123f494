"""Output forms of the tensor-core GEMM on planes: rows that are no whole 16-byte granules, with the sum
in one panel and in several (added to what the panels before wrote), a nearly empty last row of tiles,
and the site maps' bundles of 16 and 27 columns (narrower than a 32-column block, granular and not).

Tolerances: 4e-6 of sum |a b| for a split product (see test_gpu_gemm_planes). A site map chains two of
them and the split sandwich over sums of at most 500 * 27 terms, whose sum |a b| is at most 16 times
the largest output of N(0,1) data: 3 * 16 * 4e-6."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(385, 9000, 9001), (385, 9001, 9001), (500, 4097, 60000), (500, 4098, 60001), (500, 4100, 60000)])
def test_rows_of_any_length_and_several_panels(M, N, K):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    g = torch.Generator(device="cuda").manual_seed(N)
    ld = (K + 3) // 4 * 4
    A = torch.randn(M, ld, device="cuda", generator=g)
    B = torch.randn(N, ld, device="cuda", generator=g)
    C = torch.full((M, N), float("nan"), device="cuda")
    fp.fpeps_gemm_f32(fp.TF32X3, A, B, C, K=K)
    for c, b in zip(C.split(1024, 1), B.split(1024)):
        ref, mag = A[:, :K].double() @ b[:, :K].double().T, A[:, :K].double().abs() @ b[:, :K].double().abs().T
        assert ((c.double() - ref).abs() / mag).max().item() < 4e-6


@pytest.mark.parametrize("D,w,chi,k", [(2, 4, 500, 300), (3, 3, 400, 200)])
def test_narrow_bundles(D, w, chi, k):
    from paper_2511_01039_gb300 import fpeps as fp
    from paper_2511_01039_gb300 import workloads as WL
    from synth import lattice as L
    b = D * w * D
    peps = L.random_peps(3, 3, D, 4, seed=2)
    pepo = L.fsm_pepo(L.random_hamiltonian(3, 3, 4, w - 2, 2))
    g = np.random.default_rng(3)
    bnd = [g.standard_normal(s, dtype=np.float32) for s in ((1, b, chi), (chi, b, chi), (chi, b, 1))]
    e = g.standard_normal((chi, chi, b), dtype=np.float32)
    ins, outs = [(chi, b), (chi, b), (b, chi), (chi, b)], [(chi, b), (chi, b), (chi, b), (b, chi)]
    xs = [g.standard_normal((k,) + s, dtype=np.float32) for s in ins]
    res = {}
    for prec, elem in (("tf32x3", 4), ("f64", 8)):
        env = fp.Env(peps, pepo, D=D, p=4, w=w, chi=chi, prec=prec, seed=1)
        t = [x.astype(np.float64) for x in bnd] if elem == 8 else bnd
        fp.fpeps_import_boundary(env.h, WL.boundary_blob(t, 1, 1, elem), 1, 1)
        fp.fpeps_absorb_row(env.h, 1, 1)
        res[prec] = [env.apply_theta_op(op, 1, e, xs[op], outs[op]) for op in range(4)]
        env.close()
    for op in range(4):
        ref = res["f64"][op]
        assert np.abs(res["tf32x3"][op] - ref).max() < 3 * 16 * 4e-6 * np.abs(ref).max(), op
