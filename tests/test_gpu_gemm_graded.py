"""Tensor-core products whose operands are graded against each other along the sum (A falls where B
rises, in every block of 256 terms, in order or shuffled): the small elements carry the sum and keep
their 22 bits. Also where only the last panel of a long sum, or one row, is graded.

Tolerance: as for ordinary operands, 3 * 2^-22 of |a b| for the split plus the truncating FP32
accumulation of at most ~48 * 2^-23 of a chunk's partial sums: 4e-6 of sum |a b| componentwise."""
import pytest

pytestmark = pytest.mark.gpu


def _worst(C, A, B):
    worst = 0.0
    for c, b in zip(C.split(1024, 1), B.split(1024)):
        ref, mag = A.double() @ b.double().T, A.double().abs() @ b.double().abs().T
        worst = max(worst, ((c.double() - ref).abs() / mag).max().item())
    return worst


def _operands(M, N, K, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    ld = (K + 3) // 4 * 4
    return torch.randn(M, ld, device="cuda", generator=g), torch.randn(N, ld, device="cuda", generator=g)


def _product(A, B, K, mode="tf32x3"):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    C = torch.full((A.shape[0], B.shape[0]), float("nan"), device="cuda")
    fp.fpeps_gemm_f32(fp.PRECISIONS[mode], A, B, C, K=K)
    return C


@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("span", [10, 16, 17, 18, 24, 30, 36])
@pytest.mark.parametrize("M,N,K", [(2304, 2304, 4096), (2100, 2301, 4101)])
def test_opposite_grading(M, N, K, span, shuffled):
    import torch
    A, B = _operands(M, N, K, span)
    k = torch.arange(A.shape[1], device="cuda")
    if shuffled:
        k = k[torch.randperm(len(k), device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))]
    f = torch.exp2((-(k % 256) * span // 256).float())
    A, B = A * f, B / f
    assert _worst(_product(A, B, K), A[:, :K], B[:, :K]) < 4e-6


@pytest.mark.parametrize("mode", ["tf32x3", "bf16x3"])
def test_only_the_last_panel_is_graded(mode):
    import torch
    M, N, K = 500, 4096, 60000
    A, B = _operands(M, N, K, 3)
    f = torch.ones(K, device="cuda")
    f[-300:] = torch.exp2(-torch.arange(300, device="cuda").float() / 10)
    A[:, :-300] *= 1e-9   # the graded terms carry the sum
    A, B = A * f, B / f
    assert _worst(_product(A, B, K, mode), A, B) < 4e-6


def test_one_graded_row():
    import torch
    M, N, K = 2304, 2304, 4096
    A, B = _operands(M, N, K, 4)
    f = torch.exp2(-(torch.arange(K, device="cuda") % 256).float() / 8)
    A[77] *= f
    B[:, :] = B / f
    assert _worst(_product(A, B, K), A, B) < 4e-6


@pytest.mark.parametrize("kind", ["outlier", "interleaved", "one_sided", "zeros"])
def test_patterns_of_large_and_small_terms(kind):
    """A column of A that dwarfs the others and meets zeros of B; large and small terms in turn, the
    large ones against zeros; one operand alone graded; sparse operands."""
    import torch
    M, N, K = 2304, 2304, 4096
    A, B = _operands(M, N, K, 5)
    k = torch.arange(K, device="cuda")
    if kind == "outlier":
        A[:, 7::256] = 2.0 ** 30
        B[:, 7::256] = 0
    elif kind == "interleaved":
        A[:, 1::2] *= 2.0 ** -30
        B[:, 0::2] = 0
    elif kind == "one_sided":
        A *= torch.exp2(-(k % 256).float() / 8)
    else:
        A[:, k % 256 > 60] = 0
        B[:, k % 7 > 2] = 0
    assert _worst(_product(A, B, K), A, B) < 4e-6


def test_site_map_of_graded_vectors():
    """Theta^T sums over the environment's row index: powers of two on the rows of the environment, their
    inverses on the vectors, leave the map as it is. Tolerance: two maps, each of two split products and
    the sandwich, 4e-6 of sum |a b|, at most 16 times the largest output of N(0,1) data."""
    import numpy as np
    from paper_2511_01039_gb300 import fpeps as fp
    from paper_2511_01039_gb300 import workloads as WL
    from synth import lattice as L
    D, w, chi, k = 6, 4, 500, 30
    b = D * w * D
    env = fp.Env(L.random_peps(3, 3, D, 4, seed=2), L.fsm_pepo(L.random_hamiltonian(3, 3, 4, w - 2, 2)), D=D, p=4, w=w, chi=chi,
                 prec="tf32x3", seed=1)
    g = np.random.default_rng(3)
    bnd = [g.standard_normal(s, dtype=np.float32) for s in ((1, b, chi), (chi, b, chi), (chi, b, 1))]
    fp.fpeps_import_boundary(env.h, WL.boundary_blob(bnd, 1, 1, 4), 1, 1)
    fp.fpeps_absorb_row(env.h, 1, 1)
    e = g.standard_normal((chi, chi, b), dtype=np.float32)
    x = g.standard_normal((k, chi, b), dtype=np.float32)
    f = np.exp2(-((np.arange(chi) % 250) * 36 // 250)).astype(np.float32)[:, None, None]
    plain = env.apply_theta_op(1, 1, e, x, (chi, b))
    graded = env.apply_theta_op(1, 1, e * f, x / f[None, :, :, 0], (chi, b))
    env.close()
    assert np.abs(graded - plain).max() < 2 * 3 * 16 * 4e-6 * np.abs(plain).max()
