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
