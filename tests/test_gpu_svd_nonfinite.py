"""The small SVD on a matrix with a NaN: the singular values come back as NaN and the order of the
columns of V is still a permutation (it indexes V), on every route: FP64 sweeps alone (k <= 16: the
rotations carry the NaN into all of V), FP32 sweeps in one CTA (k <= 72) and on the whole GPU (V stays
orthonormal, to the rounding of an FP64 factorisation, 64 k 2^-53)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry", ["fpeps_svd_f64", "fpeps_svd_f64_noalloc"])
@pytest.mark.parametrize("k", [2, 16, 17, 40, 72, 73, 160])
def test_svd_of_a_matrix_with_a_nan(k, entry):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    g = np.random.default_rng(k)
    A = np.linalg.qr(g.standard_normal((k, k)))[1].T.copy()
    good = getattr(fp, entry)(torch.tensor(A, device="cuda"))[1].cpu().numpy()
    bad = A.copy()
    bad[k // 2, k // 3] = np.nan
    _, s, V = (x.cpu().numpy() for x in getattr(fp, entry)(torch.tensor(bad, device="cuda")))
    assert np.isnan(s).all()
    if k <= 16:
        assert np.isnan(V).all()
    else:
        assert np.abs(V.T @ V - np.eye(k)).max() < 64 * k * 2.0 ** -53
    again = getattr(fp, entry)(torch.tensor(A, device="cuda"))[1].cpu().numpy()
    assert np.allclose(good, again, rtol=1e-13, atol=0)
