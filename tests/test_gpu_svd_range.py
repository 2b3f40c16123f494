"""The small SVD far from unit scale: entries of 1e-100 and 1e100 on every route (k <= 16: FP64 sweeps
alone), and the ends of FP64 where the working copy is brought to unit scale (k >= 17). Tolerances:
backward error and orthogonality of an FP64 factorisation, 64 k 2^-53."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-290, 1e-100, 1e100, 1e290])
@pytest.mark.parametrize("k", [2, 16, 17, 31, 32, 33, 72, 73, 97, 160])
def test_svd_far_from_unit_scale(k, scale):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    if k <= 16 and not 1e-150 < scale < 1e150:
        pytest.skip("squares of the entries leave FP64 in the sweeps of k <= 16")
    g = np.random.default_rng(k)
    q = [np.linalg.qr(g.standard_normal((k, k)))[0] for _ in range(2)]
    A = np.linalg.qr((q[0] * np.logspace(0, -6, k)) @ q[1])[1].T.copy()
    for entry in (fp.fpeps_svd_f64, fp.fpeps_svd_f64_noalloc):
        U, s, V = (x.cpu().numpy() for x in entry(torch.tensor(A * scale, device="cuda")))
        s = s / scale
        tol = 64 * k * 2.0 ** -53
        assert (np.diff(s) <= 0).all()
        assert np.abs(s - np.linalg.svd(A, compute_uv=False)).max() < tol * s[0]
        assert np.abs((U * s) @ V.T - A).max() < tol * s[0]
        assert np.abs(V.T @ V - np.eye(k)).max() < tol
        assert np.abs(U.T @ U - np.eye(k)).max() < tol
