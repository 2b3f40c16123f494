"""The small SVD at the edges of its routes: FP64 sweeps alone (k <= 16), FP32 sweeps in one CTA
(k <= 72) and on the whole GPU, and spectra that need the FP64 sweeps at the end (equal singular
values), are graded over 14 decades or rank deficient. Tolerances: backward error and
orthogonality of an FP64 factorisation, 64 k 2^-53 (rotations of ~30 sweeps at most)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SPECTRA = {
    "flat": lambda k: np.linspace(1, 0.5, k),
    "graded": lambda k: np.logspace(0, -14, k),
    "pairs": lambda k: np.repeat(np.linspace(1, 0.1, (k + 1) // 2), 2)[:k],
    "rank": lambda k: np.where(np.arange(k) < (k + 1) // 2, np.linspace(1, 0.1, k), 0.0),
}


@pytest.mark.parametrize("kind", list(SPECTRA))
@pytest.mark.parametrize("k", [2, 16, 17, 31, 72, 73, 81, 160])
def test_svd_routes(k, kind):
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    g = np.random.default_rng(k)
    q = [np.linalg.qr(g.standard_normal((k, k)))[0] for _ in range(2)]
    A = np.linalg.qr((q[0] * SPECTRA[kind](k)) @ q[1])[1].T.copy() * 1e-20
    U, s, V = (x.cpu().numpy() for x in fp.fpeps_svd_f64(torch.tensor(A, device="cuda")))
    tol = 64 * k * 2.0 ** -53
    assert (np.diff(s) <= 0).all()
    assert np.abs(s - np.linalg.svd(A, compute_uv=False)).max() < tol * s[0]
    assert np.abs((U * s) @ V.T - A).max() < tol * s[0]
    assert np.abs(V.T @ V - np.eye(k)).max() < tol
    live = s > 1e-13 * s[0]
    assert np.abs(U[:, live].T @ U[:, live] - np.eye(live.sum())).max() < tol
