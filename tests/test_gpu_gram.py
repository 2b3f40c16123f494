"""The FP64-class Gram matrix of the FP32 path, seen through the isometries that CholeskyQR2 makes
of it, at column counts around the 64-column tiles. Tolerance: entries of Q^T Q are sums of k
products of FP32 columns that carry the rounding of two k-term FP32 products (Y R^-1 and the
rotation of the small SVD), 4 k 2^-24 at most."""
import numpy as np
import pytest

from synth import lattice as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi", [7, 53, 54, 55, 118, 119])   # k = chi + 10
def test_isometries_of_a_compressed_row(chi):
    from paper_2511_01039_gb300 import fpeps as fp
    peps = L.random_peps(4, 4, 3, 4, seed=7)
    pepo = L.fsm_pepo(L.random_hamiltonian(4, 4, 4, 2, seed=7))
    env = fp.Env(peps, pepo, D=3, p=4, w=4, chi=chi, prec="f32", seed=5)
    try:
        fp.fpeps_absorb_row(env.h, 0, 1)
        fp.fpeps_absorb_row(env.h, 1, 1)
        fp.fpeps_compress_rsvd(env.h, fp.params(10, 1, 0, 0, 0))
        blob = bytes(fp.fpeps_export_boundary(env.h))
        shapes = [fp.fpeps_boundary_shape(env.h, c) for c in range(4)]
    finally:
        env.close()
    off = 8 * (5 + 5 + 4) + 8
    tol = 4 * (chi + 10) * 2.0 ** -24
    left = right = 0
    for c, (t, u, tp) in enumerate(shapes):
        T = np.frombuffer(blob, np.float32, t * u * tp, off).astype(np.float64).reshape(t, u, tp)
        off += 4 * t * u * tp
        a, b = T.reshape(t * u, tp), T.reshape(t, u * tp)
        left += np.abs(a.T @ a - np.eye(tp)).max() < tol
        right += np.abs(b @ b.T - np.eye(t)).max() < tol
    assert max(left, right) >= 3   # every site but the centre
