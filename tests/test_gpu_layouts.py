"""Layout changes of the site maps (tiled transposes from 16 columns on, the general kernel below;
PEPO-outermost bundles) at vector counts around the tile edges: every map against the oracle, with
FP64's tolerance of the maps (sums of at most 36 * 36 * 4 terms: 1e-11)."""
import numpy as np
import pytest

from oracle import boundary as B
from synth import lattice as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a", [1, 15, 16, 17, 33, 64])
def test_site_maps_at_tile_edges(a):
    from paper_2511_01039_gb300 import fpeps as fp
    peps = L.random_peps(4, 4, 3, 4, seed=21)
    pepo = L.fsm_pepo(L.random_hamiltonian(4, 4, 4, 2, seed=21))
    T, _ = B.first_row_boundary(peps[0], pepo[0])
    env = fp.Env(peps, pepo, D=3, p=4, w=4, chi=36, prec="f64", seed=5)
    fp.fpeps_absorb_row(env.h, 0, 1)
    fp.fpeps_absorb_row(env.h, 1, 1)
    g = np.random.default_rng(a)
    for c in (0, 2):
        A, W = peps[1][c], pepo[1][c]
        t, tp = T[c].shape[0], T[c].shape[2]
        dL, dR, dD = B.bdim(A, W, 0), B.bdim(A, W, 2), B.bdim(A, W, 3)
        el, er = g.standard_normal((a, t, dL)), g.standard_normal((a, tp, dR))
        x = [g.standard_normal((5, *s)) for s in ((tp, dR), (a, dD), (dD, a), (t, dL))]
        out = [(a, dD), (tp, dR), (t, dL), (dD, a)]
        for op, f in enumerate((B.theta, B.theta_t, B.theta_r, B.theta_r_t)):
            o = env.apply_theta_op(op, c, er if op >= 2 else el, x[op], out[op])
            r = np.moveaxis(f(er if op >= 2 else el, T[c], A, W, np.moveaxis(x[op], 0, -1)), -1, 0)
            assert np.abs(o - r).max() <= 1e-11 * np.abs(r).max(), (op, c)
    env.close()
