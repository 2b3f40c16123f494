"""The tensor-core site maps hand their tiles between warps in a fixed order: repeated calls give the
same bits, on interior and edge sites and for few and many vectors."""
import numpy as np
import pytest

from synth import lattice as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c,chi,k", [(0, 40, 7), (1, 33, 1), (1, 96, 40), (1, 200, 130), (2, 64, 50)])
def test_site_maps_repeat_bit_for_bit(c, chi, k):
    from paper_2511_01039_gb300 import fpeps as fp
    from paper_2511_01039_gb300 import workloads as WL
    D, w = 6, 4
    b = D * w * D
    env = fp.Env(L.random_peps(3, 3, D, 4, seed=2), L.fsm_pepo(L.random_hamiltonian(3, 3, 4, w - 2, 2)), D=D, p=4, w=w, chi=chi,
                 prec="tf32x3", seed=1)
    g = np.random.default_rng(3)
    bnd = [g.standard_normal(s, dtype=np.float32) for s in ((1, b, chi), (chi, b, chi), (chi, b, 1))]
    fp.fpeps_import_boundary(env.h, WL.boundary_blob(bnd, 1, 1, 4), 1, 1)
    fp.fpeps_absorb_row(env.h, 1, 1)
    t, tp, bl, br = (1 if c == 0 else chi), (1 if c == 2 else chi), (1 if c == 0 else b), (1 if c == 2 else b)
    el, er = g.standard_normal((chi, t, bl), dtype=np.float32), g.standard_normal((chi, tp, br), dtype=np.float32)
    ins = [(tp, br), (chi, b), (b, chi), (t, bl)]
    outs = [(chi, b), (tp, br), (t, bl), (b, chi)]
    for op in range(4):
        e, x = (el if op < 2 else er), g.standard_normal((k,) + ins[op], dtype=np.float32)
        first = env.apply_theta_op(op, c, e, x, outs[op])
        assert np.isfinite(first).all() and np.abs(first).max() > 0
        for _ in range(3):
            assert np.array_equal(first, env.apply_theta_op(op, c, e, x, outs[op]))
    env.close()
