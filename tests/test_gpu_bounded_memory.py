"""Site maps and a row whose large tensor-core products do not get the memory that their split copies
would take (half a gigabyte): they run with less (on-chip split) instead of failing. The allocator
refuses beyond a limit 100 MB below the peak of an unbounded run."""
import numpy as np
import pytest

from synth import lattice as L

pytestmark = pytest.mark.gpu


class _Bounded:
    """Torch-backed allocator with a limit on the bytes held at once."""

    def __init__(self, fp, limit=None):
        import torch
        self.inner = fp.TorchAllocator(torch.device("cuda", torch.cuda.current_device()))
        self.limit, self.live, self.held, self.peak, self.refused, self.stray = limit, {}, 0, 0, 0, 0
        self._a, self._f = fp.ALLOC_FN(self._alloc), fp.FREE_FN(self._free)
        self.struct = fp.fpeps_allocator(None, self._a, self._f)

    def _alloc(self, ctx, nbytes, stream):
        if self.limit is not None and self.held + nbytes > self.limit:
            self.refused += 1
            return None
        p = self.inner._alloc(ctx, nbytes, stream)
        self.live[p] = nbytes
        self.held += nbytes
        self.peak = max(self.peak, self.held)
        return p

    def _free(self, ctx, ptr, stream):
        if ptr not in self.live:
            self.stray += 1   # not a block of ours, or given back twice
            return
        self.held -= self.live.pop(ptr)
        self.inner._free(ctx, ptr, stream)


D, W = 6, 4
B = D * W * D
LESS = 100 << 20


def _handle(fp, al, Lx, Ly, chi):
    import torch
    peps = L.random_peps(Lx, Ly, D, 4, seed=2)
    pepo = L.fsm_pepo(L.random_hamiltonian(Lx, Ly, 4, W - 2, 2))
    pk, wk = (torch.cat([torch.as_tensor(t).reshape(-1) for row in x for t in row]).cuda() for x in (peps, pepo))
    cfg = fp.fpeps_config(Lx, Ly, D, 4, W, chi, fp.TF32X3, 1, 0, 1)
    torch.cuda.synchronize()
    return fp.fpeps_env_create(cfg, pk, wk, 0, torch.cuda.current_stream().cuda_stream, al)


def _maps(fp, al, ks, chi=500):
    """The site map (op 0) on k vectors for each k, one handle: results and peaks of the calls."""
    from paper_2511_01039_gb300 import workloads as WL
    h = _handle(fp, al, 3, 3, chi)
    g = np.random.default_rng(3)
    bnd = [g.standard_normal(s, dtype=np.float32) for s in ((1, B, chi), (chi, B, chi), (chi, B, 1))]
    fp.fpeps_import_boundary(h, WL.boundary_blob(bnd, 1, 1, 4), 1, 1)
    fp.fpeps_absorb_row(h, 1, 1)
    e = g.standard_normal((chi, chi, B), dtype=np.float32)
    out, peaks = [], []
    try:
        for k in ks:
            x = g.standard_normal((k, chi, B), dtype=np.float32)
            al.peak = al.held
            out.append(fp.fpeps_apply_theta_op(h, 0, 1, e, x, (chi, B), 4))
            peaks.append(al.peak)
    finally:
        fp.fpeps_env_destroy(h)
    return out, peaks


@pytest.mark.parametrize("ks", [(30,), (30, 120)])
def test_site_maps_without_room_for_the_planes(ks):
    from paper_2511_01039_gb300 import fpeps as fp
    free = _Bounded(fp)
    ref, peaks = _maps(fp, free, ks)
    tight = _Bounded(fp, peaks[-1] - LESS)
    out, _ = _maps(fp, tight, ks)
    assert tight.refused
    for r, o in zip(ref, out):
        assert np.abs(o - r).max() < 4e-5 * np.abs(r).max()   # two split products, 4e-6 of sum |a b| each


def test_row_without_room_for_the_planes():
    from paper_2511_01039_gb300 import fpeps as fp
    from paper_2511_01039_gb300 import workloads as WL
    chi, n = 200, 4
    bonds = L.boundary_bond_profile(n, chi, B)
    bnd = L.random_boundary(bonds, [B] * n, seed=1)

    def row(al):
        h = _handle(fp, al, n, n, chi)
        try:
            fp.fpeps_import_boundary(h, WL.boundary_blob([t.astype(np.float32) for t in bnd], 1, 1, 4), 1, 1)
            fp.fpeps_absorb_row(h, 1, 1)
            al.peak = al.held
            st = fp.fpeps_compress_rsvd(h, fp.params(10, 1, 0, 1, 0))
            return st.log_scale, al.peak
        finally:
            fp.fpeps_env_destroy(h)

    want, peak = row(_Bounded(fp))
    tight = _Bounded(fp, peak - (16 << 20))   # the copies of this size take some 50 MB
    got, _ = row(tight)
    assert tight.refused and abs(got - want) < 1e-4


def test_refused_growth_leaves_the_handle_usable():
    """A call that runs out of memory while an intermediate grows gives every block back once, and the
    handle computes the smaller call as before."""
    from paper_2511_01039_gb300 import fpeps as fp
    from paper_2511_01039_gb300 import workloads as WL
    chi = 60
    al = _Bounded(fp)
    h = _handle(fp, al, 3, 3, chi)
    g = np.random.default_rng(3)
    bnd = [g.standard_normal(s, dtype=np.float32) for s in ((1, B, chi), (chi, B, chi), (chi, B, 1))]
    fp.fpeps_import_boundary(h, WL.boundary_blob(bnd, 1, 1, 4), 1, 1)
    fp.fpeps_absorb_row(h, 1, 1)
    e = g.standard_normal((chi, chi, B), dtype=np.float32)
    x = g.standard_normal((80, chi, B), dtype=np.float32)
    call = lambda k: fp.fpeps_apply_theta_op(h, 0, 1, e, x[:k], (chi, B), 4)
    want = call(2)
    big = []
    for room in range(8, 200, 8):   # MB beyond what is held: the refusal falls on one block after the other
        al.limit = al.held + (room << 20)
        try:
            big.append(call(80))
            break
        except fp.FpepsError as err:
            assert err.status == 3
        al.limit = None
        assert np.array_equal(call(2), want)
    assert al.refused and al.stray == 0
    fp.fpeps_env_destroy(h)
    assert al.stray == 0 and not al.live


def test_scratch_of_calls_without_a_handle_is_given_back():
    """A large product leaves its scratch with the library (at most 640 MB) until the caller asks for it."""
    import torch
    from paper_2511_01039_gb300 import fpeps as fp
    A, B, C = (torch.ones(s, device="cuda") for s in ((500, 40000), (8000, 40000), (500, 8000)))
    fp.fpeps_release_scratch()
    torch.cuda.synchronize()
    start = torch.cuda.mem_get_info()[0]
    fp.fpeps_gemm_f32(fp.TF32X3, A, B, C)
    kept = start - torch.cuda.mem_get_info()[0]
    assert kept <= 700 << 20
    fp.fpeps_release_scratch()
    assert start - torch.cuda.mem_get_info()[0] <= 32 << 20 < kept
    fp.fpeps_gemm_f32(fp.TF32X3, A, B, C)
    assert (C == 40000).all()
