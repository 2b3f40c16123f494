"""Performance cases of the framework: what its users have it do, through its public entry points.

A case is a dict of plain values with a ``kind``:

  gemm    one contraction GEMM of the path on device buffers (``fpeps_gemm_f32``)
  theta   one site map of a staged row on a block of vectors (``Env.apply_theta_op``)
  svd     the small dense SVD of the path (``fpeps_svd_f64``)
  row     one interior row absorbed into a stored boundary, compressed, and the last row closed
  sweep   a whole top-to-bottom boundary sweep, row by row
  expect  the expectation value <psi|O|psi> / <psi|psi> in one call

The sizes are those of the repository's tests and benchmark: 3x3 and 4x4 lattices at D = 2..4,
the 6x6 D = 6 w = 4 chi = 256 and the 8x8 D = 6 w = 6 chi = 500 workloads, and what lies between.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_01039_gb300 import fpeps as fp
from paper_2511_01039_gb300 import workloads as WL
from synth import lattice as L
from synth import u1


def listed():
    return [
        # The smallest whole call: <H> of a 3x3 lattice without truncation, in FP64 (how a user checks
        # an operator). Launches, synchronisations and one-block factorisations.
        dict(name="expect_3x3_D2_f64", kind="expect", Lx=3, Ly=3, D=2, K=2, chi=256, prec="f64", q=1, exact_svd=1),
        # A small truncated sweep in the mixed precision that production runs use.
        dict(name="sweep_4x4_D3_chi24", kind="sweep", Lx=4, Ly=4, D=3, K=2, chi=24, prec="tf32x3", q=2, n_fit=1, u1=False),
        # The charge-sector mode (U(1) x U(1), Hubbard operator): many small factorisations, one per sector.
        dict(name="sweep_u1_3x3_D2_chi32", kind="sweep", Lx=3, Ly=3, D=2, K=4, chi=32, prec="f64", q=2, n_fit=1, u1=True),
        # A production row: the last interior row of the 6x6, chi = 256 workload, from a stored boundary.
        dict(name="row_6x6_D6_chi256", kind="row", Lx=6, Ly=6, D=6, K=2, chi=256, prec="tf32x3", q=2, n_fit=1),
        # One application of the zip-up at the central site of the 8x8, chi = 500 workload.
        dict(name="theta_8x8_chi500", kind="theta", op=0, c=1, D=6, K=4, chi=500, k=46, prec="tf32x3"),
        # Its transpose at the 6x6, chi = 256 size on a whole sketch (chi + 10 columns).
        dict(name="theta_t_6x6_chi256", kind="theta", op=1, c=1, D=6, K=2, chi=256, k=266, prec="tf32x3"),
        # The fit's right-environment map at the 4x4, D = 4, chi = 64 size: a small application.
        dict(name="theta_r_4x4_chi64", kind="theta", op=2, c=1, D=4, K=2, chi=64, k=74, prec="tf32x3"),
        # Environment x vectors of the 8x8 workload: few rows, a very long sum.
        dict(name="gemm_environment", kind="gemm", M=500, N=9936, K=108000, pad=0, mode="tf32x3"),
        # Boundary x vectors of the same site: many rows, a short sum, a large output; 3xBF16.
        dict(name="gemm_boundary_bf16x3", kind="gemm", M=108000, N=1728, K=500, pad=0, mode="bf16x3"),
        # A ragged product of an edge site, rows not packed.
        dict(name="gemm_ragged", kind="gemm", M=1000, N=2000, K=500, pad=4, mode="tf32x3"),
        # The plain FP32 path: a tall-times-small product of the QR of a chi = 256 row.
        dict(name="gemm_tall_f32", kind="gemm", M=36864, N=266, K=266, pad=0, mode="f32"),
        # The small SVD of a chi = 500 row (sketch width 510).
        dict(name="svd_510", kind="svd", k=510),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "theta", "theta", "theta", "svd", "row", "sweep", "expect"])
    if kind == "gemm":
        mode = rng.choice(["tf32x3", "tf32x3", "bf16x3", "f32"])
        while True:
            M, N, K = _log_int(rng, 16, 108000), _log_int(rng, 16, 10000), _log_int(rng, 32, 108000)
            # rows start on 16-byte boundaries (the tensor-core modes need them), sums of any length
            pad = (-K) % 4 + 4 * rng.randint(0, 2)
            if 2.0 * M * N * K <= (1e12 if mode != "f32" else 3e10) and M * N <= 4e8 and (M + N) * K <= 1.2e9:
                return dict(kind=kind, M=M, N=N, K=K, pad=pad, mode=mode)
    if kind == "theta":
        D, K = rng.choice([2, 3, 4, 5, 6, 6]), rng.choice([1, 2, 4])
        prec = rng.choice(["tf32x3", "tf32x3", "tf32x3", "bf16x3", "f32", "f64"])
        while True:
            chi, k = _log_int(rng, 12, 500), _log_int(rng, 1, 300)
            case = dict(kind=kind, op=rng.randint(0, 3), c=rng.choice([0, 1, 1, 1, 2]), D=D, K=K, chi=chi, k=k, prec=prec)
            most = dict(tf32x3=2e12, bf16x3=2e12, f32=3e11, f64=1e10)[prec]
            if work(case)["flops"] <= most:
                return case
    if kind == "svd":
        return dict(kind=kind, k=_log_int(rng, 8, 510))
    if kind == "row":
        D, K = rng.choice([3, 4, 5, 6]), rng.choice([1, 2, 4])
        Lx, Ly = rng.randint(4, 6), rng.randint(3, 6)
        top = 180 if D * (K + 2) * D > 144 else 256
        return dict(kind=kind, Lx=Lx, Ly=Ly, D=D, K=K, chi=_log_int(rng, 24, top), prec="tf32x3", q=rng.randint(0, 2),
                    n_fit=rng.randint(0, 1))
    if kind == "sweep":
        if rng.random() < 0.3:
            # chi covers the bonds: a cut through a degenerate pair of sectors has no unique answer
            return dict(kind=kind, Lx=rng.randint(3, 4), Ly=3, D=2, K=4, chi=rng.randint(24, 64), prec="f64",
                        q=rng.randint(0, 2), n_fit=rng.randint(0, 1), u1=True)
        prec = rng.choice(["tf32x3", "tf32x3", "f32", "f64"])
        return dict(kind=kind, Lx=rng.randint(3, 5), Ly=rng.randint(3, 5), D=rng.choice([2, 3] if prec == "f64" else [2, 3, 4]),
                    K=rng.choice([1, 2]), chi=_log_int(rng, 8, 32 if prec == "f64" else 96), prec=prec, q=rng.randint(0, 2),
                    n_fit=rng.randint(0, 2), u1=False)
    return dict(kind=kind, Lx=3, Ly=rng.randint(2, 3), D=2, K=rng.randint(1, 2), chi=rng.randint(16, 256), prec="f64",
                q=rng.randint(0, 1), exact_svd=rng.randint(0, 1))


# ----------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _decay(n, lo):
    """Weights 1 .. lo in geometric steps: the spread of the singular values kept on a bond."""
    return torch.logspace(0.0, math.log10(lo), n, device="cuda") if n > 1 else torch.ones(1, device="cuda")


def _lattice(case, seed, Lx, Ly):
    """PEPS, operator PEPO: Hubbard hoppings where K = 4, generic symmetric terms otherwise."""
    peps = L.random_peps(Lx, Ly, case["D"], 4, seed=seed)
    if case["K"] == 4:
        ham = L.hubbard_hamiltonian(Lx, Ly, seed=seed, K=4)
    else:
        ham = L.random_hamiltonian(Lx, Ly, 4, case["K"], seed)
    return peps, L.fsm_pepo(ham), ham


def _boundary_checkpoint(gen, bonds, phys, row, elem):
    """A stored boundary MPS in the library's checkpoint layout, on the device (entries N(0,1), unit-norm tensors)."""
    dt = torch.float64 if elem == 8 else torch.float32
    empty = [np.zeros((bonds[c], phys[c], bonds[c + 1]), dtype=np.int8) for c in range(len(phys))]
    whole = WL.boundary_blob([e[:, :0, :] for e in empty], row, 1, elem)   # header without the tensors
    head = np.frombuffer(whole, dtype=np.int64).copy()
    Ly = len(phys)
    head[5:5 + Ly + 1] = bonds
    head[5 + Ly + 1:5 + 2 * Ly + 1] = phys
    parts = [torch.from_numpy(head).cuda().view(torch.uint8)]
    tensors = []
    for c in range(Ly):
        t = torch.randn(bonds[c] * phys[c] * bonds[c + 1], device="cuda", dtype=torch.float32, generator=gen).to(dt)
        t /= t.norm()
        tensors.append(t.view(bonds[c], phys[c], bonds[c + 1]))
        parts.append(t.view(torch.uint8))
    return torch.cat(parts), tensors


def _theta_dims(case):
    """Dimensions of the site (middle row of a 3 x 3 patch): ket and PEPO legs l, u, r, d, bonds t, t'."""
    c, D, w, chi = case["c"], case["D"], case["K"] + 2, case["chi"]
    a = [1 if c == 0 else D, D, 1 if c == 2 else D, D]
    b = [1 if c == 0 else w, w, 1 if c == 2 else w, w]
    t, tp = (1 if c == 0 else chi), (1 if c == 2 else chi)
    return a, b, t, tp


def _theta_shapes(case):
    a, b, t, tp = _theta_dims(case)
    bl, bu, br, bd = (x * y * x for x, y in zip(a, b))
    n, k = case["chi"], case["k"]
    envs = (n, t, bl) if case["op"] < 2 else (n, tp, br)
    xin = {0: (k, tp, br), 1: (k, n, bd), 2: (k, bd, n), 3: (k, t, bl)}[case["op"]]
    out = {0: (n, bd), 1: (tp, br), 2: (t, bl), 3: (bd, n)}[case["op"]]
    return envs, xin, out


def _theta_inputs(case, seed):
    gen = _gen(seed)
    peps, pepo, _ = _lattice(case, seed, 3, 3)
    chi, Ly = case["chi"], 3
    phys = [peps[1][c].shape[1] * pepo[1][c].shape[1] * peps[1][c].shape[1] for c in range(Ly)]
    elem = 8 if case["prec"] == "f64" else 4
    blob, tensors = _boundary_checkpoint(gen, [1, chi, chi, 1], phys, 1, elem)
    envs, xin, _ = _theta_shapes(case)
    dt = torch.float64 if elem == 8 else torch.float32
    e = torch.randn(envs, device="cuda", generator=gen) * _decay(envs[0], 1e-3)[:, None, None]   # rows carry singular values
    x = torch.randn(xin, device="cuda", generator=gen)
    return peps, pepo, blob, tensors, (e / e.norm()).to(dt), (x / x.norm()).to(dt)


def _env(case, peps, pepo, seed, charges=None):
    return fp.Env(peps, pepo, D=case["D"], p=4, w=case["K"] + 2, chi=case["chi"], prec=case["prec"], seed=seed, charges=charges)


def _params(case):
    return fp.params(oversample=4 if case.get("u1") else 10, power_iters=case["q"], n_fit=case.get("n_fit", 1),
                     exact_svd=case.get("exact_svd", 0))


def _svd_input(case, seed):
    """What the path factorises: the transposed triangular factor of a QR, singular values over six decades."""
    k = case["k"]
    gen = _gen(seed)
    g = [torch.randn(k, k, device="cuda", dtype=torch.float64, generator=gen) for _ in range(2)]
    q = [torch.linalg.qr(x)[0] for x in g]
    s = torch.logspace(0, -6, k, dtype=torch.float64, device="cuda") if k > 1 else torch.ones(1, dtype=torch.float64, device="cuda")
    return torch.linalg.qr((q[0] * s) @ q[1])[1].T.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "gemm":
        gen = _gen(seed)
        M, N, K, ld = case["M"], case["N"], case["K"], case["K"] + case["pad"]
        s["A"] = torch.randn(M, ld, device="cuda", generator=gen) * _decay(M, 1e-3)[:, None]
        s["B"] = torch.randn(N, ld, device="cuda", generator=gen)
        s["C"] = torch.empty(M, N, device="cuda")
        s["mode"] = fp.PRECISIONS[case["mode"]]
    elif kind == "theta":
        peps, pepo, blob, _, e, x = _theta_inputs(case, seed)
        s["env"] = _env(case, peps, pepo, seed)
        fp._check(s["env"].h, fp.lib().fpeps_import_boundary(s["env"].h, blob.data_ptr(), blob.numel(), 1, 1))
        fp.fpeps_absorb_row(s["env"].h, 1, 1)
        torch.cuda.synchronize()
        s["e"], s["x"] = e.cpu().numpy(), x.cpu().numpy()
        s["out"] = _theta_shapes(case)[2]
    elif kind == "svd":
        s["M"] = _svd_input(case, seed)
    elif kind == "row":
        Lx, Ly, row = case["Lx"], case["Ly"], case["Lx"] - 2
        peps, pepo, _ = _lattice(case, seed, Lx, Ly)
        bonds = L.boundary_bond_profile(Ly, case["chi"], case["D"] * (case["K"] + 2) * case["D"])
        phys = [peps[row][c].shape[1] * pepo[row][c].shape[1] * peps[row][c].shape[1] for c in range(Ly)]
        s["blob"], _ = _boundary_checkpoint(_gen(seed), bonds, phys, row, 4)
        s["env"], s["prm"], s["row"] = _env(case, peps, pepo, seed), _params(case), row
    elif kind == "sweep":
        charges = None
        if case["u1"]:
            Lx, Ly = case["Lx"], case["Ly"]
            peps, ch = u1.u1_peps(Lx, Ly, case["D"], seed)
            ham = L.hubbard_hamiltonian(Lx, Ly, seed)
            pepo = L.fsm_pepo(ham)
            qpeps = [[u1.peps_leg_charges(ch, Lx, Ly, r, c) for c in range(Ly)] for r in range(Lx)]
            charges = fp.pack_charges(qpeps, u1.hubbard_pepo_charges(ham))
        else:
            peps, pepo, _ = _lattice(case, seed, case["Lx"], case["Ly"])
        s["env"], s["prm"] = _env(case, peps, pepo, seed, charges), _params(case)
    else:
        peps, pepo, _ = _lattice(case, seed, case["Lx"], case["Ly"])
        s["env"], s["prm"] = _env(case, peps, pepo, seed), _params(case)
    return s


# ----------------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "gemm":
        fp.fpeps_gemm_f32(s["mode"], s["A"], s["B"], s["C"], K=case["K"])
        return s["C"]
    if kind == "theta":
        return s["env"].apply_theta_op(case["op"], case["c"], s["e"], s["x"], s["out"])
    if kind == "svd":
        U, sg, V = fp.fpeps_svd_f64(s["M"])
        # a singular pair's sign is free: the caller's gauge makes V's largest entry positive
        sign = torch.sign(torch.gather(V, 0, V.abs().argmax(0, keepdim=True)))
        return U * sign, sg, V * sign
    h = s["env"].h
    if kind == "expect":
        value, sign, log_abs = s["env"].expect(s["prm"])
        return dict(value=value, num_sign=sign, num_log=log_abs)
    if kind == "row":
        fp._check(h, fp.lib().fpeps_import_boundary(h, s["blob"].data_ptr(), s["blob"].numel(), s["row"], 1))
        fp.fpeps_absorb_row(h, s["row"], 1)
        st = fp.fpeps_compress_rsvd(h, s["prm"])
        res = dict(log_scale=st.log_scale, trunc_err_est=st.trunc_err_est)
        # the spectra are returned; the boundary itself stays in the library (its bond bases are
        # defined only up to rounding where kept values are close) and goes into the closing row
        for which, name in ((0, "zip"), (1, "fit")):
            res[name] = [torch.tensor(v) for c in range(case["Ly"]) if (v := fp.fpeps_bond_spectrum(h, which, c))]
        fp.fpeps_absorb_row(h, s["row"] + 1, 1)
    else:
        res = dict(rows=[])
        for r in range(case["Lx"]):
            fp.fpeps_absorb_row(h, r, 1)
            if 0 < r < case["Lx"] - 1:
                res["rows"].append(fp.fpeps_compress_rsvd(h, s["prm"]).log_scale)
    res["sign"], res["log_abs"] = fp.fpeps_sweep_value(h)
    return res


# ----------------------------------------------------------------------------- what a pass cannot do without
def _channels(K, edge_l, edge_r):
    """Nonzero channels and (l, d) pairs of an interior-row site of the finite-state PEPO with K hoppings."""
    if edge_r:
        return 4 + 3 * K, 3 + 2 * K
    return (2 + 3 * K, 1 + K) if edge_l else (3 + 4 * K, 2 + 2 * K)


def _map_work(a, b, t, tp, n, k, K, elem):
    """(bytes, flops) of one site map on k vectors with an environment of n rows."""
    bl, bu, br, bd = (x * y * x for x, y in zip(a, b))
    nch, npair = _channels(K, b[0] == 1, b[2] == 1)
    ket = a[0] * a[1] * a[2] * a[3] * 4
    sand = 2.0 * t * k * (nch * ket * a[1] * a[2] + npair * ket * a[0] * a[3])
    flops = 2.0 * t * bu * tp * k * br + sand + 2.0 * n * t * bl * k * bd
    return elem * (n * t * bl + t * bu * tp + k * tp * br + k * n * bd), flops


def _row_work(case):
    """One interior row (zip-up, and a fit pass where there is one) plus the closing row, applications only."""
    Ly, D, w, chi, K = case["Ly"], case["D"], case["K"] + 2, case["chi"], case["K"]
    B = D * w * D
    bonds = L.boundary_bond_profile(Ly, chi, B)
    nb = nf = 0.0
    left = [1]
    for c in range(Ly):
        a = [1 if c == 0 else D, D, 1 if c == Ly - 1 else D, D]
        b = [1 if c == 0 else w, w, 1 if c == Ly - 1 else w, w]
        t, tp = bonds[c], bonds[c + 1]
        n = left[c]
        cols = tp * (a[2] * b[2] * a[2])
        new = min(chi, n * B, cols)
        k = min(new + 10, n * B, cols)
        x, f = _map_work(a, b, t, tp, n, k, K, 4)
        nf += f * (2 * case["q"] + 2 if c < Ly - 1 else 1.0)
        nb += x
        if case["n_fit"] and c < Ly - 1:
            f2 = _map_work(a, b, t, tp, n, chi, K, 4)[1]
            nf += 2 * f2 * (1 + (2 * case["q"] + 2) * 0.1)
        left.append(new)
    return nb, nf


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=4.0 * (M * K + N * K + M * N), flops=2.0 * M * N * K)
    if kind == "theta":
        a, b, t, tp = _theta_dims(case)
        nb, nf = _map_work(a, b, t, tp, case["chi"], case["k"], case["K"], 8 if case["prec"] == "f64" else 4)
        return dict(bytes=float(nb), flops=nf)
    if kind == "svd":
        k = case["k"]
        return dict(bytes=8.0 * (3 * k * k + k), flops=12.0 * k ** 3)   # a dense SVD with both sets of vectors
    if kind == "row":
        nb, nf = _row_work(case)
        return dict(bytes=nb, flops=nf)
    rows = max(1, case["Lx"] - 2) * (2 if kind == "expect" else 1)
    elem = 8 if case["prec"] == "f64" else 4
    nb, nf = _row_work(dict(case, n_fit=case.get("n_fit", 1), chi=min(case["chi"], (case["D"] ** 2 * (case["K"] + 2)) ** (case["Ly"] // 2))))
    return dict(bytes=rows * nb * elem / 4, flops=rows * nf)


# ----------------------------------------------------------------------------- the same in 64 bits
def _sandwich64(A, W, I, x, y, v, z):
    """out[n, v, V, v', z, Z, z'] of the ket-PEPO-bra sandwich on I[n, x, X, x', y, Y, y'] (legs named l, u, r, d)."""
    wl, br = dict(l="L", u="U", r="R", d="D"), dict(l="i", u="j", r="k", d="m")
    one = torch.einsum("n%s%s%s%s%s%s,lurdp->n%s%s%s%s%s%sp" % (x, wl[x], br[x], y, wl[y], br[y], wl[x], br[x], wl[y], br[y], v, z), I, A)
    two = torch.einsum("n%s%s%s%s%s%sp,LURDpq->n%s%s%s%s%s%sq" % (wl[x], br[x], wl[y], br[y], v, z, br[x], br[y], v, z, wl[v], wl[z]), one, W)
    return torch.einsum("n%s%s%s%s%s%sq,ijkmq->n%s%s%s%s%s%s" % (br[x], br[y], v, z, wl[v], wl[z], v, wl[v], br[v], z, wl[z], br[z]), two, A)


def _theta64(case, seed):
    peps, pepo, _, tensors, e, x = _theta_inputs(case, seed)
    c, op = case["c"], case["op"]
    f = torch.float32 if case["prec"] != "f64" else torch.float64   # the site tensors as the library holds them
    A = torch.from_numpy(peps[1][c]).cuda().to(f).double()
    W = torch.from_numpy(pepo[1][c]).cuda().to(f).double()
    T, e = tensors[c].double(), e.double()
    a, b, t, tp = _theta_dims(case)
    leg = {n: (a[i], b[i], a[i]) for i, n in enumerate("lurd")}
    size = {n: q[0] * q[1] * q[2] for n, q in leg.items()}
    ins, outs = {0: ("ur", "ld"), 1: ("ld", "ur"), 2: ("rd", "lu"), 3: ("lu", "rd")}[op]
    y = []
    for v in x.double():                            # one vector at a time: [t, bundle x, bundle y] blocks
        if op == 0:
            g = torch.einsum("tus,sr->tur", T, v)
        elif op == 1:
            g = torch.einsum("atl,ad->tld", e, v)
        elif op == 2:
            g = torch.einsum("asr,da->srd", e, v)
        else:
            g = torch.einsum("tus,tl->slu", T, v)
        n = g.shape[0]
        g = torch.cat([_sandwich64(A, W, q.reshape(q.shape[0], *leg[ins[0]], *leg[ins[1]]), *ins, *outs)
                       for q in g.split(max(1, 2 ** 28 // (size[ins[0]] * size[ins[1]] * 16)))])
        g = g.reshape(n, size[outs[0]], size[outs[1]])
        if op == 0:
            y.append(torch.einsum("atl,tld->ad", e, g))
        elif op == 1:
            y.append(torch.einsum("tus,tur->sr", T, g))
        elif op == 2:
            y.append(torch.einsum("tus,slu->tl", T, g))
        else:
            y.append(torch.einsum("asr,srd->da", e, g))
    return torch.stack(y)


def _expect64(case, seed):
    """<H> of a lattice small enough to write its state vector out."""
    Lx, Ly = case["Lx"], case["Ly"]
    peps, _, ham = _lattice(case, seed, Lx, Ly)
    psi = None                                      # [physical so far, open down legs of the row above / this row, right leg]
    for r in range(Lx):
        for c in range(Ly):
            A = torch.from_numpy(peps[r][c]).cuda().double()
            l, u, rr, d, p = A.shape
            if psi is None:
                psi = torch.ones((1, 1, 1), dtype=torch.float64, device="cuda")
                legs = [1] * Ly
            lead, rest = psi.shape[0], int(np.prod(legs[1:]))
            q = psi.reshape(lead, u, rest, l)
            q = torch.einsum("xuyl,lurdp->xpydr", q, A)
            psi = q.reshape(lead * p, rest * d, rr)
            legs = legs[1:] + [d]
    n = Lx * Ly
    psi = psi.reshape([4] * n)

    def act(op, site, vec):
        m = torch.from_numpy(np.ascontiguousarray(op)).cuda()
        return torch.movedim(torch.tensordot(m, vec, dims=([1], [site])), 0, site)

    h = torch.zeros_like(psi)
    for r in range(Lx):
        for c in range(Ly):
            i = r * Ly + c
            h += act(ham.onsite[r][c], i, psi)
            for k in range(ham.K):
                if c + 1 < Ly:
                    h += float(ham.t_h[k, r, c]) * act(ham.Y[k], i + 1, act(ham.X[k], i, psi))
                if r + 1 < Lx:
                    h += float(ham.t_v[k, r, c]) * act(ham.Y[k], i + Ly, act(ham.X[k], i, psi))
    num, den = float((psi * h).sum()), float((psi * psi).sum())
    return dict(value=num / den, num_sign=None, num_log=math.log(abs(num)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        if case["M"] * case["K"] > 2 ** 28:
            return None
        s, K = prepare(case, seed), case["K"]
        A = s["A"][:, :K].double()
        return torch.cat([A @ b[:, :K].double().T for b in s["B"].split(max(1, 2 ** 28 // K))], 1)
    if kind == "theta":
        return _theta64(case, seed)
    if kind == "svd":
        M = _svd_input(case, seed).cpu().numpy()
        U, sg, Vt = np.linalg.svd(M)
        V = Vt.T
        sign = np.sign(np.take_along_axis(V, np.abs(V).argmax(0)[None], 0))
        return U * sign, sg, V * sign
    if kind == "expect":
        # the sweep keeps every bond (chi covers the ranks), so the value is the state's own
        B = case["D"] ** 2 * (case["K"] + 2)
        return _expect64(case, seed) if case["chi"] >= B ** (case["Ly"] // 2) else None
    return None   # truncated sweeps: what they return is defined by the algorithm's own sketches
