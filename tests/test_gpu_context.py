"""The entry points in a second context of the same process: a child process computes a few results, ends
its own context between calls (cudaDeviceReset, nothing in flight) and computes them again. What holds for
one context only (kernel attributes, co-resident blocks, the scratch pool, pinned words, the address of the
fixed SVD array) is found again in the new one."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes as C, numpy as np
from paper_2511_01039_gb300 import fpeps as fp
from synth import lattice as L
lib = fp.lib()
rt = C.CDLL("libcudart.so.13")

def put(a):
    p = C.c_void_p()
    assert rt.cudaMalloc(C.byref(p), C.c_size_t(a.nbytes)) == 0
    assert rt.cudaMemcpy(p, a.ctypes.data_as(C.c_void_p), C.c_size_t(a.nbytes), 1) == 0
    return p

def get(p, shape, dt):
    a = np.empty(shape, dt)
    assert rt.cudaMemcpy(a.ctypes.data_as(C.c_void_p), p, C.c_size_t(a.nbytes), 2) == 0
    return a

def results():
    g = np.random.default_rng(0)
    out = []
    for M, N, K in ((200, 300, 64), (1024, 2048, 4096), (100, 64, 64)):      # on-chip split, planes, single CTA
        A, B = g.standard_normal((M, K), dtype=np.float32), g.standard_normal((N, K), dtype=np.float32)
        a, b, c = put(A), put(B), put(np.zeros((M, N), np.float32))
        assert lib.fpeps_gemm_f32(fp.TF32X3, M, N, K, a, K, b, K, c, None) == 0
        got = get(c, (M, N), np.float32)
        assert np.abs(got - A.astype(float) @ B.T.astype(float)).max() < 1e-4 * K ** 0.5
        out.append(got)
    for k, f in ((70, lib.fpeps_svd_f64), (160, lib.fpeps_svd_f64), (70, lib.fpeps_svd_f64_noalloc)):
        A = np.linalg.qr(g.standard_normal((k, k)))[1].copy()                # R^T, column by column
        m, u, s, v = put(A), put(A), put(A[0].copy()), put(A)
        assert f(m, k, u, s, v, None) == 0
        out.append(get(s, k, np.float64))
        assert np.allclose(out[-1], np.linalg.svd(A, compute_uv=False), rtol=1e-9, atol=1e-12)
    peps = L.random_peps(3, 3, 2, 4, seed=0)
    pepo = L.fsm_pepo(L.random_hamiltonian(3, 3, 4, 2, seed=0))
    pk, wk = (put(np.concatenate([np.asarray(t, float).ravel() for r in x for t in r])) for x in (peps, pepo))
    for prec in ("f64", "tf32x3"):
        cfg = fp.fpeps_config(3, 3, 2, 4, 4, 256, fp.PRECISIONS[prec], 1, 0, 1)
        h = C.c_void_p()
        assert lib.fpeps_env_create(C.byref(cfg), pk, wk, None, 0, None, None, C.byref(h)) == 0
        out.append(np.array([fp.fpeps_expect(h, fp.params(10, 1, 0, 1, 1))[0]]))
        lib.fpeps_env_destroy(h)
    assert rt.cudaDeviceSynchronize() == 0
    return out

first = results()
for _ in range(2):
    assert rt.cudaDeviceReset() == 0
    for x, y in zip(first, results()):
        assert np.allclose(x, y, rtol=1e-6, atol=1e-6)
print("same")
"""


def test_results_after_the_context_was_replaced():
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", r.stdout + r.stderr
