"""After cudaDeviceReset the library works in the new context: standalone products (scratch from a
pool of the library's own), the multi-vector product on both paths, and a solve.  In a process of
its own, with memory from the CUDA runtime."""
import os
import subprocess
import sys
import textwrap

import pytest

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu

CHILD = textwrap.dedent("""
    import ctypes as C, sys
    sys.path.insert(0, {root!r})
    import numpy as np
    import paper_2009_12101_gb300 as cb
    import workloads as W

    L = cb.lib()
    rt = C.CDLL({cudart!r})
    rt.cudaMalloc.argtypes = [C.POINTER(C.c_void_p), C.c_size_t]
    rt.cudaMemcpy.argtypes = [C.c_void_p, C.c_void_p, C.c_size_t, C.c_int]

    def ok(rc):
        assert rc == 0, rc

    def up(a):
        p = C.c_void_p()
        ok(rt.cudaMalloc(C.byref(p), a.nbytes))
        ok(rt.cudaMemcpy(p, a.ctypes.data, a.nbytes, 1))
        return p

    def down(p, like):
        out = np.empty_like(like)
        ok(rt.cudaMemcpy(out.ctypes.data, p, out.nbytes, 2))
        return out

    g = np.random.default_rng(0)
    n, nc, k = 5000, 20, 7
    ld = 8192
    V = np.zeros((nc, ld), np.float32); V[:, :n] = g.standard_normal((nc, n))
    Vh = np.zeros((nc, ld), np.float16); Vh[:, :n] = g.uniform(-1, 1, (nc, n))
    w = np.zeros(ld); w[:n] = g.standard_normal(n)
    Wm = g.standard_normal((k, n)); one = np.ones(nc)
    A = W.convdiff3d(12); b = W.random_vector(A.n, 1)

    def run():
        res = []
        dV, dVh, dw, dW, d1 = up(V), up(Vh), up(w), up(Wm), up(one)
        for arith in (0, 1):
            h = np.zeros(nc)
            ok(L.cbg_basis_dot(cb.FORMATS["f32"], arith, n, nc, dV, ld, one.ctypes.data, dw, h.ctypes.data, None))
            y = up(w)
            ok(L.cbg_basis_axpy(cb.FORMATS["f32"], arith, n, nc, dV, ld, one.ctypes.data, h.ctypes.data, y, None))
            res += [h, down(y, w)]
        ws = np.zeros(L.cbg_basis_dot_multi_workspace(ld, nc, k), np.uint8)
        dws, H = up(ws), np.zeros((nc, k))
        for fmt, d, path in (("f32", dV, 1), ("f16", dVh, 2)):
            dH = up(H)
            ok(L.cbg_basis_dot_multi_path(cb.FORMATS[fmt], n, nc, d, ld, d1, k, dW, n, dH, dws, ws.nbytes, None, path))
            res.append(down(dH, H))
        rp, ci, va = (np.ascontiguousarray(a, t) for a, t in ((A.rowptr, np.int32), (A.col, np.int32), (A.val, np.float64)))
        csr = cb.Csr(A.n, ci.size, rp.ctypes.data, ci.ctypes.data, va.ctypes.data, 0, 0)
        for profile in (0, 1):                      # the single launch, the stepwise kernels
            o = cb.Options(); L.cbgmres_options_default(C.byref(o)); o.profile = profile
            s, st = C.c_void_p(), cb.Stats()
            ok(L.cbgmres_create(C.byref(csr), 20, cb.FORMATS["f32"], C.byref(o), C.byref(s)))
            db, dx = up(b), up(np.zeros(A.n))
            ok(L.cbgmres_solve(s, db, dx, 1e-10, 2000, C.byref(st)))
            res.append(down(dx, b))
            L.cbgmres_destroy(s)
        return res

    first = run()
    for _ in range(2):
        ok(rt.cudaDeviceReset())
        again = run()
        assert all(np.array_equal(p, q) for p, q in zip(first, again))
    print("same")
""")


def test_calls_after_a_device_reset():
    torch, cb = need_gpu()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    cudart = "libcudart.so." + torch.version.cuda.split(".")[0]
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=root, cudart=cudart)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("same"), r.stdout + r.stderr
