"""The batched solver's ||w|| against its 64-bit value, through the breakdown test: the threshold
is put 8e-16 below and above the ratio ||w2|| / ||A v|| of the first step, and the step must pass
and fail.

With random data the rounding of the rows of w (double-float, 2^-48) averages out over the rows; f64
codes: omega is summed in FP64.  What is left is the sums' own rounding, some 2e-16 rms in
FP64; double-float sums of the squares were 4e-16 to 2e-15 off.  (A first form of this test took
integer values and equal entries of v: every row then rounds alike and nothing averages out.)"""
import math

import numpy as np
import pytest

import workloads as W
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _restarts(cb, torch, monkeypatch, A, b, eps, cluster):
    make = cb.options

    def opts(**kw):
        o = make(**kw)
        o.breakdown_eps = eps
        return o

    with monkeypatch.context() as m:
        m.setattr(cb, "options", opts)
        with cb.BatchedSolver([A], restart=2, fmt="f64", precond="none", use_graph=False) as s:
            s.schedule(cluster, 1)
            x = torch.zeros(A.n, dtype=torch.float64, device="cuda")
            return int(s.solve(torch.from_numpy(b).cuda(), x, tol=0.0, maxit=2)["restarts"][0])


@pytest.mark.parametrize("n,cluster", [(3000, 1), (20000, 1), (60000, 8)])
def test_first_ratio_to_fp64(n, cluster, monkeypatch):
    torch, cb = need_gpu()
    for seed in range(8):
        g = np.random.default_rng(seed)
        i = np.arange(n)
        A = W._from_coo(n, np.concatenate([i, i[1:], i[:-1]]), np.concatenate([i, i[:-1], i[1:]]),
                        g.standard_normal(3 * n - 2))
        s = g.standard_normal(n)
        w = A.to_scipy() @ s
        dot = lambda x, y: math.fsum((x * y).tolist())
        c = dot(s, w) / dot(s, s)
        w2 = w - c * s
        w2 = w2 - dot(s, w2) / dot(s, s) * s
        r = math.sqrt(dot(w2, w2) / dot(w, w))
        assert _restarts(cb, torch, monkeypatch, A, s, r * (1 - 8e-16), cluster) == 1, (n, seed)
        assert _restarts(cb, torch, monkeypatch, A, s, r * (1 + 8e-16), cluster) == 2, (n, seed)
