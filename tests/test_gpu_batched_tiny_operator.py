"""Operators so small that no power of two within the solver's range normalises them, down to
subnormal values (exact here): the same iterations as the unscaled system's."""
import numpy as np
import pytest

import workloads as W
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", ["f64", "f32"])
@pytest.mark.parametrize("cluster", [1, 2])
def test_tiny_operators_converge_alike(fmt, cluster):
    torch, cb = need_gpu()
    n = 900
    i = np.arange(n)
    b = np.ldexp(W.random_vector(n, 1), -60)
    iters = []
    for e in (0, -960, -1000, -1022, -1026, -1034):
        v = np.ldexp(np.concatenate([np.full(n, 4.0), np.full(n - 1, -1.0), np.full(n - 1, -2.0)]), e)
        A = W._from_coo(n, np.concatenate([i, i[1:], i[:-1]]), np.concatenate([i, i[:-1], i[1:]]), v)
        with cb.BatchedSolver([A], restart=20, fmt=fmt, precond="none", use_graph=False) as s:
            s.schedule(cluster, 1)
            x = torch.zeros(n, dtype=torch.float64, device="cuda")
            st = s.solve(torch.from_numpy(b).cuda(), x, tol=1e-8, maxit=300)
        assert st["status"] == 0, e
        iters.append(int(st["iters"][0]))
        r = np.ldexp(b, 60) - np.ldexp(A.to_scipy() @ x.cpu().numpy(), 60)
        assert np.linalg.norm(r) <= 1.001e-8 * np.linalg.norm(np.ldexp(b, 60)), e
    assert max(iters) - min(iters) <= 1, iters
