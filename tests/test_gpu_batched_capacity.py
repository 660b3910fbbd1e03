"""The largest systems that a block, or a cluster of 8, holds: rows of w in shared memory.  The
limits are those of the layout with 32 spare rows of 8 bytes in a block."""
import numpy as np
import pytest

import workloads as W
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", ["f64", "f32", "e4m3"])
@pytest.mark.parametrize("cluster,n", [(1, 23585), (8, 188672), (8, 188657), (8, 188609)])
def test_largest_system(fmt, cluster, n):
    torch, cb = need_gpu()
    i = np.arange(n)
    A = W._from_coo(n, np.concatenate([i, i[1:], i[:-1]]), np.concatenate([i, i[:-1], i[1:]]),
                    np.concatenate([4.0 + np.sin(i), np.full(n - 1, -1.3), np.full(n - 1, -0.7)]))
    b = W.random_vector(n, 1)
    with cb.BatchedSolver([A], restart=8, fmt=fmt, use_graph=False) as s:
        s.schedule(cluster, 1)
        x = torch.zeros(n, dtype=torch.float64, device="cuda")
        st = s.solve(torch.from_numpy(b).cuda(), x, tol=1e-8, maxit=400)
    assert st["status"] == 0
    assert np.linalg.norm(b - A.to_scipy() @ x.cpu().numpy()) <= 1.001e-8 * np.linalg.norm(b)
