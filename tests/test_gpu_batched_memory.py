"""A batch whose sliced-ELL copy does not fit in the free device memory is solved from its CSR
values, not refused."""
import numpy as np
import pytest

import workloads as W
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", ["f32", "f64"])
def test_no_room_for_the_sliced_ell_copy(fmt):
    torch, cb = need_gpu()
    n, k = 150000, 24
    i = np.arange(n)
    A = W._from_coo(n, np.concatenate([i, i[1:], i[:-1]]), np.concatenate([i, i[:-1], i[1:]]),
                    np.concatenate([4.0 + np.sin(i), np.full(n - 1, -1.3), np.full(n - 1, -0.7)]))
    b1 = W.random_vector(n, 1)
    b = torch.from_numpy(np.tile(b1, k)).cuda()
    copy = 12 * k * (3 * n - 2)                          # bytes of the copy, up to its padding

    def solve():
        with cb.BatchedSolver([A] * k, restart=4, fmt=fmt, use_graph=False) as s:
            used = free - torch.cuda.mem_get_info()[0]
            x = x0.zero_()
            st = s.solve(b, x, tol=1e-8, maxit=400)
            assert st["status"] == 0
            return used, x.cpu().numpy()

    x0 = torch.zeros_like(b)
    torch.cuda.empty_cache()                             # (nothing is given back under pressure later)
    free = torch.cuda.mem_get_info()[0]
    solve()                                              # (kernels loaded)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    used, x = solve()
    assert used > copy
    ballast = torch.empty(free - (used - copy // 2), dtype=torch.uint8, device="cuda")
    try:
        free = torch.cuda.mem_get_info()[0]
        less, xc = solve()
    finally:
        del ballast
        torch.cuda.empty_cache()
    assert less < used - copy // 2
    r = [np.linalg.norm(b1 - A.to_scipy() @ v[:n]) / np.linalg.norm(b1) for v in (x, xc)]
    assert max(r) <= 1.001e-8
