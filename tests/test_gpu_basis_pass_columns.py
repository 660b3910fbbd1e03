"""Every Hessenberg column of a cycle against FP64 Gram-Schmidt on the same stored columns: all
widths of the one-pass kernel's tiles, column counts that fill its groups of four partly, and the
two kernels beyond 112 columns, for every format; the single launch as well."""
import numpy as np
import pytest

from gpu_common import FORMATS, need_gpu, to_dev
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("n,k,profile", [(300, 114, True), (5003, 114, True), (5003, 114, False), (40961, 113, True),
                                         (400000, 61, True)])
def test_columns_from_the_stored_basis(fmt, n, k, profile):
    torch, cb = need_gpu()
    i = np.arange(n)
    A = W._from_coo(n, np.concatenate([i, i[1:], i[:-1]]), np.concatenate([i, i[:-1], i[1:]]),
                    np.concatenate([3.0 + np.sin(i), np.full(n - 1, -1.3), np.full(n - 1, -0.7)]))
    b = to_dev(torch, W.random_vector(n, 5))
    with cb.Solver.from_csr(A, restart=115, fmt=fmt, profile=profile) as s:
        H = torch.from_numpy(s.arnoldi(b, torch.zeros_like(b), k)).cuda()
        V = torch.stack([s.basis_column(j) for j in range(k)])
        worst = 0.0
        for j in range(k):
            w = s.spmv(V[j].contiguous())
            h = V[:j + 1] @ w
            w1 = w - V[:j + 1].T @ h
            u = V[:j + 1] @ w1
            hn = (w1 - V[:j + 1].T @ u).norm()
            ref = torch.cat([h + u, hn[None]])
            worst = max(worst, float((H[:j + 2, j] - ref).norm() / ref.norm()))
    # products and sums to 2^-46 relative each (the bound the arithmetic states), one of either
    assert worst <= 2 * 2.0 ** -46, worst
