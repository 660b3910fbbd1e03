"""The first subtraction and the second projection in one pass over the basis: the Arnoldi
relation and the orthogonality of its columns (up to the format's rounding), from one column to
past the most that a tile holds, for every format and tile width, and the Hessenberg columns
against FP64 arithmetic.  The profiling option selects the stepwise kernels at every size."""
import numpy as np
import pytest

from gpu_common import FORMATS, col_relerr, need_gpu, to_dev
import workloads as W

pytestmark = pytest.mark.gpu

# relative rounding of a stored column (for the integers, of its largest element)
EPS = {"f64": 2.0 ** -53, "f32": 2.0 ** -24, "f16": 2.0 ** -11, "bf16": 2.0 ** -8, "e4m3": 2.0 ** -4,
       "i32": 2.0 ** -31, "i16": 2.0 ** -15}


def _tridiagonal(n):
    i = np.arange(n)
    rows = np.concatenate([i, i[1:], i[:-1]])
    cols = np.concatenate([i, i[:-1], i[1:]])
    return W._from_coo(n, rows, cols, np.concatenate([3.0 + np.sin(i), np.full(n - 1, -1.3), np.full(n - 1, -0.7)]))


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("n,k", [(300, 114), (5000, 114), (40961, 59), (400000, 30)])
def test_arnoldi_relation(fmt, n, k):
    torch, cb = need_gpu()
    A = _tridiagonal(n)
    b = to_dev(torch, W.random_vector(n, 1))
    with cb.Solver.from_csr(A, restart=115, fmt=fmt, precond="none", profile=True) as s:
        H = torch.from_numpy(s.arnoldi(b, torch.zeros_like(b), k)).cuda()
        V = torch.stack([s.basis_column(j) for j in range(k + 1)], 1)
        AV = torch.stack([s.spmv(V[:, j].contiguous()) for j in range(k)], 1)
    # A v_j = V h_j + h_{j+1,j} (stored - exact v_{j+1}); the largest element of a random-like unit
    # vector of n rows is below 6 / sqrt(n), so an integer column rounds within 6 EPS of its norm
    slack = 8 * EPS[fmt] * float(H.abs().max()) + 1e-13
    assert float((AV - V @ H).norm(dim=0).max()) <= slack
    # a new column is orthogonal to the stored ones up to its own rounding
    G = V.T @ V
    assert float((G.triu(1)).abs().max()) <= 8 * EPS[fmt] + 1e-13
    assert float((G.diagonal() - 1).abs().max()) <= 20 * EPS[fmt] + 1e-13


@pytest.mark.parametrize("fmt,n,k", [("f64", 400000, 12), ("f32", 800000, 12), ("f16", 1600000, 10), ("e4m3", 3200000, 4),
                                     ("f64", 5000, 20), ("i32", 100001, 20), ("bf16", 4096, 9), ("i16", 65537, 17)])
def test_columns_match_fp64_arithmetic(fmt, n, k):
    """Every tile width (eight spans down to one) against FP64 products of the same codes."""
    torch, cb = need_gpu()
    A = _tridiagonal(n)
    b = to_dev(torch, W.random_vector(n, 2))
    H = []
    for arith in ("df32", "fp64"):
        with cb.Solver.from_csr(A, restart=k + 1, fmt=fmt, precond="none", arith=arith, profile=True) as s:
            H.append(s.arnoldi(b, torch.zeros_like(b), k))
    assert col_relerr(H[0], H[1], k).max() <= 1e-10
