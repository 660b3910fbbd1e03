"""The sums over blocks of the stepwise kernels in double-float (column sums of the pipelined
dot, ||w|| of the axpy, omega of the SpMV) against FP64 arithmetic, from two rows to more blocks
than SMs."""
import numpy as np
import pytest

from gpu_common import col_relerr, need_gpu, to_dev
import workloads as W

pytestmark = pytest.mark.gpu


def _tridiagonal(n):
    i = np.arange(n)
    rows = np.concatenate([i, i[1:], i[:-1]])
    cols = np.concatenate([i, i[:-1], i[1:]])
    return W._from_coo(n, rows, cols, np.concatenate([3.0 + 0.1 * np.sin(i), np.full(n - 1, -1.3), np.full(n - 1, -0.7)]))


@pytest.mark.parametrize("fmt", ["f64", "f32", "i32"])
@pytest.mark.parametrize("n", [2, 33, 257, 4095, 155649, 1000003])
def test_block_sums_match_fp64(fmt, n):
    torch, cb = need_gpu()
    A = _tridiagonal(n)
    b, x0 = to_dev(torch, W.random_vector(n, 1)), to_dev(torch, W.random_vector(n, 2))
    k = min(9, n - 1)
    H = []
    for arith in ("df32", "fp64"):
        with cb.Solver.from_csr(A, restart=12, fmt=fmt, arith=arith, profile=True) as s:   # (stepwise)
            H.append(s.arnoldi(b, x0, k))
    # both evaluate the same columns to FP64 class, the bar the solver is held to everywhere
    assert col_relerr(H[0], H[1], k).max() <= 1e-10
