"""The sums over blocks of the stepwise kernels in double-float (column sums of the pipelined
dot, ||w|| of the axpy, omega of the SpMV) against FP64 arithmetic, from two rows to more blocks
than SMs, and the row limits between the stepwise kernels and the single-launch cycle."""
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


@pytest.mark.parametrize("fmt,n,restart,single", [
    ("f64", 600000, 12, True), ("f64", 600001, 12, False), ("f16", 599999, 12, True), ("f32", 600000, 12, True),
    ("f32", 600001, 12, False), ("i16", 600007, 12, False), ("f64", 149999, 99, True), ("f64", 150001, 99, False),
    ("f32", 587500, 99, True), ("i32", 587501, 99, False)])
def test_row_limits_of_the_single_launch(fmt, n, restart, single):
    """Either side of the limits: the same columns as the stepwise kernels, and the route."""
    torch, cb = need_gpu()
    A = _tridiagonal(n)
    b = to_dev(torch, W.random_vector(n, 3))
    out = []
    for profile in (False, True):
        with cb.Solver.from_csr(A, restart=restart, fmt=fmt, profile=profile) as s:
            x = torch.zeros_like(b)
            H = s.arnoldi(b, x, 10)
            st = s.solve(b, x, tol=1e-9, maxit=2000)
            out.append((H, st, x))
    (Hc, sc, xc), (Hs, ss, xs) = out
    assert col_relerr(Hc, Hs, Hc.shape[1]).max() <= 1e-10
    assert sc["status"] == ss["status"] == 0
    assert (sc["kernel_launches"] < ss["kernel_launches"]) == single
    # diagonally dominant by 0.9 of a norm of 5.1: residuals of 1e-9 ||b|| each
    assert float((xc - xs).norm()) <= 2e-9 / 0.9 * float(b.norm())
