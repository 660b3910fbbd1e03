"""The restart cycle as one cooperative launch (small matrices) against the stepwise kernels,
which the profiling option selects: Hessenberg columns and solutions at the edges of the
row partition (blocks of 64 rows or a multiple of 16, chunks of 2 to 16 rows), of the column
groups and of the preconditioner stages."""
import numpy as np
import pytest

import workloads as W
from gpu_common import FORMATS, col_relerr, need_gpu, to_dev

pytestmark = pytest.mark.gpu


def _matrix(n):
    """1D upwind convection-diffusion (well conditioned enough for tight comparison)."""
    a = np.zeros((n, n)) if n <= 8 else None
    if a is not None:
        for i in range(n):
            a[i, i] = 3.0
            if i:
                a[i, i - 1] = -1.3
            if i + 1 < n:
                a[i, i + 1] = -0.7
        return W.from_dense(a)
    i = np.arange(n)
    rows = np.concatenate([i, i[1:], i[:-1]])
    cols = np.concatenate([i, i[:-1], i[1:]])
    vals = np.concatenate([np.full(n, 3.0) + 0.1 * np.sin(i), np.full(n - 1, -1.3), np.full(n - 1, -0.7)])
    return W._from_coo(n, rows, cols, vals)


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("n,restart,precond", [
    (5, 3, "none"), (64, 8, "jacobi"), (65, 31, "bj4"), (4097, 32, "none"), (9728, 12, "jacobi"),
    (9729, 33, "bj4"), (40003, 100, "none"), (299999, 20, "none")])
def test_cycle_matches_stepwise(fmt, n, restart, precond):
    torch, cb = need_gpu()
    A = _matrix(n)
    b, x0 = to_dev(torch, W.random_vector(n, 3)), to_dev(torch, W.random_vector(n, 4))
    k = min(10, restart, n - 1)
    out = []
    for profile in (False, True):
        with cb.Solver.from_csr(A, restart=restart, fmt=fmt, precond=precond, profile=profile) as s:
            H = s.arnoldi(b, x0, k)
            x = x0.clone()
            st = s.solve(b, x, tol=1e-9, maxit=4000)
            out.append((H, x.cpu().numpy(), st))
    (Hc, xc, sc), (Hs, xs, ss) = out
    # two FP64-class evaluations of the same columns (the bar the solver is held to against
    # the oracle), and two solutions of the same residual tolerance
    assert Hc.shape == Hs.shape
    assert col_relerr(Hc, Hs, Hc.shape[1]).max() <= 1e-10
    assert sc["status"] == ss["status"] == 0
    assert abs(sc["iters"] - ss["iters"]) <= max(1, 0.02 * ss["iters"])
    assert sc["true_relres"] <= 1e-9 and ss["true_relres"] <= 1e-9
    # A is diagonally dominant by 1 of a norm of 5: ||x - x'|| <= 2e-9 ||b|| ||A^-1||
    assert np.linalg.norm(xc - xs) <= 2e-9 * 1.25 * np.linalg.norm(b.cpu().numpy())
    assert sc["kernel_launches"] < ss["kernel_launches"]


@pytest.mark.parametrize("fmt", ["f64", "f16"])
def test_cycle_longest_restart_and_maxit(fmt):
    """319 columns in one cycle, a cycle cut short by maxit, and a restart of one step."""
    torch, cb = need_gpu()
    A = W.poisson2d(40)
    b = to_dev(torch, W.random_vector(A.n, 5))
    for restart, maxit in ((319, 10000), (100, 7), (1, 30)):
        xs, st = [], []
        for profile in (False, True):
            with cb.Solver.from_csr(A, restart=restart, fmt=fmt, profile=profile) as s:
                x = torch.zeros_like(b)
                st.append(s.solve(b, x, tol=1e-10, maxit=maxit))
                xs.append(x.cpu().numpy())
        assert st[0]["status"] == st[1]["status"]
        assert abs(st[0]["iters"] - st[1]["iters"]) <= 0.02 * st[1]["iters"]
        # ||A^-1|| ~ 85 on this grid: 1e-10 residuals differ by at most 2e-10 * 85 ||b|| in x;
        # capped runs agree to the rounding of a few steps
        assert np.linalg.norm(xs[0] - xs[1]) <= 2e-10 * 90 * np.linalg.norm(b.cpu().numpy())


def test_no_cycle_and_reuse():
    """b = 0 starts no cycle; the same handle then solves, and solves again to the same bits."""
    torch, cb = need_gpu()
    A = W.convdiff3d(12)
    xs = to_dev(torch, W.random_vector(A.n, 6))
    with cb.Solver.from_csr(A, restart=20, fmt="f32") as s:
        b = s.spmv(xs)
        x = xs.clone()
        assert s.solve(torch.zeros_like(b), x, tol=1e-10)["iters"] == 0 and float(x.abs().max()) == 0.0
        got = []
        for _ in range(2):
            x = torch.zeros_like(b)
            assert s.solve(b, x, tol=1e-10, maxit=2000)["status"] == 0
            got.append(x.clone())
        assert torch.equal(*got)
