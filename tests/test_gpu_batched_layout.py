"""The batched solver's sliced-ELL layout and its CSR fallback, its default schedule, and rows
at the edges of chunks (32 rows) and of the blocks' shares, against the single-system solver."""
import numpy as np
import pytest

import workloads as W
from gpu_common import FORMATS, need_gpu

pytestmark = pytest.mark.gpu


def _uneven(n, seed):
    """Diagonally dominant, 1 to 40 entries per row: sliced ELL would pad by far more than a
    quarter, so a batch of these stays in CSR."""
    g = np.random.default_rng(seed)
    rows, cols, vals = [np.arange(n)], [np.arange(n)], [np.full(n, 0.0)]
    for i in range(n):
        k = int(g.integers(0, 3)) if i % 32 else min(40, n - 1)
        if k:
            rows.append(np.full(k, i)); cols.append(g.choice(n, k, replace=False)); vals.append(g.standard_normal(k) * 0.3)
    A = W._from_coo(n, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals))
    r = np.repeat(np.arange(n), np.diff(A.rowptr))
    off = np.bincount(r, weights=np.where(A.col == r, 0.0, np.abs(A.val)), minlength=n)
    v = A.val.copy()
    v[A.col == r] = 1.0 + off
    return W.CSR(n, A.rowptr, A.col, v)


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("layout", ["stencil", "uneven"])
def test_batched_layouts_match_single_systems(fmt, layout):
    torch, cb = need_gpu()
    g = np.random.default_rng(3)
    if layout == "stencil":
        mats = [W._weighted_laplacian(s, g, 0.3) for s in ((1,), (31,), (4, 8), (33,), (5, 205), (64, 65), (9, 10, 11))]
    else:
        mats = [_uneven(n, n) for n in (2, 31, 32, 33, 1025, 4100)]
    bs = [W.rhs_from_solution(A, W.random_vector(A.n, 7 + i)) for i, A in enumerate(mats)]
    b = torch.from_numpy(np.concatenate(bs)).cuda()
    x = torch.zeros_like(b)
    with cb.BatchedSolver(mats, restart=20, fmt=fmt) as s:
        st = s.solve(b, x, tol=1e-8, maxit=4000)
        x2 = torch.zeros_like(b)
        s.solve(b, x2, tol=1e-8, maxit=4000)
    assert torch.equal(x, x2)
    assert (st["statuses"] == 0).all() and (st["relres"] <= 1e-8).all()
    off = 0
    for i, A in enumerate(mats):
        xi = x[off: off + A.n].cpu().numpy()
        off += A.n
        with cb.Solver.from_csr(A, restart=20, fmt=fmt, precond="jacobi") as one:
            xo = torch.zeros(A.n, dtype=torch.float64, device="cuda")
            so = one.solve(torch.from_numpy(bs[i]).cuda(), xo, tol=1e-8, maxit=4000)
        assert abs(int(st["iters"][i]) - so["iters"]) <= max(1, 0.02 * so["iters"])
        # both residuals are below 1e-8 ||b||: the solutions differ by at most twice that times
        # ||A^-1||, here against a bound of it from the smallest grid eigenvalue / dominance
        r = np.linalg.norm(A.to_scipy() @ (xi - xo.cpu().numpy()))
        assert r <= 2.1e-8 * np.linalg.norm(bs[i])
