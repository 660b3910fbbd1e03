"""Adaptive basis format with rows that do not fill the columns' last tile: after a promotion the
columns' padding lies over codes of the old format, and every kernel reads whole tiles."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("profile", [False, True])      # (profiling selects the stepwise kernels)
@pytest.mark.parametrize("fmt,side,m", [("e4m3", 17, 30), ("bf16", 17, 30), ("e4m3", 33, 20), ("bf16", 21, 40),
                                        ("e4m3", 12, 15)])
def test_promotion_with_padding(fmt, side, m, profile):
    torch, cb = need_gpu()
    A = W.convdiff3d(side)
    assert A.n % 4096
    b = W.rhs_from_solution(A, W.exact_solution(A.n, 2))
    tol = 1e-10
    ro = O.gmres(A, b, m=m, fmt=O.FORMATS[fmt], tol=tol, adapt=True, maxit=5000)
    bd = to_dev(torch, b)
    with cb.Solver.from_csr(A, restart=m, fmt=fmt, adapt=True, profile=profile) as s:
        for rep in range(2):                            # (the second starts in the handle's format again)
            x = torch.zeros_like(bd)
            st = s.solve(bd, x, tol=tol, maxit=5000)
            assert st["status"] == ro["status"] == 0 and ro["promotions"] > 0
            assert st["promotions"] == ro["promotions"] and st["fmt_final"] == cb.FORMAT_NAMES[ro["fmt_final"]]
            assert abs(st["iters"] - ro["iters"]) <= max(1, 0.02 * ro["iters"]), (rep, st["iters"], ro["iters"])
        H = s.arnoldi(bd, torch.zeros_like(bd), 10)     # a fresh cycle after all of it
    ref = O.gmres(A, b, m=m, fmt=O.FORMATS[fmt], tol=1e-300, maxit=10, want_H1=True)["H1"]
    err = max(np.linalg.norm(H[: j + 2, j] - ref[: j + 2, j]) / np.linalg.norm(ref[: j + 2, j]) for j in range(10))
    assert err <= 1e-10, err
