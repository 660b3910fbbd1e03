"""Failure detection without a fault in the kernels whose blocks wait on one another: one block
does not arrive at a barrier, the others' waits give up after a millisecond, the solve returns
CBG_ERR_TIMEOUT, and the next solve on the handle gives the bits of an undisturbed one."""
import pytest

import workloads as W
from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu


def _check(cb, torch, A, fmt, kernel, ats, **kw):
    b = to_dev(torch, W.random_vector(A.n, 9))
    with cb.Solver.from_csr(A, restart=8, fmt=fmt, **kw) as s:
        want = torch.zeros_like(b)
        st0 = s.solve(b, want, tol=1e-9, maxit=2000)
        assert st0["status"] == 0 and st0["iters"] > 16
        for at in ats:
            s.test_withhold(kernel, at)
            with pytest.raises(cb.CbgError) as e:
                s.solve(b, torch.zeros_like(b), tol=1e-9, maxit=2000)
            assert e.value.status == -5, at
            torch.cuda.synchronize()
            x = torch.zeros_like(b)
            st = s.solve(b, x, tol=1e-9, maxit=2000)
            assert st["status"] == 0 and st["iters"] == st0["iters"] and torch.equal(x, want), at


# four barriers a step (five with a two-stage preconditioner): every one of the first three steps, and
# the last ones of a cycle of eight (32 or 40, less the one that the last step does without)
@pytest.mark.parametrize("fmt,precond,last", [("f64", "none", 31), ("f32", "bj4", 39), ("i16", "jacobi", 31)])
@pytest.mark.parametrize("side", [4, 14, 44])           # one block, resident in shared memory, all blocks
def test_single_launch_cycle(fmt, precond, last, side):
    torch, cb = need_gpu()
    A = W.convdiff3d(side)
    _check(cb, torch, A, fmt, "cycle", [*range(1, 16), last - 1, last], precond=precond)


@pytest.mark.parametrize("fmt", ["f64", "f32", "e4m3"])
def test_one_pass_kernel(fmt):
    torch, cb = need_gpu()
    _check(cb, torch, W.convdiff3d(20), fmt, "pass", [1, 2, 8, 9])


def test_withhold_needs_the_kernel():
    torch, cb = need_gpu()
    A = W.poisson2d(20)
    with cb.Solver.from_csr(A, restart=8, fmt="f32", profile=True) as s:
        with pytest.raises(cb.CbgError) as e:
            s.test_withhold("cycle")                     # profiling keeps the kernels of a step apart
        assert e.value.status == -6
    with cb.Solver.from_csr(A, restart=8, fmt="f32", ortho="mgs") as s:
        with pytest.raises(cb.CbgError) as e:
            s.test_withhold("pass")
        assert e.value.status == -6
