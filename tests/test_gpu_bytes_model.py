"""stats.bytes_model: an SpMV and four readings of the basis a step, three where one kernel forms
w - V h and V^T of it (the stepwise kernels, up to 112 columns)."""
import pytest

import workloads as W
from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,one_pass", [({}, 0), ({"profile": True}, 112), ({"profile": True, "ortho": "mgs"}, 0),
                                         ({"arith": "fp64"}, 0)])
def test_readings_of_the_basis(kw, one_pass):
    torch, cb = need_gpu()
    A = W.convdiff3d(24)
    b = to_dev(torch, W.random_vector(A.n, 2))
    with cb.Solver.from_csr(A, restart=120, fmt="f32", **kw) as s:
        st = s.solve(b, torch.zeros_like(b), tol=0.0, maxit=115)
    assert st["iters"] == 115
    spmv = 12.0 * A.nnz + 4.0 * (A.n + 1) + 16.0 * A.n
    want = sum(spmv + (3 if c <= one_pass else 4) * c * A.n * 4.0 for c in range(1, 116))
    assert st["bytes_model"] == pytest.approx(want, rel=1e-14)
