"""Clusters with more blocks than a system has chunks of 32 rows: the blocks without rows take no
part in the sparse product.  Each used to add the last, partial chunk's rows to omega = ||A v||
once more (and to write them in front of its vector), so the breakdown test
h_{j+1,j} > eps omega is put between the true ratio and the one with those rows counted again."""
import numpy as np
import pytest

import workloads as W
from gpu_common import need_gpu

pytestmark = pytest.mark.gpu

M = 3


def _heavy_tail(n, share):
    """Five entries per row; the rows after the last whole chunk of 32 outweigh all others."""
    g = np.random.default_rng(n)
    i = np.repeat(np.arange(n), 5)
    c = np.stack([np.arange(n)] + [(np.arange(n) * 7 + 13 * k) % n for k in range(1, 5)], 1).ravel()
    v = g.standard_normal(5 * n) + 3.0 * (np.arange(5 * n) % 5 == 0)
    A = W._from_coo(n, i, c, v * np.where(i >= n // 32 * 32, share, 1.0))
    assert A.n == n
    return A


def _ratios(A, b, empty):
    """h_{j+1,j} / omega of the first M steps, and the same with the last chunk's rows counted
    `empty` more times (FP64 Arnoldi with two Gram-Schmidt passes)."""
    V, r, first = [b / np.linalg.norm(b)], [], A.n // 32 * 32
    for _ in range(M):
        w = A.to_scipy() @ V[-1]
        om2, extra = w @ w, empty * (w[first:] @ w[first:])
        for _ in range(2):
            Q = np.stack(V, 1)
            w = w - Q @ (Q.T @ w)
        hn = np.linalg.norm(w)
        r.append((hn / np.sqrt(om2), hn / np.sqrt(om2 + extra)))
        V.append(w / hn)
    return np.array(r)


@pytest.mark.parametrize("fmt", ["f64", "f32", "i16"])
@pytest.mark.parametrize("cluster", [8, 16])
def test_blocks_without_rows_leave_omega_alone(fmt, cluster, monkeypatch):
    torch, cb = need_gpu()
    make = cb.options
    for n in (5, 33, 1089, 1331, 2197):
        chunk = (-(-n // cluster) + 31) // 32 * 32
        empty = sum(rank * chunk >= n for rank in range(cluster))
        A = _heavy_tail(n, 30.0 * n ** 0.5)
        b = W.random_vector(n, 5)
        r = _ratios(A, b, empty)
        eps = float(r[:, 0].min()) * 0.9
        if empty:
            assert r[:, 1].min() < 0.8 * eps, (n, r)   # counting the rows again would end the cycle

        def opts(**kw):
            o = make(**kw)
            o.breakdown_eps = eps
            return o

        monkeypatch.setattr(cb, "options", opts)
        with cb.BatchedSolver([A, A], restart=M, fmt=fmt, precond="none", use_graph=False) as s:
            s.schedule(cluster, 1)
            x = torch.zeros(2 * n, dtype=torch.float64, device="cuda")
            st = s.solve(torch.from_numpy(np.concatenate([b, b])).cuda(), x, tol=0.0, maxit=M)
        monkeypatch.setattr(cb, "options", make)
        # one cycle of M steps: no step was taken for a breakdown
        assert (st["iters"] == M).all() and (st["restarts"] == 1).all(), (n, cluster, st)
        assert torch.equal(x[:n], x[n:])
