"""Sums across warps and blocks keep FP64's precision: the projection of one-signed data and the
norm of a new basis vector against exactly rounded sums (math.fsum) of the same codes.

Thread chains are double-float, 2^-46 an addition at the worst; tens of thousands of them average
out to below 1e-16.  Above them at most 14 additions in FP64 (eight row groups, five blocks a lane,
a warp) round by 2^-53 each: 2^-53 sqrt(14 / 3) = 2.4e-16 rms of one-signed sums, half of it in a
norm.  4e-16 rms allows for both; sums across blocks in double-float gave 7e-16 to 1e-15.  (Codes of
64 and 32 bits carry 2^-48 per product, one-sided, and are left out; so does a row of the sparse
product with an integer format's scale, which leaves i16 out of the norms.)"""
import math

import numpy as np
import pytest

from gpu_common import need_gpu, to_dev
import workloads as W

pytestmark = pytest.mark.gpu

FORMATS = ["f32", "f16", "bf16", "i16", "e4m3"]


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("n", [50000, 1 << 20])
def test_projection_of_one_signed_data(fmt, n):
    torch, cb = need_gpu()
    ld, ncols = (n + 4095) // 4096 * 4096, 40
    g = np.random.default_rng(7)
    w = np.zeros(ld)
    w[:n] = g.random(n)
    V, err = [], []
    for _ in range(ncols):
        v = np.zeros(ld)
        v[:n] = g.random(n)
        codes, scale = cb.encode(fmt, to_dev(torch, v), 1.0)
        V.append(codes)
    h = cb.basis_dot(fmt, "df32", n, torch.stack(V), ld, np.ones(ncols), to_dev(torch, w))
    for c in range(ncols):
        ref = math.fsum((cb.decode(fmt, V[c], 1.0).cpu().numpy() * w).tolist())
        err.append((h[c] - ref) / ref)
    assert np.sqrt(np.mean(np.square(err))) <= 4e-16, err


def _new_vector_norms(cb, torch, fmt, n, profile, k=16):
    i = np.arange(n)
    A = W._from_coo(n, np.concatenate([i, i[1:], i[:-1]]), np.concatenate([i, i[:-1], i[1:]]),
                    np.concatenate([3.0 + np.sin(i), np.full(n - 1, -1.3), np.full(n - 1, -0.7)]))
    err = []
    for seed in range(3):
        b = to_dev(torch, W.random_vector(n, 20 + seed))
        with cb.Solver.from_csr(A, restart=30, fmt=fmt, profile=profile) as s:
            H = s.arnoldi(b, torch.zeros_like(b), k)
            V = torch.stack([s.basis_column(j) for j in range(k + 1)])
            for j in range(k):
                w = s.spmv(V[j].contiguous())
                for _ in range(2):
                    w = w - V[:j + 1].T @ (V[:j + 1] @ w)
                ref = math.sqrt(math.fsum(np.square(w.cpu().numpy()).tolist()))
                err.append((H[j + 1, j] - ref) / ref)
    return err


@pytest.mark.parametrize("fmt", ["f32", "f16", "bf16", "e4m3"])
@pytest.mark.parametrize("n", [40000, 900000])
def test_norm_of_the_new_vector_stepwise(fmt, n):
    torch, cb = need_gpu()
    err = _new_vector_norms(cb, torch, fmt, n, profile=True)
    assert np.sqrt(np.mean(np.square(err))) <= 4e-16, err


@pytest.mark.parametrize("fmt", ["f32", "e4m3"])
def test_norm_of_the_new_vector_single_launch(fmt):
    torch, cb = need_gpu()
    err = _new_vector_norms(cb, torch, fmt, 262144, profile=False)
    assert np.sqrt(np.mean(np.square(err))) <= 4e-16, err
