"""What the framework is timed on: the calls a program makes of it, over the range of sizes,
storage formats and options it makes them with.

Each case is a dict of plain values; `prepare` builds the inputs and the handle a user's
program keeps (the solver of one matrix, the trained network's data), `run` is one call
through the public entry points, `exact` the same result from plain torch in 64 bits.

* ``solve``   restarted GMRES with a compressed basis on one matrix (the framework's main
              path): SpMV, the basis products of classical Gram-Schmidt with
              re-orthogonalisation, the store of the new vector, restarts.  x is returned.
* ``batch``   many small uneven systems in one call.  The packed x is returned.
* ``project`` one classical Gram-Schmidt pass through the basis products:
              h = V^T w, then w -= V h.  h and w are returned.
* ``multi``   H = V^T W for several vectors that share one basis (block Krylov methods).
* ``train``   optimiser steps of the learned preconditioner's network.  Weights are returned.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2009_12101_gb300 as cb

BYTES = cb.FORMAT_BYTES
ROW_PAD = cb.TILE_ROWS


# ---------------------------------------------------------------------------- matrices
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _csr(cols, vals, mask):
    """CSR (int32, int32, float64 CUDA tensors) of a candidate table: row i keeps the
    entries of cols[i], vals[i] where mask[i]; columns ascend along a row."""
    rowptr = torch.zeros(cols.shape[0] + 1, dtype=torch.int32, device=cols.device)
    rowptr[1:] = torch.cumsum(mask.sum(1), 0)
    return rowptr, cols[mask].to(torch.int32), vals[mask]


def _grid(shape):
    """Index tensors of a grid whose last axis runs fastest, the offset of a neighbour along
    each axis, and the row numbers."""
    n = math.prod(shape)
    idx = torch.arange(n, device="cuda")
    coord, stride, rest = [], [], n
    for s in shape:
        rest //= s
        coord.append(idx // rest % s)
        stride.append(rest)
    return idx, coord, stride


def _stencil(shape, low, high, diag):
    """low[a] / high[a]: the coefficient of the neighbour before / after a row along axis a
    (a number, or a value per row)."""
    idx, coord, stride = _grid(shape)
    one = torch.ones(idx.numel(), dtype=torch.float64, device="cuda")
    cols, vals, mask = [], [], []
    for a in range(len(shape)):
        cols.append(idx - stride[a]); vals.append(one * low[a]); mask.append(coord[a] > 0)
    cols.append(idx); vals.append(one * diag); mask.append(one > 0)
    for a in reversed(range(len(shape))):
        cols.append(idx + stride[a]); vals.append(one * high[a]); mask.append(coord[a] < shape[a] - 1)
    return _csr(torch.stack(cols, 1), torch.stack(vals, 1), torch.stack(mask, 1))


def _poisson2d(side, g):
    return _stencil((side, side), [-1.0] * 2, [-1.0] * 2, 4.0)


def _convdiff3d(side, g):
    """Upwind convection-diffusion, Peclet number 10, velocity (1, 0.5, 0.25) along (x, y, z)."""
    h, beta = 1.0 / (side + 1), (2.5, 5.0, 10.0)              # z, y, x
    return _stencil((side,) * 3, [-1.0 - h * b for b in beta], [-1.0] * 3, 6.0 + h * sum(beta))


def _diffusion3d(side, g):
    """Cell-centred diffusion, lognormal(0, 1) cell coefficients, harmonic face means."""
    shape = (side,) * 3
    kap = torch.exp(torch.randn(shape, dtype=torch.float64, device="cuda", generator=g))
    low, high, diag = [], [], torch.zeros_like(kap)
    for a in range(3):
        prev, nxt = torch.roll(kap, 1, a), torch.roll(kap, -1, a)
        lo, hi = 2 * kap * prev / (kap + prev), 2 * kap * nxt / (kap + nxt)
        lo.select(a, 0).copy_(2 * kap.select(a, 0))
        hi.select(a, side - 1).copy_(2 * kap.select(a, side - 1))
        diag += lo + hi
        low.append(-lo.reshape(-1)); high.append(-hi.reshape(-1))
    return _stencil(shape, low, high, diag.reshape(-1))


def _random27(n, g):
    """A band of nine and 18 random columns per row, N(0, 1) off the diagonal, diagonal 1.1
    times the row's absolute sum."""
    i = torch.arange(n, device="cuda")
    lo = (i - 4).clamp(0, n - 9)
    far = torch.randint(0, n - 9, (n, 18), device="cuda", generator=g)
    far = torch.where(far >= lo[:, None], far + 9, far)
    cols = torch.sort(torch.cat([lo[:, None] + torch.arange(9, device="cuda"), far], 1), 1).values
    vals = torch.randn(n, 27, dtype=torch.float64, device="cuda", generator=g)
    on = cols == i[:, None]
    vals = torch.where(on, 1.1 * vals.abs().masked_fill(on, 0.0).sum(1, keepdim=True), vals)
    return _csr(cols, vals, torch.ones_like(on))


def _laplacian(shape, g):
    """Weighted graph Laplacian of a grid, lognormal(0, 0.5) conductances, Dirichlet edges."""
    n, low, high = math.prod(shape), [], []
    diag = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for a in range(len(shape)):
        ext = list(shape)
        ext[a] += 1                                            # the edges between rows and at both walls
        c = torch.exp(0.5 * torch.randn(ext, dtype=torch.float64, device="cuda", generator=g))
        lo, hi = c.narrow(a, 0, shape[a]), c.narrow(a, 1, shape[a])
        diag += lo + hi
        low.append(-lo.reshape(n)); high.append(-hi.reshape(n))
    return _stencil(shape, low, high, diag.reshape(n))


PROBLEMS = {"poisson2d": _poisson2d, "convdiff3d": _convdiff3d, "diffusion3d": _diffusion3d, "random27": _random27}


def _rows(case):
    return case["side"] ** {"poisson2d": 2, "random27": 1}.get(case["problem"], 3)


def _nnz(case):
    s = case["side"]
    return {"poisson2d": 5 * s * s - 4 * s, "random27": 27 * s}.get(case["problem"], 7 * s ** 3 - 6 * s * s)


def _matvec(A):
    rowptr, col, val = A
    n = rowptr.numel() - 1
    M = torch.sparse_csr_tensor(rowptr.long(), col.long(), val, size=(n, n))
    return lambda x: torch.mv(M, x)


def _uniform(n, g):
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * 2 - 1


def _system(case, seed):
    g = _gen(seed)
    A = PROBLEMS[case["problem"]](case["side"], g)
    return A, _matvec(A)(_uniform(_rows(case), g)), g


def _batch_sizes(case):
    """The grids of a batch: log-uniform rows, 2D or 3D."""
    r, shapes = random.Random(case["sizes"]), []
    for _ in range(case["systems"]):
        n = math.exp(r.uniform(math.log(case["nmin"]), math.log(case["nmax"])))
        d = r.choice((2, 3))
        shapes.append((max(2, round(n ** (1.0 / d))),) * d)
    return shapes


class _Host:
    """One system of a batch as the host arrays a user's program assembles."""

    def __init__(self, A):
        self.rowptr, self.col, self.val = (t.cpu().numpy() for t in A)


def _batch_system(case, seed):
    g = _gen(seed)
    mats = [_laplacian(s, g) for s in _batch_sizes(case)]
    return mats, [_matvec(A)(_uniform(A[0].numel() - 1, g)) for A in mats]


# ------------------------------------------------------------------------------- bases
def _basis(case, g):
    """Codes and scales of `cols` random unit columns, padded rows zero."""
    n, cols, fmt = case["n"], case["cols"], case["fmt"]
    ld = -(-n // ROW_PAD) * ROW_PAD
    v = torch.zeros(cols, ld, dtype=torch.float32, device="cuda")
    v[:, :n] = torch.randn(cols, n, device="cuda", generator=g) / math.sqrt(n)
    top = v.abs().amax(1, keepdim=True).double()
    scale = np.ones(cols)
    if fmt in ("f64", "f32"):
        V = v.double() if fmt == "f64" else v
    elif fmt == "f16":
        V = v.half()
    elif fmt in ("bf16", "e4m3"):                              # a power of two brings the column to the format's top
        s = torch.exp2(torch.ceil(torch.log2(top / (1.0 if fmt == "bf16" else 448.0))))
        scale = s.reshape(-1).cpu().numpy()
        V = (v / s.float()).to(torch.bfloat16 if fmt == "bf16" else torch.float8_e4m3fn)
    else:                                                      # fixed point: the column's largest entry is the largest code
        s = top / (2147483647.0 if fmt == "i32" else 32767.0)
        scale = s.reshape(-1).cpu().numpy()
        V = torch.empty(cols, ld, dtype=torch.int32 if fmt == "i32" else torch.int16, device="cuda")
        for c in range(cols):
            V[c] = torch.round(v[c].double() / s[c]).to(V.dtype)
    return V.contiguous(), ld, scale


def _decoded(V, scale, n):
    for c in range(V.shape[0]):
        yield V[c, :n].double() * float(scale[c])


# ------------------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest solve: launches and latency count
        dict(name="solve_poisson64_f64", op="solve", problem="poisson2d", side=64, fmt="f64", restart=100,
             precond="none", tol=1e-10, maxit=20000, steps=255),
        # a small engineering grid, odd size, 16-bit basis; the restarts recover what the basis
        # loses, down to a residual near the limit of 64 bits
        dict(name="solve_convdiff31_f16", op="solve", problem="convdiff3d", side=31, fmt="f16", restart=50,
             precond="jacobi", tol=1e-12, maxit=20000, steps=170),
        # an ordinary heterogeneous problem
        dict(name="solve_diffusion64_f32", op="solve", problem="diffusion3d", side=64, fmt="f32", restart=100,
             precond="jacobi", tol=1e-10, maxit=20000, steps=320),
        # the uncompressed basis
        dict(name="solve_convdiff96_f64", op="solve", problem="convdiff3d", side=96, fmt="f64", restart=100,
             precond="none", tol=1e-10, maxit=20000, steps=385),
        # fixed-point codes, block-Jacobi, odd size
        dict(name="solve_convdiff101_i16", op="solve", problem="convdiff3d", side=101, fmt="i16", restart=100,
             precond="bj4", tol=1e-12, maxit=20000, steps=370),
        # the headline solve
        dict(name="solve_convdiff128_f32", op="solve", problem="convdiff3d", side=128, fmt="f32", restart=100,
             precond="none", tol=1e-10, maxit=20000, steps=514),
        # wide rows, quick convergence, 16-bit basis with scales
        dict(name="solve_random27_bf16", op="solve", problem="random27", side=1 << 20, fmt="bf16", restart=100,
             precond="none", tol=1e-10, maxit=20000, steps=54),
        # many small systems at once, over a restart
        dict(name="batch96_f32", op="batch", systems=96, sizes=4, nmin=1024, nmax=65536, fmt="f32", restart=30,
             tol=1e-8, maxit=40),
        # one projection against a long basis
        dict(name="project_e4m3_200", op="project", fmt="e4m3", n=1 << 20, cols=200),
        # several right-hand sides: half-precision codes, and single-precision ones at odd sizes
        dict(name="multi_f16_k8", op="multi", fmt="f16", n=1 << 21, cols=100, k=8),
        dict(name="multi_f32_k5", op="multi", fmt="f32", n=999983, cols=67, k=5),
        # training of the learned preconditioner
        dict(name="train_diffusion64", op="train", side=64, steps=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("solve", "solve", "solve", "solve", "batch", "project", "multi", "train"))
    fmt = rng.choice(("f64", "f32", "f16", "bf16", "e4m3", "i32", "i16"))
    if op == "solve":
        # to convergence, as a program runs it; an 8-bit basis is for the quickly converging
        # matrices (elsewhere it takes many restarts)
        problem = "random27" if fmt == "e4m3" else rng.choice(("poisson2d", "convdiff3d", "convdiff3d", "diffusion3d", "random27"))
        lo, hi = {"poisson2d": (32, 96), "convdiff3d": (16, 101), "diffusion3d": (16, 64), "random27": (4096, 1 << 20)}[problem]
        side = _log(rng, lo, hi)
        precond = "none" if problem == "random27" else rng.choice(("none", "jacobi", "bj4"))
        steps = {"poisson2d": 5 * side, "convdiff3d": 4 * side, "diffusion3d": 6 * side}.get(problem, 60)
        return dict(op="solve", problem=problem, side=side, fmt=fmt, restart=rng.choice((50, 100, 150)), precond=precond,
                    tol=1e-10 if BYTES[fmt] > 2 else 1e-12, maxit=20000, steps=steps)
    if op == "batch":
        return dict(op="batch", systems=rng.randint(24, 128), sizes=rng.randint(1, 10 ** 6), nmin=1024,
                    nmax=_log(rng, 4096, 65536), fmt=rng.choice(("f64", "f32", "f16")), restart=rng.choice((20, 30, 40)),
                    tol=1e-8, maxit=rng.randint(20, 40))
    if op == "project":
        return dict(op="project", fmt=fmt, n=_log(rng, 4096, 1 << 20), cols=rng.randint(1, 200))
    if op == "multi":
        return dict(op="multi", fmt=rng.choice(("f16", "f16", fmt)), n=_log(rng, 16384, 1 << 20), cols=rng.randint(8, 120),
                    k=rng.randint(1, 16))
    return dict(op="train", side=rng.randint(16, 72), steps=rng.randint(5, 20))


# ----------------------------------------------------------------------------- measure
def prepare(case, seed):
    op = case["op"]
    if op == "solve":
        A, b, _ = _system(case, seed)
        s = cb.Solver(*A, restart=case["restart"], fmt=case["fmt"], precond=case["precond"])
        return dict(case=case, solver=s, b=b)
    if op == "batch":
        mats, bs = _batch_system(case, seed)
        s = cb.BatchedSolver([_Host(A) for A in mats], restart=case["restart"], fmt=case["fmt"], precond="jacobi")
        return dict(case=case, solver=s, b=torch.cat(bs))
    g = _gen(seed)
    if op == "project":
        V, ld, scale = _basis(case, g)
        w = torch.zeros(ld, dtype=torch.float64, device="cuda")
        w[:case["n"]] = torch.randn(case["n"], dtype=torch.float64, device="cuda", generator=g)
        return dict(case=case, V=V, ld=ld, scale=scale, w=w, out=torch.empty_like(w))
    if op == "multi":
        V, ld, scale = _basis(case, g)
        W = torch.randn(case["k"], case["n"], dtype=torch.float64, device="cuda", generator=g)
        return dict(case=case, V=V, ld=ld, scale=torch.from_numpy(scale).cuda(), W=W)
    A = _diffusion3d(case["side"], g)
    spai = cb.LearnedSpai(_Host(A), case["side"], case["side"] ** 2)
    for noise in (1.0, 0.3):                                   # errors of a start and of an early iterate
        xs = _uniform(spai.n, g)
        spai.add_pair(xs, (xs - noise * _uniform(spai.n, g)).contiguous())
    return dict(case=case, spai=spai, w0=spai.params())


def run(state):
    case = state["case"]
    op, fmt = case["op"], case.get("fmt")
    if op in ("solve", "batch"):
        x = torch.zeros_like(state["b"])
        state["solver"].solve(state["b"], x, tol=case["tol"], maxit=case["maxit"])
        return x
    if op == "project":
        w = state["out"].copy_(state["w"])
        h = cb.basis_dot(fmt, "df32", case["n"], state["V"], state["ld"], state["scale"], w)
        cb.basis_axpy(fmt, "df32", case["n"], state["V"], state["ld"], state["scale"], h, w)
        return {"h": h, "w": w}
    if op == "multi":
        return cb.basis_dot_multi(fmt, case["n"], state["V"], state["ld"], state["scale"], state["W"])
    state["spai"].set_params(state["w0"])
    state["spai"].train(case["steps"], lr=1e-3)
    return state["spai"].params()


def _solve_work(n, nnz, steps, restart, size):
    """Bytes and operations of `steps` Arnoldi steps: the matrix, and the j basis columns of
    a step three times (projection; its subtraction and the re-orthogonalisation's
    projection share a pass; the second subtraction), once more per cycle for x."""
    full, rest = divmod(steps, restart)
    cols = full * restart * (restart + 1) // 2 + rest * (rest + 1) // 2
    cycle = full * restart + rest
    return (steps * (12.0 * nnz + 4.0 * n + size * n) + (3.0 * cols + cycle) * n * size,
            2.0 * steps * nnz + (8.0 * cols + 2.0 * cycle) * n)


def work(case):
    op = case["op"]
    size = BYTES.get(case.get("fmt"), 4)
    if op == "solve":
        b, f = _solve_work(_rows(case), _nnz(case), case["steps"], case["restart"], size)
    elif op == "batch":
        b = f = 0.0
        for s in _batch_sizes(case):
            n = math.prod(s)
            db, df = _solve_work(n, n + 2 * len(s) * (n - n // s[0]), case["maxit"], case["restart"], size)
            b, f = b + db, f + df
    elif op == "project":
        n, c = case["n"], case["cols"]
        b, f = 2.0 * n * c * size + 16.0 * n, 4.0 * n * c
    elif op == "multi":
        n, c, k = case["n"], case["cols"], case["k"]
        b, f = n * c * size + 8.0 * n * k + 8.0 * c * k, 2.0 * n * c * k
    else:
        n = case["side"] ** 3
        per_row = 4.0 * (7 + 49 + 7 + 1) + 8 + 1               # features, statistics, diagonal, pattern
        b, f = case["steps"] * n * per_row, case["steps"] * n * 6.0 * (7 * 64 + 64 * 64 + 64 * 7)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------- exact
def _gmres(mv, precond, b, restart, tol, maxit):
    """GMRES(m) in 64 bits, right-preconditioned, classical Gram-Schmidt twice."""
    n, x, left = b.numel(), torch.zeros_like(b), maxit
    target = tol * float(b.norm())
    V = torch.empty(restart + 1, n, dtype=torch.float64, device=b.device)
    while True:
        r = b - mv(x)
        beta = float(r.norm())
        if not beta > target or left <= 0:
            return x
        V[0] = r / beta
        H, g, k = np.zeros((restart + 1, restart)), np.zeros(restart + 1), 0
        cs, sn = np.zeros(restart), np.zeros(restart)
        g[0] = beta
        for j in range(min(restart, left)):
            w = mv(precond(V[j]))
            h = V[: j + 1] @ w
            w -= h @ V[: j + 1]
            u = V[: j + 1] @ w
            w -= u @ V[: j + 1]
            hn = w.norm()
            V[j + 1] = w / hn
            H[: j + 2, j] = torch.cat([h + u, hn[None]]).cpu().numpy()
            for i in range(j):
                H[i, j], H[i + 1, j] = cs[i] * H[i, j] + sn[i] * H[i + 1, j], -sn[i] * H[i, j] + cs[i] * H[i + 1, j]
            rr = math.hypot(H[j, j], H[j + 1, j])
            cs[j], sn[j] = H[j, j] / rr, H[j + 1, j] / rr
            H[j, j], H[j + 1, j] = rr, 0.0
            g[j], g[j + 1] = cs[j] * g[j], -sn[j] * g[j]
            k = j + 1
            if abs(g[k]) <= target:
                break
        left -= k
        y = np.linalg.solve(H[:k, :k], g[:k])
        x = x + precond(torch.from_numpy(y).to(b.device) @ V[:k])


def _preconditioner(A, kind):
    rowptr, col, val = A
    n = rowptr.numel() - 1
    if kind == "none":
        return lambda v: v
    row = torch.repeat_interleave(torch.arange(n, device=val.device), rowptr[1:] - rowptr[:-1])
    if kind == "jacobi":
        d = torch.ones(n, dtype=torch.float64, device=val.device)
        on = row == col
        d[row[on]] = val[on]
        return lambda v: v / d
    nb = -(-n // 4)                                            # diagonal blocks of four rows
    D = torch.eye(4, dtype=torch.float64, device=val.device).repeat(nb, 1, 1)
    on = row // 4 == col // 4
    D[row[on] // 4, row[on] % 4, col[on] % 4] = val[on]
    inv = torch.linalg.inv(D)

    def apply(v):
        t = torch.zeros(4 * nb, dtype=torch.float64, device=v.device)
        t[:n] = v
        return torch.bmm(inv, t.view(nb, 4, 1)).reshape(-1)[:n]

    return apply


def exact(case, seed):
    op = case["op"]
    if op == "solve":
        A, b, _ = _system(case, seed)
        return _gmres(_matvec(A), _preconditioner(A, case["precond"]), b, case["restart"], case["tol"], case["maxit"])
    if op == "batch":
        mats, bs = _batch_system(case, seed)
        return torch.cat([_gmres(_matvec(A), _preconditioner(A, "jacobi"), b, case["restart"], case["tol"], case["maxit"])
                          for A, b in zip(mats, bs)])
    g = _gen(seed)
    if op == "project":
        V, ld, scale = _basis(case, g)
        n = case["n"]
        w = torch.zeros(ld, dtype=torch.float64, device="cuda")
        w[:n] = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
        h = torch.stack([(v * w[:n]).sum() for v in _decoded(V, scale, n)])
        for v, c in zip(_decoded(V, scale, n), h):
            w[:n] -= c * v
        return {"h": h.cpu().numpy(), "w": w}
    if op == "multi":
        V, ld, scale = _basis(case, g)
        W = torch.randn(case["k"], case["n"], dtype=torch.float64, device="cuda", generator=g)
        return torch.stack([(W * v).sum(1) for v in _decoded(V, scale, case["n"])])
    return None                                                # the weights after training: the path's own 16-bit operands
