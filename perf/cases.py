"""Workloads of the MBPCG library that are timed and compared: solves, the iterations of a solve on
their own, single products and a batch, through the package's public entry points.

A case is a matrix family with its size, a block width s, the options of the handle, and what is done:

  do = "solve"    Solver.solve(b) on the device to a tolerance: the call a user makes. The output is x.
  do = "cg"       Solver.solve with the Chronopoulos-Gear CG algorithm, stopped after `iters` iterations.
  do = "iterate"  mbpcg_run_iterations_dev: set-up and exactly `iters` iterations of Algorithm 1; the
                  outputs are the whole state (X0, X~, R, W, P, Sigma). The number of iterations of a
                  full solve depends on rounding where the system is ill-conditioned, so most cases
                  time the iteration itself, which is what a long solve consists of (few enough of
                  them that rounding has not yet grown to the size of the state).
  do = "gram"     mbpcg_k_spmm_gram: one A P product with the Gram P^T (A P), a single call on a user's
                  own device buffers.
  do = "batch"    Batch.solve: uneven systems in one graph launch, from host arrays.

The matrices are the library's own workloads (2D and 3D Poisson, variable-coefficient diffusion with
Jacobi scaling, a 27-point stencil, dense Q diag(lambda) Q^T), drawn on the GPU from the seed.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2608_07327_gb300 as mb

PRECISION = {"fp64": mb.MBPCG_FP64, "mixed": mb.MBPCG_MIXED_FP32, "tc": mb.MBPCG_FP64_TC}


def listed():
    return [
        # the smallest solve: a 64 x 64 Poisson problem, 4 copies; every kernel is a few microseconds
        # and launches, gaps and serial k x k steps are what a user waits for
        dict(name="poisson2d_64_s4", do="solve", matrix="poisson2d", m=64, s=4, precision="fp64", jacobi=False, tol=1e-8),
        # a dense system with the default options (FP64 throughout), 8 copies
        dict(name="dense_2304_s8", do="iterate", matrix="dense", n=2304, cond=4.0, s=8, precision="fp64", jacobi=False,
             implicit=False, iters=10),
        # a large sparse system in FP64: variable-coefficient diffusion on 128^3 cells, Jacobi scaling
        dict(name="diffusion3d_128_s4", do="iterate", matrix="diffusion3d", m=128, s=4, precision="fp64", jacobi=True,
             implicit=False, iters=12),
        # odd sizes and the implicit-residual option: 77^3 cells, 11 copies (padded to 16)
        dict(name="diffusion3d_77_s11_implicit", do="iterate", matrix="diffusion3d", m=77, s=11, precision="fp64",
             jacobi=True, implicit=True, iters=8),
        # the densest sparse rows: the 27-point stencil on 96^3 points, 16 copies, in FP64
        dict(name="stencil27_96_s16", do="iterate", matrix="stencil27", m=96, s=16, precision="fp64", jacobi=False,
             implicit=False, iters=8),
        # the same system solved in mixed precision (FP32 inner solves, FP64 refinement), a whole call
        dict(name="stencil27_96_s16_mixed", do="solve", matrix="stencil27", m=96, s=16, precision="mixed", jacobi=False,
             tol=1e-12),
        # the CG baseline on the large diffusion system
        dict(name="diffusion3d_128_cg", do="cg", matrix="diffusion3d", m=128, jacobi=True, iters=96),
        # the headline system: dense n = 4096, condition number 1e6, 32 copies, tensor-core product
        dict(name="dense_4096_s32_tc", do="iterate", matrix="dense", n=4096, cond=6.0, s=32, precision="tc", jacobi=False,
             implicit=False, iters=8),
        # a ragged dense system with 12 copies (padded to 16), Jacobi scaling
        dict(name="dense_1531_s12_tc", do="iterate", matrix="dense", n=1531, cond=4.0, s=12, precision="tc", jacobi=True,
             implicit=False, iters=10),
        # the CG baseline on the headline system
        dict(name="dense_4096_cg", do="cg", matrix="dense", n=4096, cond=6.0, jacobi=False, iters=48),
        # one product with its Gram on a caller's buffers: a small system, 4 copies
        dict(name="gram_poisson2d_120_s4", do="gram", matrix="poisson2d", m=120, s=4),
        # twelve uneven requests solved as one graph launch, host arrays in and out
        dict(name="batch_12", do="batch", members=12, n_lo=1000, n_hi=60000, tol=1e-8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(("solve", "iterate", "iterate", "iterate", "dense", "dense", "cg", "densecg", "gram", "batch", "mixed"))
    if do == "solve":  # small Poisson solves
        return dict(do="solve", matrix="poisson2d", m=rng.randint(48, 128), s=rng.choice((1, 2, 3, 4)), precision="fp64",
                    jacobi=rng.random() < 0.3, tol=1e-8)
    if do == "iterate":
        kind = rng.choice(("poisson3d", "diffusion3d", "stencil27", "diffusion3d"))
        s = rng.choice((1, 2, 3, 4, 6, 8, 12, 16, 23, 32))
        hi = {"poisson3d": 120, "diffusion3d": 128, "stencil27": 96}[kind]
        hi = min(hi, int((1.6e7 / s) ** (1.0 / 3.0)))  # no larger than the largest listed blocks
        return dict(do="iterate", matrix=kind, m=_log_int(rng, 24, hi), s=s, precision="fp64", jacobi=kind == "diffusion3d",
                    implicit=rng.random() < 0.25, iters=rng.randint(4, 10))
    if do == "dense":
        return dict(do="iterate", matrix="dense", n=_log_int(rng, 700, 4096), cond=rng.choice((2.0, 4.0, 6.0)),
                    s=rng.choice((4, 8, 12, 16, 20, 32)), precision=rng.choice(("tc", "tc", "fp64")),
                    jacobi=rng.random() < 0.25, implicit=False, iters=rng.randint(4, 8))
    if do == "cg":
        kind = rng.choice(("poisson3d", "diffusion3d", "stencil27"))
        hi = 96 if kind == "stencil27" else 128
        return dict(do="cg", matrix=kind, m=_log_int(rng, 24, hi), jacobi=kind == "diffusion3d", iters=rng.randint(32, 96))
    if do == "densecg":
        return dict(do="cg", matrix="dense", n=_log_int(rng, 500, 4096), cond=rng.choice((2.0, 4.0, 6.0)),
                    jacobi=rng.random() < 0.25, iters=rng.randint(24, 48))
    if do == "gram":
        kind = rng.choice(("poisson2d", "poisson3d", "stencil27"))
        m = {"poisson2d": (64, 1000), "poisson3d": (16, 96), "stencil27": (16, 64)}[kind]
        return dict(do="gram", matrix=kind, m=_log_int(rng, *m), s=rng.choice((1, 2, 4, 7, 8, 16, 32)))
    if do == "batch":
        return dict(do="batch", members=rng.randint(4, 16), n_lo=1000, n_hi=rng.randint(20000, 60000), tol=1e-8)
    return dict(do="solve", matrix=rng.choice(("stencil27", "poisson3d")), m=rng.randint(40, 80), s=rng.choice((4, 8, 16)),
                precision="mixed", jacobi=False, tol=1e-12)


# ------------------------------------------------------------------------------------ matrices


def _grid_csr(m, dim, offsets, values):
    """CSR arrays (device) of a stencil on an m^dim grid: offsets in column order, values(k, keep) the
    n values of offset k, keep its mask of neighbours inside the grid."""
    n = m ** dim
    i = torch.arange(n, device="cuda")
    x = [i // m ** (dim - 1 - a) % m for a in range(dim)]
    keep = torch.empty((n, len(offsets)), dtype=torch.bool, device="cuda")
    cols = torch.empty((n, len(offsets)), dtype=torch.int32, device="cuda")
    for k, off in enumerate(offsets):
        ok = torch.ones(n, dtype=torch.bool, device="cuda")
        flat = 0
        for a, d in enumerate(off):
            ok &= (x[a] + d >= 0) & (x[a] + d < m)
            flat += d * m ** (dim - 1 - a)
        keep[:, k] = ok
        cols[:, k] = i + flat
    vals = torch.stack([values(k, keep[:, k]) for k in range(len(offsets))], 1)
    rp = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum(keep.sum(1), 0)
    return n, rp, cols[keep], vals[keep]


def _flat(off, m):
    return sum(d * m ** (len(off) - 1 - a) for a, d in enumerate(off))


def _faces(dim):
    off = []
    for a in range(dim):
        for d in (-1, 1):
            off.append(tuple(d if b == a else 0 for b in range(dim)))
    off.append((0,) * dim)
    return sorted(off)


def _sparse(kind, m, gen):
    """(n, row_ptr, col_idx, val) on the device."""
    if kind in ("poisson2d", "poisson3d"):
        dim = 2 if kind == "poisson2d" else 3
        off = _faces(dim)
        n = m ** dim
        return _grid_csr(m, dim, off, lambda k, keep: torch.full(
            (n,), 2.0 * dim if not any(off[k]) else -1.0, dtype=torch.float64, device="cuda"))
    n = m ** 3
    if kind == "diffusion3d":  # harmonic means of 10^U[-2,2], the cell's own value at a boundary face
        kap = 10.0 ** (4.0 * torch.rand(n, generator=gen, dtype=torch.float64, device="cuda") - 2.0)
        off = _faces(3)
        diag = torch.zeros_like(kap)
        face = {}
        i = torch.arange(n, device="cuda")
        x = [i // m ** (2 - a) % m for a in range(3)]
        for o in off:
            if not any(o):
                continue
            ok = torch.ones(n, dtype=torch.bool, device="cuda")
            for a, d in enumerate(o):
                ok &= (x[a] + d >= 0) & (x[a] + d < m)
            nb = torch.where(ok, i + _flat(o, m), i)
            f = 2.0 * kap * kap[nb] / (kap + kap[nb])  # nb = i at a boundary: the cell's own value
            diag += f
            face[o] = -f
        face[(0, 0, 0)] = diag
        return _grid_csr(m, 3, off, lambda k, keep: face[off[k]])
    # 27-point: -U[0,1) per undirected edge, diagonal = sum |off-diagonal| + 1e-2
    off = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
    w = {o: torch.rand(n, generator=gen, dtype=torch.float64, device="cuda") for o in off if o > (0, 0, 0)}
    diag = torch.full((n,), 1e-2, dtype=torch.float64, device="cuda")
    order = [k for k in range(27) if any(off[k])] + [13]
    vals = {}

    def edge(o):
        if o > (0, 0, 0):
            return w[o]
        p = tuple(-d for d in o)
        return torch.roll(w[p], _flat(p, m))

    i = torch.arange(n, device="cuda")
    x = [i // m ** (2 - a) % m for a in range(3)]
    for k in order[:-1]:
        ok = torch.ones(n, dtype=torch.bool, device="cuda")
        for a, d in enumerate(off[k]):
            ok &= (x[a] + d >= 0) & (x[a] + d < m)
        e = edge(off[k])
        diag += torch.where(ok, e, torch.zeros_like(e))
        vals[k] = -e
    vals[13] = diag
    return _grid_csr(m, 3, off, lambda k, keep: vals[k])


def _dense(n, cond, gen):
    """Q diag(lambda) Q^T, lambda = 10^U[0, cond], symmetric (device, FP64)."""
    g = torch.randn((n, n), generator=gen, dtype=torch.float64, device="cuda")
    q, _ = torch.linalg.qr(g)
    lam = 10.0 ** (cond * torch.rand(n, generator=gen, dtype=torch.float64, device="cuda"))
    a = (q * lam) @ q.T
    return 0.5 * (a + a.T)


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _uniform(shape, gen):
    return 2.0 * torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda") - 1.0


def _members(case, seed):
    """The requests of a batch: (kind, m, s, seed); sizes and widths cycle so that they are uneven."""
    out = []
    for i in range(case["members"]):
        kind = ("poisson2d", "poisson3d", "diffusion3d")[i % 3]
        t = (i * 0.618034) % 1.0
        n = case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** t
        m = max(10, int(round(n ** (1.0 / (2 if kind == "poisson2d" else 3)))))
        out.append((kind, m, (1, 4, 8, 2)[(i // 2) % 4], 1000 * int(seed) + i))
    return out


def _host(csr):
    n, rp, ci, av = csr
    return SimpleNamespace(n=n, row_ptr=rp.cpu().numpy(), col_idx=ci.cpu().numpy(), val=av.cpu().numpy())


def _matrix(case, gen):
    if case["matrix"] == "dense":
        return _dense(case["n"], case["cond"], gen)
    return _sparse(case["matrix"], case["m"], gen)


def _solver(A, case, seed):
    algo = mb.MBPCG_ALGO_CG if case["do"] == "cg" else mb.MBPCG_ALGO_MBPCG
    host = SimpleNamespace(n=A.shape[0], a=A.cpu().numpy().T) if torch.is_tensor(A) else _host(A)
    return mb.Solver(host, s=case.get("s", 1), precond=mb.MBPCG_PRECOND_JACOBI if case["jacobi"] else mb.MBPCG_PRECOND_NONE,
                     algo=algo, seed=int(seed), precision=PRECISION[case.get("precision", "fp64")],
                     residual_mode=mb.MBPCG_RESIDUAL_IMPLICIT if case.get("implicit") else mb.MBPCG_RESIDUAL_EXPLICIT)


# ------------------------------------------------------------------------------------ the passes


def prepare(case, seed):
    do = case["do"]
    if do == "batch":
        solvers, bs = [], []
        for kind, m, s, sd in _members(case, seed):
            gen = _generator(sd)
            A = _sparse(kind, m, gen)
            solvers.append(_solver(A, dict(do="solve", s=s, jacobi=kind == "diffusion3d"), sd))
            bs.append(_uniform(A[0], gen).cpu().numpy())
        return dict(do=do, solvers=solvers, bs=bs, batch=mb.Batch(solvers), tol=case["tol"])
    gen = _generator(seed)
    A = _matrix(case, gen)
    n = A.shape[0] if torch.is_tensor(A) else A[0]
    if do == "gram":
        s = case["s"]
        kp = mb.mbpcg_k_padded_width(s)
        P = torch.zeros((n, kp), dtype=torch.float64, device="cuda")
        P[:, :s] = torch.randn((n, s), generator=gen, dtype=torch.float64, device="cuda") / math.sqrt(n)
        bytes_ = mb.mbpcg_k_scratch_bytes(n, s)
        return dict(do=do, n=n, s=s, A=A, P=P, AP=torch.empty_like(P),
                    G=torch.empty((s, s), dtype=torch.float64, device="cuda"),
                    scratch=torch.empty(bytes_, dtype=torch.uint8, device="cuda"), bytes=bytes_)
    b = _uniform(n, gen)
    st = dict(do=do, b=b, n=n)
    if do == "iterate":
        s = case["s"]
        st["U"] = _uniform((s, n), gen)  # row-major s x n: the column-major n x s block
        st["out"] = {k: torch.empty((s, n), dtype=torch.float64, device="cuda") for k in ("X0", "Xt", "R", "W", "P")}
        st["out"]["Sigma"] = torch.empty((s, s), dtype=torch.float64, device="cuda")
        st["iters"] = case["iters"]
    elif do == "cg":
        st["maxit"] = case["iters"]
    else:
        st["tol"] = case["tol"]
    st["solver"] = _solver(A, case, seed)
    torch.cuda.synchronize()
    return st


def run(state):
    do = state["do"]
    if do == "gram":
        _, rp, ci, av = state["A"]
        rc = mb.mbpcg_k_spmm_gram(state["n"], rp, ci, av, state["s"], state["P"], state["AP"], state["G"],
                                  state["scratch"], state["bytes"], torch.cuda.current_stream().cuda_stream)
        if rc != mb.MBPCG_OK:
            raise mb.MBPCGError(rc, "mbpcg_k_spmm_gram")
        return {"AP": state["AP"], "G": state["G"]}
    if do == "batch":
        return [x for x, _ in state["batch"].solve(state["bs"], tol=state["tol"])]
    sv = state["solver"]
    if do == "iterate":
        o = state["out"]
        rc = mb.mbpcg_run_iterations_dev(sv.h, state["b"], state["U"], state["iters"], o["X0"], o["Xt"], o["R"], o["W"],
                                         o["P"], o["Sigma"])
        if rc != mb.MBPCG_OK:
            raise mb.MBPCGError(rc, "mbpcg_run_iterations_dev")
        return o
    if do == "cg":
        x, _ = sv.solve(state["b"], tol=1e-14, maxit=state["maxit"])
    else:
        x, _ = sv.solve(state["b"], tol=state["tol"])
    return x


# ------------------------------------------------------------------------------------ floors


def _entries(case):
    if case["matrix"] == "dense":
        return case["n"], case["n"] ** 2
    m, k = case["m"], case["matrix"]
    if k == "poisson2d":
        return m ** 2, 5 * m ** 2 - 4 * m
    return (m ** 3, (3 * m - 2) ** 3) if k == "stencil27" else (m ** 3, 7 * m ** 3 - 6 * m ** 2)


def work(case):
    """Bytes: A once and every block that an iteration reads or writes once per iteration (P, A P, W, R,
    X~, V); FLOPs: the products and the upper triangles of the Grams."""
    if case["do"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for kind, m, s, _ in _members(case, 0):
            w = work(dict(do="solve", matrix=kind, m=m, s=s, precision="fp64"))
            for k in total:
                total[k] += w[k]
        return total
    n, nnz = _entries(case)
    s = case.get("s", 1)
    word = 4 if case.get("precision") == "mixed" else 8
    a_bytes = word * nnz if case["matrix"] == "dense" else (word + 4) * nnz + 4 * (n + 1)
    if case["do"] == "gram":
        return {"bytes": float(a_bytes + 16 * n * s), "flops": float(2 * nnz * s + n * s * (s + 1))}
    if "iters" in case:
        iters = case["iters"]
    elif case["matrix"] == "stencil27":
        iters = 220  # about what the solves of these families take
    else:
        iters = 2.3 * case["m"]
    if case["do"] == "cg":
        return {"bytes": float(iters * (a_bytes + 10 * 8 * n)), "flops": float(iters * (2 * nnz + 14 * n))}
    return {"bytes": float(iters * (a_bytes + 14 * word * n * s)), "flops": float(iters * (2 * nnz * s + 10 * n * s * s))}


# ------------------------------------------------------------------------------------ in 64 bits


def _operator(A, jacobi):
    """(apply, n, d): the scaled operator of the case in torch, d = 1/sqrt(diag) or None."""
    if torch.is_tensor(A):
        d = 1.0 / torch.sqrt(torch.diagonal(A)) if jacobi else None
        M = A if d is None else d[:, None] * A * d[None, :]
        return (lambda X: M @ X), A.shape[0], d
    n, rp, ci, av = A
    d = None
    if jacobi:
        rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
        diag = torch.zeros(n, dtype=torch.float64, device="cuda")
        on = rows == ci
        diag[rows[on]] = av[on]
        d = 1.0 / torch.sqrt(diag)
        av = d[rows] * av * d[ci.long()]
    M = torch.sparse_csr_tensor(rp, ci, av, size=(n, n))
    return (lambda X: M @ X), n, d


def _qr(X):
    """Q, R with a positive diagonal, by two passes of Cholesky QR."""
    r1 = torch.linalg.cholesky(X.T @ X).T
    q = torch.linalg.solve_triangular(r1, X, upper=True, left=False)
    r2 = torch.linalg.cholesky(q.T @ q).T
    return torch.linalg.solve_triangular(r2, q, upper=True, left=False), r2 @ r1


def _algorithm1(apply, b, U, d, iters):
    bs = b if d is None else d * b
    s = U.shape[1]
    AU = apply(U)
    X0 = (math.sqrt(s) * torch.linalg.norm(bs) / torch.linalg.norm(AU)) * U
    R = bs[:, None] - (X0[0, 0] / U[0, 0]) * AU
    W, Sigma = _qr(R)
    P, Xt = W.clone(), torch.zeros_like(X0)
    for _ in range(iters):
        Q = apply(P)
        Xi = torch.linalg.inv(P.T @ Q)
        T = Xi @ Sigma
        Xt = Xt + P @ T
        R = R - Q @ T
        W, zeta = _qr(W - Q @ Xi)
        Sigma = zeta @ Sigma
        P = W + P @ zeta.T
    return X0, Xt, R, W, P, Sigma


def _cg(apply, b, iters, tol=0.0):
    """Plain conjugate gradients from zero: after `iters` steps, or until the residual is below tol."""
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), r @ r
    stop = tol * tol * float(rr)
    for k in range(iters):
        q = apply(p[:, None])[:, 0]
        a = rr / (p @ q)
        x = x + a * p
        r = r - a * q
        new = r @ r
        if tol and k % 16 == 0 and float(new) < stop:
            break
        p, rr = r + (new / rr) * p, new
    return x


def _solution(A, b, jacobi):
    apply, n, d = _operator(A, jacobi)
    x = torch.zeros_like(b)
    for _ in range(2):  # one refinement step
        xs = x if d is None else x / d
        r = (b if d is None else d * b) - apply(xs[:, None])[:, 0]
        x = x + (1.0 if d is None else d) * _cg(apply, r, 6000, 1e-13)
    return x


def exact(case, seed):
    do = case["do"]
    if do == "batch":
        out = []
        for kind, m, s, sd in _members(case, seed):
            gen = _generator(sd)
            A = _sparse(kind, m, gen)
            out.append(_solution(A, _uniform(A[0], gen), kind == "diffusion3d").cpu().numpy())
        return out
    gen = _generator(seed)
    A = _matrix(case, gen)
    n = A.shape[0] if torch.is_tensor(A) else A[0]
    if do == "gram":
        s = case["s"]
        kp = 1 << (s - 1).bit_length()
        P = torch.zeros((n, kp), dtype=torch.float64, device="cuda")
        P[:, :s] = torch.randn((n, s), generator=gen, dtype=torch.float64, device="cuda") / math.sqrt(n)
        AP = _operator(A, False)[0](P)
        return {"AP": AP, "G": P[:, :s].T @ AP[:, :s]}
    b = _uniform(n, gen)
    if do == "solve":
        return _solution(A, b, case["jacobi"])
    apply, n, d = _operator(A, case["jacobi"])
    if do == "cg":
        x = _cg(apply, b if d is None else d * b, case["iters"])
        return x if d is None else d * x
    U = _uniform((case["s"], n), gen).T.contiguous()
    X0, Xt, R, W, P, Sigma = _algorithm1(apply, b, U, d, case["iters"])
    out = {"X0": X0.T, "Xt": Xt.T, "R": R.T, "W": W.T, "P": P.T}
    out = {k: v.contiguous() for k, v in out.items()}
    out["Sigma"] = Sigma.T.contiguous()  # the library writes it column by column
    return out
