"""Performance cases of the ROR-BK library: what a user's program asks of it.

A case is a dict of plain values.  ``prepare`` makes the inputs and the handle
that a program holds before the call, ``run`` is one pass through the public
Python entry points, ``work`` the bytes and operations the path cannot do
without, and ``exact`` the same result in 64 bits from plain torch.

Kinds of case:

* ``solve``          -- one right-hand side: ``iters`` iterations of Algorithm 1
                        from x = 0 or, with ``warm`` > 0, a solve resumed from
                        the iterate after ``warm`` iterations (start_iter);
                        FP64, or the mixed-precision form.
* ``multi``          -- a block of ``nr`` right-hand sides of one system.
* ``batch``          -- ``count`` systems of uneven size, each with a block of
                        ``nr`` right-hand sides, in one graph launch.
* ``residual``       -- one residual r = b - A x and ||r||^2 (a host-driven
                        outer method, or a check of a returned solution).
* ``residual_multi`` -- the residual of a block of columns.
* ``refresh``        -- new values of A in a handle that is kept
                        (update_values), then the proposal and the residual.
* ``train``          -- one training step through the differentiable solve:
                        forward, backward, gradients of the values and of b.

Matrices: ``laplace`` (row-scaled 5-point Laplacian on a grid), ``powerlaw``
(square CSR, power-law row lengths, diagonal shift, row scales over decades,
FP32-stored values) and ``usv`` (dense, U diag(s) V^T with a geometric
spectrum).
"""
import math

import numpy as np
import torch

from paper_2510_02156_gb300 import autograd as AG
from paper_2510_02156_gb300 import binding as B

SEED = 1          # the solver's Philox key


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the small Laplacian: launches and latency only
        {"name": "laplace_2025_fp64", "kind": "solve", "matrix": "laplace", "m": 2025, "n": 2025,
         "blocks": 32, "lam": 1e-6, "precision": "fp64", "warm": 0, "iters": 200},
        # a small sparse system in blocks of 256 rows: most rows of the dynamic block share columns
        {"name": "sparse_16384_fp64", "kind": "solve", "matrix": "powerlaw", "m": 16384, "n": 16384,
         "blocks": 64, "dmax": 200, "decades": 4.0, "lam": 1e-8, "precision": "fp64", "warm": 0, "iters": 50},
        # a mid-size sparse system in the plain method, in the middle of its solve
        {"name": "sparse_262144_fp64", "kind": "solve", "matrix": "powerlaw", "m": 262144, "n": 262144,
         "blocks": 1024, "dmax": 200, "decades": 4.0, "lam": 1e-8, "precision": "fp64", "warm": 300,
         "iters": 100},
        # the benchmark system in the mixed form, in the middle of its solve
        {"name": "sparse_1048576_mixed", "kind": "solve", "matrix": "powerlaw", "m": 1048576,
         "n": 1048576, "blocks": 4096, "dmax": 200, "decades": 4.0, "lam": 1e-8, "precision": "mixed",
         "warm": 400, "iters": 200},
        # 16 right-hand sides of a system of the batched workload's size
        {"name": "multi16_100003_mixed", "kind": "multi", "matrix": "powerlaw", "m": 100003, "n": 100003,
         "blocks": 390, "dmax": 50, "decades": 4.0, "lam": 1e-8, "precision": "mixed", "nr": 16,
         "warm": 0, "iters": 60},
        # uneven systems with 16 right-hand sides each in one launch
        {"name": "batch_10x16_mixed", "kind": "batch", "count": 10, "nmin": 5000, "nmax": 200000,
         "dmax": 50, "decades": 4.0, "lam": 1e-8, "precision": "mixed", "nr": 16, "iters": 30},
        # dense least squares, strongly over-determined, mixed form (tensor-core Gram)
        {"name": "dense_200000x2048_mixed", "kind": "solve", "matrix": "usv", "m": 200000, "n": 2048,
         "blocks": 781, "smin": 1e-8, "lam": 2.56e-4, "precision": "mixed", "warm": 0, "iters": 30},
        # the same form in the plain method at an eighth of the rows
        {"name": "dense_25600x2048_fp64", "kind": "solve", "matrix": "usv", "m": 25600, "n": 2048,
         "blocks": 100, "smin": 1e-8, "lam": 2.56e-4, "precision": "fp64", "warm": 0, "iters": 30},
        # dense under-determined: the minimum-norm member of the batched workload
        {"name": "dense_2048x100000_mixed", "kind": "solve", "matrix": "usv", "m": 2048, "n": 100000,
         "blocks": 8, "smin": 0.1, "lam": 1e-10, "precision": "mixed", "warm": 0, "iters": 6},
        # one FP64 residual over FP32-stored values
        {"name": "residual_1048576", "kind": "residual", "matrix": "powerlaw", "m": 1048576, "n": 1048576,
         "blocks": 4096, "dmax": 200, "decades": 4.0, "lam": 1e-8},
        # new values in a kept handle (every forward of a training loop)
        {"name": "refresh_262144_fp64", "kind": "refresh", "matrix": "powerlaw", "m": 262144, "n": 262144,
         "blocks": 1024, "dmax": 200, "decades": 4.0, "lam": 1e-8, "precision": "fp64"},
        # forward and backward of a small differentiable solve
        {"name": "train_2025", "kind": "train", "matrix": "powerlaw", "m": 2025, "n": 2025, "blocks": 32,
         "dmax": 50, "decades": 1.0, "lam": 1e-6, "precision": "fp64", "tol": 1e-10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "dense", "dense", "multi", "batch", "residual", "residual_multi",
                       "refresh", "train"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "dense":
        if rng.random() < 0.7:        # over-determined
            m, n = _log(rng, 2000, 100000), _log(rng, 100, 2048)
            blocks, smin, lam = max(2, m // 256), 1e-8, 2.56e-4
        else:                         # under-determined
            m, n = _log(rng, 500, 2048), _log(rng, 3000, 50000)
            blocks, smin, lam = max(2, m // 256), 0.1, 1e-10
        return {"kind": "solve", "matrix": "usv", "m": m, "n": n, "blocks": blocks, "smin": smin,
                "lam": lam, "precision": prec, "warm": 0, "iters": rng.randint(4, 20)}
    if kind == "train":
        n = _log(rng, 300, 2000)
        return {"kind": "train", "matrix": "powerlaw", "m": n, "n": n, "blocks": max(2, n // 64),
                "dmax": 50, "decades": 1.0, "lam": 1e-6, "precision": "fp64", "tol": 1e-10}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 8), "nmin": 5000, "nmax": _log(rng, 20000, 200000),
                "dmax": 50, "decades": 4.0, "lam": 1e-8, "precision": "mixed",
                "nr": rng.choice([2, 4, 8, 16]), "iters": rng.randint(10, 30)}
    n = _log(rng, 2000, 1000000)
    c = {"kind": kind, "matrix": "powerlaw", "m": n, "n": n, "blocks": max(4, n // 256),
         "dmax": rng.choice([50, 200]), "decades": 4.0, "lam": 1e-8, "precision": prec}
    if kind == "multi":
        c.update(nr=rng.choice([2, 4, 8, 16, 32]), warm=0, iters=rng.randint(10, 50))
    elif kind == "residual":
        del c["precision"]
    elif kind == "residual_multi":
        del c["precision"]
        c["nr"] = rng.choice([2, 4, 8, 16, 32])
    elif kind == "solve":
        if rng.random() < 0.3:
            g = _log(rng, 20, 400)
            c = {"kind": "solve", "matrix": "laplace", "m": g * g, "n": g * g, "blocks": max(4, g * g // 100),
                 "lam": 1e-6, "precision": prec}
        # small systems couple more of the dynamic block's rows: an iteration costs more
        c.update(warm=rng.choice([0, 200]), iters=rng.randint(30, 200) if c["n"] > 60000 else rng.randint(10, 40))
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _spmv(rp, ci, vals, x):
    """A x in FP64 (each row one reduction; the same on every run)."""
    return torch.segment_reduce(vals.double() * x[ci.long()], "sum", offsets=rp.long(), initial=0.0)


def _laplace(g, gen):
    """5-point Laplacian on a g x g grid, rows scaled by 10**U(-3, 0)."""
    n = g * g
    r = torch.arange(n, device="cuda")
    i, j = r // g, r % g
    scale = 10.0 ** (-3.0 * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64))
    keys, vals = [], []
    for di, dj, v in ((-1, 0, -1.0), (0, -1, -1.0), (0, 0, 4.0), (0, 1, -1.0), (1, 0, -1.0)):
        ok = (i + di >= 0) & (i + di < g) & (j + dj >= 0) & (j + dj < g)
        rr = r[ok]
        keys.append(rr * n + rr + di * g + dj)
        vals.append(v * scale[ok])
    key, order = torch.sort(torch.cat(keys))
    return _csr(key, torch.cat(vals)[order], n)


def _csr(key, vals, n):
    rows = key // n
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return rp.int(), (key % n).int(), vals


def _powerlaw(n, dmax, decades, gen, pattern):
    """Power-law row lengths (alpha = 2.5, at least 3), values N(0,1), diagonal
    1 + sum |off-diagonal|, rows scaled by 10**U(-decades, 0), FP32.  The
    pattern comes from the generator `pattern`, the values from `gen`."""
    u = 1.0 - torch.rand(n, generator=pattern, device="cuda", dtype=torch.float64)
    d = torch.clamp(torch.round(3.0 * u ** (-1.0 / 1.5)), max=float(min(dmax, n - 1))).long()
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), d)
    cols = torch.randint(0, n, (rows.numel(),), generator=pattern, device="cuda")
    key = torch.unique(rows * n + cols)                # repeated draws of a column dropped
    key = key[key // n != key % n]
    rows = key // n
    v = torch.randn(key.numel(), generator=gen, device="cuda", dtype=torch.float64)
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    diag = 1.0 + torch.segment_reduce(v.abs(), "sum", offsets=rp, initial=0.0)
    r = torch.arange(n, device="cuda")
    key, order = torch.sort(torch.cat([key, r * n + r]))
    scale = 10.0 ** (-decades * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64))
    vals = (torch.cat([v, diag])[order] * scale[key // n]).float()
    return _csr(key, vals, n)


def _usv(m, n, smin, gen):
    """Dense U diag(s) V^T, s geometric from 1 to smin: the long factor's
    columns are scaled Gaussians (orthonormal up to sampling), the short one an
    orthogonal matrix."""
    k, big = min(m, n), max(m, n)
    s = smin ** (torch.arange(k, device="cuda", dtype=torch.float32) / max(k - 1, 1))
    Q = torch.linalg.qr(torch.randn(k, k, generator=gen, device="cuda"))[0]
    L = torch.randn(big, k, generator=gen, device="cuda") / math.sqrt(big)
    return ((L * s) @ Q.T if m >= n else (Q * s) @ L.T).double().contiguous()


def _system(case, seed, n=None):
    """{"rp", "ci", "vals"} or {"dense"}, on the device, and a generator for what follows."""
    gen = _gen(seed)
    n = n or case["n"]
    kind = case.get("matrix", "powerlaw")
    if kind == "usv":
        return {"dense": _usv(case["m"], n, case["smin"], gen)}, gen
    if kind == "laplace":
        rp, ci, v = _laplace(math.isqrt(n), gen)
    else:
        # a training loop keeps its pattern and changes the values
        pattern = _gen(n) if case["kind"] == "train" else gen
        rp, ci, v = _powerlaw(n, case["dmax"], case["decades"], gen, pattern)
    return {"rp": rp, "ci": ci, "vals": v}, gen


def _apply(A, x):
    if "dense" in A:
        return A["dense"] @ x
    if x.dim() == 1:
        return _spmv(A["rp"], A["ci"], A["vals"], x)
    return torch.stack([_spmv(A["rp"], A["ci"], A["vals"], x[:, j].contiguous()) for j in range(x.shape[1])], 1)


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float64)


def _prec(case):
    return B.PREC_MIXED if case.get("precision") == "mixed" else B.PREC_FP64


def _handle(A, m, n, blocks, lam, prec):
    if "dense" in A:
        return B.Handle(None, None, A["dense"].cpu().numpy(), m, n, blocks, lam, precision=prec)
    return B.Handle(A["rp"], A["ci"], A["vals"], m, n, blocks, lam, precision=prec)


def _b(A, gen, n, nr=0):
    return _apply(A, _randn(gen, n, nr) if nr else _randn(gen, n)).contiguous()


def prepare(case, seed):
    kind, prec = case["kind"], _prec(case)
    if kind == "batch":
        sizes = np.random.default_rng(42).integers(case["nmin"], case["nmax"] + 1, case["count"])
        hs, bs, xs = [], [], []
        for i, n in enumerate(int(v) for v in sizes):
            A, gen = _system(case, seed * 1000 + i, n)
            h = _handle(A, n, n, max(1, n // 256), case["lam"], prec)
            hs.append(h.multi(case["nr"]))
            h.close()
            bs.append(_b(A, gen, n, case["nr"]))
            xs.append(torch.zeros(n, case["nr"], dtype=torch.float64, device="cuda"))
        return {"kind": kind, "case": case, "batch": B.Batch(hs, precision=prec), "hs": hs, "b": bs, "x": xs}

    m, n = case["m"], case["n"]
    A, gen = _system(case, seed)
    if kind == "train":
        spec = AG.SolveSpec(A["rp"].cpu().numpy(), A["ci"].cpu().numpy(), m, n, case["blocks"], case["lam"],
                            tol=case["tol"], seed=SEED, precision=prec)
        v = A["vals"].double().requires_grad_(True)
        b = _b(A, gen, n).requires_grad_(True)
        return {"kind": kind, "case": case, "spec": spec, "vals": v, "b": b, "target": _randn(gen, n)}
    s = {"kind": kind, "case": case, "h": _handle(A, m, n, case["blocks"], case["lam"], prec)}
    nr = case.get("nr", 0)
    if nr:
        s["one"], s["h"] = s["h"], s["h"].multi(nr)
    s["b"] = _b(A, gen, n, nr)
    if kind == "residual":
        s["x"], s["r"] = _randn(gen, n), torch.empty(m, dtype=torch.float64, device="cuda")
    elif kind == "residual_multi":
        s["x"], s["r"] = _randn(gen, n, nr), torch.empty(m, nr, dtype=torch.float64, device="cuda")
    elif kind == "refresh":
        # the next step's values: a few percent away, as after an optimizer step
        v = A["vals"]
        s["vals"] = (v * (1.0 + 0.05 * torch.randn(v.numel(), generator=gen, device="cuda", dtype=torch.float64)).to(v.dtype))
        s["x"], s["r"] = _randn(gen, n), torch.empty(m, dtype=torch.float64, device="cuda")
    else:
        shape = (n, nr) if nr else (n,)
        s["x"] = torch.zeros(*shape, dtype=torch.float64, device="cuda")
        s["x0"] = None
        if case["warm"]:              # the iterate of the solve that is resumed
            s["x0"] = torch.zeros(n, dtype=torch.float64, device="cuda")
            s["h"].solve(s["b"], s["x0"], tol=0.0, maxit=case["warm"], seed=SEED, precision=prec)
    return s


# --------------------------------------------------------------------- run
def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "solve":
        res = s["h"].solve(s["b"], s["x"], x0=s["x0"], tol=0.0, maxit=case["iters"], seed=SEED,
                           start_iter=case["warm"], precision=_prec(case))
        return {"x": s["x"], "rrn": res.rrn, "iters": int(res.iters)}
    if kind == "multi":
        res = s["h"].solve_multi(s["b"], s["x"], tol=0.0, maxit=case["iters"], seed=SEED, precision=_prec(case))
        return {"x": s["x"], "rrn": np.array([r.rrn for r in res], dtype=np.float32),
                "iters": np.array([r.iters for r in res])}
    if kind == "batch":
        _, res = s["batch"].solve(s["b"], s["x"], tol=0.0, maxit=case["iters"], seed=SEED)
        return {"x": s["x"], "iters": np.array([r.iters for r in res])}
    if kind == "residual":
        rr = s["h"].residual(s["b"], s["x"], s["r"])
        return {"r": s["r"], "rr": rr}
    if kind == "residual_multi":
        rr = s["h"].residual_multi(s["b"], s["x"], s["r"])
        return {"r": s["r"], "rr": rr}
    if kind == "refresh":
        s["h"].update_values(s["vals"])
        cdf, rowsum = s["h"].proposal()
        rr = s["h"].residual(s["b"], s["x"], s["r"])
        return {"cdf": cdf, "rowsum": rowsum, "r": s["r"], "rr": rr}
    v, b = s["vals"], s["b"]
    v.grad = b.grad = None
    x = AG.RorbkSolve.apply(v, b, s["spec"])
    loss = 0.5 * (x - s["target"]).square().sum()
    loss.backward()
    return {"x": x.detach(), "gv": v.grad, "gb": b.grad}


# -------------------------------------------------------------------- work
def _nnz(case, n):
    """Stored entries, on average over the seeds."""
    if case.get("matrix") == "usv":
        return float(case["m"]) * n
    if case.get("matrix") == "laplace":
        return 5.0 * n - 4.0 * math.sqrt(n)
    # E[min(dmax, 3 U^(-2/3))] + 1: integral of the truncated Pareto tail
    d, a = float(min(case["dmax"], n - 1)), 1.5
    p = (3.0 / d) ** a
    return n * (a / (a - 1.0) * (3.0 - d * p) + d * p + 1.0)


def work(case):
    """One iteration reads A once (the residual) and the vectors; a value is 4
    bytes where it is stored or used in FP32, 8 otherwise, an index 4 bytes."""
    kind = case["kind"]
    if kind == "batch":
        n = 0.5 * (case["nmin"] + case["nmax"])
        z, nr, it = _nnz(case, n), case["nr"], case["iters"]
        return {"bytes": case["count"] * it * (8.0 * z + nr * 4.0 * 3 * n),
                "flops": case["count"] * it * nr * 2.0 * z}
    m, n = case["m"], case["n"]
    dense = case["matrix"] == "usv"
    mixed = case.get("precision") == "mixed"
    z = _nnz(case, n)
    vec = 4.0 if mixed and kind in ("solve", "multi") else 8.0
    if dense:
        entry = 4.0 if mixed else 8.0
    else:
        entry = 4.0 + (8.0 if case["matrix"] == "laplace" and not mixed else 4.0)
    if kind == "residual":
        return {"bytes": entry * z + vec * (n + 2 * m), "flops": 2.0 * z}
    if kind == "residual_multi":
        return {"bytes": entry * z + case["nr"] * vec * (n + 2 * m), "flops": 2.0 * z * case["nr"]}
    if kind == "refresh":
        # values in, every copy of A and the block operators out, one residual
        return {"bytes": 4.0 * z * 4 + entry * z + vec * (n + 2 * m), "flops": 6.0 * z}
    if kind == "train":
        # some hundred iterations each way on a system that stays on the chip
        return {"bytes": 100 * (entry * z + vec * 3 * n) * 2, "flops": 100 * 4.0 * z}
    nr, it = case.get("nr", 1), case["iters"]
    rows = m // case["blocks"]
    flops = nr * 2.0 * z
    if dense:      # three sampled blocks, the dynamic block's Gram and factor
        flops += 3 * (4.0 * rows * n + 2.0 * rows * rows) + rows * rows * n + rows ** 3 / 3.0 + 2.0 * rows * n
    return {"bytes": it * (entry * z + nr * vec * (n + 2 * m)), "flops": it * flops}


# ------------------------------------------------------------------- exact
_M64 = (1 << 64) - 1


def _philox(it, draw_, key0, key1):
    """First word of Philox4x64-10 for counter (it, draw, 0, 0)."""
    c = [it & _M64, draw_, 0, 0]
    k = [key0, key1]
    for rnd in range(10):
        p0, p1 = c[0] * 0xD2E7470EE14C6C93, c[2] * 0xCA5A826395121157
        c = [(p1 >> 64) ^ c[1] ^ k[0], p1 & _M64, (p0 >> 64) ^ c[3] ^ k[1], p0 & _M64]
        k = [(k[0] + 0x9E3779B97F4A7C15) & _M64, (k[1] + 0xBB67AE8584CAA73B) & _M64]
    return c[0]


def _offsets(m, k):
    q, rem = divmod(m, k)
    return [t * q + min(t, rem) for t in range(k + 1)]


def _proposal(A, m, n, k):
    """cdf and C's row sums."""
    off = torch.tensor(_offsets(m, k), device="cuda")
    if "dense" in A:
        Z = torch.stack([A["dense"][int(off[t]):int(off[t + 1])].sum(0) for t in range(k)])
    else:
        rows = torch.repeat_interleave(torch.arange(m, device="cuda"), (A["rp"][1:] - A["rp"][:-1]).long())
        blk = torch.searchsorted(off, rows, right=True) - 1
        Z = torch.zeros(k, n, dtype=torch.float64, device="cuda")
        Z.index_put_((blk, A["ci"].long()), A["vals"].double(), accumulate=True)
    nrm = Z.norm(dim=1)
    C = (Z @ Z.T).abs()
    d = nrm[:, None] * nrm[None, :]
    C = torch.where(d > 0, C / torch.where(d > 0, d, torch.ones_like(d)), torch.zeros_like(C))
    C.fill_diagonal_(1.0)
    rowsum = C.sum(1)
    return torch.cumsum(torch.exp(-2.0 * rowsum / n), 0), rowsum


def _rows(A, idx):
    """(M, cols): rows idx as a dense matrix over their distinct columns."""
    if "dense" in A:
        return A["dense"][idx], None
    p0 = A["rp"][idx].long()
    ln = A["rp"][idx + 1].long() - p0
    local = torch.repeat_interleave(torch.arange(idx.numel(), device="cuda"), ln)
    start = torch.cumsum(ln, 0) - ln
    p = p0[local] + torch.arange(local.numel(), device="cuda") - start[local]
    cols, inv = torch.unique(A["ci"][p].long(), return_inverse=True)
    M = torch.zeros(idx.numel(), cols.numel(), dtype=torch.float64, device="cuda")
    M[local, inv] = A["vals"][p].double()
    return M, cols


def _update(A, idx, lam, r, x):
    """x += A_I^T (A_I A_I^T + lam I)^{-1} r_I (the n x n form for wide I)."""
    M, cols = _rows(A, idx)
    s, w = M.shape
    if s >= x.numel():
        d = torch.linalg.solve(M.T @ M + lam * torch.eye(w, dtype=M.dtype, device="cuda"), M.T @ r)
    else:
        d = M.T @ torch.linalg.solve(M @ M.T + lam * torch.eye(s, dtype=M.dtype, device="cuda"), r)
    if cols is None:
        x += d
    else:
        x[cols] += d


def _iterate(A, b, m, n, k, lam, iters):
    """`iters` iterations of Algorithm 1 from x = 0; (x, the last tested relative residual)."""
    off = _offsets(m, k)
    cdf = _proposal(A, m, n, k)[0].cpu().numpy()
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    bn, K, rrn = b.norm(), m // k, 0.0
    for it in range(iters):
        for d in range(3):
            u = (_philox(it, d, SEED, 0) >> 11) * 2.0 ** -53
            t = min(int(np.searchsorted(cdf, u * cdf[-1], side="right")), k - 1)
            idx = torch.arange(off[t], off[t + 1], device="cuda")
            M, cols = _rows(A, idx)
            _update(A, idx, lam, b[idx] - M @ (x if cols is None else x[cols]), x)
        r = b - _apply(A, x)
        rrn = float(r.norm() / bn)
        idx = torch.sort(torch.sort(r.abs(), descending=True, stable=True)[1][:K])[0]
        _update(A, idx, lam, r[idx], x)
    return x, rrn


def exact(case, seed):
    kind = case["kind"]
    if kind in ("multi", "batch"):
        return None
    m, n = case["m"], case["n"]
    A, gen = _system(case, seed)
    if kind == "solve":
        total = case["warm"] + case["iters"]
        heavy = total * (m * n / 2e10 if "dense" in A else 0.01 + A["vals"].numel() / 2e10)
        if heavy > 12 or (case["matrix"] != "usv" and (case["precision"] == "mixed" or case["blocks"] * n > 3e8)):
            return None
        b = _b(A, gen, n)
        x, rrn = _iterate(A, b, m, n, case["blocks"], case["lam"], total)
        return {"x": x, "rrn": rrn if case["precision"] == "fp64" else None, "iters": None}
    if kind == "train":
        D = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        rows = torch.repeat_interleave(torch.arange(m, device="cuda"), (A["rp"][1:] - A["rp"][:-1]).long())
        D[rows, A["ci"].long()] = A["vals"].double()
        b = _b(A, gen, n)
        target = _randn(gen, n)
        x = torch.linalg.solve(D, b)
        g = torch.linalg.solve(D.T, x - target)
        return {"x": x, "gv": -(g[rows] * x[A["ci"].long()]), "gb": g}
    nr = case.get("nr", 0)
    b = _b(A, gen, n, nr)
    if kind == "refresh":
        v = A["vals"]
        A["vals"] = (v * (1.0 + 0.05 * torch.randn(v.numel(), generator=gen, device="cuda", dtype=torch.float64)).to(v.dtype))
    x = _randn(gen, n, nr) if nr else _randn(gen, n)
    r = b - _apply(A, x)
    out = {"r": r, "rr": r.square().sum(0).cpu().numpy() if nr else float(r.square().sum())}
    if kind == "refresh":
        cdf = rowsum = None
        if case["blocks"] * n <= 3e8:
            cdf, rowsum = _proposal(A, m, n, case["blocks"])
        out.update(cdf=cdf, rowsum=rowsum)
    return out
