"""Timed workloads of the Top-K sparse eigensolver, through its public Python entry points.

A case is a dict of plain values; ``kind`` names the entry point:

* ``plan``     - ``Plan.solve``: a plan kept by the program, one complete solve per pass (the serving form of a
  solver embedded in an application: the matrix layout, work memory and CUDA graph exist already);
* ``oneshot``  - ``topk_eigs``: one call from a CSR to the eigenpairs, the layout built inside it; the CSR on the
  device, or (``host``) in pinned host memory with pinned results, as a program does whose data arrives from disk;
* ``lanczos``  - ``lanczos``: the Lanczos phase with its basis (for programs that go on from T and V themselves);
* ``spmv``     - ``spmv_noalloc``: y = M x straight from a CSR (an application's own iteration around the operator);
* ``tridiag``  - ``tridiag_eigs``: the Jacobi phase on a T the program has;
* ``serve``    - ``Server``: a burst of small solves of mixed sizes submitted together, collected as they finish.

Matrices: ``uniform`` (every row draws ``deg`` columns: road- and mesh-like row lengths), ``rmat`` (R-MAT with
(0.57, 0.19, 0.19, 0.05): power-law rows, empty rows, hubs; vertex ids permuted, ids past ``n`` dropped) and
``planted`` (uniform background plus disjoint unit cliques of sizes in a geometric progression: community
structure, what spectral clustering looks for).  Off-diagonal values are uniform(0, 1), the matrix is symmetric.
Everything is drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2201_07498_gb300 as te

RMAT = (0.57, 0.19, 0.19, 0.05)
L2_BYTES = 100e6  # working sets below this stay on chip between a solve's steps


def listed():
    return [
        # the smallest complete solve: binary64 parity size of the configurations (latency, many tiny launches)
        dict(name="plan_small_ddd", kind="plan", graph="uniform", n=10_000, deg=10, K=8, m=16, prec="ddd",
             reorth="full", order="keep", refine=False),
        # an ordinary mixed-precision solve, odd row count, power-law rows, default options
        dict(name="plan_mid_fdf", kind="plan", graph="rmat", n=200_003, deg=16, K=12, m=24, prec="fdf",
             reorth="full", order="keep", refine=False),
        # the headline size and options (2^24 rows, K = 24, m = 48, delayed sweep, rows by degree)
        dict(name="plan_large_fdf", kind="plan", graph="rmat", n=1 << 24, deg=8, K=24, m=48, prec="fdf",
             reorth="delayed", order="degree", refine=False),
        # the plain binary64 form that the mixed forms are compared with, at the precision sweep's size
        dict(name="plan_large_ddd", kind="plan", graph="rmat", n=1 << 22, deg=16, K=16, m=32, prec="ddd",
             reorth="delayed", order="degree", refine=False),
        # the same size in the mixed form with the binary64 refinement and true residuals
        dict(name="plan_refined_fdf", kind="plan", graph="rmat", n=1 << 22, deg=16, K=16, m=32, prec="fdf",
             reorth="delayed", order="degree", refine=True),
        # one call on a device CSR: FP8 values with row scales, communities, odd sizes
        dict(name="oneshot_8df", kind="oneshot", graph="planted", n=1_000_003, deg=8, K=10, m=30, prec="8df",
             reorth="delayed", order="degree", refine=False, host=False),
        # one call from pinned host memory to pinned host results (end to end over the host link)
        dict(name="oneshot_host_fdf", kind="oneshot", graph="rmat", n=1 << 20, deg=8, K=8, m=16, prec="fdf",
             reorth="delayed", order="degree", refine=False, host=True),
        # the Lanczos phase alone in binary64, classical Gram-Schmidt twice, with its basis
        dict(name="lanczos_ddd", kind="lanczos", graph="uniform", n=524_287, deg=12, m=40, prec="ddd",
             reorth="full", order="keep"),
        # y = M x on a large power-law matrix, binary32 values
        dict(name="spmv_large_fdf", kind="spmv", graph="rmat", n=1 << 22, deg=16, prec="fdf"),
        # y = M x on a small binary64 matrix (launch latency counts)
        dict(name="spmv_small_ddd", kind="spmv", graph="uniform", n=30_011, deg=10, prec="ddd"),
        # the Jacobi phase at the headline's order
        dict(name="tridiag_48", kind="tridiag", m=48),
        # a burst of the serving mix
        dict(name="serve_mix", kind="serve", count=32, mix=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plan", "plan", "plan", "oneshot", "lanczos", "spmv", "tridiag", "serve"])
    if kind == "tridiag":
        return dict(kind="tridiag", m=rng.randint(4, 64))
    if kind == "serve":
        return dict(kind="serve", count=rng.randint(4, 32), mix=rng.randint(2, 1 << 30))
    graph = rng.choice(["uniform", "rmat"])
    c = dict(kind=kind, graph=graph)
    if kind == "spmv":
        c.update(n=_log_int(rng, 4_000, 4_000_000), deg=rng.randint(4, 16), prec=rng.choice(["ddd", "fdf"]))
        return c
    big = {"plan": 3_500_000, "oneshot": 1_500_000, "lanczos": 1_500_000}[kind]
    K = rng.randint(2, 24)
    c.update(n=_log_int(rng, 4_000, big), deg=rng.randint(6, 16), K=K, m=min(48, K * rng.choice([2, 2, 3])),
             prec=rng.choice(["ddd", "fdf", "fdf", "bdf", "8df"]), reorth=rng.choice(["full", "delayed"]),
             order=rng.choice(["keep", "degree"]))
    if kind == "lanczos":
        del c["K"]
        c["prec"] = rng.choice(["ddd", "fdf"])
        return c
    c["refine"] = c["prec"] != "ddd" and rng.random() < 0.25
    if kind == "oneshot":
        c["host"] = rng.random() < 0.3
    return c


# ---------------------------------------------------------------------------
# matrices
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _edges(graph, n, deg, g):
    """`deg * n` undirected edges (i, j) before duplicates merge."""
    if graph != "rmat":
        i = torch.arange(n, device="cuda").repeat_interleave(deg)
        return i, torch.randint(0, n, (n * deg,), device="cuda", generator=g)
    scale = max(1, (n - 1).bit_length())
    E = n * deg
    i = torch.zeros(E, dtype=torch.int64, device="cuda")
    j = torch.zeros(E, dtype=torch.int64, device="cuda")
    a, b, c, _ = RMAT
    for _ in range(scale):
        u = torch.rand(E, device="cuda", generator=g)
        i = i.mul_(2).add_(u >= a + b)
        j = j.mul_(2).add_(((u >= a) & (u < a + b)) | (u >= a + b + c))
    if n != 1 << scale:
        ok = (i < n) & (j < n)
        i, j = i[ok], j[ok]
    p = torch.randperm(n, device="cuda", generator=g)
    return p[i], p[j]


def _matrix(graph, n, deg, seed):
    """(row_ptr, col, val float64) on the GPU."""
    g = _gen(seed)
    i, j = _edges(graph, n, deg, g)
    key = torch.minimum(i, j).mul_(n).add_(torch.maximum(i, j))
    key = key[i != j]
    del i, j
    key = torch.unique(key)
    w = torch.rand(key.numel(), device="cuda", generator=g, dtype=torch.float64)
    if graph == "planted":  # unit cliques on disjoint random vertices, sizes 16 * 1.25^k
        p = torch.randperm(n, device="cuda", generator=g)
        at, more = 0, []
        for k in range(24):
            s = int(round(16 * 1.25 ** k))
            if at + s > n // 4:
                break
            v = p[at:at + s].sort().values
            t = torch.triu_indices(s, s, 1, device="cuda")
            more.append(v[t[0]] * n + v[t[1]])
            at += s
        ck = torch.cat(more)
        fresh = key[~torch.isin(key, ck)]
        w = torch.cat([w[:fresh.numel()], torch.ones(ck.numel(), device="cuda", dtype=torch.float64)])
        key = torch.cat([fresh, ck])
    lo, hi = key // n, key % n
    key = torch.cat([lo * n + hi, hi * n + lo])
    del lo, hi
    key, at = torch.sort(key)
    val = torch.cat([w, w])[at]
    del w, at
    row = key // n
    col = (key - row * n).to(torch.int32)
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.bincount(row, minlength=n).cumsum(0)
    return rp, col, val


def _csr(case, seed, host=False):
    rp, col, val = _matrix(case["graph"], case["n"], case["deg"], seed)
    if case["prec"] == "fdf" and not case.get("refine"):
        val = val.float()  # binary32 data; every other form takes the binary64 values
    if host:
        rp, col, val = (t.cpu().pin_memory() for t in (rp, col, val))
    return te.CSR(case["n"], rp, col, val)


def _start(n, seed):
    return torch.rand(n, device="cuda", generator=_gen(seed ^ 0x5EED), dtype=torch.float64) * 2 - 1


def _tridiag(m, seed):
    """A T as the Lanczos phase leaves it: one leading value, then a band of nearly constant width."""
    g = _gen(seed)
    a = 0.3 * torch.randn(m, device="cuda", generator=g, dtype=torch.float64)
    a[1 % m] += 9.0
    b = 2.0 + 0.4 * torch.rand(m + 1, device="cuda", generator=g, dtype=torch.float64)
    b[0] = 0.0
    return a, b


def _requests(case):
    """The serving mix: n log-uniform in 2^10..2^18, mean degree 4..64, K in {4, 8, 16}, m = 2K, binary32 or bfloat16
    values, uniform or R-MAT.  The case says which sizes, prepare()'s seed which matrices."""
    r = np.random.RandomState(case["mix"])
    out = []
    for _ in range(case["count"]):
        n = int(2 ** r.uniform(10, 18))
        deg = int(r.randint(4, 65)) // 2
        K = int(r.choice([4, 8, 16]))
        out.append(dict(graph=str(r.choice(["uniform", "rmat"])), n=n, deg=deg, K=K, m=2 * K,
                        prec=str(r.choice(["fdf", "bdf"]))))
    return out


# ---------------------------------------------------------------------------
# the interface
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "tridiag":
        a, b = _tridiag(case["m"], seed)
        return dict(kind=kind, alpha=a, beta=b)
    if kind == "serve":
        srv = te.Server(max_slots=64, max_krylov_steps=32, budget=4 << 30)
        reqs = []
        for i, q in enumerate(_requests(case)):
            csr = _csr(q, seed * 64 + i)
            A = _HostCSR(q["n"], *(t.cpu().numpy() for t in (csr.row_ptr, csr.col, csr.val)))
            out = torch.empty(q["n"] * q["K"], dtype=torch.float64, pin_memory=True)
            reqs.append((A, q["K"], q["m"], q["prec"], seed * 64 + i, out))
        return dict(kind=kind, srv=srv, reqs=reqs)
    if kind == "spmv":
        csr = _csr(case, seed)
        x = _start(case["n"], seed)
        x = x if case["prec"] == "ddd" else x.float()
        return dict(kind=kind, csr=csr, x=x, y=torch.empty(case["n"], dtype=torch.float64, device="cuda"),
                    prec=case["prec"])
    csr = _csr(case, seed, host=bool(case.get("host")))
    v1 = _start(case["n"], seed)
    s = dict(kind=kind, case=case, csr=csr, v1=v1)
    if kind == "plan":
        s["plan"] = te.Plan(csr, case["K"], case["m"], case["prec"], reorth=case["reorth"], order=case["order"],
                            refine=case["refine"])
    elif kind == "oneshot" and case["host"]:
        s["out"] = (torch.empty(case["K"], dtype=torch.float64),
                    torch.empty((case["K"], case["n"]), dtype=torch.float64, pin_memory=True))
    return s


class _HostCSR:
    def __init__(self, n, row_ptr, col, val):
        self.n, self.row_ptr, self.col, self.val = n, row_ptr, col, val


def run(s):
    kind = s["kind"]
    if kind == "tridiag":
        return te.tridiag_eigs(s["alpha"], s["beta"])
    if kind == "spmv":
        return te.spmv_noalloc(s["csr"], s["x"], s["y"], s["prec"])
    if kind == "plan":
        return s["plan"].solve(v1=s["v1"], residuals=s["case"]["refine"])
    if kind == "oneshot":
        c = s["case"]
        return te.topk_eigs(s["csr"], c["K"], c["m"], c["prec"], v1=s["v1"], reorth=c["reorth"], order=c["order"],
                            refine=c["refine"], residuals=c["refine"], out=s.get("out"))
    if kind == "lanczos":
        c = s["case"]
        return te.lanczos(s["csr"], c["m"], c["prec"], v1=s["v1"], reorth=c["reorth"], order=c["order"])
    srv, got = s["srv"], {}
    tickets = {srv.submit(A, K, m, prec, seed): (q, out)
               for q, (A, K, m, prec, seed, out) in enumerate(s["reqs"])}
    while len(got) < len(tickets):
        srv.step()
        for t in srv.completed():
            q, out = tickets[t]
            got[q] = srv.poll(t, out=out)
    order = range(len(got))
    return ([got[q][1] for q in order], np.concatenate([got[q][0] for q in order]),
            np.concatenate([got[q][2] for q in order]))


def work(case):
    kind = case["kind"]
    if kind == "tridiag":
        m = case["m"]
        return {"bytes": 8.0 * (3 * m + m * m), "flops": 9.0 * m ** 3}
    if kind == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        for q in _requests(case):
            w = work(dict(q, kind="plan", prec="fdf", refine=False))
            for k in total:
                total[k] += w[k]
        return total
    n, nnz = case["n"], 2.0 * case["n"] * case["deg"]
    sv = {"ddd": 8, "fdf": 4, "bdf": 2, "8df": 1}[case["prec"]]
    sb = 8 if case["prec"] == "ddd" else 4
    matrix = nnz * (4 + sv) + 8.0 * (n + 1)
    if kind == "spmv":
        return {"bytes": matrix + n * (sb + 8.0), "flops": 2 * nnz}
    m, K = case["m"], case.get("K", case["m"])
    flops = 2 * nnz * m + 8.0 * n * m * (m + 1) / 2 + 2.0 * n * m * K
    basis = n * (m + 1.0) * sb
    if matrix + basis < L2_BYTES:  # read once, then kept on chip
        by = matrix + n * 8.0 * K
    else:  # every step reads the matrix and twice the basis so far; the vectors read it once more
        by = m * (matrix + n * (sb + 8.0)) + n * sb * (m * (m + 1.0) + m) + n * 8.0 * K
    if case.get("refine"):  # one binary64 product per returned pair; the matrix serves all pairs at once
        by += nnz * 12.0 + 2 * n * 8.0 * K
        flops += 2 * nnz * K
    if kind == "oneshot":
        by += nnz * (4 + (4 if case["prec"] == "fdf" else 8)) + 8.0 * n
    return {"bytes": by, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, without the package
# ---------------------------------------------------------------------------
def _stored_values(val, rp, prec):
    """The binary64 values of the matrix a form computes with."""
    if prec == "ddd":
        return val
    if prec == "fdf":
        return val.float().double()
    if prec == "bdf":
        return _round_to(val, 8, -133)
    n = rp.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device=val.device), rp[1:] - rp[:-1])
    big = torch.zeros(n, dtype=torch.float64, device=val.device).scatter_reduce_(0, row, val.abs(), "amax")
    s = torch.where(big > 0, (big / 448.0).float().double(), torch.ones_like(big))[row]
    return _round_to(val / s, 4, -9).clamp(-448.0, 448.0) * s


def _round_to(x, bits, least):
    """Round to nearest even at `bits` significant bits, quantum at least 2^least."""
    q = (torch.frexp(x).exponent - bits).clamp(min=least)
    return torch.ldexp(torch.round(torch.ldexp(x, -q)), q)


def _lanczos64(rp, col, val, v1, m):
    n = rp.numel() - 1
    A = torch.sparse_csr_tensor(rp, col.long(), val, size=(n, n), check_invariants=False)
    V = torch.empty((m + 1, n), dtype=torch.float64, device=val.device)
    V[0] = v1 / v1.norm()
    alpha, beta = [], [0.0]
    for i in range(m):
        w = A @ V[i]
        h = V[:i + 1] @ w
        w = w - h @ V[:i + 1]
        h2 = V[:i + 1] @ w
        w = w - h2 @ V[:i + 1]
        alpha.append(float(h[i] + h2[i]))
        beta.append(float(w.norm()))
        V[i + 1] = w / beta[-1]
    return torch.tensor(alpha, dtype=torch.float64), torch.tensor(beta, dtype=torch.float64), V[:m], A


def _top(alpha, beta, K):
    """The K eigenpairs of T largest in modulo, each vector's largest entry positive."""
    T = torch.diag(alpha) + torch.diag(beta[1:alpha.numel()], 1) + torch.diag(beta[1:alpha.numel()], -1)
    th, Y = torch.linalg.eigh(T.cpu())
    at = th.abs().argsort(descending=True, stable=True)[:K]
    th, Y = th[at], Y[:, at]
    return th, Y * torch.sign(Y.gather(0, Y.abs().argmax(0, keepdim=True)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None  # the server draws its own start vectors
    if kind == "tridiag":
        a, b = _tridiag(case["m"], seed)
        th, Y = _top(a.cpu(), b.cpu(), case["m"])
        return th, Y, None
    rp, col, val = _matrix(case["graph"], case["n"], case["deg"], seed)
    stored = _stored_values(val, rp, case["prec"])
    v1 = _start(case["n"], seed)
    if kind == "spmv":
        x = v1 if case["prec"] == "ddd" else v1.float().double()
        return torch.sparse_csr_tensor(rp, col.long(), stored, size=(case["n"],) * 2, check_invariants=False) @ x
    alpha, beta, V, A = _lanczos64(rp, col, stored, v1, case["m"])
    if kind == "lanczos":
        return alpha, beta, V.t(), None
    th, Y = _top(alpha, beta, case["K"])
    U = Y.to(V.device).t() @ V
    res = None
    if case["refine"]:  # the quotients and residuals against the unrounded matrix
        if case["prec"] != "ddd":
            A = torch.sparse_csr_tensor(rp, col.long(), val, size=(case["n"],) * 2, check_invariants=False)
        quot, off = [], []
        for u in U:
            y = A @ u
            quot.append(float(u @ y / (u @ u)))
            off.append(float((y - quot[-1] * u).norm() / u.norm()))
        th, res = torch.tensor(quot, dtype=torch.float64), torch.tensor(off, dtype=torch.float64)
    return th, U.t(), res
