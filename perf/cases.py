"""The work that programs have this solver do, as cases that can be timed.

Every case goes through the public entry points of ``paper_2103_00736_gb300.capi``.  The kinds:

* ``residuals`` -- KKT residuals of a point held on the device, without allocation: the monitor of
  a program that runs a method of its own;
* ``solve`` -- one problem, created once and solved from x = z = e, results read back: the paper's
  dense LPs and SOCPs (Sections V-A, V-C), the sparse LPs of the batched and large workloads;
* ``end_to_end`` -- create from host arrays, solve, read back, destroy: a problem solved once;
* ``batch`` -- many uneven LPs in one launch;
* ``serve`` -- a burst of requests through the serving loop, all results read back.

Solves stop at a KKT tolerance, or at an iteration budget where a program has only so much time for
an answer (a budgeted solve reports ``ACS_MAX_ITER`` with a valid iterate and its residuals).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2103_00736_gb300 import capi, instances

LP = dict(capi.LP_SCHEDULE)
SOCP = dict(capi.SOCP_SCHEDULE)


def listed():
    return [
        # a monitoring call on a small problem: nothing but latency
        dict(name="residuals_500", kind="residuals", m=200, n=500, per_col=10, cones=False),
        # the same at the size of the large LP (1e7 nonzeros), near the entry point's limit on n
        dict(name="residuals_1m", kind="residuals", m=200_000, n=1_000_000, per_col=10, cones=False),
        # the smallest complete solve: a dense SOCP of Section V-C, cached projection operator
        dict(name="socp_dense_200", kind="solve", recipe="socp_dense", n=200, h=10, budget=3000),
        # the small sparse LP (200 x 500) with an iteration budget
        dict(name="lp_sparse_500", kind="solve", recipe="lp_bernoulli", m=200, n=500, density=0.05, budget=250),
        # Section V-C with small cones: CG that hands over to the cached operator
        dict(name="socp_dense_1000", kind="solve", recipe="socp_dense", n=1000, h=4, budget=3000),
        # the largest dense SOCP of the paper: CG passes over full rows
        dict(name="socp_dense_2900", kind="solve", recipe="socp_dense", n=2900, h=10, budget=3000),
        # a sparse LP whose user asks for exact projections: factor and inverse of a 2000 x 2000 operator
        dict(name="lp_exact_5000", kind="solve", recipe="lp_bernoulli", m=2000, n=5000, density=0.02, budget=250,
             exact_projection=True),
        # a mid-sized LP (rows scaled over four decades) solved to 1e-6 with the crossover polish
        dict(name="lp_polish_10000", kind="solve", recipe="lp_scaled", m=2000, n=10_000, per_col=10, budget=5000,
             exact_projection=True, polish_tol=2e-2),
        # the SOCP workload (100000 orthant coordinates, 20000 cones of 3 to 64) with an iteration budget
        dict(name="socp_770k", kind="solve", recipe="socp_large", m=150_000, n_orth=100_000, n_soc=20_000, per_col=8,
             budget=150),
        # an LP of the large LP's size once, from host arrays to host arrays, FP64 throughout, an iteration budget
        dict(name="lp_1m_end_to_end", kind="end_to_end", recipe="lp_large", m=200_000, n=1_000_000, per_col=10,
             budget=30, fp64=True),
        # many uneven LPs in one launch (the batched workload's recipe, m of 50 to 500)
        dict(name="batch_256", kind="batch", count=256, mmin=50, mmax=500, budget=250),
        # a burst of dense SOCP requests through the serving loop
        dict(name="serve_48", kind="serve", count=48, nmin=50, nmax=600, h=10, budget=3000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residuals", "socp_dense", "lp_sparse", "lp_exact", "lp_polish", "socp_large", "end_to_end",
                       "batch", "serve"])
    if kind == "residuals":
        n = _log_int(rng, 300, 1_000_000)
        return dict(kind="residuals", m=max(3, int(n / rng.uniform(2, 6))), n=n, per_col=rng.randint(3, 10),
                    cones=rng.random() < 0.5)
    if kind == "socp_dense":
        h = rng.choice([4, 5, 10])
        n = _log_int(rng, 100, 2900 if h == 10 else 1000)
        return dict(kind="solve", recipe="socp_dense", n=h * max(10, n // h), h=h, budget=3000)
    if kind == "lp_sparse":
        m = _log_int(rng, 50, 500)
        return dict(kind="solve", recipe="lp_bernoulli", m=m, n=int(m * rng.uniform(2, 3)), density=0.05,
                    budget=rng.randint(50, 250))
    if kind == "lp_exact":
        m = _log_int(rng, 520, 2000)
        return dict(kind="solve", recipe="lp_bernoulli", m=m, n=int(2.5 * m), density=0.02,
                    budget=rng.randint(50, 250), exact_projection=True)
    if kind == "lp_polish":
        m = _log_int(rng, 600, 2000)
        return dict(kind="solve", recipe="lp_scaled", m=m, n=5 * m, per_col=10, budget=5000, exact_projection=True,
                    polish_tol=2e-2)
    if kind == "socp_large":
        f = math.exp(rng.uniform(math.log(0.02), 0.0))
        return dict(kind="solve", recipe="socp_large", m=int(150_000 * f), n_orth=int(100_000 * f),
                    n_soc=int(20_000 * f), per_col=8, budget=rng.randint(100, 150))
    if kind == "end_to_end":
        m = _log_int(rng, 4000, 200_000)
        return dict(kind="end_to_end", recipe="lp_large", m=m, n=5 * m, per_col=rng.randint(5, 10),
                    budget=rng.randint(10, 30), fp64=True)
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 16, 256), mmin=50, mmax=_log_int(rng, 100, 500),
                    budget=rng.randint(50, 250))
    return dict(kind="serve", count=_log_int(rng, 8, 48), nmin=50, nmax=_log_int(rng, 100, 600), h=10, budget=3000)


# ---------------------------------------------------------------------------
# instances
# ---------------------------------------------------------------------------

class _Problem:
    """min c'x, Ax = b, x in K, in CSR form; x_star / y_star / s_star where an optimum is planted."""

    def __init__(self, m, n, row_ptr, col, val, n_orth, soc_dims):
        self.m, self.n, self.row_ptr, self.col, self.val = m, n, row_ptr, col, val
        self.n_orth, self.soc_dims = n_orth, soc_dims

    def plant(self, x, y, s):
        self.x_star, self.y_star, self.s_star = x, y, s
        rows = np.repeat(np.arange(self.m), np.diff(self.row_ptr))
        self.b = np.add.reduceat(self.val * x[self.col], self.row_ptr[:-1])
        self.c = np.bincount(self.col, weights=self.val * y[rows], minlength=self.n) + s
        return self


def _orthant_pair(rng, n):
    """x*_j in [0.5, 2] on 30 % of the coordinates, s*_j in [0.5, 2] on the others."""
    on = np.zeros(n, bool)
    on[rng.permutation(n)[: int(round(0.3 * n))]] = True
    v = rng.uniform(0.5, 2.0, n)
    return np.where(on, v, 0.0), np.where(on, 0.0, v)


def _cone_pair(rng, dims):
    """Complementary pairs x*, s* per Lorentz cone: 80 % on the boundary, 10 % x* and 10 % s* interior."""
    off = np.concatenate([[0], np.cumsum(dims)])
    heads = off[:-1]
    u = rng.standard_normal(off[-1])
    u[heads] = 0.0
    u /= np.repeat(np.sqrt(np.add.reduceat(u * u, heads)), dims)
    a, b, kind = rng.uniform(0.5, 2.0, dims.size), rng.uniform(0.5, 2.0, dims.size), rng.random(dims.size)
    fx = np.where(kind < 0.8, 1.0, np.where(kind < 0.9, 0.5, 0.0))
    fs = np.where(kind < 0.8, -1.0, np.where(kind < 0.9, 0.0, 0.5))
    x, s = np.repeat(a * fx, dims) * u, np.repeat(b * fs, dims) * u
    x[heads], s[heads] = np.where(kind < 0.9, a, 0.0), np.where((kind < 0.8) | (kind >= 0.9), b, 0.0)
    return x, s


def _random_columns(rng, m, n, per_col, row_scale):
    """CSR with per_col entries in every column, one in each of per_col equal ranges of rows (so the rows
    are distinct), and at least one entry in every row; N(0,1) values, rows scaled by 10^U[-2,2]."""
    k = min(per_col, m)
    lo = (np.arange(k) * m) // k
    hi = (np.arange(1, k + 1) * m) // k
    rows = torch.from_numpy((lo + rng.random((n, k)) * (hi - lo)).astype(np.int64)).cuda().reshape(-1)
    cols = torch.arange(n, device="cuda").repeat_interleave(k)
    empty = torch.nonzero(torch.bincount(rows, minlength=m) == 0).reshape(-1)
    if empty.numel():
        extra = torch.from_numpy(rng.integers(0, n, empty.numel())).cuda()
        rows, cols = torch.cat([rows, empty]), torch.cat([cols, extra])
    key = torch.sort(rows * n + cols).values
    rows, col = (key // n).cpu().numpy(), (key % n).to(torch.int32).cpu().numpy()
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))]).astype(np.int64)
    val = rng.standard_normal(rows.size)
    if row_scale:
        val *= np.repeat(10.0 ** rng.uniform(-2.0, 2.0, m), np.diff(row_ptr))
    return row_ptr, col, val


def _instance(case, seed):
    recipe = case["recipe"]
    if recipe == "socp_dense":
        return instances.dense_socp(case["n"], case["h"], seed=seed)
    if recipe == "lp_bernoulli":
        return instances.bernoulli_lp(seed, case["m"], case["n"], case["density"])
    rng = np.random.default_rng(seed)
    if recipe.startswith("lp_"):
        dims, n = np.zeros(0, np.int32), case["n"]
        n_orth = n
    else:
        dims = np.random.default_rng(case["n_soc"]).integers(3, 65, size=case["n_soc"]).astype(np.int32)
        n_orth = case["n_orth"]
        n = n_orth + int(dims.sum())
    m = case["m"]
    p = _Problem(m, n, *_random_columns(rng, m, n, case["per_col"], recipe == "lp_scaled"), n_orth, dims)
    x, s = _orthant_pair(rng, n_orth)
    if dims.size:
        xc, sc = _cone_pair(rng, dims)
        x, s = np.concatenate([x, xc]), np.concatenate([s, sc])
    return p.plant(x, rng.standard_normal(m), s)


def _options(case):
    o = dict(SOCP if "socp" in case["recipe"] else LP)
    if case.get("exact_projection"):
        o["projection"] = 2                              # ACS_PROJ_DENSE
    if case.get("fp64"):
        o["precision"] = 2                               # ACS_PREC_FP64
    if case.get("polish_tol"):
        o["polish_tol"] = case["polish_tol"]
    return o


def _sizes(count, lo, hi):
    """Log-uniform sizes, the same for every seed of a case."""
    u = np.random.default_rng(count).uniform(math.log(lo), math.log(hi), count)
    return np.rint(np.exp(u)).astype(int).tolist()


def _batch_members(case, seed):
    ms = _sizes(case["count"], case["mmin"], case["mmax"])
    return [instances.bernoulli_lp(seed * 4096 + i, m, int(round(2.5 * m))) for i, m in enumerate(ms)]


def _requests(case, seed):
    h = case["h"]
    ns = _sizes(case["count"], case["nmin"], case["nmax"])
    return [instances.dense_socp(h * max(2, n // h), h, seed=seed * 4096 + i) for i, n in enumerate(ns)]


def _residual_inputs(case, seed):
    """A sparse problem and a point about 1 % away from its optimum."""
    rng = np.random.default_rng(seed)
    m, n = case["m"], case["n"]
    dims = np.zeros(0, np.int32)
    if case["cones"]:
        dims = np.full(max(1, n // 40), 20, np.int32)
    n_orth = n - int(dims.sum())
    p = _Problem(m, n, *_random_columns(rng, m, n, case["per_col"], False), n_orth, dims)
    x, s = _orthant_pair(rng, n_orth)
    if dims.size:
        xc, sc = _cone_pair(rng, dims)
        x, s = np.concatenate([x, xc]), np.concatenate([s, sc])
    p.plant(x, rng.standard_normal(m), s)
    at = [v + 0.01 * rng.standard_normal(v.size) for v in (x, p.y_star, s)]
    return p, at


def prepare(case, seed):
    kind = case["kind"]
    if kind == "residuals":
        p, at = _residual_inputs(case, seed)
        off = p.n_orth + np.concatenate([[0], np.cumsum(p.soc_dims)])
        arrays = [p.row_ptr.astype(np.int32), p.col, p.val, p.b, p.c, *at, off.astype(np.int32)]
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]
        return dict(kind=kind, m=p.m, n=p.n, n_orth=p.n_orth, n_soc=int(p.soc_dims.size), dev=dev,
                    out=torch.zeros(6, dtype=torch.float64, device="cuda"))
    if kind == "solve":
        return dict(kind=kind, budget=case["budget"], solver=capi.Solver(_instance(case, seed), **_options(case)))
    if kind == "end_to_end":
        return dict(kind=kind, budget=case["budget"], problem=_instance(case, seed), options=_options(case))
    if kind == "batch":
        return dict(kind=kind, budget=case["budget"], batch=capi.Batch(_batch_members(case, seed), share=None, **LP))
    return dict(kind=kind, budget=case["budget"], requests=_requests(case, seed), server=capi.Server())


def _result(got):
    status, x, y, z, iterations, res = got[:6]
    return dict(status=status, iterations=iterations, x=x, y=y, z=z, residuals=res[:6])


def _results(got):
    """The results of many problems, one after the other."""
    return dict(status=np.array([g[0] for g in got]), iterations=np.array([g[4] for g in got]),
                x=np.concatenate([g[1] for g in got]), y=np.concatenate([g[2] for g in got]),
                z=np.concatenate([g[3] for g in got]), residuals=np.stack([g[5][:6] for g in got]))


def run(state):
    kind = state["kind"]
    if kind == "residuals":
        d = state["dev"]
        rc = capi.acs_kkt_residuals_noalloc(state["m"], state["n"], *[t.data_ptr() for t in d[:8]], state["n_orth"],
                                            state["n_soc"], d[8].data_ptr(), state["out"].data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
        if rc != capi.SOLVED:
            raise capi.AcsError(rc, "acs_kkt_residuals_noalloc")
        return state["out"]
    if kind == "solve":
        state["solver"].solve(tol=1e-6, max_iter=state["budget"])
        return _result(state["solver"].get())
    if kind == "end_to_end":
        with capi.Solver(state["problem"], **state["options"]) as s:
            s.solve(tol=1e-6, max_iter=state["budget"])
            return _result(s.get())
    if kind == "batch":
        b = state["batch"]
        b.solve(tol=1e-6, max_iter=state["budget"])
        return _results([b.get(i) for i in range(b.count)])
    server = state["server"]
    ids = [server.submit(r, tol=1e-6, max_iter=state["budget"]) for r in state["requests"]]
    for i in ids:
        server.wait(i)
    return _results([server.result(i) for i in ids])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _one(m, n, nnz, iterations, factor):
    """Bytes and operations of one problem: its data read and its results written once; two products with
    A per iteration, and where the projection is exact, its operator formed once and applied."""
    b = 12.0 * nnz + 8.0 * (m + n) + 8.0 * (2 * n + m)
    f = iterations * (4.0 * nnz + 10.0 * n)
    if factor:
        f += 2.0 * m ** 3 / 3.0 + iterations * 2.0 * m * m
    return b, f


def work(case):
    kind = case["kind"]
    if kind == "residuals":
        m, n = case["m"], case["n"]
        nnz = n * min(case["per_col"], m)
        return {"bytes": 12.0 * nnz + 4.0 * m + 16.0 * m + 24.0 * n, "flops": 4.0 * nnz + 10.0 * n}
    if kind in ("solve", "end_to_end"):
        r = case["recipe"]
        if r == "socp_dense":                            # solved in about 100 iterations
            m, n = (4 * case["n"]) // 5, case["n"]
            b, f = _one(m, n, m * n, 100, m <= 512)
        elif r == "lp_bernoulli":
            m, n = case["m"], case["n"]
            b, f = _one(m, n, case["density"] * m * n, case["budget"], True)
        else:
            m = case["m"]
            n = case["n"] if r.startswith("lp_") else case["n_orth"] + 33.5 * case["n_soc"]
            b, f = _one(m, n, n * case["per_col"], min(case["budget"], 60), bool(case.get("exact_projection")))
        return {"bytes": b, "flops": f}
    if kind == "batch":                                  # mean of m and m^2, m^3 under a log-uniform m
        lo, hi = case["mmin"], case["mmax"]
        mean = [(hi ** k - lo ** k) / (k * math.log(hi / lo)) if hi > lo else lo ** k for k in (1, 2, 3)]
        m, m2, m3 = mean
        it = case["budget"]
        nnz = 0.05 * m2
        return {"bytes": case["count"] * (12.0 * nnz + 8.0 * 9.5 * m),
                "flops": case["count"] * (2.0 * m3 / 3.0 + it * (4.0 * nnz + 25.0 * m + 2.0 * m2))}
    lo, hi = case["nmin"], case["nmax"]
    n, n2, n3 = [(hi ** k - lo ** k) / (k * math.log(hi / lo)) if hi > lo else lo ** k for k in (1, 2, 3)]
    return {"bytes": case["count"] * (12.0 * 0.8 * n2 + 8.0 * 4.6 * n),
            "flops": case["count"] * (0.34 * n3 + 100 * (4.0 * 0.8 * n2 + 10.0 * n + 1.28 * n2))}


# ---------------------------------------------------------------------------
# the same results from plain FP64 arithmetic
# ---------------------------------------------------------------------------

def _reflect(v, n_orth, starts, dims):
    """abs_K: |v| on the orthant; per Lorentz cone (v1, vbar), t = |vbar|: v, -v, or (t, (v1/t) vbar)."""
    out = torch.empty_like(v)
    out[:n_orth] = v[:n_orth].abs()
    if starts is not None:
        tail = v[n_orth:].clone()
        v1 = tail[starts].clone()
        tail[starts] = 0.0
        owner = torch.repeat_interleave(torch.arange(dims.numel(), device=v.device), dims)
        t = torch.zeros_like(v1).index_add_(0, owner, tail * tail).sqrt()
        inside, polar = t <= v1, t <= -v1
        f = torch.where(inside, torch.ones_like(t), torch.where(polar, -torch.ones_like(t), v1 / t))
        head = torch.where(inside, v1, torch.where(polar, -v1, t))
        w = f[owner] * tail
        w[starts] = head
        out[n_orth:] = w
    return out


def _cone_distance2(v, n_orth, starts, dims):
    d = (v[:n_orth].clamp(max=0.0) ** 2).sum()
    if starts is not None:
        p = 0.5 * (v + _reflect(v, n_orth, starts, dims))
        d = d + ((v - p)[n_orth:] ** 2).sum()
    return d


def _algorithm2(p, t_cap, first, period, tol, budget):
    """Algorithm 2 with exact projections in FP64 on dense data, its KKT test every 10 iterations."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    A = torch.zeros(p.m, p.n, dtype=torch.float64)
    A[torch.from_numpy(np.repeat(np.arange(p.m), np.diff(p.row_ptr))), torch.from_numpy(p.col).long()] = \
        torch.from_numpy(np.ascontiguousarray(p.val))
    A = A.to(dev)
    b, c = torch.from_numpy(p.b).to(dev), torch.from_numpy(p.c).to(dev)
    k = int(p.n_orth)
    dims = torch.from_numpy(np.asarray(p.soc_dims)).long().to(dev)
    starts = torch.cat([dims.new_zeros(1), dims.cumsum(0)[:-1]]) if dims.numel() else None
    owner = torch.repeat_interleave(torch.arange(dims.numel(), device=dev), dims) if dims.numel() else None
    x = torch.zeros(p.n, dtype=torch.float64, device=dev)
    x[:k] = 1.0
    if starts is not None:
        x[k + starts] = 1.0
    z = x.clone()
    for it in range(1, budget + 1):
        if it == 1 or (first and it >= first and (it - first) % period == 0):
            o = x[:k].abs() / z[:k].abs()
            if starts is not None:
                tail = x[k:].clone()
                tail[starts] = 0.0
                nb = torch.zeros(dims.numel(), dtype=torch.float64, device=dev).index_add_(0, owner, tail * tail).sqrt()
                o = torch.cat([o, (x[k + starts] - nb).abs() / z[k + starts].abs()])
            lo = o.log()
            fine = torch.isfinite(lo)
            hi_, lo_ = (lo[fine].max(), lo[fine].min()) if fine.any() else (0.0, 0.0)
            spread = float(hi_ - lo_)
            alpha = min(1.0, t_cap / spread) if spread > 0 else (1.0 if fine.any() else 0.0)
            e = torch.where(torch.isnan(lo), torch.full_like(lo, 0.5 * float(hi_ + lo_)),
                            lo.clamp(min=float(lo_), max=float(hi_)))
            O = (alpha * e).exp()
            if starts is not None:
                O = torch.cat([O[:k], O[k:][owner]])
            Ah = A * O
            ch = O * c
            s = x / O - O * z
            L = torch.linalg.cholesky(Ah @ Ah.T)
            bt = b + Ah @ ch
        pr = _reflect(s, k, starts, dims)
        w = torch.cholesky_solve((bt - Ah @ pr)[:, None], L)[:, 0]
        s = 0.5 * (s + pr) - ch + Ah.T @ w
        if it % 10 and it != budget and not (first and it + 1 >= first and (it + 1 - first) % period == 0):
            continue
        x, z = O * (pr + s) * 0.5, (pr - s) / (2.0 * O)
        if it % 10 == 0 or it == budget:
            cx, by = c @ x, b @ w
            dx, dz = _cone_distance2(x, k, starts, dims).sqrt(), _cone_distance2(z, k, starts, dims).sqrt()
            res = torch.stack([(A @ x - b).norm() / (1 + b.norm()), (A.T @ w + z - c).norm() / (1 + c.norm()),
                               (cx - by).abs() / (1 + cx.abs() + by.abs()),
                               torch.maximum(dx, dz) / (1 + torch.maximum(x.norm(), z.norm())), cx, by])
            xr, zr = x, z
            if float(res[:4].max()) <= tol:
                break
    return [v.cpu().numpy() for v in (xr, w, zr, res)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "residuals":
        p, (x, y, z) = _residual_inputs(case, seed)
        rows = np.repeat(np.arange(p.m), np.diff(p.row_ptr))
        rp = np.add.reduceat(p.val * x[p.col], p.row_ptr[:-1]) - p.b
        rd = np.bincount(p.col, weights=p.val * y[rows], minlength=p.n) + z - p.c
        dims = torch.from_numpy(p.soc_dims).long()
        starts = torch.cat([dims.new_zeros(1), dims.cumsum(0)[:-1]]) if dims.numel() else None
        dx, dz = (math.sqrt(float(_cone_distance2(torch.from_numpy(v), p.n_orth, starts, dims))) for v in (x, z))
        n2 = np.linalg.norm
        cx, by = float(p.c @ x), float(p.b @ y)
        return np.array([n2(rp) / (1 + n2(p.b)), n2(rd) / (1 + n2(p.c)), abs(cx - by) / (1 + abs(cx) + abs(by)),
                         max(dx, dz) / (1 + max(n2(x), n2(z))), cx, by])
    if kind in ("solve", "end_to_end"):
        p = _instance(case, seed)
        none = dict(status=None, iterations=None, x=None, y=None, z=None, residuals=None)
        if case.get("polish_tol"):                       # |support| >= m: the multipliers are unique
            return dict(none, y=p.y_star, z=p.s_star)
        # Where CG applies the projection, an iterate depends on where its inexact solves stopped.
        if p.m > 512 and not case.get("exact_projection"):
            return None
        o = _options(case)
        x, y, z, res = _algorithm2(p, o["t"], o["cond_first"], o["cond_period"], 1e-6, case["budget"])
        return dict(none, x=x, y=y, z=z, residuals=res)
    return None
