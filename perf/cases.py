"""Workloads of the Monte Carlo nodal stage: what its users run, over the range they run it in.

Every case is one call (or one batch of serving requests) through the public
Python entry points.  Sizes come from the repository's own workloads (the
24-node and 256-node problems, the 3D cascade, the anisotropic 513^2 problem,
the paper's example, Algorithm 3's cloud, the serving request ranges).  Work is
counted in Euler path-steps: nodes x paths x mean exit index.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1512_02818_gb300 import pdd
from paper_1512_02818_gb300 import workloads as W

CFG0, ANISO, CUBE, PAPER = "cfg0", "aniso", "cube", "paper"
KIND = {CFG0: pdd.PDD_PROBLEM_CFG0_2D, ANISO: pdd.PDD_PROBLEM_ANISO_2D,
        CUBE: pdd.PDD_PROBLEM_CUBE_3D, PAPER: pdd.PDD_PROBLEM_PAPER_EX_2D}
# mean exit time of the paths that start on the interfaces
MEAN_TAU = {CFG0: 0.10, ANISO: 0.07, CUBE: 0.05, PAPER: 0.045}
FIELDS = pdd.STAT_FIELDS + pdd.COUNT_FIELDS


def _case(name, call, problem, nodes, paths, dt, grid=0, eps=0.0, parts=1, precision="f32",
          host=False):
    c = dict(call=call, problem=problem, nodes=nodes, paths=paths, dt=dt, grid=grid, eps=eps,
             parts=parts, precision=precision, host=host)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one node of a request, coarse step, host arrays in and out
        _case("one_node", "estimate", CFG0, 1, 1000, 1e-2, host=True),
        # the 24-node problem: plain estimator, host arrays in and out
        _case("nodes_24", "estimate", CFG0, 24, 10_000, 1e-3, host=True),
        # a batch of serving requests of mixed sizes, submitted together and polled
        _case("serve_12", "serve", CFG0, 256, 8000, 1e-3, grid=129, eps=1e-2, parts=12),
        # the paper's own PDE on 18 nodes with a previous iterate, host arrays
        _case("paper_18", "estimate", PAPER, 18, 100_000, 1e-4, grid=129, eps=1e-2, host=True),
        # a run at a fixed error: every group of nodes with its own balanced path count
        _case("fixed_error_128", "groups", CFG0, 256, 2000, 1e-4, grid=129, eps=1e-2, parts=128),
        # plain estimator on the 256-node problem, device arrays
        _case("plain_256", "estimate", CFG0, 256, 20_000, 1e-4),
        # the same with the control variate: the largest ordinary call
        _case("cv_256", "estimate", CFG0, 256, 100_000, 1e-4, grid=129, eps=1e-2),
        # anisotropic diffusion on every interface node of 32 x 32 subdomains, fine grid
        _case("aniso_31744", "estimate", ANISO, 31_744, 500, 1e-4, grid=513, eps=1e-2),
        # three levels of the 3D cascade in one launch
        _case("cascade_3d", "cascade", CUBE, 9216, 1000, 1e-4, grid=65, eps=1e-3, parts=3),
        # Algorithm 3: the cloud of 100 time steps and the fits on the host
        _case("fit_24", "fit", CFG0, 24, 1000, 1e-3, grid=129, eps=1.0, parts=100),
        # one coupled level of the multilevel estimator
        _case("coupled_256", "coupled", CFG0, 256, 4000, 1e-3, grid=129, eps=1e-2),
        # FP64 paths of the precision comparison
        _case("f64_64", "estimate", CFG0, 64, 1000, 1e-3, grid=129, eps=1e-2, precision="f64"),
    ]


def _steps(c):
    """Expected path-steps of one pass."""
    per = MEAN_TAU[c["problem"]] / c["dt"]
    w = c["nodes"] * c["paths"] * per
    if c["call"] == "serve":  # sizes log-uniform up to the largest
        return c["parts"] * w * 0.04
    if c["call"] == "groups":
        return 0.6 * w
    if c["call"] == "fit":  # dt .. 10 dt
        return w * c["parts"] * 0.26
    if c["call"] == "coupled":  # fine at dt / 2, coarse at dt
        return 3 * w
    return w


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["estimate"] * 6 + ["groups", "cascade", "serve", "fit", "coupled", "coupled"])
    dt = rng.choice([1e-2, 3e-3, 1e-3, 4e-4, 1e-4])
    cv = rng.random() < 0.6
    precision = "f32"
    if call == "cascade":
        problem, grid, parts = rng.choice([CUBE, CFG0]), 0, rng.randint(2, 4)
        grid = rng.choice([33, 65]) if problem == CUBE else rng.choice([129, 200])
        dt, cv = rng.choice([1e-3, 4e-4, 1e-4]), True
    elif call in ("groups", "serve", "fit"):
        problem, parts = CFG0, {"groups": rng.randint(3, 128), "serve": rng.randint(2, 24),
                                "fit": rng.randint(10, 130)}[call]
        grid, cv = 129, cv or call == "fit"
        dt = 1e-3 if call == "fit" else dt
    else:
        problem, parts = rng.choice([CFG0, CFG0, ANISO, CUBE, PAPER]), 1
        grid = rng.choice([33, 65]) if problem == CUBE else rng.choice([65, 129, 257, 513])
        if call == "estimate" and rng.random() < 0.2:
            precision = "f64"
    nodes = int(_log(rng, 1, 600 if call in ("serve", "fit", "groups") else 20_000))
    nodes = max(nodes, parts if call == "groups" else 1)
    most = 3e7 if precision == "f64" else 1.5e9 if call == "serve" else 8e9
    c = _case("", call, problem, nodes, 100, dt, grid if cv else 0, rng.choice([1e-1, 1e-2, 1e-3]),
              parts, precision, call == "estimate" and rng.random() < 0.5)
    target = min(_log(rng, 3e5, most), most)
    c["paths"] = max(20, min(1_000_000, int(100 * target / max(_steps(c), 1.0))))
    while _steps(c) > most and c["nodes"] > max(1, parts if call == "groups" else 1):
        c["nodes"] = max(c["nodes"] // 2, parts if call == "groups" else 1)
    return c


# ---- inputs ------------------------------------------------------------------
def _nodes(problem, n, rng):
    if problem == PAPER:
        t = rng.uniform(0.02, 0.98, n)
        return np.stack([rng.integers(1, 4, n) / 4.0, t], 1).astype(np.float32)
    if problem == CUBE:
        all_ = W.nodes_3d(4, 8)
    else:
        all_ = W.workload_nodes("c4") if problem == ANISO else None
    if all_ is None:
        fixed = {24: "c0", 256: "c1"}.get(n)
        return W.workload_nodes(fixed) if fixed else W.random_interface_nodes(rng, n)
    if n >= len(all_):
        return all_
    return all_[np.sort(rng.permutation(len(all_))[:n])]


def _inputs(c, seed):
    """Nodes, seed and the list of parts: dicts of (index into nodes, paths, dt, eps, tag)."""
    rng = np.random.default_rng([11, seed])
    nodes = _nodes(c["problem"], c["nodes"], rng)
    n = len(nodes)
    every = np.arange(n)
    P = c["parts"]
    if c["call"] == "groups":
        sizes = np.array_split(rng.permutation(n), P)
        need = np.sort(np.exp(rng.uniform(math.log(c["paths"] / 3), math.log(c["paths"]), P)))
        parts = [dict(idx=g, paths=max(2, int(m)), dt=c["dt"], eps=c["eps"], tag=1000 + i)
                 for i, (g, m) in enumerate(zip(sizes, need))]
    elif c["call"] == "cascade":  # 10x fewer paths and 10x longer steps per coarser level
        parts = [dict(idx=every, paths=max(20, c["paths"] // 10 ** l), dt=min(c["dt"] * 10 ** l, 1e-2),
                      eps=c["eps"] * 10 ** l, tag=l) for l in range(P)]
    elif c["call"] == "serve":
        parts, sizes = [], np.random.default_rng([13, c["nodes"], c["paths"], P])  # of the case
        for i in range(P):
            m = max(1, int(math.exp(sizes.uniform(0, math.log(c["nodes"] + 0.5)))))
            N = max(2, int(math.exp(sizes.uniform(math.log(c["paths"] / 20), math.log(c["paths"])))))
            dt = c["dt"] * (1, 3)[i % 2]
            parts.append(dict(idx=np.sort(rng.permutation(n)[:m]), paths=N, dt=dt,
                              eps=c["eps"] if i % 3 else 0.0, tag=i + 1))
    else:
        parts = [dict(idx=every, paths=c["paths"], dt=c["dt"], eps=c["eps"], tag=0)]
    if not c["grid"]:
        for p in parts:
            p["eps"] = 0.0
    return nodes, 1234 + seed, parts


def _grid(c, eps):
    """Values of the previous iterate on the control grid ([y, x] or [z, y, x])."""
    k = KIND[c["problem"]]
    v = W.control_grid(k, c["grid"], eps)
    return v - W.control_grid(k, c["grid"], 0.0) if c["call"] == "fit" else v


def prepare(case, seed):
    nodes, rng_seed, parts = _inputs(case, seed)
    ctx = pdd.Context(0)
    prob = pdd.Problem(ctx, KIND[case["problem"]],
                       precision=pdd.PDD_PATH_FP64 if case["precision"] == "f64" else
                       pdd.PDD_PATH_FP32)
    slot = {0.0: pdd.PDD_CV_NONE}
    for eps in sorted({p["eps"] for p in parts} - {0.0}):
        slot[eps] = len(slot) - 1
        prob.set_control_grid(slot[eps], _grid(case, eps))
    st = dict(case=case, ctx=ctx, prob=prob, nodes=nodes, seed=rng_seed, parts=parts)
    for p in parts:
        p["gid"] = slot[p["eps"]]
        own = nodes[p["idx"]]
        p["nodes"] = own
        p["cols"] = [torch.from_numpy(np.ascontiguousarray(own[:, j])) for j in range(own.shape[1])]
        if not case["host"]:
            p["cols"] = [x.cuda() for x in p["cols"]]
    if case["call"] == "groups":
        # one buffer per result, a slice for every group
        n = len(nodes)
        st["out"] = {f: torch.empty(n, dtype=torch.float64 if f in pdd.STAT_FIELDS else torch.int64,
                                    device="cuda") for f in FIELDS}
        st["levels"], st["outs"], at = [], [], 0
        for p in parts:
            a, o = pdd.EstimateArgs(), pdd.NodeStats()
            a.n_nodes, a.coords_on_device, a.grid_id = len(p["idx"]), 1, p["gid"]
            a.coords[0], a.coords[1], a.coords[2] = p["cols"][0].data_ptr(), p["cols"][1].data_ptr(), None
            a.n_paths, a.dt, a.kappa, a.seed, a.stream_tag = p["paths"], p["dt"], 1.0, rng_seed, p["tag"]
            o.on_device = 1
            for f in FIELDS:
                setattr(o, f, st["out"][f].data_ptr() + 8 * at)
            at += len(p["idx"])
            st["levels"].append(a)
            st["outs"].append(o)
    if case["call"] == "serve":
        st["server"] = pdd.Server(ctx)
    return st


def _stats(res):
    return {f: res[f] for f in FIELDS}


def run(state):
    c, prob, seed, parts = state["case"], state["prob"], state["seed"], state["parts"]
    call = c["call"]
    if call == "estimate":
        p = parts[0]
        return _stats(prob.estimate(p["cols"], p["paths"], p["dt"], grid_id=p["gid"], seed=seed,
                                    device_out=not c["host"], host_inputs=c["host"]))
    if call == "groups":
        pdd.pdd_estimate_levels(prob.handle, state["levels"], state["outs"])
        return state["out"]
    if call == "cascade":
        _, res = prob.estimate_levels([dict(nodes=p["cols"], n_paths=p["paths"], dt=p["dt"],
                                            grid_id=p["gid"], seed=seed, stream_tag=p["tag"])
                                       for p in parts])
        return [_stats(r) for r in res]
    if call == "coupled":
        p = parts[0]
        fine, diff = prob.estimate_coupled(p["cols"], p["paths"], p["dt"], grid_id=p["gid"], seed=seed)
        return [_stats(fine), _stats(diff)]
    if call == "fit":
        p = parts[0]
        r = prob.fit_constants(p["nodes"], p["paths"], p["dt"], 10 * p["dt"], c["parts"],
                               grid_id=p["gid"], seed=seed)
        return {f: r[f] for f in pdd.FIT_FIELDS + ["cloud"]}
    srv = state["server"]
    tickets = [srv.submit(prob, p["nodes"], p["paths"], p["dt"], grid_id=p["gid"], seed=seed,
                          stream_tag=p["tag"]) for p in parts]
    got = []
    for t, p in zip(tickets, parts):
        status, res = srv.poll(t, len(p["nodes"]), 60_000_000)
        if status != pdd.PDD_OK:
            raise RuntimeError(f"request {t}: status {status}")
        got.append(res)
    return {f: np.concatenate([r[f] for r in got]) for f in FIELDS}


def work(case):
    """Operations of the path-steps (the random numbers, the coefficients, the
    update and the control variate's interpolation), and the inputs and results."""
    three = case["problem"] == CUBE
    per = (130 if three else 90) + (70 if three else 35) * bool(case["grid"])
    nodes = case["nodes"] * (case["parts"] if case["call"] in ("cascade", "fit") else 1)
    table = (16 * case["grid"] ** 3 if three else 8 * case["grid"] ** 2) if case["grid"] else 0
    levels = case["parts"] if case["call"] == "cascade" else 1
    return {"bytes": nodes * (14 * 8 + 12) + levels * table, "flops": per * _steps(case)}


# ---- the same in plain torch, 64 bits ------------------------------------------
MASK = 0xFFFFFFFF


def _philox(block, path, node, seed, tag):
    c0, c1, c2 = torch.full_like(path, block), path, node
    c3 = torch.full_like(path, (seed >> 32) & MASK)
    k0, k1 = seed & MASK, tag
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & MASK) ^ c1 ^ k0, p1 & MASK,
                          ((p0 >> 32) & MASK) ^ c3 ^ k1, p0 & MASK)
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c0, c1, c2, c3


def _normals(block, path, node, seed, tag):
    u = [((w >> 9).double() + 0.5) * 2.0 ** -23 for w in _philox(block, path, node, seed, tag)]
    out = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r, t = torch.sqrt(-2 * torch.log(a)), 2 * math.pi * b
        out += [r * torch.cos(t), r * torch.sin(t)]
    return out


def _u(problem, x):
    if problem in (CFG0, ANISO):
        return torch.exp(x[0] + x[1]) * torch.cos(x[0] - x[1])
    if problem == CUBE:
        return torch.exp(x[0]) * torch.sin(x[1]) * torch.cos(x[2]) + x[0] * x[1] * x[2]
    return 2 * torch.cos(2 * (x[1] - 2) * x[0]) + torch.sin(3 * (x[0] - 2) * x[1]) + 3.1


def _coefficients(problem, x):
    """b, c, f and the factor of |sigma^T N| at x."""
    if problem in (CFG0, ANISO):
        X, Y = x
        E, sn, cs = torch.exp(X + Y), torch.sin(X - Y), torch.cos(X - Y)
        b = [torch.sin(Y) / 2, torch.cos(X) / 2]
        c = 1 + X * X + Y * Y
        f = b[0] * E * (cs - sn) + b[1] * E * (cs + sn) - c * E * cs
        if problem == CFG0:
            return b, c, f, 1.0
        a = 1 + torch.sin(2 * math.pi * X) / 2
        return b, c, f + a * E * cs, torch.sqrt(a)
    if problem == CUBE:
        e = torch.exp(x[0]) * torch.sin(x[1]) * torch.cos(x[2])
        return [0.0, 0.0, 0.0], 1.0, -1.5 * e - x[0] * x[1] * x[2], 1.0
    X, Y = x
    p, q, s = 2 * X * (Y - 2), 3 * Y * (X - 2), 1.1 + torch.sin(X + Y)
    sp, cp, sq, cq = torch.sin(p), torch.cos(p), torch.sin(q), torch.cos(q)
    b = torch.cos(X + Y) / s
    c = (X * X + Y * Y) / s
    ux, uy = -4 * (Y - 2) * sp + 3 * Y * cq, -4 * X * sp + 3 * (X - 2) * cq
    lap = -8 * (X * X + (Y - 2) ** 2) * cp - 9 * ((X - 2) ** 2 + Y * Y) * sq
    return [b, b], c, lap + b * (ux + uy) - c * _u(PAPER, x), math.sqrt(2.0)


def _table(v):
    """Gradient of grid values: centred differences, second-order one-sided ones on the edges."""
    v = torch.from_numpy(v).cuda()
    d = 1.0 / (v.shape[0] - 1)
    out = []
    for axis in reversed(range(v.dim())):  # x is the last axis
        w = v.movedim(axis, 0)
        g = torch.empty_like(w)
        g[1:-1] = (w[2:] - w[:-2]) / (2 * d)
        g[0] = (-3 * w[0] + 4 * w[1] - w[2]) / (2 * d)
        g[-1] = (3 * w[-1] - 4 * w[-2] + w[-3]) / (2 * d)
        out.append(g.movedim(0, axis).reshape(-1))
    return torch.stack(out, 1), v.shape[0]


def _interpolate(table, n, x):
    D = len(x)
    cell, frac = [], []
    for c in x:
        i = (c * (n - 1)).floor().clamp(0, n - 2)
        cell.append(i.long())
        frac.append((c * (n - 1) - i)[:, None])
    total = 0.0
    for corner in range(2 ** D):
        at, w = 0, 1.0
        for j in reversed(range(D)):
            bit = corner >> j & 1
            at = at * n + cell[j] + bit
            w = w * (frac[j] if bit else 1 - frac[j])
        total = total + w * table[at]
    return total.unbind(1)


class _Paths:
    """Paths in lock step, each with its own time step; those that have left keep their state."""

    def __init__(self, problem, x, h, cv, table):
        self.problem, self.table, self.x = problem, table, list(x)
        self.h, self.cv = h, cv
        self.alive = torch.ones_like(x[0], dtype=torch.bool)
        self.Y, self.Z, self.xi, self.k = (torch.full_like(x[0], v) for v in (1.0, 0.0, 0.0, 0.0))

    def step(self, dW):
        x = self.x
        b, c, f, scale = _coefficients(self.problem, x)
        d = torch.stack([torch.minimum(v, 1 - v) for v in x]).amin(0)
        self.alive = self.alive & (d > 0.5826 * torch.sqrt(self.h) * scale)
        on = self.alive.double()
        dW, h = [w * on for w in dW], self.h * on
        if self.problem == ANISO:
            dW = [scale * dW[0], scale * (0.5 * dW[0] + math.sqrt(0.75) * dW[1])]
        elif self.problem == PAPER:
            dW = [scale * w for w in dW]
        if self.table is not None:
            g = _interpolate(*self.table, x)
            self.xi = self.xi - self.cv * self.Y * sum(p * q for p, q in zip(g, dW))
        self.Z = self.Z - h * self.Y * f
        self.x = [v + (h * bj + w) for v, bj, w in zip(x, b, dW)]
        self.Y = self.Y * (1 - h * c)
        self.k = self.k + on

    def take(self, keep):
        new = object.__new__(_Paths)
        new.problem, new.table, new.x = self.problem, self.table, [v[keep] for v in self.x]
        for f in ("h", "cv", "alive", "Y", "Z", "xi", "k"):
            setattr(new, f, getattr(self, f)[keep])
        return new

    def scores(self):
        x = torch.stack(self.x)
        out = ((x < 0) | (x > 1)).any(0)
        best = torch.stack([v for c in self.x for v in (c, 1 - c)]).argmin(0)
        moved = [torch.where(best == 2 * j, 0.0, torch.where(best == 2 * j + 1, 1.0, c))
                 for j, c in enumerate(self.x)]
        p = [torch.where(out, c.clamp(0, 1), m) for c, m in zip(self.x, moved)]
        return torch.stack([_u(self.problem, p) * self.Y + self.Z, self.xi, self.k])


def _simulate(problem, nodes, parts, seed, table, coupled=False):
    """Scores (phi, xi, k) of every part's paths, each of shape (3, nodes, paths); coupled: of
    the paths at dt / 2 and of those at dt that the same increments drive."""
    D = nodes.shape[1]

    def spread(values, dtype=torch.float64):
        return torch.cat([torch.as_tensor(np.asarray(v), dtype=dtype).cuda().expand(len(p["idx"]) * p["paths"])
                          for v, p in zip(values, parts)])

    x0 = torch.cat([torch.from_numpy(nodes[p["idx"]].astype(np.float64)).cuda().repeat_interleave(p["paths"], 0)
                    for p in parts]).unbind(1)
    node = torch.cat([torch.arange(len(p["idx"])).repeat_interleave(p["paths"]) for p in parts]).cuda()
    path = torch.cat([torch.arange(p["paths"]).repeat(len(p["idx"])) for p in parts]).cuda()
    tag = spread([p["tag"] for p in parts], torch.int64)
    h = spread([p["dt"] for p in parts])
    cv = spread([float(p["eps"] != 0) for p in parts])
    sets = [_Paths(problem, x0, s, cv, table) for s in ([h / 2, h] if coupled else [h])]
    rt = torch.sqrt(sets[0].h)
    where = torch.arange(len(h), device="cuda")
    res = [torch.zeros(3, len(h), dtype=torch.float64, device="cuda") for _ in sets]
    spare, block, k, before = [], 0, 0, None
    while len(where):
        while len(spare) < D:
            spare += _normals(block, path, node, seed, tag)
            block += 1
        dW, spare = [rt * z for z in spare[:D]], spare[D:]
        sets[0].step(dW)
        if coupled and k % 2:
            sets[1].step([a + b for a, b in zip(before, dW)])
        before, k = dW, k + 1
        if k % 32 == 0:  # an even number of steps: both sets are at the same time
            on = sets[0].alive | sets[-1].alive
            for s, r in zip(sets, res):
                r[:, where[~on]] = s.take(~on).scores()
            sets = [s.take(on) for s in sets]
            node, path, tag, rt, where = node[on], path[on], tag[on], rt[on], where[on]
            spare = [z[on] for z in spare]
    sizes = [len(p["idx"]) * p["paths"] for p in parts]
    return [[v.view(3, len(p["idx"]), p["paths"]) for v, p in zip(r.split(sizes, 1), parts)] for r in res]


def _moments(phi, psi, k):
    N = phi.shape[1]
    vp, vs = phi.var(1), psi.var(1)
    xi = psi - phi
    cov = ((phi - phi.mean(1, True)) * (xi - xi.mean(1, True))).sum(1) / (N - 1)
    vx = xi.var(1)
    return dict(mean_phi=phi.mean(1), var_phi=vp, mean_cv=psi.mean(1), var_cv=vs, cov_phi_xi=cov,
                var_xi=vx, rho=cov / torch.sqrt(vp * vx), se_phi=torch.sqrt(vp / N),
                se_cv=torch.sqrt(vs / N), vr=vs / vp, pred_speedup=vp / vs, mean_steps=k.mean(1),
                n_paths=None, n_truncated=None)


def exact(case, seed):
    """Algorithm 1 in 64 bits on the same streams, where that is quick."""
    nodes, rng_seed, parts = _inputs(case, seed)
    call, n_h = case["call"], case["parts"]
    if call == "fit":
        parts = [dict(parts[0], dt=10 * case["dt"] - 9 * case["dt"] * j / (n_h - 1), tag=j)
                 for j in range(n_h)]
    dt = min(p["dt"] for p in parts) / (2 if call == "coupled" else 1)
    batches = [[p] for p in parts] if call == "cascade" else [parts]
    if _steps(case) > 4e8 or MEAN_TAU[case["problem"]] / dt > 1001:
        return None
    got = []
    for batch in batches:
        eps = max(p["eps"] for p in batch)
        r = _simulate(case["problem"], nodes, batch, rng_seed,
                      _table(_grid(case, eps)) if eps else None, call == "coupled")
        got += [_moments(s[0], s[0] + s[1], s[2]) for s in r[0]]
        if call == "coupled":
            (f,), (c,) = r
            got.append(_moments(f[0] - c[0], (f[0] + f[1]) - (c[0] + c[1]), c[2]))
    if call == "fit":
        rows = [torch.stack([torch.full_like(m["rho"], p["dt"]), m["mean_phi"], m["var_phi"],
                             m["mean_steps"] * p["dt"], m["cov_phi_xi"], m["var_xi"]], 1)
                for m, p in zip(got, parts)]
        return {**{f: None for f in pdd.FIT_FIELDS}, "cloud": torch.stack(rows, 1)}
    if call in ("cascade", "coupled"):
        return got
    return {f: None if got[0][f] is None else torch.cat([g[f] for g in got]) for f in FIELDS}
