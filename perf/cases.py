"""The work that users of this library have it do, as cases to be timed.

A case is one call (or one batch of calls) through the public Python API on
inputs that live on the GPU:

- ``solve``: ``Solver.solve`` with a pass budget (``max_iter``): restarted PDHG
  with the adaptive step, restarts, primal weight and checks that every solve
  runs.  A solve to tolerance takes thousands of such passes; the budget keeps
  a case short and its work the same for every input.
- ``steps``: ``Solver.pdhg_steps``, the inner iterations of such a solve alone,
  at a constant step.
- ``batch``: ``BatchSolver.submit`` for a mix of uneven instances, then ``run``.
- ``kkt``: ``Solver.kkt``, the error measures of a plan and its duals.
- ``round``: ``Solver.round``, Algorithm 3 (a feasible plan from an iterate).
- ``bound``: ``Solver.dual_bound``, the certified lower bound of a row dual.

The inputs follow the repository's generators: point clouds in the unit cube
with uniform marginals, pixel grids with blob marginals (the paper's image
workloads: 32 x 32, 64 x 64 and 128 x 128 pixels, so 1024, 4096 and 16384 rows
and columns), and log-uniform mixes of sizes with Dirichlet marginals.
"""
import math

import numpy as np
import torch

from paper_2407_19689_gb300 import instances, pdot

DEV = "cuda:0"


def listed():
    return [
        # the smallest problem of the configurations: 64 points against 64, an iteration is pure latency
        dict(name="steps_points64", kind="steps", cost="f32", shape="points", m=64, n=64, d=2, dist="sqeuclid",
             passes=256),
        # a ragged rectangle with the L1 cost in three dimensions
        dict(name="steps_rect", kind="steps", cost="f32", shape="points", m=517, n=301, d=3, dist="l1", passes=256),
        # 32 x 32 images, the paper's smallest: a whole call
        dict(name="solve_grid32", kind="solve", cost="f32", shape="grid", m=1024, n=1024, d=2, dist="sqeuclid",
             passes=512, warm=False),
        # 64 x 64 images, the benchmark's headline workload: a whole call, and the iterations with the cost in the
        # other two storages that the library offers (BF16, and generated from the pixels' coordinates)
        dict(name="solve_grid64", kind="solve", cost="f32", shape="grid", m=4096, n=4096, d=2, dist="sqeuclid",
             passes=256, warm=False),
        dict(name="steps_grid64_bf16", kind="steps", cost="bf16", shape="grid", m=4096, n=4096, d=2, dist="sqeuclid",
             passes=128),
        dict(name="steps_grid64_points", kind="steps", cost="points", shape="grid", m=4096, n=4096, d=2,
             dist="sqeuclid", passes=128),
        # 128 x 128 images: the largest configuration (1 GB of cost)
        dict(name="steps_grid128", kind="steps", cost="f32", shape="grid", m=16384, n=16384, d=2, dist="sqeuclid",
             passes=64),
        # double-precision plans, for a user who wants the objective to many digits
        dict(name="steps_f64", kind="steps", cost="f64", shape="points", m=600, n=801, d=2, dist="sqeuclid",
             passes=128),
        # uneven instances through the continuous-batching engine
        dict(name="batch16", kind="batch", cost="f32", count=16, lo=64, hi=2048, passes=256),
        # what follows a solve: its error measures, a feasible plan, and the certified bound
        dict(name="kkt_grid64", kind="kkt", cost="f32", shape="grid", m=4096, n=4096, d=2, dist="sqeuclid"),
        dict(name="round_grid64", kind="round", cost="f32", m=4096, n=4096),
        dict(name="bound_rect", kind="bound", cost="f32", shape="points", m=3000, n=2001, d=2, dist="sqeuclid"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    kind = rng.choice(["solve", "steps"])
    if u < 0.15:      # image pairs
        G = _log_int(rng, 20, 96)
        mn = G ** 4
        c = dict(kind=kind, cost=rng.choice(["f32", "f32", "points"]), shape="grid", m=G * G, n=G * G, d=2,
                 dist=rng.choice(["sqeuclid", "l1"]), passes=256 if mn <= 1 << 20 else 128 if mn <= 1 << 24 else 64)
    elif u < 0.55:    # point clouds, stored or generated costs
        cost = rng.choice(["f32", "f32", "bf16", "points"])
        m, n = _log_int(rng, 40, 4096), _log_int(rng, 40, 4096)
        c = dict(kind=kind, cost=cost, shape="points", m=m, n=n, d=rng.choice([2, 3, 8]),
                 dist=rng.choice(["sqeuclid", "l1"]), passes=256 if m * n <= 1 << 20 else 128)
    elif u < 0.65:    # double-precision plans
        c = dict(kind=kind, cost="f64", shape="points", m=_log_int(rng, 40, 1024), n=_log_int(rng, 40, 1024), d=2,
                 dist="sqeuclid", passes=128)
    if u < 0.65:
        return dict(c, warm=rng.random() < 0.3) if kind == "solve" else c
    if u < 0.75:
        return dict(kind="batch", cost=rng.choice(["f32", "bf16"]), count=rng.randint(6, 20), lo=64,
                    hi=_log_int(rng, 512, 2048), passes=256)
    m, n = _log_int(rng, 64, 8192), _log_int(rng, 64, 8192)
    if u < 0.85:
        return dict(kind="round", cost=rng.choice(["f32", "f32", "f64"]), m=m, n=n)
    kind = "kkt" if u < 0.93 else "bound"
    return dict(kind=kind, cost=rng.choice(["f32", "f32", "bf16", "points"]), shape="points", m=m, n=n,
                d=rng.choice([2, 3]), dist=rng.choice(["sqeuclid", "l1"]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _distances(xs, ys, dist):
    """FP32 distances, coordinates accumulated in order."""
    acc = None
    for k in range(xs.shape[1]):
        t = xs[:, k, None] - ys[None, :, k]
        t = t.mul_(t) if dist == "sqeuclid" else t.abs_()
        acc = t if acc is None else acc.add_(t)
    return acc


def _points(case, seed):
    """Coordinates, marginals and the divisor of the cost (the largest distance on a grid)."""
    m, n = case["m"], case["n"]
    if case["shape"] == "grid":
        G = math.isqrt(m)
        rng = np.random.default_rng(seed)
        f, g = (torch.tensor(instances.blob_marginal(G, rng), device=DEV) for _ in range(2))
        xs = torch.tensor(instances.grid_coords(G), dtype=torch.float32, device=DEV)
        return xs, xs, f, g, float(2 * (G - 1) ** 2 if case["dist"] == "sqeuclid" else 2 * (G - 1))
    r = _gen(seed)
    xs = torch.rand((m, case["d"]), device=DEV, generator=r)
    ys = torch.rand((n, case["d"]), device=DEV, generator=r)
    f = 0.1 + 0.9 * torch.rand(m, device=DEV, dtype=torch.float64, generator=r)
    g = 0.1 + 0.9 * torch.rand(n, device=DEV, dtype=torch.float64, generator=r)
    return xs, ys, f / f.sum(), g / g.sum(), 1.0


def _instance(case, seed):
    """(cost as the caller holds it, f, g)"""
    xs, ys, f, g, div = _points(case, seed)
    if case["cost"] == "points":
        return pdot.Points(xs, ys, case["dist"], div), f, g
    if case["cost"] == "f64":
        C = _distances(xs.double(), ys.double(), case["dist"])
    else:
        C = _distances(xs, ys, case["dist"])
    if div != 1.0:
        C.div_(div)
    return (C.bfloat16() if case["cost"] == "bf16" else C), f, g


def _batch(case, seed):
    """Uneven point clouds with Dirichlet(1) marginals; the sizes of a case are the same for every seed."""
    out = []
    rng = np.random.default_rng(seed)
    for m, n in instances.batch_sizes(case["count"], case["count"] * 7 + case["hi"], case["lo"], case["hi"]):
        xs, ys = (torch.tensor(rng.random((k, 2)), dtype=torch.float32, device=DEV) for k in (m, n))
        f, g = (torch.tensor(rng.dirichlet(np.ones(k)), device=DEV) for k in (m, n))
        C = _distances(xs, ys, "sqeuclid")
        out.append((C.bfloat16() if case["cost"] == "bf16" else C, f / f.sum(), g / g.sum()))
    return out


def _plan(m, n, f, g, dtype, r):
    """An iterate late in a solve: about a third of the entries positive, marginals a few per cent off."""
    X = torch.rand((m, n), device=DEV, generator=r)
    X = (X - 0.65).clamp_(min=0.0).mul_(2.0 / 0.35 ** 2)
    X.mul_((f[:, None] * (0.97 + 0.06 * torch.rand((m, 1), device=DEV, generator=r))).float()).mul_(g[None, :].float())
    return X.to(dtype)


def _duals(m, n, r):
    return [0.2 * torch.rand(k, device=DEV, dtype=torch.float64, generator=r) - 0.05 for k in (m, n)]


def prepare(case, seed):
    kind, xt = case["kind"], pdot.F64 if case["cost"] == "f64" else pdot.F32
    st = {"kind": kind}
    if kind == "batch":
        st["solver"] = pdot.BatchSolver(device=0, tol=1e-9, max_iter=case["passes"])
        st["requests"] = _batch(case, seed)
        return st
    if kind == "solve":
        st["solver"] = pdot.Solver(device=0, x_dtype=xt, tol=1e-9, max_iter=case["passes"])
        st["C"], st["f"], st["g"] = _instance(case, seed)
        st["start"] = _start(st["f"], st["g"], xt) if case["warm"] else {}
        return st
    if kind == "steps":   # from the product plan, at the step of Theorem 1
        st["solver"] = pdot.Solver(device=0, x_dtype=xt)
        st["C"], st["f"], st["g"] = _instance(case, seed)
        st["start"] = _start(st["f"], st["g"], xt)
        st["k"], st["eta"] = case["passes"], 0.5 / math.sqrt(case["m"] + case["n"])
        return st
    st["solver"] = pdot.Solver(device=0, x_dtype=xt)
    m, n = case["m"], case["n"]
    r = _gen(seed + 1)
    if kind == "round":
        f, g = (0.1 + 0.9 * torch.rand(k, device=DEV, dtype=torch.float64, generator=r) for k in (m, n))
        st["f"], st["g"] = f / f.sum(), g / g.sum()
        st["X"] = _plan(m, n, st["f"], st["g"], torch.float64 if xt == pdot.F64 else torch.float32, r)
        return st
    st["C"], st["f"], st["g"] = _instance(case, seed)
    st["p"], st["q"] = _duals(m, n, r)
    if kind == "kkt":
        st["X"] = _plan(m, n, st["f"], st["g"], torch.float32, r)
    return st


def _start(f, g, xt):
    X = (f[:, None] * g[None, :]).to(torch.float64 if xt == pdot.F64 else torch.float32)
    return dict(X0=X, p0=torch.zeros_like(f), q0=torch.zeros_like(g))


def run(state):
    s, kind = state["solver"], state["kind"]
    if kind == "batch":
        ids = [s.submit(C, f, g) for C, f, g in state["requests"]]
        done = s.run()
        return [_solution(done[i]) for i in ids]
    if kind == "solve":
        return _solution(s.solve(state["C"], state["f"], state["g"], **state["start"]))
    if kind == "steps":
        s0 = state["start"]
        return s.pdhg_steps(state["C"], state["f"], state["g"], s0["X0"], s0["p0"], s0["q0"], state["k"],
                            state["eta"])
    if kind == "kkt":
        return s.kkt(state["C"], state["f"], state["g"], state["X"], state["p"], state["q"])
    if kind == "round":
        return s.round(state["X"], state["f"], state["g"])
    lower, q = s.dual_bound(state["C"], state["f"], state["g"], state["p"])
    return {"lower": lower, "q": q}


def _solution(sol):
    return {"X": sol.X, "p": sol.p, "q": sol.q}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
ON_CHIP = 126e6       # bytes that can stay in the last-level cache from pass to pass


def _solve_work(m, n, cost, passes):
    """The cost and the plan are read once and the plan written once; where the two together do not fit on the chip,
    every pass has to read them (the plan's next value can be recomputed, but not without them).  Ten operations per
    entry and pass: the reduced cost, the projection, the change, its square and its row and column sums."""
    c, x = {"f32": 4, "bf16": 2, "f64": 8, "points": 0}[cost], 8 if cost == "f64" else 4
    once = m * n * (c + x) + 32 * (m + n)
    each = m * n * (c + x) if m * n * (c + x) > ON_CHIP else 0
    return {"bytes": once + each * passes, "flops": 10.0 * m * n * passes}


def work(case):
    if case["kind"] == "batch":
        sizes = instances.batch_sizes(case["count"], case["count"] * 7 + case["hi"], case["lo"], case["hi"])
        w = [_solve_work(m, n, case["cost"], case["passes"]) for m, n in sizes]
        return {"bytes": sum(v["bytes"] for v in w), "flops": sum(v["flops"] for v in w)}
    m, n = case["m"], case["n"]
    if case["kind"] in ("solve", "steps"):
        return _solve_work(m, n, case["cost"], case["passes"])
    c = {"f32": 4, "bf16": 2, "f64": 8, "points": 0}[case["cost"]]
    if case["kind"] == "round":   # the plan in, the feasible plan out
        return {"bytes": 2 * m * n * c + 16 * (m + n), "flops": 8.0 * m * n}
    if case["kind"] == "kkt":
        return {"bytes": m * n * (c + 4) + 16 * (m + n), "flops": 9.0 * m * n}
    return {"bytes": m * n * c + 16 * m + 24 * n, "flops": 2.0 * m * n}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _cost64(C):
    if isinstance(C, pdot.Points):
        return _distances(C.xs.double(), C.ys.double(), C.dist).div_(C.divisor)
    return C.double()


def _kkt64(C, f, g, X, p, q):
    """Error measures of Sec. 3.1 and their relative forms."""
    r, c = X.sum(1), X.sum(0)
    rp2 = ((r - f) ** 2).sum() + ((c - g) ** 2).sum()
    rd2 = torch.linalg.vector_norm((p[:, None] - C).add_(q[None, :]).clamp_(min=0.0)) ** 2
    cx = torch.dot(C.reshape(-1), X.reshape(-1))
    dual = (f * p).sum() + (g * q).sum()
    rp2, rd2, cx, dual = (float(v) for v in (rp2, rd2, cx, dual))
    gap = cx - dual
    nb = math.sqrt(float((f * f).sum() + (g * g).sum())) or 1.0
    nc = float(torch.linalg.vector_norm(C)) or 1.0
    rel = dict(rel_p=math.sqrt(rp2) / nb, rel_d=math.sqrt(rd2) / nc, rel_gap=abs(gap) / ((abs(cx) + abs(dual)) or 1.0))
    return dict(rp2=rp2, rd2=rd2, cx=cx, dual=dual, gap=gap, kkt=math.sqrt(rp2 + rd2 + gap * gap), **rel,
                rel_kkt=max(rel.values()))


def _steps64(C, f, g, X, p, q, k, eta):
    """k iterations of Algorithm 2 at a constant step, and the average of the iterates."""
    X = X.double()
    Xb, Xn = torch.zeros_like(X), torch.empty_like(X)
    pb, qb = torch.zeros_like(p), torch.zeros_like(q)
    r, c = X.sum(1), X.sum(0)
    for t in range(1, k + 1):
        torch.sub(C, p[:, None], out=Xn).sub_(q[None, :]).mul_(-eta).add_(X).clamp_(min=0.0)
        X, Xn = Xn, X
        rn, cn = X.sum(1), X.sum(0)
        p, q, r, c = p + eta * (f - (2 * rn - r)), q + eta * (g - (2 * cn - c)), rn, cn
        Xb.lerp_(X, 1.0 / t)
        pb, qb = pb + (p - pb) / t, qb + (q - qb) / t
    return X, p, q, Xb, pb, qb


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "batch"):
        # The step rule and the restarts branch on the iterates: a last-bit difference grows by about ten orders of
        # magnitude in 256 passes, in double precision too, so such a call has no value to be near to.
        return None
    st = prepare(case, seed)
    if kind == "steps":
        s0 = st["start"]
        return _steps64(_cost64(st["C"]), st["f"], st["g"], s0["X0"], s0["p0"], s0["q0"], st["k"], st["eta"])
    f, g = st["f"], st["g"]
    if kind == "kkt":
        C = _cost64(st["C"])
        return _kkt64(C, f, g, st["X"].double(), st["p"], st["q"])
    if kind == "round":   # Algorithm 3
        X = st["X"].double()
        X *= torch.clamp(f / X.sum(1), max=1.0)[:, None]
        X *= torch.clamp(g / X.sum(0), max=1.0)[None, :]
        er, ec = f - X.sum(1), g - X.sum(0)
        return X.addr_(er, ec, alpha=1.0 / float(er.abs().sum()))
    q = (_cost64(st["C"]) - st["p"][:, None]).amin(0)
    return {"lower": float((f * st["p"]).sum() + (g * q).sum()), "q": q}
