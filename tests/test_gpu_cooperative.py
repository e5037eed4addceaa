"""The cooperative kernel (csrc/pdot_persist.cuh: all passes of a check period
in one launch) takes the same operations in the same order as an iteration of
two kernels, so results are equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import instances as I
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


def _two(monkeypatch, **opts):
    """A solver whose iterations are two kernels, and one with the cooperative kernel."""
    monkeypatch.setenv("PDOT_COOP", "0")
    a = pdot.Solver(device=0, **opts)
    monkeypatch.setenv("PDOT_COOP", "1")
    return a, pdot.Solver(device=0, **opts)


def _cost(ins, cost, seed):
    if cost.startswith("points"):
        d = int(cost[6:])
        r = np.random.default_rng(seed)
        xs, ys = (torch.tensor(r.random((k, d)), dtype=torch.float32, device="cuda:0") for k in ins.C.shape)
        return pdot.Points(xs, ys, "sqeuclid")
    C = torch.tensor(ins.C, dtype=torch.float32, device="cuda:0")
    return C.bfloat16() if cost == "bf16" else C


# one entry; fewer tiles than a CTA's warps; ragged columns and rows; tiles of
# 4 rows, of more rows than stay in shared memory with the compensated cost (8)
# and without it (12), and more vector tiles than CTAs
SHAPES = [(1, 1), (5, 3), (64, 64), (130, 517), (1021, 301), (1300, 1311), (2050, 1030), (40, 9000), (2300, 2001)]


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("cost", ["f32", "bf16", "points2", "points3", "points7"])
@pytest.mark.parametrize("comp", [0, 1])
def test_steps_equal_two_kernels(monkeypatch, m, n, cost, comp):
    ins = I.points_instance(m, n, I.seed_for(0, m + 3 * n))
    C = _cost(ins, cost, m)
    X = np.outer(ins.f, ins.g).astype(np.float32)
    out = []
    for s in _two(monkeypatch, compensated_cost=comp):
        for k in (1, 11):
            out.append(s.pdhg_steps(C, ins.f, ins.g, X, np.zeros(m), np.zeros(n), k=k, eta=0.5 / np.sqrt(m + n)))
        s.close()
    for a, b in zip(out[0] + out[1], out[2] + out[3]):
        assert torch.equal(a, b)


@pytest.mark.parametrize("m,n,cost", [(64, 64, "f32"), (300, 517, "f32"), (1200, 900, "bf16"), (2304, 2304, "f32"),
                                      (2304, 2304, "points2"), (5776, 5776, "f32")])
def test_adaptive_solve_equals_two_kernels(monkeypatch, m, n, cost):
    """Accepted and rejected steps, restarts to the current point and to the
    average, and the checks between launches."""
    if m == n and m > 2000:
        G = int(round(m ** 0.5))
        ins = I.grid_blob_instance(G, I.seed_for(1, G), build_cost=False)
        P = torch.tensor(I.grid_coords(G), dtype=torch.float32, device="cuda:0")
        C = pdot.Points(P, P, "sqeuclid", float(2 * (G - 1) ** 2))
        if cost == "f32":
            C = ((P[:, None, 0] - P[None, :, 0]) ** 2 + (P[:, None, 1] - P[None, :, 1]) ** 2) / C.divisor
    else:
        ins = I.points_instance(m, n, I.seed_for(0, m + n))
        C = _cost(ins, cost, m)
    sols = []
    for s in _two(monkeypatch, max_iter=448):
        sols.append(s.solve(C, ins.f, ins.g, tol=1e-9))
        s.close()
    a, b = sols
    for k in ("passes", "iters", "restarts", "rejected_steps", "eta", "omega", "rel_kkt"):
        assert a.result[k] == b.result[k], k
    assert a.result["restarts"] > 0
    assert torch.equal(a.X, b.X) and torch.equal(a.p, b.p) and torch.equal(a.q, b.q)


@pytest.mark.parametrize("coop", ["0", "1"])
def test_numeric_failure_returns_the_last_accepted_plan(monkeypatch, coop):
    """A start of 1e25 leaves the plan as it is in the first step (which is
    accepted) and overflows the second one's change: the solve ends with the
    numeric status and the plan after the first step, pending or written."""
    monkeypatch.setenv("PDOT_COOP", coop)
    m, n = 70, 90
    X0 = torch.full((m, n), 1e25, device="cuda:0")
    C = torch.rand((m, n), device="cuda:0")
    f, g = np.full(m, 1 / m), np.full(n, 1 / n)
    s = pdot.Solver(device=0, max_iter=128)
    sol = s.solve(C, f, g, tol=1e-9, X0=X0)
    assert sol.status == pdot.ERR_NUMERIC and sol.result["iters"] == 1
    assert torch.equal(sol.X, X0)
    assert s.solve(C, f, g, tol=1e-2).status in (pdot.OK, pdot.MAX_ITER)   # the handle stays usable
    s.close()
