"""Batched instances in the cooperative kernel (several instances per launch,
csrc/pdot_persist.cuh) take the same operations in the same order as in the
tile kernels: results are equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import instances as I
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu

# one launch; more vector tiles than CTAs and ragged edges; three launches
# (the largest instance alone fills most of one); too many tiles for the kernel
SETS = {
    "small": [(1, 1), (5, 3), (64, 64), (130, 517), (70, 90)],
    "ragged": [(1, 4000), (3000, 2), (1021, 301), (257, 129), (16, 128), (17, 129)],
    "waves": [(1943, 1629), (1500, 1501), (722, 1358), (900, 901), (64, 700), (2000, 95)],
    "large": [(5000, 8200), (300, 301)],
}


def _instances(name, cost):
    out = []
    for k, (m, n) in enumerate(SETS[name]):
        ins = I.points_instance(m, n, I.seed_for(0, m + 3 * n))
        kind = cost if cost != "mix" else ("f32", "bf16", "points2")[k % 3]
        if kind.startswith("points"):
            r = np.random.default_rng(m)
            xs, ys = (torch.tensor(r.random((s, int(kind[6:]))), dtype=torch.float32, device="cuda:0") for s in (m, n))
            C = pdot.Points(xs, ys, "sqeuclid")
        else:
            C = torch.tensor(ins.C, dtype=torch.float32, device="cuda:0")
            C = C.bfloat16() if kind == "bf16" else C
        out.append((C, ins.f, ins.g))
    return out


@pytest.mark.parametrize("name,cost,comp", [("small", "f32", 1), ("small", "mix", 1), ("ragged", "f32", 1),
                                            ("ragged", "mix", 0), ("waves", "f32", 1), ("waves", "bf16", 0),
                                            ("waves", "mix", 1), ("ragged", "points3", 1), ("small", "points7", 1),
                                            ("large", "f32", 1)])
def test_batch_equals_tile_kernels(monkeypatch, name, cost, comp):
    insts = _instances(name, cost)
    got = []
    for coop in ("0", "1"):
        monkeypatch.setenv("PDOT_COOP", coop)
        b = pdot.BatchSolver(device=0, max_iter=192, tol=1e-9, compensated_cost=comp)
        ids = [b.submit(*x) for x in insts]
        done = b.run()
        got.append([done[i] for i in ids])
        b.close()
    for x, y in zip(*got):
        for k in ("status", "passes", "iters", "restarts", "rejected_steps", "eta", "rel_kkt"):
            assert x.result[k] == y.result[k] or x.result[k] != x.result[k], k
        assert torch.equal(x.X, y.X) and torch.equal(x.p, y.p) and torch.equal(x.q, y.q)
