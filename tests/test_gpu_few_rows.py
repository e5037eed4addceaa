"""Plans of a few long rows in the cooperative kernel: CTAs that hold vector tiles
but no plan tile, as many vector tiles as CTAs and more than the device holds
CTAs.  The same bits as an iteration of two kernels."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(1, 300), (1, 5000), (2, 9700), (3, 20001), (21, 4096)])
@pytest.mark.parametrize("cost", ["f32", "points"])
@pytest.mark.parametrize("comp", [0, 1])
def test_steps_equal_two_kernels(monkeypatch, m, n, cost, comp):
    r = np.random.default_rng(m + n)
    xs, ys = (torch.tensor(r.random((k, 2)), dtype=torch.float32, device="cuda:0") for k in (m, n))
    C = pdot.Points(xs, ys, "l1") if cost == "points" else (xs[:, None] - ys[None]).abs().sum(2)
    f, g = (v / v.sum() for v in (r.random(m) + 0.1, r.random(n) + 0.1))
    X = np.outer(f, g).astype(np.float32)
    out = []
    for coop in ("0", "1"):
        monkeypatch.setenv("PDOT_COOP", coop)
        s = pdot.Solver(device=0, compensated_cost=comp)
        out.append(s.pdhg_steps(C, f, g, X, np.zeros(m), np.zeros(n), k=11, eta=0.5 / np.sqrt(m + n)))
        s.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
