"""Vector tiles that two CTAs update by halves (csrc/pdot_persist.cuh) give the
same bits as the dual-update kernel, which takes whole tiles."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import instances as I
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


# around 32 partial sums per column (tiles of two rows); a tile with rows and
# columns and none; one column; a last tile of one entry; the longest sums;
# the most CTAs that all halves fit, and more halves than CTAs
@pytest.mark.parametrize("m,n", [(62, 64), (64, 64), (66, 64), (96, 65), (127, 33), (64, 1), (1137, 155), (1024, 1024),
                                 (2000, 97), (300, 2600), (300, 4000)])
def test_halves_equal_whole_tiles(monkeypatch, m, n):
    ins = I.points_instance(m, n, I.seed_for(0, m + 3 * n))
    C = torch.tensor(ins.C, dtype=torch.float32, device="cuda:0")
    got = []
    for coop in ("0", "1"):
        monkeypatch.setenv("PDOT_COOP", coop)
        s = pdot.Solver(device=0, compensated_cost=1, max_iter=192)
        sol = s.solve(C, ins.f, ins.g, tol=1e-9)
        X = torch.tensor(np.outer(ins.f, ins.g), dtype=torch.float32, device="cuda:0")
        st = s.pdhg_steps(C, ins.f, ins.g, X, np.zeros(m), np.zeros(n), k=5, eta=0.5 / np.sqrt(m + n))
        got.append((sol, st))
        s.close()
    (a, sa), (b, sb) = got
    for k in ("passes", "iters", "restarts", "rejected_steps", "eta", "omega", "rel_kkt"):
        assert a.result[k] == b.result[k] or a.result[k] != a.result[k], k
    assert torch.equal(a.X, b.X) and torch.equal(a.p, b.p) and torch.equal(a.q, b.q)
    for x, y in zip(sa, sb):
        assert torch.equal(x, y)
