"""A solve whose first step after a restart to the average is not finite: the
reported point is the restart point, which has been formed once."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import instances as I
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu

K = 16
# Fixed restarts to the average at every check; a smoothing exponent that makes
# the primal weight infinite at the first restart (||dy|| > ||dX|| there).
OPTS = dict(restart_check_every=K, adaptive_restart=0, beta=1e30, theta=1e4)


@pytest.mark.parametrize("coop", ["0", "1"])
@pytest.mark.parametrize("xt", [pdot.F32, pdot.F64])
@pytest.mark.parametrize("batch", [False, True])
def test_first_step_after_a_restart_is_not_finite(monkeypatch, coop, xt, batch):
    monkeypatch.setenv("PDOT_COOP", coop)
    ins = I.points_instance(90, 130, I.seed_for(0, 5))
    C = torch.tensor(ins.C, dtype=torch.float64 if xt == pdot.F64 else torch.float32, device="cuda:0")

    def run(**o):
        if not batch:
            s = pdot.Solver(device=0, x_dtype=xt, **OPTS, **o)
            sol = s.solve(C, ins.f, ins.g, tol=1e-12)
        else:
            s = pdot.BatchSolver(device=0, x_dtype=xt, **OPTS, **o)
            s.submit(C, ins.f, ins.g, tol=1e-12)
            (sol,) = s.run().values()
        s.close()
        return sol

    at = run(max_iter=K)   # stopped at that check: reports the average
    assert at.status == pdot.MAX_ITER and at.result["returned_average"] == 1
    sol = run(max_iter=8 * K)
    assert sol.status == pdot.ERR_NUMERIC and sol.result["restarts"] == 1 and sol.result["passes"] == K + 1
    assert torch.equal(sol.X, at.X) and torch.equal(sol.p, at.p) and torch.equal(sol.q, at.q)
