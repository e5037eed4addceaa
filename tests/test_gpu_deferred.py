"""Deferred plan writes (csrc/pdot_pass.cuh): the plan pass leaves up to three
accepted steps unapplied in the stored plan and recomputes them from the
entries it reads.  Checked against the oracle after every number of steps a
cycle can end at, at the edges of its tiles, groups and strips."""
import numpy as np
import pytest
import torch

import oracle
from paper_2407_19689_gb300 import instances as I
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu

# rows: one, fewer than a group of four, a ragged last group; columns: one, a
# ragged lane, the last lane of a strip, the first of the next
SHAPES = [(1, 1), (1, 130), (3, 5), (7, 127), (9, 128), (66, 129), (130, 257)]


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 7])
@pytest.mark.parametrize("kernel,cost", [(2, "f32"), (3, "f32"), (3, "bf16")])
def test_every_cycle_position_matches_oracle(m, n, k, kernel, cost):
    ins = I.points_instance(m, n, I.seed_for(0, 7 * m + n))
    C = torch.tensor(ins.C, dtype=torch.float32, device="cuda:0")
    if cost == "bf16":
        C = C.bfloat16()
    r = np.random.default_rng(m + n)
    X, p, q = np.outer(ins.f, ins.g).astype(np.float32), 0.1 * r.random(m), 0.1 * r.random(n)
    eta = 0.5 / np.sqrt(m + n)
    s = pdot.Solver(device=0, pass_kernel=kernel)
    got = s.pdhg_steps(C, ins.f, ins.g, X, p, q, k=k, eta=eta)
    s.close()
    want = oracle.pdhg_steps(C.double().cpu().numpy(), ins.f, ins.g, X.astype(np.float64), p, q, k=k, eta=eta)
    # FP32 entries of size <= ~1 with a few roundings of 6e-8 per step, seven
    # steps at most: 1e-5 of the largest entry leaves a factor of ten.
    for a, b in zip(got, want):
        a = a.double().cpu().numpy()
        assert np.abs(a - b).max() <= 1e-5 * max(np.abs(b).max(), 1e-30)


@pytest.mark.parametrize("tile_rows", [2, 6, 34, 64])
def test_row_order_changes_no_more_than_rounding(tile_rows):
    """Rows in order and groups in order (bottom-up passes differ in the order
    of the FP32 column sums only) over tiles whose 32-row sums end inside a
    group, with adaptive steps, a restart check and a rejected step's path."""
    ins = I.points_instance(101, 140, I.seed_for(0, 5))
    C = torch.tensor(ins.C, dtype=torch.float32, device="cuda:0")
    sols = []
    for kernel in (2, 3):
        s = pdot.Solver(device=0, pass_kernel=kernel, tile_rows=tile_rows, max_iter=64)
        sols.append(s.solve(C, ins.f, ins.g, tol=1e-9))
        s.close()
    k = oracle.kkt(C.double().cpu().numpy(), ins.f, ins.g, sols[0].X.double().cpu().numpy(), sols[0].p.cpu().numpy(),
                   sols[0].q.cpu().numpy())
    # The reported measures are those of the returned plan (one that was not
    # written back in full would miss by whole steps).
    assert abs(k.rel_kkt - sols[0].result["rel_kkt"]) <= 1e-4 * k.rel_kkt
    # 64 adaptive passes amplify a rounding of 6e-8 by about 1e4.
    assert float((sols[0].X - sols[1].X).norm() / sols[0].X.norm()) < 1e-2
