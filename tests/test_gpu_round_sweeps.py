"""The rounding's sweeps (csrc/pdot_round.cu): aligned and unaligned rows, a
warp or a block per row, many and few row groups, in place, and plans whose
sums leave FP32's range, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (1, 5000), (5000, 1), (3, 4), (33, 127), (17, 1030), (700, 1028), (2433, 260), (130, 8192), (64, 8195)]


def _plan(m, n, seed, scale=1.0):
    r = np.random.default_rng(seed)
    f, g = r.random(m) + 0.1, r.random(n) + 0.1
    f, g = f / f.sum(), g / g.sum()
    X = np.outer(f, g) * scale * r.uniform(0.5, 1.6, (m, n)) * (r.random((m, n)) < 0.7)
    return X, f, g


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("xt", [pdot.F32, pdot.F64])
@pytest.mark.parametrize("inplace", [False, True])
def test_round_matches_oracle(m, n, xt, inplace):
    X, f, g = _plan(m, n, m + n)
    Xd = torch.tensor(X, device="cuda:0", dtype=torch.float64 if xt == pdot.F64 else torch.float32)
    want = oracle.round_plan(Xd.double().cpu().numpy(), f, g)
    s = pdot.Solver(device=0, x_dtype=xt)
    if inplace:
        fd, gd = (torch.tensor(v, device="cuda:0") for v in (f, g))
        assert pdot.pdot_round(s.h, m, n, Xd.data_ptr(), fd.data_ptr(), gd.data_ptr(), Xd.data_ptr()) == pdot.OK
        got = Xd
    else:
        got = s.round(Xd, f, g)
    s.close()
    # FP32: each entry is the exact one rounded once (2^-24) and the pairs'
    # error far below it; FP64: a few roundings of sums of at most 8192 terms.
    tol = 1e-7 if xt == pdot.F32 else 1e-12
    assert np.abs(got.double().cpu().numpy() - want).max() <= tol * np.abs(want).max()


def test_round_beyond_fp32_sums():
    """Row sums of about 1e38 (the pairs would overflow): FP64 arithmetic."""
    m, n = 40, 300
    X, f, g = _plan(m, n, 3, scale=1e38 * m * n / 8)
    Xd = torch.tensor(X.clip(max=3e38), device="cuda:0", dtype=torch.float32)
    want = oracle.round_plan(Xd.double().cpu().numpy(), f, g)
    s = pdot.Solver(device=0)
    got = s.round(Xd, f, g).double().cpu().numpy()
    s.close()
    assert np.abs(got - want).max() <= 1e-7 * np.abs(want).max()


@pytest.mark.parametrize("cost", ["f32", "bf16", "points"])
def test_rounded_objective(cost):
    m, n = 150, 205
    r = np.random.default_rng(1)
    xs, ys = (torch.tensor(r.random((k, 2)), dtype=torch.float32, device="cuda:0") for k in (m, n))
    f, g = (v / v.sum() for v in (r.random(m) + 0.1, r.random(n) + 0.1))
    C = ((xs[:, None] - ys[None]) ** 2).sum(2)
    arg = pdot.Points(xs, ys) if cost == "points" else C.bfloat16() if cost == "bf16" else C
    Cd = (C.bfloat16() if cost == "bf16" else C).double().cpu().numpy()
    s = pdot.Solver(device=0, round_plan=1, max_iter=256)
    sol = s.solve(arg, f, g, tol=1e-9)
    s.close()
    want = float((Cd * sol.X.double().cpu().numpy()).sum())
    # The stored cost is exact; the generated one differs from torch's by a few FP32 roundings.
    assert abs(sol.result["rounded_obj"] - want) <= (1e-6 if cost == "points" else 1e-12) * want
