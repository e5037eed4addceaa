"""Rounding of FP32 plans whose scales leave the range of an FP32 pair: row
scales f_i / (X 1)_i, column scales and error scales far below FP32's smallest
numbers, with entries so large that the products are ordinary numbers; column
errors beyond its largest.  And marginals that are not finite, and the FP64 sum
of the objective."""
import numpy as np
import pytest
import torch

import oracle
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


def _case(kind, m, n):
    r = np.random.default_rng(m + n)
    X = r.uniform(0.5, 1.5, (m, n)).astype(np.float32).astype(np.float64)
    f, g = r.uniform(0.5, 1.5, m), r.uniform(0.5, 1.5, n)
    f, g = f / f.sum(), g / g.sum()
    if kind == "rows":          # all row scales about 1e-46
        X, f, g = X * 1e22, f * 1e-24, g * 1e-24
    elif kind == "one_row":     # one row scale of about 1e-46, beside ordinary ones
        f[m // 2] *= 1e-46
    elif kind == "columns":     # all column scales but one about 1e-46
        X, f, g = X * 1e22, f * 1e22, g * 1e-24
        g[n // 2] = f.sum()
    elif kind == "errors":      # err_r of one row against all: about 1e-45
        X, f, g = X * 1e-30, f * 1e-25, g * 1e20
        f[m // 2] = 1e20
    elif kind == "beyond":      # column errors beyond FP32, entries within it
        g = np.full(n, 1e39)
        f = np.full(m, n * 1e39 / m)
    X = X.astype(np.float32).astype(np.float64)
    return X, f, g


@pytest.mark.parametrize("kind", ["rows", "one_row", "columns", "errors", "beyond"])
@pytest.mark.parametrize("m,n", [(6, 6), (70, 1030), (2500, 36)])
def test_round_with_tiny_scales(kind, m, n):
    X, f, g = _case(kind, m, n)
    want = oracle.round_plan(X, f, g)
    s = pdot.Solver(device=0)
    got = s.round(torch.tensor(X, device="cuda:0", dtype=torch.float32), f, g).double().cpu().numpy()
    s.close()
    # Every entry is the FP64 one rounded once (2^-24, or half of the smallest
    # FP32 number); the sums behind it differ by about 1e-12 of their terms'.
    scale = np.minimum(np.abs(want).max(axis=1, keepdims=True), np.abs(want).max(axis=0, keepdims=True))
    assert (np.abs(got - want) <= 1e-7 * scale + 1e-45).all()


@pytest.mark.parametrize("xt", [pdot.F32, pdot.F64])
@pytest.mark.parametrize("where", ["f", "g"])
def test_round_with_a_marginal_that_is_not_a_number(xt, where):
    """min(f / r, 1) of a NaN is NaN: it reaches the error terms of every row
    and column, so no entry of the plan looks like a rounded one."""
    X, f, g = _case("plain", 40, 300)
    (f if where == "f" else g)[7] = np.nan
    s = pdot.Solver(device=0, x_dtype=xt)
    got = s.round(torch.tensor(X, device="cuda:0"), f, g)
    s.close()
    assert got.isnan().all()


def test_rounded_objective_of_equal_terms():
    """<C, plan> of a constant plan and cost: the terms' rounding errors all have
    the same sign.  In FP64 a thread adds at most 264 terms (67 rows of four
    columns), a warp, block and the host 5 + 8 + 608 more sums, each of relative
    error 2^-53 at most."""
    m, n = 40000, 256
    f, g = np.full(m, 1 / m), np.full(n, 1 / n)
    X0 = torch.full((m, n), 1 / (m * n), dtype=torch.float32, device="cuda:0")
    s = pdot.Solver(device=0, round_plan=1)
    for c in (0.2718282, 0.5405107, 0.7697867, 0.8889214, 1.1231872, 1.4127556):
        C = torch.full((m, n), c, dtype=torch.float32, device="cuda:0")
        sol = s.solve(C, f, g, tol=1e9, X0=X0)   # (the start is accepted as it is)
        assert sol.result["passes"] == 0
        values, counts = sol.X.double().unique(return_counts=True)
        want = float(C[0, 0].double()) * float((values * counts).sum())
        assert abs(sol.result["rounded_obj"] - want) <= 900 * 2.0 ** -53 * want
    s.close()


def test_round_with_an_infinite_marginal():
    """Its column has an infinite error and infinite entries, as in FP64 (a pair's
    low part, inf - inf, made them not a number)."""
    X, f, g = _case("plain", 40, 300)
    g[7] = np.inf
    s = pdot.Solver(device=0)
    got = s.round(torch.tensor(X, device="cuda:0"), f, g).cpu().numpy()
    s.close()
    want = oracle.round_plan(X, f, g)
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
    np.testing.assert_array_equal(np.isinf(got), np.isinf(want))
