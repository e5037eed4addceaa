"""The dual bound of generated costs: small and large matrices, coordinate counts
on both sides of the choice between one FP64 sweep and the FP32 screen, few and
many row groups.  Whole-number coordinates make the cost exact."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 3, 4, 5, 8])
@pytest.mark.parametrize("m,n", [(1, 1), (17, 300), (100000, 3), (1500, 1501), (3, 800000)])
def test_bound_is_exact(m, n, d):
    r = np.random.default_rng(m + n + d)
    xs, ys = (r.integers(0, 30, (k, d)) for k in (m, n))
    p = r.standard_normal(m) * 20
    C = sum(np.abs(xs[:, k, None] - ys[None, :, k]) for k in range(d))
    want = (C - p[:, None]).min(0)
    f, g = np.full(m, 1 / m), np.full(n, 1 / n)
    s = pdot.Solver(device=0)
    cost = pdot.Points(*(torch.tensor(v, dtype=torch.float32, device="cuda:0") for v in (xs, ys)), "l1")
    lower, q = s.dual_bound(cost, f, g, p)
    s.close()
    np.testing.assert_array_equal(q.cpu().numpy(), want)
    terms = np.concatenate([f * p, g * want])
    assert abs(lower - terms.sum()) <= 1e-13 * np.abs(terms).sum()


@pytest.mark.parametrize("m,n,d,launches", [(300, 200, 2, 2), (1500, 1501, 2, 3), (1500, 1501, 4, 2)])
def test_launches_are_counted_as_they_are_made(m, n, d, launches):
    """One sweep or two (see above), and the value."""
    s = pdot.Solver(device=0)
    xs, ys = (torch.rand((k, d), device="cuda:0") for k in (m, n))
    n0 = s.launch_count()
    s.dual_bound(pdot.Points(xs, ys), np.full(m, 1 / m), np.full(n, 1 / n), np.zeros(m))
    assert s.launch_count() - n0 == launches
    s.close()
