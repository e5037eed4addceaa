"""The dual bound's candidate sweep (csrc/pdot_round.cu): the FP64 minimum is
taken over the entries whose FP32 difference is within its rounding error of
the FP32 minimum, so it has to be exact whatever the duals' size, with ties,
near ties, infinities and every alignment."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu

CASES = ["plain", "ties", "near_ties", "large", "beyond_fp32", "tiny", "inf_cost", "minus_inf_cost", "nan_dual"]


@pytest.mark.parametrize("m,n,ldc", [(1, 1, 1), (5, 1023, 1023), (70, 1030, 1032), (4097, 6, 8), (300, 257, 301),
                                     (1100, 2030, 2032), (2101, 1003, 1003)])
@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("bf16", [False, True])
def test_bound_is_exact(m, n, ldc, case, bf16):
    r = np.random.default_rng(m + n)
    C = torch.tensor(r.random((m, ldc)), dtype=torch.bfloat16 if bf16 else torch.float32, device="cuda:0")
    p = r.standard_normal(m)
    if case == "ties":
        p = np.round(p)
        C = (C * 4).round()
    elif case == "near_ties":      # differences that agree to 2^-40
        C = torch.full_like(C, 0.75)
        p = 0.5 + r.standard_normal(m) * 2.0 ** -40
    elif case == "large":
        p = p * 1e12
    elif case == "beyond_fp32":
        p = p * 1e60
    elif case == "tiny":
        C = C * 1e-38
        p = p * 1e-42
    elif case == "inf_cost":
        C[r.integers(m), :] = float("inf")
        C[:, 0] = float("inf")
    elif case == "minus_inf_cost":
        C[r.integers(m), n // 2] = float("-inf")
    elif case == "nan_dual" and m > 1:
        p[r.integers(m)] = np.nan
    f, g = np.full(m, 1 / m), np.full(n, 1 / n)
    fd, gd, pd = (torch.tensor(v, device="cuda:0") for v in (f, g, p))
    q = torch.empty(n, dtype=torch.float64, device="cuda:0")
    s = pdot.Solver(device=0)
    st, lower = pdot.pdot_dual_bound(s.h, m, n, C.data_ptr(), pdot.BF16 if bf16 else pdot.F32, ldc, fd.data_ptr(),
                                     gd.data_ptr(), pd.data_ptr(), q.data_ptr())
    s.close()
    assert st == pdot.OK
    D = C[:, :n].double().cpu().numpy() - p[:, None]
    want = np.nanmin(np.where(np.isnan(D), np.inf, D), axis=0)   # (a NaN difference is never a minimum)
    np.testing.assert_array_equal(q.cpu().numpy(), want)
    if np.isfinite(want).all() and np.isfinite(p).all():
        terms = np.concatenate([f * p, g * want])
        assert abs(lower - terms.sum()) <= 1e-13 * np.abs(terms).sum()
