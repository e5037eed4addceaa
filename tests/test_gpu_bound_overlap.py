"""The bound's column dual written over one of its own inputs."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", ["p", "f", "g", "p_shifted"])
@pytest.mark.parametrize("n", [700, 20000])
def test_q_over_an_input(over, n):
    m = n if n == 700 else n + 40
    r = np.random.default_rng(n)
    xs, ys = (torch.tensor(r.random((k, 1)), dtype=torch.float32, device="cuda:0") for k in (m, n))
    cost = pdot.Points(xs, ys, "l1")
    f, g, p = np.full(m, 1 / m), np.full(n, 1 / n), r.standard_normal(m)
    s = pdot.Solver(device=0)
    lower, q = s.dual_bound(cost, f, g, p)
    c, fd, gd = s._prep(cost, f, g)
    buf = torch.empty(m + 8, dtype=torch.float64, device="cuda:0")
    pd = buf[4:4 + m]
    pd.copy_(torch.tensor(p))
    torch.cuda.synchronize()
    out = {"p": pd, "f": fd, "g": gd, "p_shifted": buf[1:]}[over]
    st, got = pdot.pdot_dual_bound(s.h, m, n, c.ptr, c.dtype, c.ldc, fd.data_ptr(), gd.data_ptr(), pd.data_ptr(),
                                   out.data_ptr())
    s.close()
    assert st == pdot.OK and got == lower
    assert torch.equal(out[:n], q)
