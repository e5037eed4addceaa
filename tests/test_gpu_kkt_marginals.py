"""pdot_kkt refuses invalid marginals (tested on the device) and says why."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what,text", [("negative f", "f has a negative"), ("nan g", "g has a negative or non-finite"),
                                       ("inf f", "f has a negative or non-finite"), ("sums", "sum(f) != sum(g)")])
def test_invalid_marginals(what, text):
    m, n = 30, 50
    f, g = np.full(m, 1 / m), np.full(n, 1 / n)
    if what == "negative f":
        f[3] = -f[3]
    elif what == "nan g":
        g[n - 1] = np.nan
    elif what == "inf f":
        f[0] = np.inf
    else:
        g *= 1 + 1e-6
    C = torch.rand((m, n), device="cuda:0")
    s = pdot.Solver(device=0)
    with pytest.raises(pdot.PdotError) as e:
        s.kkt(C, f, g, torch.zeros((m, n), device="cuda:0"), np.zeros(m), np.zeros(n))
    assert e.value.status == pdot.ERR_ARG and text in str(e.value)
    s.kkt(C, np.full(m, 1 / m), np.full(n, 1 / n), torch.zeros((m, n), device="cuda:0"), np.zeros(m), np.zeros(n))
    s.close()
