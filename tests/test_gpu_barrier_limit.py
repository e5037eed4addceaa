"""The cooperative kernel's barrier gives up: with one poll per barrier, a call
whose instance has many CTAs ends with the device status, and an instance of
one CTA, which meets nobody, is solved on the same handle as on any other."""
import pytest
import torch

from paper_2407_19689_gb300 import instances as I
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


def _instance(m, n):
    ins = I.points_instance(m, n, I.seed_for(0, m + n))
    return torch.tensor(ins.C, dtype=torch.float32, device="cuda:0"), ins.f, ins.g


def test_solve(monkeypatch):
    big, small = _instance(2100, 2000), _instance(6, 20)
    s = pdot.Solver(device=0, max_iter=64)
    want = s.solve(*small, tol=1e-9)
    s.close()
    monkeypatch.setenv("PDOT_BARRIER_POLLS", "1")
    s = pdot.Solver(device=0, max_iter=64)
    for _ in range(3):   # (the launches take two barrier counters in turn)
        with pytest.raises(pdot.PdotError) as e:
            s.solve(*big, tol=1e-9)
        assert e.value.status == pdot.ERR_CUDA
        got = s.solve(*small, tol=1e-9)
        assert torch.equal(got.X, want.X) and torch.equal(got.p, want.p)
    s.close()
    monkeypatch.delenv("PDOT_BARRIER_POLLS")
    s = pdot.Solver(device=0, max_iter=64)
    assert s.solve(*big, tol=1e-9).status == pdot.MAX_ITER
    s.close()


def test_batch(monkeypatch):
    """The instances of a launch have barriers of their own."""
    out = []
    for polls in (None, "1"):
        if polls:
            monkeypatch.setenv("PDOT_BARRIER_POLLS", polls)
        B = pdot.BatchSolver(device=0, max_iter=64, tol=1e-9)
        for _ in range(2):
            big, one = B.submit(*_instance(2100, 2000)), B.submit(*_instance(1, 1))
            done = B.run()
            out.append((done[big], done[one]))
        B.close()
    for i, (big, one) in enumerate(out):
        assert big.status == (pdot.MAX_ITER if i < 2 else pdot.ERR_CUDA)
        assert one.status == out[0][1].status and torch.equal(one.X, out[0][1].X) and torch.equal(one.p, out[0][1].p)


def test_constant_steps_leave_the_state(monkeypatch):
    m, n = 2100, 2000
    C, f, g = _instance(m, n)
    f, g = (torch.tensor(v, device="cuda:0") for v in (f, g))
    state = [(f[:, None] * g[None]).float(), torch.zeros_like(f), torch.zeros_like(g)]
    before = [v.clone() for v in state]
    monkeypatch.setenv("PDOT_BARRIER_POLLS", "1")
    s = pdot.Solver(device=0)
    st = pdot.pdot_pdhg_steps(s.h, m, n, C.data_ptr(), pdot.F32, n, f.data_ptr(), g.data_ptr(), 20, 0.01, 1.0,
                              *(v.data_ptr() for v in state))
    s.close()
    assert st == pdot.ERR_CUDA
    for a, b in zip(state, before):
        assert torch.equal(a, b)
