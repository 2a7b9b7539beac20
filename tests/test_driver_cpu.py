"""run_until_stop takes its steps through `step` where a subclass or the object replaces it (no device needed: the
energies are made up)."""
import pytest

torch = pytest.importorskip("torch")
from paper_2604_02550_gb300 import api


class _Fake(api.ACSE):
    """A driver without a context: E falls by 1 a step, ||A||^2 by half."""

    def __init__(self):
        self.device, self.stream, self.ctx, self.n = torch.device("cpu"), None, None, 0

    def energy(self, D):
        return torch.zeros(1, dtype=torch.float64)


class _Stepping(_Fake):
    def step(self, D, eps=0.0):
        self.n += 1
        D[0].add_(eps)
        one = torch.ones(1, dtype=torch.float64)
        return -self.n * one, 0.5 ** self.n * one, eps * one


def _check(drv, D):
    got = drv._run_until_stop(D, 3, 0.25, 1e-10)
    assert drv.n == 3 and got["E"] == [0.0, -1.0, -2.0, -3.0] and got["eps"] == [0.25] * 3 and got["reason"] == "cap"
    assert float(D[0][0]) == 0.75


def test_step_of_a_subclass():
    _check(_Stepping(), (torch.zeros(2, dtype=torch.float64),) * 3)


def test_step_of_the_object():
    drv = _Fake()
    drv.step = lambda D, eps=0.0: _Stepping.step(drv, D, eps)
    _check(drv, (torch.zeros(2, dtype=torch.float64),) * 3)


def test_own_step_uses_one_buffer(monkeypatch):
    seen = []

    def step(ctx, aa, ab, bb, eps, E, n2, e):
        seen.append((E.data_ptr(), n2.data_ptr(), e.data_ptr()))
        E.fill_(-float(len(seen)))
        n2.fill_(0.5 ** len(seen))
        e.fill_(eps)

    monkeypatch.setattr(api._lib, "acse_step", step)
    got = _Fake()._run_until_stop(tuple(torch.zeros(2, dtype=torch.float64) for _ in range(3)), 3, 0.25, 1e-10)
    assert got["E"] == [0.0, -1.0, -2.0, -3.0] and len(set(seen)) == 1
