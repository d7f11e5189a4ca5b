"""Order of the rollout's calls and what they are given, on a stand-in for the library's context whose
step multiplies by 3/2: ragged and single segments, no steps, no gradient asked for."""
import types
import weakref

import pytest

torch = pytest.importorskip("torch")
from paper_2309_12019_gb300 import adjoint  # noqa: E402


class Ctx:
    def __init__(self, rk_order=3, bc=("periodic",) * 4):
        self.problem = types.SimpleNamespace(rk_order=rk_order, bc=bc)
        self.reversed_from, self.kept = [], 0

    def rk_step(self, U, dt, n):
        U.mul_(1.5 ** n)

    def rk_step_stages(self, U, dt, U1, U2, nxt=None):
        self.kept += 1
        if nxt is not None:
            nxt.copy_(1.5 * U)

    def adjoint_step_stages(self, Un, U1, U2, lam, out, dt):
        self.reversed_from.append(float(Un[0]))
        out.copy_(1.5 * lam)


@pytest.mark.parametrize("n,every", [(8, 4), (7, 3), (1, 20), (3, 1), (0, 5)])
def test_rollout_reverses_every_step_once(n, every):
    c = Ctx()
    U0 = torch.ones(2, dtype=torch.float64, requires_grad=True)
    U = adjoint.rollout(c, U0, 0.1, n, every)
    U.sum().backward()
    assert float(U[0]) == 1.5 ** n and float(U0.grad[0]) == 1.5 ** n and float(U0[0]) == 1.0
    assert c.reversed_from == [1.5 ** i for i in reversed(range(n))]
    assert c.kept == n             # every step's stages once


@pytest.mark.parametrize("kw", [dict(rk_order=2), dict(bc=("state", "outflow", "state", "state"))])
def test_rollout_without_an_adjoint_steps_forward(kw):
    c = Ctx(**kw)
    U = adjoint.rollout(c, torch.ones(2, dtype=torch.float64, requires_grad=True), 0.1, 5, 2)
    assert float(U.detach()[0]) == 1.5 ** 5 and c.kept == 0
    c = Ctx()
    with torch.no_grad():
        U = adjoint.rollout(c, torch.ones(2, dtype=torch.float64, requires_grad=True), 0.1, 5, 2)
    assert float(U[0]) == 1.5 ** 5


def test_rollout_without_a_gradient_keeps_no_stages():
    U0 = torch.ones(2, dtype=torch.float64, requires_grad=True)
    c = Ctx()
    with torch.no_grad():
        assert float(adjoint.rollout(c, U0, 0.1, 5, 2)[0]) == 1.5 ** 5
    adjoint.rollout(c, U0.detach(), 0.1, 5, 2)
    assert c.kept == 0


def test_one_segment_is_kept_per_context():
    """Rollouts that are chained in one graph, or whose backward pass never comes, hold the stages of
    the latest one only; the others recompute theirs from the checkpoint, which stays."""
    class Watched(Ctx):
        def rk_step_stages(self, U, dt, U1, U2, nxt=None):
            super().rk_step_stages(U, dt, U1, U2, nxt)
            self.stages.append(weakref.ref(U1))

        def alive(self):
            return sum(r() is not None for r in self.stages)

    c = Watched()
    c.stages = []
    waiting = adjoint.rollout(c, torch.ones(2, dtype=torch.float64, requires_grad=True), 0.1, 4, 4)
    assert c.alive() == 4
    U0 = torch.ones(2, dtype=torch.float64, requires_grad=True)
    U = U0
    for n in (3, 5, 2):
        U = adjoint.rollout(c, U, 0.1, n, 4)
    assert c.alive() == 2
    U.sum().backward()
    assert c.reversed_from == [1.5 ** i for i in reversed(range(10))]
    waiting.sum().backward()
    assert float(U0.grad[0]) == 1.5 ** 10 and c.reversed_from[10:] == [1.5 ** i for i in reversed(range(4))]
    assert c.alive() == 0
