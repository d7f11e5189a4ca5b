"""Steps that keep their stages on 1D meshes: they take the launches of dgw_rk_step, so a rollout is
differentiated about the states it went through and its value does not depend on whether a gradient
was asked for, also with the threshold b at its default.  And dgw_rk_step on such meshes against
combinations of dgw_residual, which runs the stage kernels."""
import pytest

import test_gpu_line as TL
import helpers as H
from paper_2309_12019_gb300 import adjoint, dgw
from paper_2309_12019_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _context(flux, p, n, prec):
    if flux == "euler":
        s = dict(dim=1, nx=n, ny=1, p=p, box=(0.0, n / 64.0, 0.0, 1.0), bc=("reflect",) * 2 + ("periodic",) * 2, flux="euler")
        U, dt = I.random_euler_state(p, n, seed=n + p, amp=0.02), 0.2 * I.euler_cfl(p) / 64.0
    else:
        s = H.spec(1, p, n, flux=flux)
        U, dt = H.state_for(s, seed=n + p), 0.01 / n
    ctx = dgw.Context(dgw.Problem(**s, prec=prec))
    return ctx, torch.tensor(U, dtype=ctx.dtype, device="cuda"), dt


# one CTA and several, eight lanes a cell and one (double beyond 512 cells), the first mesh without a cluster
@pytest.mark.parametrize("prec,n", [("fp64", 33), ("fp64", 512), ("fp64", 600), ("fp64", 2049), ("fp32", 33),
                                    ("fp32", 4096), ("fp32", 4097)])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("flux", ["burgers", "kpp", "euler"])
def test_kept_stages_are_those_of_the_step(flux, p, n, prec):
    ctx, U, dt = _context(flux, p, n, prec)
    ref, U1, U2, nxt = U.clone(), torch.empty_like(U), torch.empty_like(U), torch.empty_like(U)
    ctx.rk_step(ref, dt, 1)
    ctx.rk_step_stages(U, dt, U1, U2, nxt)
    assert torch.equal(nxt, ref)
    V1, V2, V = torch.empty_like(U), torch.empty_like(U), U.clone()
    ctx.rk_step_stages(U, dt, V1, V2)          # without the third stage
    assert torch.equal(V1, U1) and torch.equal(V2, U2) and torch.equal(V, U)
    ctx.rk_step_stages(V, dt, V1, V2, V)       # in place
    assert torch.equal(V, ref)
    # U1 = U + dt L(U), U2 = 3/4 U + 1/4 (U1 + dt L(U1)) to rounding
    L = torch.empty_like(U)
    ctx.residual(U, L)
    assert flux == "kpp" or H.rel_l2((U + dt * L).cpu(), U1.cpu()) <= {"fp64": 1e-12, "fp32": 2e-5}[prec]
    if flux == "burgers":
        lam, a, b = torch.randn_like(U), torch.empty_like(U), torch.empty_like(U)
        ctx.adjoint_step(U, lam, a, dt)
        ctx.adjoint_step_stages(U, U1, U2, lam, b, dt)
        assert torch.equal(a, b)
    ctx.sync_status()
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [100, 600])
def test_rollout_value_does_not_depend_on_the_gradient(n, prec):
    ctx, U, dt = _context("burgers", 2, n, prec)
    ref = U.clone()
    ctx.rk_step(ref, dt, 10)
    plain = adjoint.rollout(ctx, U, dt, 10, 4)
    U0 = U.clone().requires_grad_(True)
    graded = adjoint.rollout(ctx, U0, dt, 10, 4)
    graded.sum().backward()
    # the states about which the first segment is linearised, and its end
    V, U1, U2 = U.clone(), torch.empty_like(U), torch.empty_like(U)
    for _ in range(10):
        ctx.rk_step_stages(V, dt, U1, U2, V)
    for x in (plain, graded.detach(), V):
        assert torch.equal(x, ref)
    assert torch.isfinite(U0.grad).all()
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("flux", list(TL.BCS))
@pytest.mark.parametrize("n", TL.SIZES)
def test_line_matches_residuals(n, flux, prec):
    for bc in TL.BCS[flux]:
        for p, stab in ((1, "weno"), (2, "weno"), (3, "weno"), (2, "dg"), (1, "lo"), (3, "zhao")):
            ctx, U, dt = TL._setup(flux, p, n, bc, stab, prec)
            V, R = U.clone(), torch.empty_like(U)
            ctx.rk_step(V, dt, 3)

            def L(u):
                ctx.residual(u.contiguous(), R)
                return R.clone()
            for _ in range(3):
                q = U + dt * L(U)
                q = 0.75 * U + 0.25 * (q + dt * L(q))
                U = U / 3.0 + 2.0 / 3.0 * (q + dt * L(q))
            ctx.sync_status()
            assert TL._close(V, U, prec), (bc, p, stab)
            ctx.close()
