"""Steps of small 1D meshes, which one thread-block cluster takes in one launch, against the
stage kernels that larger meshes run (dgw_rk_step_stages keeps the stages, so it launches them
one by one), at the edges of the cluster's CTAs: one cell, 32 cells and one more, 16 CTAs of
each size and one cell more, and the first mesh that does not fit."""
import numpy as np
import pytest

import helpers as H
from paper_2309_12019_gb300 import dgw
from paper_2309_12019_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SIZES = [1, 2, 31, 32, 33, 65, 512, 513, 1024, 1025, 2048, 2049, 4096, 4097]
BCS = {"advect": ("periodic", "inflow_zero", "outflow"), "burgers": ("periodic", "inflow_zero"),
       "rotation": ("inflow_zero",), "kpp": ("periodic", "inflow_zero"),
       "euler": ("periodic", "reflect", "outflow")}


def _setup(flux, p, n, bc, stab, prec, **kw):
    if flux == "euler":
        s = dict(dim=1, nx=n, ny=1, p=p, box=(0.0, n / 64.0, 0.0, 1.0), bc=(bc,) * 2 + ("periodic",) * 2, flux="euler",
                 stab=stab)
        U = I.random_euler_state(p, n, seed=n + p, amp=0.02)
        dt = 0.2 * I.euler_cfl(p) / 64.0
    else:
        # b = 0: with a threshold a rounding difference may move a cell across it
        s = H.spec(1, p, n, flux=flux, bc=bc, stab=stab, b=0.0)
        U = H.state_for(s, seed=n + p)
        dt = 0.01 / n
    ctx = dgw.Context(dgw.Problem(**s, prec=prec, **kw))
    return ctx, torch.tensor(U, dtype=ctx.dtype, device="cuda"), dt


def _close(a, b, prec):
    # three steps of a few hundred operations on each side: a relative rounding error of a few
    # hundred units of 2^-53, the bar of the double parity tests; in float, that of the float ones
    return H.rel_l2(a.double().cpu().numpy(), b.double().cpu().numpy()) <= {"fp64": 1e-12, "fp32": 2e-5}[prec]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("flux", list(BCS))
@pytest.mark.parametrize("n", SIZES)
def test_line_matches_stage_kernels(n, flux, prec):
    for bc in BCS[flux]:
        for p, stab in ((1, "weno"), (2, "weno"), (3, "weno"), (2, "dg"), (1, "lo"), (3, "zhao")):
            ctx, U, dt = _setup(flux, p, n, bc, stab, prec)
            V, U1, U2 = U.clone(), torch.empty_like(U), torch.empty_like(U)
            ctx.rk_step(V, dt, 3)
            for _ in range(3):
                ctx.rk_step_stages(U, dt, U1, U2, U)
            ctx.sync_status()
            assert _close(V, U, prec), (bc, p, stab)
            ctx.close()


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("flux", ["burgers", "euler"])
def test_line_other_orders_on_residuals(flux, order):
    """SSP-RK of order 2 and 4 against the same combinations of dgw_residual."""
    for n in (33, 300):
        ctx, U, dt = _setup(flux, 2, n, "periodic", "weno", "fp64", rk_order=order)
        V, R = U.clone(), torch.empty_like(U)
        ctx.rk_step(V, dt, 2)

        def L(u):
            ctx.residual(u.contiguous(), R)
            return R.clone()
        for _ in range(2):
            if order == 2:
                q = U + dt * L(U)
                U = 0.5 * U + 0.5 * (q + dt * L(q))
            else:
                q, q2 = U, U
                for _ in range(5):
                    q = q + dt / 6 * L(q)
                q2 = q2 / 25 + 9 / 25 * q
                q = 15 * q2 - 5 * q
                for _ in range(4):
                    q = q + dt / 6 * L(q)
                U = q2 + 0.6 * q + dt / 10 * L(q)
        assert _close(V, U, "fp64")
        ctx.close()


def test_line_capture_streams_and_status():
    """Inside a stream capture, on a side stream and past the launch's 1024 steps the result is
    the same; a non-finite step is reported."""
    ctx, U, dt = _setup("burgers", 2, 100, "periodic", "weno", "fp64")
    ref = U.clone()
    for _ in range(41):
        ctx.rk_step(ref, dt, 25)
    one, V, W = U.clone(), U.clone(), U.clone()
    ctx.rk_step(one, dt, 1025)
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        ctx.rk_step(V, dt, 1025)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.rk_step(W, dt, 25)
    for _ in range(41):
        g.replay()
    torch.cuda.synchronize()
    for x in (one, V, W):
        assert torch.equal(x, ref)
    ctx.sync_status()
    U[0, 40] = float("nan")
    ctx.rk_step(U, dt, 1)
    with pytest.raises(dgw.DGWError) as err:
        ctx.sync_status()
    assert err.value.status == -6
    ctx.close()
    del g
    assert np.isfinite(ref.cpu().numpy()).all()
