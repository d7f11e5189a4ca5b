"""Stage launches that overlap the one before (or not, or with padded shared memory, by the number of
CTAs and the way they are launched) compute the same: one by one on the default stream, replayed from
a graph, and one launch after a synchronisation each, at CTA counts around half the SMs, one, and a
few per SM."""
import pytest

import helpers as H
from paper_2309_12019_gb300 import dgw
from paper_2309_12019_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _spec(flux, p, n):
    if flux == "euler":
        return dict(dim=2, nx=n, ny=n, p=p, box=(0.0, 1.0, 0.0, 1.0), bc=("periodic",) * 4, flux="euler")
    return H.spec(2, p, n, flux=flux)


def _state(ctx, flux, n, p):
    K = (p + 1) ** 2
    U = torch.tensor(I.random_state(2, p, n * n, n + p, smooth=True, scale=0.1, offset=1.0), device="cuda")
    if flux == "euler":
        z = torch.zeros_like(U)
        z[0] = 3.0
        U = torch.cat([U, 0.1 * U, -0.2 * U, z + 0.1 * U])
    assert U.shape[0] == ctx.K and K
    return U.to(ctx.dtype).contiguous()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("flux,p", [("burgers", 1), ("burgers", 2), ("euler", 1), ("euler", 2)])
@pytest.mark.parametrize("n", [64, 96, 130, 192, 256])
def test_launch_modes_agree(n, flux, p, prec):
    ctx = dgw.Context(dgw.Problem(**_spec(flux, p, n), prec=prec))
    U = _state(ctx, flux, n, p)
    dt, V, W, R = 1e-5, U.clone(), U.clone(), U.clone()
    torch.cuda.synchronize()
    ctx.rk_step(V, dt, 3, stream=0)                       # launched one by one
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for _ in range(2):                                    # captured, then replayed
        W.copy_(U)
        torch.cuda.synchronize()
        ctx.rk_step(W, dt, 3, stream=st.cuda_stream)
        st.synchronize()
    U1, U2 = torch.empty_like(U), torch.empty_like(U)
    for _ in range(3):
        ctx.rk_step_stages(R, dt, U1, U2, R, stream=0)
        torch.cuda.synchronize()
    ctx.sync_status()
    assert torch.equal(V, R) and torch.equal(W, R)
    ctx.close()


def test_adjoint_launched_and_captured_agree():
    n, p = 128, 2
    for prec in ("fp64", "fp32"):
        ctx = dgw.Context(dgw.Problem(**H.spec(2, p, n, flux="burgers"), prec=prec))
        U = _state(ctx, "burgers", n, p)
        lam, a, b = torch.randn_like(U), torch.empty_like(U), torch.empty_like(U)
        ctx.adjoint_step(U, lam, a, 1e-5)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            ctx.adjoint_step(U, lam, b, 1e-5)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(a, b)
        ctx.close()
        del g
