"""The closed-form volume and face terms of the linear fluxes (2D, double) against the
oracle's quadrature: velocities of either sign and zero along an axis, every kind of side, rotation
centres inside and far outside the mesh, ragged tiles."""
import numpy as np
import pytest

import helpers as H
from oracle import oracle as O
from paper_2309_12019_gb300 import dgw

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("kw", [
    dict(flux="advect", a=(1.0, 0.0)), dict(flux="advect", a=(-0.7, 0.0)), dict(flux="advect", a=(0.0, -1.0)),
    dict(flux="advect", a=(-0.3, 0.4)), dict(flux="rotation", center=(0.4, 0.3), omega=1.0),
    dict(flux="rotation", center=(-2.0, 3.0), omega=-1.5), dict(flux="rotation", center=(0.0, 0.5), omega=0.7)])
def test_linear_fluxes_match_quadrature(kw, p):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    flux = kw["flux"]
    for bc in ("inflow_zero", "outflow") + (("periodic",) if flux == "advect" else ()):
        for nx, ny in ((33, 18), (36, 5)):
            for stab in ("dg", "lo", "weno"):
                s = H.spec(2, p, nx, ny=ny, bc=bc, stab=stab, **kw)
                U0 = H.state_for(s, seed=p + nx)
                want = O.residual(O.Problem(**s), U0)
                ctx = dgw.Context(dgw.Problem(**s, prec="fp64"))
                U = torch.tensor(U0, device="cuda")
                L = torch.empty_like(U)
                ctx.residual(U, L)
                assert H.rel_l2(L.cpu().numpy(), want) <= 1e-12, (bc, nx, stab)   # the bar of the parity tests
                ctx.close()
    assert np.isfinite(want).all()
