"""The sensor of states far from one in double, whose weights (the fourth power of 1 / U) and their
squares leave the range in which the ratio is taken through its squares: against the oracle, in the
stage kernels (dgw_sensor) and in the steps of a linear law on meshes that one cluster holds."""
import numpy as np
import pytest

import helpers as H
from paper_2309_12019_gb300 import dgw

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SCALES = [1e-9, 1e-4, 1e3, 1e20, 1e40, 1e60, 1e70]


@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("dim,p", [(1, 1), (1, 2), (1, 3), (2, 1), (2, 2), (2, 3)])
def test_sensor_of_scaled_states(oracle_mod, dim, p, scale):
    s = H.spec(dim, p, 40 if dim == 1 else 12, flux="advect", b=0.0)
    U = scale * H.state_for(s, seed=p)
    # cells of one value among the others, and cells of zeros
    U[1:, ::5] = 0.0
    U[:, ::10] = 0.0
    want = oracle_mod.sensor(oracle_mod.Problem(**s), U)[0]
    ctx = dgw.Context(dgw.Problem(**s, prec="fp64"))
    V, g = torch.tensor(U, device="cuda"), torch.empty(ctx.E, dtype=torch.float64, device="cuda")
    ctx.sensor(V, g)
    # the bar of the double sensor tests
    assert np.abs(g.cpu().numpy() - want).max() <= 1e-12
    if dim == 1:
        ref = oracle_mod.rk3(oracle_mod.Problem(**s), U, 0.01 / s["nx"], 2)
        ctx.rk_step(V, 0.01 / s["nx"], 2)
        assert H.rel_l2(V.cpu().numpy() / scale, ref / scale) <= 1e-12
    ctx.sync_status()
    ctx.close()
