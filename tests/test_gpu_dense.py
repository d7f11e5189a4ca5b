"""Float stages of meshes with more tiles than one round of CTAs run a build of the tile kernel with
fewer registers: the same bits as the other build, which the host-buffer pipeline's bands (few tiles
each) run, at one tile more and fewer than a round of 152 SMs."""
import pytest

import helpers as H
from paper_2309_12019_gb300 import dgw

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("flux", ["advect", "rotation", "burgers", "kpp"])
@pytest.mark.parametrize("p,nx,ny", [(1, 609, 384), (1, 608, 384), (2, 513, 288), (2, 512, 304)])
def test_dense_build_same_bits(p, nx, ny, flux):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = H.spec(2, p, nx, ny=ny, flux=flux, bc="outflow")
    U = torch.tensor(H.state_for(s, seed=nx), dtype=torch.float32)
    ctx = dgw.Context(dgw.Problem(**s, prec="fp32"))
    Ud = U.cuda()
    ctx.rk_step(Ud, 0.005 / nx, 1)
    Uh, out = U.pin_memory(), torch.empty_like(U).pin_memory()
    ctx.rk_step_host(Uh, out, 0.005 / nx, 1)
    torch.cuda.synchronize()
    ctx.sync_status()
    assert torch.equal(out, Ud.cpu())
    ctx.close()
