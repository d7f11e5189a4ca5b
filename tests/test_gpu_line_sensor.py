"""The one-lane line kernel of the scalar laws takes the bits of the stage kernels, the sensor's
included: steps of a periodic mesh that one cluster holds against the same state repeated on a mesh
that does not fit, with the threshold b at its default, where another rounding of the ratio could
move a cell across it."""
import pytest

import helpers as H
from paper_2309_12019_gb300 import dgw

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec,n,copies", [("fp32", 256, 32), ("fp32", 4096, 2), ("fp64", 1024, 4)])
@pytest.mark.parametrize("flux", ["advect", "burgers", "kpp"])
def test_line_steps_have_the_stage_kernels_bits(flux, prec, n, copies):
    for p in (1, 2, 3):
        for stab in ("weno", "zhao", "lo", "dg"):
            s = H.spec(1, p, n, flux=flux, stab=stab)
            U = torch.tensor(H.state_for(s, seed=n + p), device="cuda")
            big = dict(s, nx=n * copies, box=(0.0, float(copies), 0.0, 1.0))
            out = []
            for q in (s, big):
                ctx = dgw.Context(dgw.Problem(**q, prec=prec))
                V = U.to(ctx.dtype).repeat(1, q["nx"] // n).contiguous()
                ctx.rk_step(V, 0.01 / n, 4)
                ctx.sync_status()
                ctx.close()
                out.append(V)
            assert torch.equal(out[0].repeat(1, copies), out[1]), (p, stab)
