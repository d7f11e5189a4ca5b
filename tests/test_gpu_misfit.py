"""dgw_misfit, J and its gradient, against the mass matrix in NumPy: scalar laws and the Euler
system, whose components (rows component-major) are all weighted alike."""
import numpy as np
import pytest

import helpers as H
from paper_2309_12019_gb300 import dgw

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("flux", ["burgers", "euler"])
def test_misfit_weighs_every_component_alike(flux, dim, p, prec):
    s = H.spec(dim, p, 7, flux=flux)
    ctx = dgw.Context(dgw.Problem(**s, prec=prec))
    rng = np.random.default_rng(p)
    U, V = (torch.tensor(rng.standard_normal((ctx.K, ctx.E)), dtype=ctx.dtype, device="cuda") for _ in range(2))
    grad = torch.empty_like(U)
    J = ctx.misfit(U, V, grad)
    m = 1.0 / 7 / (2 * np.arange(p + 1) + 1)                  # int P_i^2 over a cell of width 1/7
    m = m if dim == 1 else np.outer(m, m).reshape(-1)
    m = np.tile(m, ctx.K // m.size)[:, None]
    d = U.double().cpu().numpy() - V.double().cpu().numpy()
    # at most 200 roundings of positive terms in double; a mass has at most eight on either side (h,
    # its quotients, their product), and the gradient is rounded once to its type
    assert abs(J - 0.5 * np.sum(m * d * d)) <= 200 * 2.0 ** -53 * J
    u = 17 * 2.0 ** -53 + (2.0 ** -24 if prec == "fp32" else 0.0)
    assert (np.abs(grad.double().cpu().numpy() - m * d) <= u * np.abs(m * d)).all()
    ctx.close()
