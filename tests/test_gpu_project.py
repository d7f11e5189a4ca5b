"""dgw_project against the oracle for every sample rule, at the edges of the kernel's blocks, and
from sample arrays that start off a 16-byte boundary (no paired loads)."""
import numpy as np
import pytest

import helpers as H
from oracle import oracle as O
from paper_2309_12019_gb300 import dgw

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nq", range(1, 9))
@pytest.mark.parametrize("dim,nx,ny", [(1, 1, 1), (1, 129, 1), (2, 16, 8), (2, 43, 3)])
def test_project_all_rules(dim, nx, ny, nq):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(nq + 10 * nx)
    for p in (1, 2, 3):
        s = H.spec(dim, p, nx, ny=ny)
        f = rng.standard_normal(nx * ny * nq ** dim)
        # the rule's sums in NumPy (the oracle divides by the rule's own norm of P_i, which is the
        # exact one from p + 1 points on)
        g, w = np.polynomial.legendre.leggauss(nq)
        M = np.polynomial.legendre.legvander(g, p) * w[:, None] * (np.arange(p + 1) + 0.5)
        v = f.reshape((nx * ny,) + (nq,) * dim)
        want = np.einsum("ea,ai->ie", v, M) if dim == 1 else np.einsum("eba,ai,bj->jie", v, M, M).reshape(-1, nx * ny)
        if nq > p:
            assert np.allclose(want, O.project(O.Problem(**s), f, nq), rtol=0, atol=1e-12)
        # |sum w_a w_b P_i P_j f| <= 4 max |f|, times minv_i minv_j <= 12.25; at most 20 roundings of
        # partial sums in double on either side, and one of the result in float
        tol = {"fp64": 2 * 20 * 4 * 2.0 ** -53, "fp32": 4 * 2.0 ** -24}
        for prec in ("fp64", "fp32"):
            ctx = dgw.Context(dgw.Problem(**s, prec=prec))
            for off in (0, 1):
                buf = torch.zeros(f.size + 1, dtype=torch.float64, device="cuda")
                buf[off:off + f.size] = torch.tensor(f)
                U = torch.empty((ctx.K, ctx.E), dtype=ctx.dtype, device="cuda")
                ctx.project(buf[off:off + f.size], U, nq=nq)
                err = np.abs(U.double().cpu().numpy() - want).max()
                assert err <= tol[prec] * 12.25 * np.abs(f).max(), (p, prec, off)
            ctx.close()


@pytest.mark.parametrize("scale", [1e-25, 1e30])
def test_project_float_outside_the_split_range(scale):
    """Float projection sums in double-float arithmetic where every sample lies in [2^-60, 2^96) or
    is zero, and in double elsewhere: cells of either kind side by side, and cells of zeros."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny, nq, p = 20, 7, 8, 3
    s = H.spec(2, p, nx, ny=ny)
    f = np.random.default_rng(5).standard_normal((nx * ny, nq * nq))
    f[::3] *= scale
    f[1::5, ::2] = 0.0
    f[7] = 0.0
    want = O.project(O.Problem(**s), f.reshape(-1), nq)
    ctx = dgw.Context(dgw.Problem(**s, prec="fp32"))
    U = torch.empty((ctx.K, ctx.E), dtype=torch.float32, device="cuda")
    ctx.project(torch.tensor(f.reshape(-1), device="cuda"), U, nq=nq)
    err = np.abs(U.double().cpu().numpy() - want).max(axis=0)
    # as above, per cell
    assert (err <= 4 * 2.0 ** -24 * 12.25 * np.abs(f).max(axis=1)).all()
    ctx.close()
