"""Float projection, mode by mode, against sums in extended precision, on data whose high modes are small
beside the samples and cancel: every stored mode within its own rounding and what sums in double over the
differences of a cell's samples may lose."""
import numpy as np
import pytest

import helpers as H
from paper_2309_12019_gb300 import dgw

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _gauss(nq):
    """Nodes and weights in extended precision, by Newton from NumPy's."""
    x = np.polynomial.legendre.leggauss(nq)[0].astype(np.longdouble)
    for _ in range(3):
        P = _legendre(nq + 1, x)
        d = nq * (x * P[nq] - P[nq - 1]) / (x * x - 1) if nq > 1 else np.ones_like(x)
        x = x - P[nq] / d
    P = _legendre(nq + 1, x)
    d = nq * (x * P[nq] - P[nq - 1]) / (x * x - 1) if nq > 1 else np.ones_like(x)
    return x, 2 / ((1 - x * x) * d * d)


def _legendre(n, x):
    P = [np.ones_like(x), x]
    for k in range(1, n):
        P.append(((2 * k + 1) * x * P[k] - k * P[k - 1]) / np.longdouble(k + 1))
    return P[:n]


def _samples(kind, nx, ny, nq):
    x, _ = np.polynomial.legendre.leggauss(nq)
    X = ((np.arange(nx)[:, None] + 0.5 + 0.5 * x) / 1024.0)[None, :, None, :]
    Y = ((np.arange(ny)[:, None] + 0.5 + 0.5 * x) / 1024.0)[:, None, :, None]
    w = 2 * np.pi
    if kind == "smooth":
        f = 2 + np.sin(w * X) * np.cos(w * Y)
    elif kind == "through_zero":
        f = np.sin(w * (X - 20 / 1024.0)) * np.cos(w * Y)
    elif kind == "nearly_constant":
        f = 3.0 * (1 + 1e-9 * np.sin(9 * w * X + 3 * w * Y))
    elif kind == "step":
        f = np.where(np.hypot(X - 0.02, Y) < 0.015, 3.5 * np.pi, 0.25 * np.pi) + 0.05 * np.sin(3 * X + Y)
    else:
        f = np.random.default_rng(nq).standard_normal((ny, nx, nq, nq))
        f[:, ::7] = 0.7                              # constant cells
        f[:, 1::7] = 0.0
        f[:, 2::7] *= 1e-25                          # cells whose sums are taken in double
        f[:, 3::7, 0] *= 1e-9                        # exponents far apart within a cell
    return np.broadcast_to(f, (ny, nx, nq, nq)).reshape(nx * ny, nq, nq).copy()


@pytest.mark.parametrize("nq", range(1, 9))
@pytest.mark.parametrize("kind", ["smooth", "through_zero", "nearly_constant", "step", "mixed"])
def test_float_modes_keep_the_double_sums_accuracy(kind, nq):
    nx, ny = 43, 5                                   # 215 cells: three full CTAs of 64 and a ragged one
    f = _samples(kind, nx, ny, nq)
    g, w = _gauss(nq)
    F = np.abs(f).max(axis=(1, 2))
    D = np.abs(f - f[:, nq // 2, nq // 2][:, None, None]).max(axis=(1, 2))
    for p in (1, 2, 3):
        P = np.stack(_legendre(p + 1, g), 1)
        M = P * w[:, None] * (np.arange(p + 1) + np.longdouble(0.5))
        want = np.einsum("eba,ai,bj->jie", f.astype(np.longdouble), M, M).reshape(-1, nx * ny)
        ctx = dgw.Context(dgw.Problem(**H.spec(2, p, nx, ny=ny), prec="fp32"))
        U = torch.empty((ctx.K, ctx.E), dtype=torch.float32, device="cuda")
        ctx.project(torch.tensor(f.reshape(-1), device="cuda"), U, nq=nq)
        err = np.abs(U.double().cpu().numpy() - want).astype(np.float64)
        ctx.close()
        # The stored float's half unit; then, relative to the sums of w_q (i + 1/2) |d| a dimension (|P_i| <= 1,
        # d the differences from the centre sample, which rules of two points or more leave out of all
        # modes but the mean), at most 24 roundings of 2^-53 and four units in each of the two weights.
        # The mean and the one-point rule take the samples themselves.  Last, the reference's roundings.
        i, j = np.tile(np.arange(p + 1), p + 1), np.repeat(np.arange(p + 1), p + 1)
        S = ((2 * i + 1) * (2 * j + 1))[:, None]
        rough = np.where(((i + j == 0) | (nq == 1))[:, None], F, D)
        bar = np.abs(want).astype(np.float64) * 2.0 ** -24 + S * 32 * 2.0 ** -53 * rough
        bar = bar + S * 128 * float(np.finfo(np.longdouble).eps) * F + 1e-44
        assert (err <= bar).all(), (p, float((err / bar).max()), int((err / bar).max(axis=1).argmax()))
