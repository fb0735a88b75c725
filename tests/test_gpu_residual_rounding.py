"""The FP64 residual's rounding where arithmetic leaves none: a gas at rest under constant pressure whose density
grows by the same amount from cell to cell (in few enough bits that its differences are exact) has third
differences of zero, so its dissipation is zero, bit for bit.  And the convective part of FP64 contexts, summed in
an order of its own, against extended precision: its rounding error (rms) is no larger than that of mixed contexts,
whose residual takes the two cells' fluxes one after the other (a sum that meets the pressure first and is rounded
at its size three times instead of once has 1.2 to 1.4 times the error)."""
import numpy as np
import pytest

import paper_1710_04875_gb300 as P
from helpers import perturbed_state
from synth.cgrid import make_rect_grid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ni,nj", [(40, 12), (64, 100)])  # tiles of one row, of four
def test_dissipation_of_a_linear_density_is_zero(ni, nj, precision):
    i = np.arange(ni)
    rho = (1.0 + 5.0 * i / 256.0)[None].repeat(nj, axis=0)
    s = P.Solver(make_rect_grid(ni, nj, ni * 3.0 / 32.0, nj * 5.0 / 64.0),
                 P.default_params(mach=0.5, nlevels=1, precision=precision))
    s.set_state(np.stack([rho, 0.0 * rho, 0.0 * rho, 2.5 + 0.0 * rho]))
    Fv = s.residual()[2]
    s.close()
    assert not np.any(Fv[:, :nj - 2, 2:ni - 2])   # two cells from the far field's ghosts
    assert np.any(Fv)


def _convective(g, u):
    """F^c of the cells that touch no boundary, in extended precision."""
    x, y, u = (a.astype(np.longdouble) for a in (g.x, g.y, u))
    gam = np.longdouble(1.4)
    p = (gam - 1) * (u[3] - (u[1] ** 2 + u[2] ** 2) / u[0] / 2)
    w = np.stack([u[0], u[1], u[2], u[3] + p])

    def flux(sx, sy, c):
        q = (u[1][c] * sx + u[2][c] * sy) / u[0][c]
        return w[(slice(None),) + c] * q + p[c] * np.stack([0 * sx, sx, sy, 0 * sx])

    def faces(sx, sy, a, b):
        return (flux(sx, sy, a) + flux(sx, sy, b)) / 2

    o, m = slice(1, -1), slice(None)
    i = faces((y[1:] - y[:-1])[:, 1:-1], (x[:-1] - x[1:])[:, 1:-1], (m, slice(0, -1)), (m, slice(1, None)))
    j = faces((y[:, :-1] - y[:, 1:])[1:-1], (x[:, 1:] - x[:, :-1])[1:-1], (slice(0, -1), m), (slice(1, None), m))
    d1x, d1y = x[1:, 1:] - x[:-1, :-1], y[1:, 1:] - y[:-1, :-1]
    d2x, d2y = x[1:, :-1] - x[:-1, 1:], y[1:, :-1] - y[:-1, 1:]
    vol = (d1x * d2y - d1y * d2x) / 2
    return ((i[:, o, 1:] - i[:, o, :-1]) + (j[:, 1:, o] - j[:, :-1, o])) / vol[o, o]


@pytest.mark.parametrize("ni,nj", [(64, 48), (130, 72)])
def test_convective_sums_are_as_accurate_as_the_fluxes_one_by_one(ni, nj):
    g = make_rect_grid(ni, nj, 4.0, 1.0, jitter=0.2, seed=ni)
    u = perturbed_state(0.5, 1.0, nj, ni, amp=0.01, seed=nj)
    want, err = _convective(g, u), {}
    for precision in ("fp64", "mixed"):
        s = P.Solver(g, P.default_params(mach=0.5, alpha_deg=1.0, nlevels=1, precision=precision))
        s.set_state(u)
        d = s.residual()[1][:, 1:-1, 1:-1] - want
        s.close()
        err[precision] = np.sqrt((d ** 2).mean(axis=(1, 2)))
    assert np.all(err["mixed"] < 1e-12 * np.abs(want).max())
    assert np.all(err["fp64"] <= err["mixed"]), err
