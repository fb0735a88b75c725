"""The residual of states on the way to divergence: a cell of negative pressure has no sound speed (a NaN), and
its faces take the radii of the cells beside it, as fmax does.  The residual stays finite, and outside the
cell's stencil it is that of the good state, bit for bit."""
import numpy as np
import pytest

import paper_1710_04875_gb300 as P
from helpers import perturbed_state
from synth.cgrid import make_cgrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sensor", [0, 1])
@pytest.mark.parametrize("j", [1, 7])
def test_residual_around_a_cell_of_negative_pressure(precision, sensor, j):
    ni, nj, i = 64, 16, 30
    u = perturbed_state(0.8, 1.0, nj, ni, amp=0.01, seed=4)
    s = P.Solver(make_cgrid(ni, nj, n_wake=8), P.default_params(mach=0.8, alpha_deg=1.0, nlevels=1, sensor=sensor,
                                                                precision=precision))
    s.set_state(u)
    good = s.residual()
    u[3, j, i] = 0.4 * (u[1, j, i] ** 2 + u[2, j, i] ** 2) / u[0, j, i]  # p = -0.04 rho |v|^2
    s.set_state(u)
    bad = s.residual()
    s.close()
    far = np.ones((nj, ni), bool)
    far[max(0, j - 2):j + 3, i] = far[j, i - 2:i + 3] = False
    for a, b in zip(bad, good):
        assert np.all(np.isfinite(a))
        assert np.array_equal(a[:, far], b[:, far])
        assert not np.array_equal(a[:, ~far], b[:, ~far])
