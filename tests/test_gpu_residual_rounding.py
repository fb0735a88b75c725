"""The FP64 residual's rounding where arithmetic leaves none: a gas at rest under constant pressure whose density
grows by the same amount from cell to cell (in few enough bits that its differences are exact) has third
differences of zero, so its dissipation is zero, bit for bit."""
import numpy as np
import pytest

import paper_1710_04875_gb300 as P
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
