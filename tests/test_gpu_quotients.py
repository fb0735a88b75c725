"""The quotients of FP64 contexts against IEEE division, where every other operation on the way is exact or
rounds as on the host: the volume-weighted restriction of a state that is constant on each block of four cells
(its sums are exact, so it is that state, bit for bit; at a CFL number of 1e-30 the smoothing steps before and
after change nothing), and the pseudo time step of a gas at rest on a rectangular grid."""
import numpy as np
import pytest

import paper_1710_04875_gb300 as P
from synth.cgrid import make_rect_grid

pytestmark = pytest.mark.gpu

NI, NJ, HX, HY = 48, 24, 3.0 / 32.0, 5.0 / 64.0   # volumes 15/2048: powers of two would divide exactly


def _solver(precision, **kw):
    return P.Solver(make_rect_grid(NI, NJ, NI * HX, NJ * HY),
                    P.default_params(mach=0.5, precision=precision, cfl_ramp=1e-30, **kw))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_restriction_keeps_a_state_constant_on_its_blocks(precision):
    rng = np.random.default_rng(7)
    c = rng.integers(0, 2**20, (4, NJ // 2, NI // 2)) / 2.0**22
    c += np.array([1.0, 0.0, 0.0, 2.0])[:, None, None]
    s = _solver(precision, nlevels=2, cfl=1e-30)
    s.set_state(np.ascontiguousarray(c.repeat(2, axis=1).repeat(2, axis=2)))
    s.fas_cycle(0)
    assert np.array_equal(s.get_state(0), c)
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_time_step_of_a_gas_at_rest(precision):
    E = np.random.default_rng(8).uniform(2.0, 3.0, (NJ, NI))
    s = _solver(precision, nlevels=1, cfl=7.3)
    s.set_state(np.stack([np.ones_like(E), 0.0 * E, 0.0 * E, E]))
    a = np.sqrt(1.4 * ((1.4 - 1.0) * E))
    assert np.array_equal(s.pseudo_dt(7.3), 7.3 * (HX * HY) / (a * HY + a * HX))
    s.close()
