"""The adjoint's FP64 sweeps on a level of more rows than the warp strips take (256): the strip-pipelined FP64
sweep, its finish and the transposed smoothing step around it.  P^-T r against the triangular solves on the
oracle's blocks (tolerance as in test_gpu_adjoint_precision); the smoothing step and, with a coarse level that
the warp strips take, the cycle against their transposes, <S^T a, b> = <a, S b>: two sums of 16,640 products
whose factors carry some 1e-13 of rounding, 1e-11 of the sum of their absolute values."""
import numpy as np
import pytest

from helpers import make_pair, perturbed_state
from synth.cgrid import make_cgrid
from test_gpu_adjoint_precision import _solve_transposed

pytestmark = pytest.mark.gpu

NI, NJ, NW = 16, 260, 4


def _pair(levels):
    o, s = make_pair(make_cgrid(NI, NJ, n_wake=NW, wall_spacing=1e-3), nlevels=levels, mach=0.6, alpha_deg=1.0)
    u = perturbed_state(0.6, 1.0, NJ, NI, amp=0.01, seed=NI)
    o.set_state(u)
    s.set_state(u)
    return o, s


def test_transposed_preconditioner_on_a_tall_level():
    o, s = _pair(1)
    r = np.random.default_rng(NJ).standard_normal((4, NJ, NI))
    for cfl in (5.0, 100.0):
        want = _solve_transposed(o, r, cfl, NW)
        assert np.abs(s.adjoint_precond_apply(r, cfl) - want).max() < 5e-15 * np.abs(want).max()
    s.close()


@pytest.mark.parametrize("kind,levels", [("smoother", 1), ("cycle", 2)])
def test_smoother_and_cycle_are_transposes_on_a_tall_level(kind, levels):
    _, s = _pair(levels)
    s.adjoint_jacobian()
    rng = np.random.default_rng(3)
    a, b = rng.standard_normal((2, 4, NJ, NI))
    t = s.adjoint_cycle_apply(a, 5.0, kind=kind) * b
    f = s.adjoint_cycle_apply(b, 5.0, kind=kind, transpose=False) * a
    s.close()
    assert np.all(np.isfinite(t)) and abs(t.sum() - f.sum()) < 1e-11 * np.abs(f).sum()
