"""The warp-strip sweep (strips of 8 rows, two per CTA) at the sizes where its strips, stages and
buffers end: fewer rows than a strip, odd numbers of strips, one strip, the most strips a cluster
holds, steps that do not fill a stage, a wake cut that leaves two wall cells, no cut, and grids too
long for an edge buffer per pass and for the deeper ring; against the oracle's lexicographic sweep.

Tolerances: in FP64 the FP32 solve (relative error up to 3e-7) and one defect correction leave
(3e-7)^2 times the sweep's amplification, 1e-13; 1e-11 as in the other sweep parity tests.  In mixed
precision the FP32 solve itself: 3e-7 amplified by up to a hundred steps' rounding, 2e-5."""
import numpy as np
import pytest

from helpers import make_pair, perturbed_state, rel_err
from synth.cgrid import make_cgrid, make_rect_grid

pytestmark = pytest.mark.gpu

SIZES = [(10, 13, 4), (34, 5, 16), (24, 9, 4), (70, 17, 8), (66, 24, 0), (40, 8, 0), (50, 2, 0), (130, 72, 12),
         (64, 250, 8), (48, 256, 6), (2100, 20, 100), (4200, 10, 0)]


def _grid(ni, nj, nw):
    return make_cgrid(ni, nj, n_wake=nw, wall_spacing=1e-3) if nw else make_rect_grid(ni, nj, 4.0, 1.0, jitter=0.05)


@pytest.mark.parametrize("kind", ["warp", "warp8"])
@pytest.mark.parametrize("ni,nj,nw", SIZES)
def test_strip_sweep_equals_the_lexicographic_sweep(ni, nj, nw, kind):
    g = _grid(ni, nj, nw)
    u = perturbed_state(0.6, 1.0, nj, ni, amp=0.01, seed=ni)
    r = np.random.default_rng(nj).standard_normal((4, nj, ni))
    for precision, tol in (("fp64", 1e-11), ("mixed", 2e-5)):
        o, s = make_pair(g, nlevels=1, mach=0.6, alpha_deg=1.0, precision=precision)
        s.set_sweep(kind)
        o.set_state(u)
        s.set_state(u)
        z = s.precond_apply(r, 50.0)
        assert rel_err(z, o.precond_apply(r, 50.0)[0]) < tol
        assert np.array_equal(z, s.precond_apply(r, 50.0))  # a second pass finds the buffers as the first did
        s.close()
