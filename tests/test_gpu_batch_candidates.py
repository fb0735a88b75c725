"""What the batch autotuner chooses among: the warp strips with the smaller ring (kind 10), which let strips of
different cases share an SM, also in mixed precision where the batch has more strips than the device SMs; and a
batch that takes them runs as its cases do by themselves."""
import numpy as np
import pytest

import paper_1710_04875_gb300 as P
from helpers import rel_err
from synth.cgrid import make_cgrid

pytestmark = pytest.mark.gpu


def _batch(n, precision):
    g = make_cgrid(32, 8)
    p = P.default_params(mach=0.6, alpha_deg=1.0, nlevels=1, cfl=20.0, precision=precision)
    return g, p, P.fasw.Batch([g] * n, [p] * n)


@pytest.mark.parametrize("precision,n,kinds", [("mixed", 4, {2, 6, 7, 9}), ("mixed", 160, {2, 6, 7, 9, 10}),
                                               ("fp64", 4, {2, 9, 10}), ("fp64", 160, {2, 9, 10})])
def test_candidates_of_small_and_full_batches(precision, n, kinds):
    g, p, b = _batch(n, precision)
    assert set(b.candidates(precision)) == kinds
    if n > 4 and precision == "mixed":
        assert set(b.autotune()) <= kinds
        b.cycle(0)
        s = P.Solver(g, p)
        s.fas_cycle(0)
        want = s.get_state()
        assert all(rel_err(b.get_state(k), want) < 1e-5 for k in (0, n // 2, n - 1))
        s.close()
    b.close()
