"""The warp-strip sweep's warps pass stages, edge entries and decisions among themselves while they run: many
applications side by side, on streams of three host threads and of sizes whose strips wait on one another for
most of their steps, give the same bits every time."""
import threading

import numpy as np
import pytest

import paper_1710_04875_gb300 as P
from helpers import perturbed_state
from synth.cgrid import make_cgrid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_many_applications_side_by_side_give_the_same_bits(precision):
    torch = pytest.importorskip("torch")
    bad = []

    def apply(ni, nj, nw):
        stream = torch.cuda.Stream()
        s = P.Solver(make_cgrid(ni, nj, n_wake=nw, wall_spacing=1e-3),
                     P.default_params(mach=0.6, alpha_deg=1.0, nlevels=1, precision=precision), stream=stream.cuda_stream)
        s.set_state(perturbed_state(0.6, 1.0, nj, ni, amp=0.01, seed=ni))
        r = np.random.default_rng(nj).standard_normal((4, nj, ni))
        z = s.precond_apply(r, 50.0)
        same = all(np.array_equal(s.precond_apply(r, 50.0), z) for _ in range(60))
        s.close()
        if not (same and np.all(np.isfinite(z))):
            bad.append((ni, nj))

    threads = [threading.Thread(target=apply, args=a) for a in ((96, 256, 16), (130, 72, 12), (40, 200, 4))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
