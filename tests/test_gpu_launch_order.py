"""Launches that overlap against launches one after the other (fasw_ordered_launches): several kernels read, and
one writes, before they wait for the kernel before, on the rule that no writer or reader of that memory comes
directly before them.  A launch sequence that breaks the rule is a race; here every sequence of the library runs
both ways and gives the same bits."""
import numpy as np
import pytest

import paper_1710_04875_gb300 as P
from helpers import perturbed_state
from synth.cgrid import make_cgrid
from test_zz_no_alloc import _noalloc_residual

pytestmark = pytest.mark.gpu

RANS = dict(viscous=1, turb=1, sensor=1, re=1e6, mach=0.6, gamma_cycle=2, cfl=50.0, nlevels=3)
EULER = dict(mach=0.6, alpha_deg=1.0, cfl=50.0, nlevels=2)


def _state(ni, nj, alpha=0.0):
    return perturbed_state(0.6, alpha, nj, ni, amp=0.005, seed=ni)


def _solver(ni, nj, nw, torch, **kw):
    s = P.Solver(make_cgrid(ni, nj, n_wake=nw, wall_spacing=1e-3), P.default_params(**kw),
                 stream=torch.cuda.current_stream().cuda_stream)
    s.set_state(_state(ni, nj))
    return s


def _cycles(torch, ni, nj, nw, graphs, **kw):
    s = _solver(ni, nj, nw, torch, **kw)
    s.use_graphs(graphs)
    out = [s.fas_cycle(k) for k in range(2)] + [s.get_state()]
    out += list(s.residual()) + [s.precond_apply(_state(ni, nj), 10.0), s.pseudo_dt(3.0)]
    s.close()
    return out


def _smooth(torch, ni, nj, nw, **kw):
    s = _solver(ni, nj, nw, torch, **kw)
    s.smooth(3, 2.0)
    out = [s.get_state()]
    s.close()
    return out


def _pitch(torch, **kw):
    s = _solver(128, 32, 16, torch, **kw)
    out = []
    for k in range(2):
        s.set_motion(0.01 * (k + 1), 0.02)
        out += [s.dual_time_step(0.05, 1e-9, 2)[2], s.get_state()]
    s.close()
    return out


def _batch(torch, precision):
    sizes = [(64, 16, 8), (96, 24, 12), (128, 32, 16), (64, 16, 0), (256, 64, 32)]
    b = P.fasw.Batch([make_cgrid(*z[:2], n_wake=z[2]) for z in sizes],
                     [P.default_params(precision=precision, **EULER) for _ in sizes])
    out = [b.cycle(0), b.cycle(3)] + [b.get_state(k) for k in range(len(sizes))]
    b.close()
    return out


def _adjoint(torch, jacobian, **kw):
    s = _solver(64, 16, 8, torch, **kw)
    s.adjoint_set_jacobian(jacobian)
    s.adjoint_jacobian()
    v = _state(64, 16)
    lam = s.adjoint_solve(which=1, tol=1e-14, max_iters=4)[0]
    out = [lam, s.adjoint_apply(v), s.adjoint_apply(v, transpose=True), s.adjoint_precond_apply(v, 5.0),
           s.adjoint_cycle_apply(v, 5.0), s.adjoint_cycle_apply(v, 5.0, kind="smoother", transpose=False)]
    out += list(s.adjoint_vertex_gradient(1, lam))
    s.close()
    return out


def _noalloc(torch):
    g = make_cgrid(128, 32, n_wake=16, wall_spacing=1e-3)
    u = torch.from_numpy(_state(128, 32).ravel()).cuda()
    return [_noalloc_residual(P.library(), g, P.default_params(nlevels=1, viscous=1, re=1e5, mach=0.6), u, torch)[1]]


RUNS = {f"cycles-{n}-{p}-{g}": (_cycles, (*size, g), dict(precision=p, **kw))
        for p in ("fp64", "mixed") for g in (True, False)
        for n, size, kw in (("euler64x16", (64, 16, 8), EULER), ("rans256x64", (256, 64, 32), RANS),
                            ("rans512x128", (512, 128, 64), RANS))}
RUNS.update({f"smooth-{s}-{p}": (_smooth, (66, 18, 8), dict(precision=p, scheme=s, nlevels=1, mach=0.6))
             for p in ("fp64", "mixed") for s in ("AW51", "ARK3J")})
RUNS.update({f"pitch-{p}": (_pitch, (), dict(precision=p, **RANS)) for p in ("fp64", "mixed")})
RUNS.update({f"batch-{p}": (_batch, (p,), {}) for p in ("fp64", "mixed")})
RUNS.update({f"adjoint-{j}-{p}": (_adjoint, (j,), dict(precision=p, **RANS)) for p in ("fp64", "mixed")
             for j in ("tangent", "differences")})
RUNS["noalloc"] = (_noalloc, (), {})


@pytest.mark.parametrize("name", RUNS)
def test_overlapping_launches_give_the_bits_of_ordered_ones(name):
    torch = pytest.importorskip("torch")
    run, args, kw = RUNS[name]
    lib, out = P.library(), []
    with torch.cuda.stream(torch.cuda.Stream()):
        for ordered in (1, 0, 0):
            assert lib.fasw_ordered_launches(ordered) == 0
            try:
                out.append(run(torch, *args, **kw))
            finally:
                assert lib.fasw_ordered_launches(0) == ordered
    for got in out[1:]:
        assert all(np.array_equal(a, b, equal_nan=True) for a, b in zip(got, out[0]))
    assert all(np.all(np.isfinite(a)) for a in out[0])
