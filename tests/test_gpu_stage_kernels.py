"""The smoothing stage's kernels around the warp-strip sweep against the general path (the one-CTA sweep,
whose blocks, right-hand side and update are kernels of their own): the stage update that waits for the
next launch over schemes that read dt* in it (ARK) and that do not (AW), cycle shapes and repeated
smoothing, callers' buffers in place, and the FP64 block preparation where its last block is partly
filled and where it changes (up to 16,384 cells it forms the diagonal blocks too).

Tolerance: in FP64 the two sweeps agree to 1e-14 of the state; a cycle of two levels amplifies that (ARK
by up to 500, between any two FP64 sweeps): 1e-11."""
import numpy as np
import pytest

import paper_1710_04875_gb300 as P
from helpers import rel_err
from synth.cgrid import make_cgrid

pytestmark = pytest.mark.gpu


def _solver(ni, nj, nw, kind, **kw):
    s = P.Solver(make_cgrid(ni, nj, n_wake=nw, wall_spacing=1e-3),
                 P.default_params(mach=0.6, alpha_deg=1.0, precision="fp64", cfl=2.0, **kw))
    s.set_sweep(kind)  # from the free stream
    return s


@pytest.mark.parametrize("scheme", ["AW3", "ARK51"])
@pytest.mark.parametrize("nlevels,nu1,gamma", [(1, 1, 1), (1, 3, 1), (2, 1, 2), (2, 2, 1)])
def test_waiting_update_equals_the_update_kernel(scheme, nlevels, nu1, gamma):
    u = []
    for kind in ("warp", "cta"):
        s = _solver(64, 16, 8, kind, scheme=scheme, nlevels=nlevels, nu1=nu1, gamma_cycle=gamma)
        s.fas_cycle(0)
        u.append(s.get_state())
        s.close()
    assert rel_err(u[0], u[1]) < 1e-11


@pytest.mark.parametrize("scheme", ["AW51", "ARK3J"])
def test_repeated_smoothing_equals_the_update_kernel(scheme):
    u = []
    for kind in ("warp", "cta"):
        s = _solver(36, 9, 4, kind, scheme=scheme, nlevels=1)
        s.smooth(3, 2.0)
        u.append(s.get_state())
        s.close()
    assert rel_err(u[0], u[1]) < 1e-11


@pytest.mark.parametrize("ni,nj,nw", [(10, 2, 2), (34, 3, 6), (152, 16, 20), (256, 64, 32), (258, 64, 32)])
def test_block_rows_equal_the_cell_kernel(ni, nj, nw):
    r = np.random.default_rng(ni).standard_normal((4, nj, ni))
    z = []
    for kind in ("warp", "cta"):
        s = _solver(ni, nj, nw, kind, nlevels=1)
        z.append(s.precond_apply(r, 20.0))
        s.close()
    assert rel_err(z[0], z[1]) < 1e-11


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("offset", [0, 4])
def test_callers_device_buffers_in_any_place(precision, offset):
    """State and preconditioner calls on the caller's device memory, aligned (used as it is) and four bytes
    off (copied), with the result over the right-hand side: the bits of the calls on host arrays."""
    torch = pytest.importorskip("torch")
    ni, nj = 36, 9
    s = P.Solver(make_cgrid(ni, nj, n_wake=4, wall_spacing=1e-3),
                 P.default_params(mach=0.6, alpha_deg=1.0, precision=precision, cfl=2.0, nlevels=1))
    rng = np.random.default_rng(3)
    u = s.get_state() * (1.0 + 1e-3 * rng.standard_normal((4, nj, ni)))
    r = rng.standard_normal((4, nj, ni))
    s.set_state(u)
    z = s.precond_apply(r, 20.0)
    raw = [torch.zeros(8 * u.size + 8, dtype=torch.uint8, device="cuda") for _ in range(2)]
    for t, a in zip(raw, (u, r)):
        t[offset:offset + 8 * a.size] = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).ravel()).cuda()
    torch.cuda.synchronize()
    at = [t.data_ptr() + offset for t in raw]
    lib = P.fasw.library()
    assert lib.fasw_set_state(s.h, 0, at[0], 1) == 0
    assert lib.fasw_precond_apply(s.h, 0, 20.0, at[1], at[1], 1) == 0
    assert lib.fasw_get_state(s.h, 0, at[0], 1) == 0
    got = [t[offset:offset + 8 * u.size].cpu().numpy().view(np.float64).reshape(u.shape) for t in raw]
    s.close()
    assert np.array_equal(got[0], u) and np.array_equal(got[1], z)
