"""The transposed preconditioner P^-T r of FP64 contexts against the two block-triangular solves in FP64 on
the oracle's blocks: P = S^-1 (D + L) D^-1 (D + U), S = eta dt*.

Tolerance (largest error over largest entry): a cell's unknown is a sum of 16 products and a 4x4 solve, whose
roundings (1.1e-16 each) and whose blocks' (up to 8e-16 an entry, theirs and the oracle's) the two solves
amplify by up to three: 5e-15.  An FP32 solve with one FP64 correction leaves (1.2e-7)^2 = 1.4e-14 and more."""
import numpy as np
import pytest

from helpers import make_pair, perturbed_state
from synth.cgrid import make_cgrid

pytestmark = pytest.mark.gpu


def _solve_transposed(o, r, cfl, nw, eta=0.8):
    axp, axm, aep, aem = o.face_blocks()
    dts, vol = o.pseudo_dt(cfl), o.metrics(o.finest)[4]
    nj, ni = dts.shape
    c = (eta * dts / vol)[..., None, None]
    W, E, S, N = -c * axp[:, :-1], c * axm[:, 1:], -c * aep[:-1], c * aem[1:]
    DT = np.swapaxes(np.eye(4) + c * ((axp[:, 1:] - axm[:, :-1]) + (aep[1:] - aem[:-1])), -1, -2).copy()
    r = r.transpose(1, 2, 0).copy()
    a, z = np.zeros_like(r), np.zeros_like(r)
    for j in range(nj):                      # (D + U)^T a = r
        for i in range(ni):
            x = a[j, i] = np.linalg.solve(DT[j, i], r[j, i])
            if i < ni - 1:
                r[j, i + 1] -= E[j, i].T @ x
            if j < nj - 1:
                r[j + 1, i] -= N[j, i].T @ x
            if j == 0 and i < nw:            # the lower wake's cells come before their mirrors
                r[0, ni - 1 - i] -= S[0, i].T @ x
    r = (DT @ a[..., None])[..., 0]
    for j in range(nj - 1, -1, -1):          # (D + L)^T z = D^T a
        for i in range(ni - 1, -1, -1):
            x = z[j, i] = np.linalg.solve(DT[j, i], r[j, i])
            if i > 0:
                r[j, i - 1] -= W[j, i].T @ x
            if j > 0:
                r[j - 1, i] -= S[j, i].T @ x
            if j == 0 and i >= ni - nw:
                r[0, ni - 1 - i] -= S[0, i].T @ x
    return (eta * dts) * z.transpose(2, 0, 1)


@pytest.mark.parametrize("ni,nj,nw,viscous", [(64, 16, 8, 0), (150, 43, 18, 1), (40, 9, 0, 0)])
def test_transposed_preconditioner_is_exact_to_fp64(ni, nj, nw, viscous):
    g = make_cgrid(ni, nj, n_wake=nw, wall_spacing=1e-3)
    o, s = make_pair(g, nlevels=1, mach=0.6, alpha_deg=1.0, viscous=viscous, re=5e4)
    u = perturbed_state(0.6, 1.0, nj, ni, amp=0.01, seed=ni)
    r = np.random.default_rng(nj).standard_normal((4, nj, ni))
    o.set_state(u)
    s.set_state(u)
    for cfl in (5.0, 100.0):
        want = _solve_transposed(o, r, cfl, nw)
        assert np.abs(s.adjoint_precond_apply(r, cfl) - want).max() < 5e-15 * np.abs(want).max()
    s.close()


@pytest.mark.parametrize("levels", [1, 2])
def test_operators_take_right_hand_sides_of_any_size(levels):
    """The operators are linear: of a right-hand side times a power of two they give the result times it, bit
    for bit, beyond the range of FP32 too; a right-hand side of zeros gives zeros."""
    import paper_1710_04875_gb300 as P
    ni, nj = 64, 16
    s = P.Solver(make_cgrid(ni, nj, n_wake=8, wall_spacing=1e-3),
                 P.default_params(mach=0.6, alpha_deg=1.0, nlevels=levels, gamma_cycle=2))
    s.set_state(perturbed_state(0.6, 1.0, nj, ni, amp=0.01, seed=1))
    s.adjoint_jacobian()
    r = np.random.default_rng(2).standard_normal((4, nj, ni))
    kind = "cycle" if levels > 1 else "smoother"
    for apply in (lambda v: s.adjoint_precond_apply(v, 5.0), lambda v: s.adjoint_precond_apply(v, 5.0, steps=1),
                  lambda v: s.adjoint_cycle_apply(v, 5.0, kind=kind), lambda v: s.adjoint_cycle_apply(v, 5.0, kind=kind, transpose=False)):
        z = apply(r)
        assert np.all(np.isfinite(z)) and np.any(z)
        for e in (-700.0, -130.0, 130.0, 700.0):
            assert np.array_equal(apply(r * 2.0**e), z * 2.0**e)
        assert not np.any(apply(0.0 * r))
    s.close()


def test_stage_loops_that_amplify_stay_in_the_range_of_fp64():
    """The stage loop on J^T is not a convergent iteration: many steps of it leave FP32's range, not FP64's.  The
    result is finite, linear in the right-hand side, and the step after it is that of the steps' recurrence."""
    import paper_1710_04875_gb300 as P
    ni, nj = 64, 16
    s = P.Solver(make_cgrid(ni, nj, n_wake=8, wall_spacing=1e-3), P.default_params(mach=0.6, alpha_deg=1.0, nlevels=1))
    s.set_state(perturbed_state(0.6, 1.0, nj, ni, amp=0.01, seed=1))
    s.adjoint_jacobian()
    r = np.random.default_rng(2).standard_normal((4, nj, ni))
    n = 1
    while np.abs(z := s.adjoint_precond_apply(r, 200.0, steps=n)).max() < 1e60 and n < 4096:
        n *= 2
    assert np.all(np.isfinite(z)) and np.abs(z).max() > 1e60
    assert np.array_equal(s.adjoint_precond_apply(r * 2.0**-60, 200.0, steps=n), z * 2.0**-60)
    # x_(n+1) = x_n + S (r - J^T x_n), S the step from zero
    more = s.adjoint_precond_apply(r, 200.0, steps=n + 1)
    want = z + s.adjoint_precond_apply(r - s.adjoint_apply(z, transpose=True), 200.0, steps=1)
    assert np.abs(more - want).max() < 1e-10 * np.abs(more).max()
    s.close()
