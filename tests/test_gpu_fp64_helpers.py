"""The FP64 helpers that keep off the FP64 pipe, against IEEE arithmetic on the host: the conversions
between FP64 and FP32 are exact in every bit (ties, carries into the exponent, overflow, subnormals,
infinities, NaNs, signed zeros), and the reciprocal is within two units in the last place (two Newton
steps from an 18-bit estimate leave a truncation error of 2^-72 and two roundings)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _values(seed):
    rng = np.random.default_rng(seed)
    bits = rng.integers(0, 2**64, 200000, dtype=np.uint64).view(np.float64)
    x32 = rng.integers(0, 2**32, 200000, dtype=np.uint64).astype(np.uint32).view(np.float32)
    with np.errstate(all="ignore"):
        near = x32.astype(np.float64)
        ties = np.nextafter(x32, np.float32(np.inf)).astype(np.float64)
        mid = np.where(np.isfinite(near) & np.isfinite(ties), 0.5 * near + 0.5 * ties, near)
        edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0**-126, -2.0**-126, 2.0**-127, 2.0**-149, 2.0**-150,
                         2.0**127, 2.0**128 - 2.0**103, 2.0**128 - 2.0**104, -(2.0**128), 1.0 - 2.0**-25,
                         1.0 - 2.0**-53, 1.0 + 2.0**-24, 1.0 + 3 * 2.0**-24, 5e-324, 1.7e308])
        scale = rng.standard_normal(200000) * 10.0 ** rng.uniform(-12, 12, 200000)
    return np.concatenate([bits, near, mid, np.nextafter(mid, np.inf), np.nextafter(mid, -np.inf), edge, scale])


def test_conversions_are_exact_and_the_reciprocal_is_close():
    import paper_1710_04875_gb300 as P
    a = _values(5)
    rcp, div, low, wide = P.fasw.check_fp64(a)
    with np.errstate(all="ignore"):
        want = a.astype(np.float32).astype(np.float64)
    for got in (low, wide):
        nan = np.isnan(want)
        assert np.array_equal(nan, np.isnan(got))
        assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))
    normal = np.isfinite(a) & (np.abs(a) > 1e-300) & (np.abs(a) < 1e300)
    assert np.all(np.abs(rcp[normal] - div[normal]) <= 2 * np.spacing(np.abs(div[normal])))
    assert not np.any(np.isfinite(rcp[np.isnan(a)]))
