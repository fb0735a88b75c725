"""The library's FP64 reciprocal at the arguments whose reciprocal is not a normal number, and around them: the
division's result (zeros, infinities, subnormals, NaNs), on the host in IEEE arithmetic."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_reciprocal_outside_the_normal_range():
    import paper_1710_04875_gb300 as P
    a = np.array([0.0, np.inf, 5e-324, 1e-310, 2.0**-1024, 2.0**-1023, np.nextafter(2.0**-1022, 0.0), 2.0**-1022,
                  np.nextafter(2.0**-1022, 1.0), 2.0**1021, np.nextafter(2.0**1022, 0.0), 2.0**1022, 2.0**1023, 1.7e308,
                  np.finfo(float).max, 3.0 * 2.0**1020, 3.0 * 2.0**-1022])
    a = np.concatenate([a, -a, [np.nan]])
    rcp = P.fasw.check_fp64(a)[0]
    with np.errstate(all="ignore"):
        want = 1.0 / a
    assert np.isnan(rcp[-1])
    assert np.array_equal(rcp[:-1].view(np.uint64), want[:-1].view(np.uint64))
