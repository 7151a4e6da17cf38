"""phi of the Cholesky cache at the ends of its argument: zero, far beyond underflow, and
NaN, which the Matern kernels hand on (whatever its sign bit)."""
import numpy as np
import pytest

import paper_2310_17137_gb300 as ap
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kern", [wl.RBF, wl.MATERN32, wl.MATERN52])
def test_ends_of_the_argument(kern):
    got = ap.ap_phi_fp64_eval(kern, [0.0, 1e-300, 1e-40, 1e13, 1e300, np.inf])
    assert np.array_equal(got, [1.0, 1.0, 1.0, 0.0, 0.0, 0.0])


@pytest.mark.parametrize("kern", [wl.MATERN32, wl.MATERN52])
def test_a_nan_stays_a_nan(kern):
    got = ap.ap_phi_fp64_eval(kern, [np.nan, -np.nan, 1.0])
    assert np.isnan(got[0]) and np.isnan(got[1]) and 0.0 < got[2] < 1.0
