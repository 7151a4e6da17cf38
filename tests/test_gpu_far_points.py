"""The compensated product where every other point is very far: squared distances of 1e25
and more, whose kernel values are exactly 0, so the residual is B - (s + sigma^2) W.  An
odd number of points, so that the last pair of columns is half empty.  Tolerance: the
parity tests' own for this form (the output's rounding and 1e-9 of the terms)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2310_17137_gb300 as ap
import workloads as wl

pytestmark = pytest.mark.gpu


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to("cuda:0")


@pytest.mark.parametrize("kern", [wl.RBF, wl.MATERN32, wl.MATERN52])
@pytest.mark.parametrize("c", [1, 4])
def test_compensated_product_of_far_points(kern, c):
    p = wl.random_problem(301, 3, 128, c, kern, 0.1, 51, ell_range=(1e-14, 2e-14))
    ctx = ap.ap_create(_t(p.X), ap.Hyper(kern, p.lengthscale, p.outputscale, p.noise),
                       ap.ap_opts_default(block=128, residual_mode=ap.AP_RESID_COMPENSATED))
    W = np.random.default_rng(11).standard_normal(p.B.shape).astype(np.float32)
    R = ap.ap_residual(ctx, _t(p.B), _t(W)).cpu().numpy()
    X, B, W = p.X.astype(np.float64), p.B.astype(np.float64), W.astype(np.float64)
    h = oracle.Hyper.of(p)
    ref = oracle.residual_rows(h, X, B, W)
    mag = np.abs(oracle.gram(h, X)) @ np.abs(W) + np.abs(B)
    assert np.all(np.abs(R - ref) <= 2.0 ** -23 * np.abs(ref) + 1e-9 * mag)
    ap.ap_destroy(ctx)
