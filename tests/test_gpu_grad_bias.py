"""The gradient contraction has no lean towards zero.  With all points equal phi is exactly
1, so the outputscale form is sum_ij G_ij = sum_c alpha_c (sum_i U_ic) (sum_j V_jc), and what
is left of its error is that of the contraction and of the sums.  Entries of one sign:

  - FP32 sums of 128 entries, every addition rounded to nearest: a relative error of about
    2^-24 sqrt(128 / 3) = 3.9e-7 each, independent over the n^2 / 256 = 2^20 of them, 3.9e-10
    in all; five of those are 2e-9;
  - an accumulation that cuts off leaves a mean error of the same sign everywhere, which the
    n^2 entries do not average out: 3.4e-9 at c = 32 with the parts' own cut-off."""
import numpy as np
import pytest
import torch

import paper_2310_17137_gb300 as ap
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kern", [wl.RBF, wl.MATERN32, wl.MATERN52])
@pytest.mark.parametrize("c", [4, 16, 32])
def test_same_sign_sums_have_no_mean_error(kern, c):
    n = 16384
    rng = np.random.default_rng(61)
    X = torch.zeros(n, 3, device="cuda:0")
    ctx = ap.ap_create(X, ap.Hyper(kern, np.ones(3), 1.0, 0.5), ap.ap_opts_default(block=256))
    U, V = rng.uniform(0.5, 1.5, (2, n, c)).astype(np.float32)
    alpha = np.ones(c)
    got = ap.ap_grad_quadforms(ctx, torch.from_numpy(U).cuda(), torch.from_numpy(V).cuda(), alpha)
    want = (U.astype(np.float64).sum(0) * V.astype(np.float64).sum(0)).sum()
    assert np.all(got[:3] == 0.0)
    assert abs(got[3] - want) <= 2e-9 * want, (got[3] - want) / want
    ap.ap_destroy(ctx)
