"""The tensor-core contraction has little of a mean error.  Columns lie at 64 distinct
distances from 128 equal row points, so every entry is one of 64 values, which single unit
vectors give back exactly; sums over W > 0 are compared with the float64 sums of those
values, on average over 128 of them.

  - The FP32 additions of 74 drained sums are rounded to nearest: at most 2^-24 sqrt(74 / 3)
    = 3.0e-7 each, 2.6e-8 of the average of 128; two of those are 5e-8 (the sums differ in W).
  - A tensor-core step that is added to a running sum cuts off half a unit in the last place
    on average, 0.5 * 2^-23 * 0.72 = 4.3e-8 of that sum: 4.3e-8 in all when every step of a
    drain has its own accumulator, 6.4e-8 with two for four steps, 1.07e-7 with one.

The bounds are the cut-off's mean plus two standard deviations where each step has its own
accumulator (16 columns), and likewise with two (32 columns)."""
import numpy as np
import pytest
import torch

import paper_2310_17137_gb300 as ap
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kern,ell", [(wl.RBF, 0.2), (wl.MATERN32, 0.12), (wl.MATERN52, 0.12)])
@pytest.mark.parametrize("c,bound", [(16, 4.3e-8 + 5e-8), (32, 6.4e-8 + 5e-8)])
def test_mean_error_of_positive_sums(kern, ell, c, bound):
    rows, n, d = 128, 4864, 8
    rng = np.random.default_rng(111)
    X = np.zeros((n, d), np.float32)
    pos = np.concatenate([np.zeros(rows, np.int64), rng.integers(0, 64, n - rows)])
    X[:, 0] = np.where(np.arange(n) < rows, 0.0, (pos + 1) / 64.0)
    ctx = ap.ap_create(torch.from_numpy(X).cuda(), ap.Hyper(kern, np.full(d, ell), 1.0, 0.5), ap.ap_opts_default(block=64))
    Z = torch.zeros(n, c, device="cuda")
    phi = np.zeros(64)
    for k0 in range(0, 64, c):
        W = torch.zeros(n, c)
        for k in range(c):
            W[rows + int(np.flatnonzero(pos[rows:] == k0 + k)[0]), k] = 1.0
        phi[k0:k0 + c] = -ap.ap_residual(ctx, Z, W.cuda())[0].cpu().numpy().astype(np.float64)
    assert np.all(np.diff(phi) < 0) and phi[0] < 1.0
    errs = []
    for _ in range(128 // c):
        W = np.zeros((n, c), np.float32)
        W[rows:] = rng.uniform(0.5, 1.5, (n - rows, c)).astype(np.float32)
        got = -ap.ap_residual(ctx, Z, torch.from_numpy(W).cuda())[:rows].cpu().numpy().astype(np.float64)
        assert np.all(got == got[0])
        want = phi[pos[rows:]] @ W[rows:].astype(np.float64)
        errs.append((got[0] - want) / want)
    assert abs(np.mean(errs)) <= bound, np.mean(errs)
    ap.ap_destroy(ctx)
