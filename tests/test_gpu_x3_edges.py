"""The FP32 product's two forms with more than four right-hand sides on both sides of the
line between them (2.2e7 entries for 16 columns, 8e6 for 32): rows and columns at the
edges of tiles and chunks, every padded dimension, short last blocks, non-finite values,
timings aside the same results.  Against float64 rows at the bound of the plain product,
2e-5 (sum_j |K_ij| |w_j| + |b_i|)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2310_17137_gb300 as ap
import workloads as wl

pytestmark = pytest.mark.gpu
TOL_PROD = 2e-5


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to("cuda:0")


def _ctx(p, trace_cap=0, **kw):
    return ap.ap_create(_t(p.X), ap.Hyper(p.kernel, p.lengthscale, p.outputscale, p.noise),
                        ap.ap_opts_default(block=p.block, **kw), trace_cap=trace_cap)


@pytest.mark.parametrize("n,d,c,kern", [
    (4690, 8, 16, wl.RBF), (4691, 3, 16, wl.MATERN52), (4736, 4, 16, wl.RBF), (4737, 6, 9, wl.MATERN32),
    (4865, 11, 16, wl.MATERN52), (4991, 15, 5, wl.RBF), (5000, 22, 16, wl.MATERN32), (5121, 32, 16, wl.MATERN52),
    (2828, 8, 32, wl.MATERN32), (2829, 8, 32, wl.MATERN32), (2944, 2, 32, wl.RBF), (2945, 9, 17, wl.MATERN52),
    (3073, 14, 32, wl.RBF), (3199, 24, 32, wl.MATERN32), (3000, 29, 31, wl.RBF), (300, 17, 32, wl.MATERN32),
    (129, 30, 16, wl.RBF), (1793, 12, 32, wl.RBF), (2900, 5, 16, wl.MATERN52)])
def test_residual_on_both_sides_of_the_line(n, d, c, kern):
    p = wl.random_problem(n, d, 64, c, kern, 0.1, 101)
    h, X, B = oracle.Hyper.of(p), p.X.astype(np.float64), p.B.astype(np.float64)
    ctx = _ctx(p)
    W = np.random.default_rng(11).standard_normal((n, c)).astype(np.float32)
    R = ap.ap_residual(ctx, _t(p.B), _t(W))
    assert torch.equal(R, ap.ap_residual(ctx, _t(p.B), _t(W)))  # fixed-order sums
    rows = np.unique(np.r_[0, n - 1, np.arange(0, n, max(1, n // 250))])
    K = np.concatenate([oracle.gram(h, X[i:i + 1], X, row0=int(i)) for i in rows])
    W = W.astype(np.float64)
    assert np.all(np.abs(R.cpu().numpy()[rows] - (B[rows] - K @ W)) <= TOL_PROD * (np.abs(K) @ np.abs(W) + np.abs(B[rows])))
    ap.ap_destroy(ctx)


@pytest.mark.parametrize("n,d,b,c,kern", [(7000, 3, 3400, 16, wl.MATERN32), (6000, 12, 4000, 9, wl.RBF),
                                          (3500, 5, 2400, 32, wl.MATERN52), (4000, 20, 2100, 32, wl.MATERN32),
                                          (2400, 8, 1000, 32, wl.RBF), (2600, 3, 700, 16, wl.MATERN52),
                                          (1500, 25, 400, 32, wl.MATERN32)])
def test_steps_with_short_last_blocks(n, d, b, c, kern):
    p = wl.random_problem(n, d, b, c, kern, 0.1, 102)
    k = -(-n // b) + 1
    ctx = _ctx(p, trace_cap=k, tol=1e-30, min_epochs=0, max_steps=k, select=ap.AP_SEL_CYCLIC)
    st, W, info, trace = ap.ap_solve(ctx, _t(p.B))
    assert st == ap.AP_ERR_NOT_CONVERGED and info["steps"] == k
    r = oracle.ap_solve(oracle.Hyper.of(p), p.X.astype(np.float64), p.B.astype(np.float64), b,
                        select=oracle.SEL_FORCED, forced=trace, max_steps=k, trace_cap=k)
    assert np.abs(W.cpu().numpy() - r.W).max() <= 2e-4 * np.abs(r.W).max()
    ap.ap_destroy(ctx)


@pytest.mark.parametrize("n,c", [(4800, 16), (3000, 32)])
def test_every_split_product_is_there(n, c):
    """All terms positive and of equal mantissa, so that a split product that is missing
    shows: hm, mh weigh 2^-9 of the result or more, hl, lh, mm at least 2^-18 = 3.8e-6.  The
    FP32 entries' own error here (|t| <= 3) is at most 3.8e-7 + 2.4e-7, the sums' 2e-7."""
    p = wl.random_problem(n, 3, 500, c, wl.RBF, 0.1, 103, ell_range=(1.0, 3.0))
    ctx = _ctx(p)
    scale = 2.0 ** np.random.default_rng(6).integers(-3, 3, (n, c))
    W = (scale * (1.0 + 2.0 ** -8 + 2.0 ** -9 + 2.0 ** -16 + 2.0 ** -17 + 2.0 ** -23)).astype(np.float32)
    R = -ap.ap_residual(ctx, torch.zeros(n, c, device="cuda"), _t(W)).cpu().numpy().astype(np.float64)
    ref = oracle.gram(oracle.Hyper.of(p), p.X.astype(np.float64)) @ W.astype(np.float64)
    assert np.max(np.abs(R - ref) / ref) <= 1.5e-6
    ap.ap_destroy(ctx)


@pytest.mark.parametrize("n,c", [(4800, 16), (3000, 32)])
def test_infinities_and_nans_reach_their_column_only(n, c):
    p = wl.random_problem(n, 3, 300, c, wl.MATERN52, 0.1, 104)
    ctx = _ctx(p)
    W = np.random.default_rng(7).standard_normal((n, c)).astype(np.float32)
    good = ap.ap_residual(ctx, _t(p.B), _t(W)).cpu().numpy()
    bad = [(450, 1), (3, 4), (n - 1, 4), (200, 9), (128, 12), (n - 2, c - 1)]
    for (i, k), v in zip(bad, [np.inf, -np.inf, np.inf, np.nan, 3.4e38, -np.inf]):
        W[i, k] = v
    R = ap.ap_residual(ctx, _t(p.B), _t(W)).cpu().numpy()
    rest = [k for k in range(c) if k not in (1, 4, 9, 12, c - 1)]
    assert np.array_equal(R[:, rest], good[:, rest])
    assert np.all(R[:, 1] == -np.inf) and np.all(R[:, c - 1] == np.inf)
    assert np.all(np.isnan(R[:, 4])) and np.all(np.isnan(R[:, 9]))
    # 3.4e38 stays finite but on its own row, where (1 + noise) 3.4e38 is above the largest float
    others = np.arange(n) != 128
    assert np.all(np.isfinite(R[others, 12])) and np.all(R[others, 12] < -1e34) and R[128, 12] == -np.inf
    for i, k in bad:  # the flags do not stay behind
        W[i, k] = 0.5
    R = ap.ap_residual(ctx, _t(p.B), _t(W)).cpu().numpy()
    assert np.all(np.isfinite(R)) and np.array_equal(R[:, rest], good[:, rest])
    ap.ap_destroy(ctx)
