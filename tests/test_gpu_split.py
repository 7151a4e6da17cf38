"""The FP32 product's split into row tiles, cluster splits and column groups: shapes at
the edges of the split rule (fewer rows than a tile, one row more than a tile, columns
that leave the last ranges empty or short, groups and no groups), against the oracle.
Every output sums n terms in FP32 whatever the split, so the tolerance is that of the
plain product: 2e-5 (sum_j |K_ij| |v_j| + |base_i|)."""
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


@pytest.mark.parametrize("n,d,M,kern", [(63, 3, 1, wl.RBF), (65, 4, 129, wl.MATERN52), (1023, 11, 16, wl.MATERN32),
                                        (1025, 17, 513, wl.RBF), (5000, 2, 1, wl.MATERN52), (20003, 9, 1024, wl.RBF),
                                        (3001, 25, 4100, wl.MATERN32)])
def test_mean_over_split_shapes(n, d, M, kern):
    p = wl.random_problem(n, d, 256, 1, kern, 0.05, 21)
    ctx = ap.ap_create(_t(p.X), ap.Hyper(kern, p.lengthscale, 1.3, p.noise, 0.25), ap.ap_opts_default(block=256))
    w = np.random.default_rng(3).standard_normal(n).astype(np.float32)
    Xt = wl.test_points(p, m=M)
    h = oracle.Hyper(kern, p.lengthscale.astype(np.float64), 1.3, p.noise, 0.25)
    K = oracle.gram(h, Xt.astype(np.float64), p.X.astype(np.float64), noise=False)
    ref = oracle.predict_mean(h, p.X.astype(np.float64), w.astype(np.float64), Xt.astype(np.float64))
    bound = TOL_PROD * (np.abs(K) @ np.abs(w.astype(np.float64)) + 0.25)
    first = ap.ap_predict_mean(ctx, _t(w), _t(Xt)).cpu().numpy()
    again = ap.ap_predict_mean(ctx, _t(w), _t(Xt)).cpu().numpy()
    assert np.all(np.abs(first - ref) <= bound), np.max(np.abs(first - ref) / bound)
    assert np.array_equal(first, again)  # fixed-order sums; the tickets are back at zero
    ap.ap_destroy(ctx)


@pytest.mark.parametrize("n,d,b,c,kern", [(600, 3, 600, 1, wl.MATERN52), (1281, 6, 640, 4, wl.RBF),
                                          (4097, 5, 2048, 1, wl.MATERN32), (700, 19, 100, 1, wl.RBF)])
def test_steps_and_residual_over_split_shapes(n, d, b, c, kern):
    p = wl.random_problem(n, d, b, c, kern, 0.1, 22)
    h = oracle.Hyper.of(p)
    X, B = p.X.astype(np.float64), p.B.astype(np.float64)
    k = 2 * (-(-n // b)) + 1
    ctx = ap.ap_create(_t(p.X), ap.Hyper(kern, p.lengthscale, p.outputscale, p.noise),
                       ap.ap_opts_default(block=b, tol=1e-30, min_epochs=0, max_steps=k), trace_cap=k)
    st, W, info, trace = ap.ap_solve(ctx, _t(p.B))
    assert st == ap.AP_ERR_NOT_CONVERGED and info["steps"] == k
    R = ap.ap_residual(ctx, _t(p.B), W).cpu().numpy()
    W = W.cpu().numpy().astype(np.float64)
    r = oracle.ap_solve(h, X, B, b, select=oracle.SEL_FORCED, forced=trace, max_steps=k, trace_cap=k)
    assert np.abs(W - r.W).max() <= 2e-4 * np.abs(r.W).max()
    K = oracle.gram(h, X)
    bound = TOL_PROD * (np.abs(K) @ np.abs(W) + np.abs(B))
    assert np.all(np.abs(R - oracle.residual_rows(h, X, B, W)) <= bound)
    ap.ap_destroy(ctx)


def test_groups_are_given_back_when_the_budget_needs_the_bytes():
    """The group sums are optional: a context whose budget has no room left for a
    required buffer releases them and computes the same result without groups."""
    n, M = 6000, 40000
    p = wl.random_problem(n, 3, 512, 1, wl.RBF, 0.05, 23)
    hyper = ap.Hyper(wl.RBF, p.lengthscale, 1.0, p.noise)
    w = _t(np.random.default_rng(4).standard_normal(n))
    Xt = _t(wl.test_points(p, m=M))
    free = ap.ap_create(_t(p.X), hyper, ap.ap_opts_default(block=512))
    ref = ap.ap_predict_mean(free, w, Xt)
    need = M * 4 * 4  # the scaled test inputs
    tight = ap.ap_create(_t(p.X), hyper, ap.ap_opts_default(block=512, hbm_budget=64 << 20))
    few = ap.ap_predict_mean(tight, w, Xt[:100].contiguous())
    tight2 = ap.ap_create(_t(p.X), hyper, ap.ap_opts_default(
        block=512, hbm_budget=max(ap.ap_device_bytes(tight), (16 << 20)) + need))
    ap.ap_predict_mean(tight2, w, Xt[:100].contiguous())
    out = ap.ap_predict_mean(tight2, w, Xt)
    assert float((out - ref).abs().max()) <= TOL_PROD * float(w.abs().sum())
    assert float((few - ref[:100]).abs().max()) <= TOL_PROD * float(w.abs().sum())
    for c in (free, tight, tight2):
        ap.ap_destroy(c)
