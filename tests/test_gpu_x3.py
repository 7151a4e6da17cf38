"""The split-precision tensor-core form of the FP32 product (more than four right-hand
sides) against the oracle, at the edges of its tiles: rows and columns that are not
multiples of 128 or 256, one chunk and many, one and two rows per thread, every padded
dimension, row groups cut between CTAs and (without memory for the parts) whole.

Tolerance of the shapes: that of the plain FP32 product, 2e-5 (sum_j |K_ij| |v_j| + |b_i|)."""
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


def _ctx(p, **kw):
    opts = {k: kw.pop(k) for k in ("trace_cap",) if k in kw}
    return ap.ap_create(_t(p.X), ap.Hyper(p.kernel, p.lengthscale, p.outputscale, p.noise),
                        ap.ap_opts_default(block=p.block, **kw), **opts)


@pytest.mark.parametrize("n,d,b,c,kern", [(1, 1, 1, 5, wl.RBF), (127, 3, 127, 16, wl.MATERN52),
                                          (129, 4, 64, 17, wl.MATERN32), (385, 8, 200, 32, wl.RBF),
                                          (1030, 11, 300, 9, wl.MATERN52), (2500, 15, 1100, 32, wl.MATERN32),
                                          (700, 22, 350, 16, wl.RBF), (900, 32, 256, 32, wl.MATERN52),
                                          (20600, 2, 10300, 16, wl.MATERN32)])
def test_residual_and_steps_over_shapes(n, d, b, c, kern):
    p = wl.random_problem(n, d, b, c, kern, 0.1, 31)
    h = oracle.Hyper.of(p)
    X, B = p.X.astype(np.float64), p.B.astype(np.float64)
    rows = np.arange(0, n, max(1, n // 400))
    ctx = _ctx(p)
    W = np.random.default_rng(5).standard_normal(p.B.shape).astype(np.float32)
    R = ap.ap_residual(ctx, _t(p.B), _t(W)).cpu().numpy()[rows]
    W = W.astype(np.float64)
    K = np.concatenate([oracle.gram(h, X[i:i + 1], X, row0=int(i)) for i in rows])
    bound = TOL_PROD * (np.abs(K) @ np.abs(W) + np.abs(B[rows]))
    assert np.all(np.abs(R - oracle.residual_rows(h, X, B, W, rows=rows)) <= bound)
    ap.ap_destroy(ctx)
    if n > 3000:
        return
    k = 2 * (-(-n // b)) + 1
    ctx = _ctx(p, trace_cap=k, tol=1e-30, min_epochs=0, max_steps=k)
    st, Ws, info, trace = ap.ap_solve(ctx, _t(p.B))
    assert st == ap.AP_ERR_NOT_CONVERGED and info["steps"] == k
    r = oracle.ap_solve(h, X, B, b, select=oracle.SEL_FORCED, forced=trace, max_steps=k, trace_cap=k)
    assert np.abs(Ws.cpu().numpy() - r.W).max() <= 2e-4 * np.abs(r.W).max()
    ap.ap_destroy(ctx)


@pytest.mark.parametrize("c", [16, 32])
def test_every_split_product_is_there(c):
    """All terms positive and of equal mantissa, so that a split product that is missing
    shows: hm, mh weigh 2^-9 of the result or more, hl, lh, mm at least 2^-18 = 3.8e-6.
    The FP32 entries' own error here: |t| <= 3 carries 3 t 2^-24 ln 2 <= 3.8e-7 and
    ex2.approx 2.4e-7 relative; sums 2e-7: 1.5e-6 in all."""
    n, d = 1500, 3
    p = wl.random_problem(n, d, 500, c, wl.RBF, 0.1, 32, ell_range=(1.0, 3.0))
    ctx = _ctx(p)
    scale = 2.0 ** np.random.default_rng(6).integers(-3, 3, (n, c))
    W = (scale * (1.0 + 2.0 ** -8 + 2.0 ** -9 + 2.0 ** -16 + 2.0 ** -17 + 2.0 ** -23)).astype(np.float32)
    Z = torch.zeros(n, c, device="cuda")
    R = -ap.ap_residual(ctx, Z, _t(W)).cpu().numpy().astype(np.float64)
    ref = oracle.gram(oracle.Hyper.of(p), p.X.astype(np.float64)) @ W.astype(np.float64)
    assert np.max(np.abs(R - ref) / ref) <= 1.5e-6
    ap.ap_destroy(ctx)


def test_infinities_and_nans_reach_their_column_only():
    n, c = 700, 16
    p = wl.random_problem(n, 3, 300, c, wl.MATERN52, 0.1, 33)
    ctx = _ctx(p)
    W = np.random.default_rng(7).standard_normal((n, c)).astype(np.float32)
    good = ap.ap_residual(ctx, _t(p.B), _t(W)).cpu().numpy()
    W[450, 1], W[3, 4], W[699, 4], W[200, 9], W[128, 12] = np.inf, -np.inf, np.inf, np.nan, 3.4e38
    R = ap.ap_residual(ctx, _t(p.B), _t(W)).cpu().numpy()
    touched = [1, 4, 9, 12]
    rest = [k for k in range(c) if k not in touched]
    assert np.array_equal(R[:, rest], good[:, rest])
    assert np.all(R[:, 1] == -np.inf) and np.all(np.isnan(R[:, 4])) and np.all(np.isnan(R[:, 9]))
    # 3.4e38 stays finite but on its own row, where (1 + noise) 3.4e38 is above the largest float
    others = np.arange(n) != 128
    assert np.all(np.isfinite(R[others, 12])) and np.all(R[others, 12] < -1e34) and R[128, 12] == -np.inf
    # the flags do not stay behind
    W[[450, 3, 699, 200, 128], [1, 4, 4, 9, 12]] = 0.5
    R = ap.ap_residual(ctx, _t(p.B), _t(W)).cpu().numpy()
    assert np.all(np.isfinite(R)) and np.array_equal(R[:, rest], good[:, rest])
    ap.ap_destroy(ctx)


def test_whole_row_groups_without_memory_for_parts():
    """A budget that leaves nothing for the parts of shared row groups: the groups stay
    whole and the result agrees to the order of the sums."""
    n, c = 5000, 16
    p = wl.random_problem(n, 5, 64, c, wl.MATERN32, 0.1, 34)
    W = _t(np.random.default_rng(8).standard_normal((n, c)))
    ref_ctx = _ctx(p)
    ref = ap.ap_residual(ref_ctx, _t(p.B), W)
    need = ap.ap_device_bytes(ref_ctx) - 2 * 152 * 256 * c * 4  # less the parts
    ctx = _ctx(p, hbm_budget=need + (1 << 18))
    out = ap.ap_residual(ctx, _t(p.B), W)
    assert ap.ap_device_bytes(ctx) < need + (1 << 18)
    scale = oracle.gram(oracle.Hyper.of(p), p.X[:50].astype(np.float64), p.X.astype(np.float64), noise=False)
    bound = TOL_PROD * float((scale @ np.abs(W.cpu().numpy().astype(np.float64))).max())
    assert float((out - ref).abs().max()) <= bound
    for x in (ref_ctx, ctx):
        ap.ap_destroy(x)
