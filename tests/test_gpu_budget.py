"""Contexts at the edge of their HBM budget: the optional column-group sums never cost a
required buffer or the factorisation's workspace, and come back when there is room.
Products are compared with float64 rows, at the plain product's bound
2e-5 (sum_j |K_ij| |v_j| + |base_i|)."""
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


def _workspace(b, cache_gemm):
    """Bytes of one block's factorisation workspace: the FP64 block and its tile inverses,
    and the slice planes and row exponents of the tensor-core products."""
    nt = -(-b // 64)
    edge = 64 * nt
    ws = 8 * (edge * edge + 64 * edge)
    return ws + (8 * (edge + 64) * 128 + 4 * (edge + 64) if cache_gemm == ap.AP_CACHE_TC_EXACT else 0)


def _check_mean(ctx, p, w, Xt, rows):
    out = ap.ap_predict_mean(ctx, _t(w), _t(Xt)).cpu().numpy()[rows]
    h = oracle.Hyper.of(p)
    K = oracle.gram(h, Xt[rows].astype(np.float64), p.X.astype(np.float64), noise=False)
    w = w.astype(np.float64)
    assert np.all(np.abs(out - K @ w) <= TOL_PROD * (np.abs(K) @ np.abs(w)))


@pytest.mark.parametrize("cache_gemm", [ap.AP_CACHE_TC_EXACT, ap.AP_CACHE_FP64], ids=["tc", "fp64"])
@pytest.mark.parametrize("c", [1, 16])
def test_set_hyper_after_a_solve_fits_the_budget_that_held_it_without_group_sums(c, cache_gemm):
    p = wl.random_problem(6000, 3, 512, c, wl.MATERN52, 0.1, 51)
    hyper = ap.Hyper(p.kernel, p.lengthscale, p.outputscale, p.noise)
    w = np.random.default_rng(5).standard_normal(p.n).astype(np.float32)
    Xt = wl.test_points(p, m=200)

    def used(budget):
        ctx = ap.ap_create(_t(p.X), hyper, ap.ap_opts_default(block=512, max_epochs=3, hbm_budget=budget,
                                                              cache_gemm=cache_gemm))
        _, W, _, _ = ap.ap_solve(ctx, _t(p.B))
        ap.ap_predict_mean(ctx, _t(w), _t(Xt))
        return ctx, W, ap.ap_device_bytes(ctx)

    free, W0, held = used(0)
    # one byte short of one block's workspace beside everything, group sums included
    ctx, W1, held1 = used(held + _workspace(512, cache_gemm) - 1)
    assert held1 == held and torch.equal(W0, W1)
    ap.ap_set_hyper(ctx, hyper)
    _check_mean(ctx, p, w, Xt, np.arange(200))
    # the areas are asked for again: the same split and the same bits as before
    _, W2, _, _ = ap.ap_solve(ctx, _t(p.B))
    assert torch.equal(W0, W2) and ap.ap_device_bytes(ctx) == held
    for x in (free, ctx):
        ap.ap_destroy(x)


def test_a_refused_set_hyper_leaves_the_context_as_it_was():
    """Work buffers that grew since the context was made leave less than one block's
    workspace: NOMEM, and the old hyperparameters stay in force throughout."""
    p = wl.random_problem(6000, 3, 512, 16, wl.RBF, 0.1, 52)
    hyper = ap.Hyper(p.kernel, p.lengthscale, p.outputscale, p.noise)
    twin = ap.ap_create(_t(p.X), hyper, ap.ap_opts_default(block=512))
    created = ap.ap_device_bytes(twin)
    budget = created + _workspace(512, ap.AP_CACHE_TC_EXACT)  # (the solve buffers take some 2 MB of those 3)
    ctx = ap.ap_create(_t(p.X), hyper, ap.ap_opts_default(block=512, hbm_budget=budget))
    W = _t(np.random.default_rng(6).standard_normal((p.n, 16)))
    want = ap.ap_residual(twin, _t(p.B), W)
    ap.ap_residual(ctx, _t(p.B), W)
    with pytest.raises(ap.ApError) as e:
        ap.ap_set_hyper(ctx, ap.Hyper(p.kernel, 2 * p.lengthscale, 3.0, 0.2))
    assert e.value.status == ap.AP_ERR_NOMEM
    got = ap.ap_residual(ctx, _t(p.B), W)
    scale = (want - _t(p.B)).abs().max()
    assert float((got - want).abs().max()) <= 1e-5 * float(scale)
    for x in (twin, ctx):
        ap.ap_destroy(x)


def test_group_sums_are_given_back_to_a_required_buffer():
    """The scaled test inputs of a large prediction need bytes that the group sums of
    earlier calls hold: those are released, and the result is that of the plain product."""
    n, M = 6000, 400_000
    p = wl.random_problem(n, 3, 512, 1, wl.RBF, 0.05, 23)
    hyper = ap.Hyper(wl.RBF, p.lengthscale, p.outputscale, p.noise)
    w = np.random.default_rng(4).standard_normal(n).astype(np.float32)
    Xt = wl.test_points(p, m=M)
    xt_bytes = M * 4 * 4

    def small(budget):
        ctx = ap.ap_create(_t(p.X), hyper, ap.ap_opts_default(block=512, hbm_budget=budget))
        ap.ap_predict_mean(ctx, _t(w), _t(Xt[:500]))
        return ctx, ap.ap_device_bytes(ctx)

    free, held = small(0)
    budget = held - 500 * 4 * 4 + xt_bytes - 1  # one byte short beside the group sums
    assert xt_bytes > _workspace(512, ap.AP_CACHE_TC_EXACT)  # (or the budget would bind at ap_create)
    ctx, held1 = small(budget)
    assert held1 == held
    rows = np.random.default_rng(8).integers(0, M, 300)
    _check_mean(ctx, p, w, Xt, rows)
    assert ap.ap_device_bytes(ctx) <= budget
    _check_mean(free, p, w, Xt, rows)
    for x in (free, ctx):
        ap.ap_destroy(x)
