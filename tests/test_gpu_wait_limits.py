"""opts.wait_limit_cycles in the FP32 product for more than 4 right-hand sides and in the
gradient forms: with a one-cycle bound the copy issuer, which runs ahead of the pipeline
until it must wait for a stage, gives up (every CTA here has more chunks than stages); the
kernel lets its copies and MMAs land, frees its tensor memory and returns, the call reports
AP_ERR_TIMEOUT, and neither the context nor the library's fixed scratch keeps anything of
it: calls without such waits are right on the same context, all calls on another one."""
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


def _ctx(p, limit, **kw):
    return ap.ap_create(_t(p.X), ap.Hyper(p.kernel, p.lengthscale, p.outputscale, p.noise),
                        ap.ap_opts_default(block=p.block, wait_limit_cycles=limit, **kw))


def _times_out(call):
    with pytest.raises(ap.ApError) as e:
        call()
    assert e.value.status == ap.AP_ERR_TIMEOUT


def _check_residual(ctx, p, B, W):
    """Rows of B - K_hat W against float64, at the plain product's bound."""
    R = ap.ap_residual(ctx, _t(B), _t(W)).cpu().numpy()
    rows = np.random.default_rng(1).integers(0, p.n, 200)
    h, X, W = oracle.Hyper.of(p), p.X.astype(np.float64), W.astype(np.float64)
    K = oracle.gram(h, X[rows], X, noise=False)
    K[np.arange(len(rows)), rows] += p.noise
    want = B[rows].astype(np.float64) - K @ W
    assert np.all(np.abs(R[rows] - want) <= TOL_PROD * (np.abs(K) @ np.abs(W) + np.abs(B[rows])))


@pytest.mark.parametrize("kern,d,c", [(wl.MATERN52, 3, 16), (wl.RBF, 20, 32), (wl.MATERN32, 8, 32)])
def test_residual_times_out_and_the_next_ones_are_right(kern, d, c):
    p = wl.random_problem(40000, d, 1024, c, kern, 0.05, 91)
    ctx = _ctx(p, 1)
    W = np.random.default_rng(2).standard_normal((p.n, c)).astype(np.float32)
    for _ in range(2):
        _times_out(lambda: ap.ap_residual(ctx, _t(p.B), _t(W)))
        for k in (1, 4):
            _check_residual(ctx, p, np.ascontiguousarray(p.B[:, :k]), np.ascontiguousarray(W[:, :k]))
    ap.ap_destroy(ctx)
    ctx = _ctx(p, 0)
    _check_residual(ctx, p, p.B, W)
    ap.ap_destroy(ctx)


def test_fp32_solve_times_out_and_a_narrow_one_is_right():
    p = wl.random_problem(40000, 3, 4096, 16, wl.MATERN32, 0.1, 92, ell_range=(0.02, 0.05))
    ctx = _ctx(p, 1, max_epochs=2)
    _times_out(lambda: ap.ap_solve(ctx, _t(p.B)))
    st, W, info, _ = ap.ap_solve(ctx, _t(p.B[:, :1]))
    assert st in (ap.AP_OK, ap.AP_ERR_NOT_CONVERGED)
    _check_residual(ctx, p, np.ascontiguousarray(p.B[:, :1]), W.cpu().numpy())
    R = ap.ap_residual(ctx, _t(p.B[:, :1]), W)
    rel = float(R.norm() / _t(p.B[:, :1]).norm())
    assert abs(rel - info["rel_res_tracked"][0]) <= 1e-4
    ap.ap_destroy(ctx)


@pytest.mark.parametrize("kern,d,c", [(wl.RBF, 3, 1), (wl.MATERN32, 8, 32), (wl.MATERN52, 20, 16)])
def test_gradient_forms_time_out_and_leave_nothing_behind(kern, d, c):
    p = wl.random_problem(20000, d, 1024, 1, kern, 0.1, 93)
    short, free = _ctx(p, 1, max_epochs=1, min_epochs=1), _ctx(p, 0)
    U, V = (_t(a) for a in np.random.default_rng(3).standard_normal((2, p.n, c)))
    alpha = np.linspace(-1, 1, c) if c > 1 else np.ones(1)
    want = ap.ap_grad_quadforms(free, U, V, alpha)
    _times_out(lambda: ap.ap_grad_quadforms(short, U, V, alpha))
    _times_out(lambda: ap.ap_grad_quadforms_static(short, U, V, alpha))
    _times_out(lambda: ap.ap_mll_grad(short, _t(p.y), 0))
    assert np.array_equal(ap.ap_grad_quadforms_static(free, U, V, alpha), want)
    assert np.array_equal(ap.ap_grad_quadforms(free, U, V, alpha), want)
    B, W = p.B, U[:, :1].cpu().numpy()
    _check_residual(short, p, np.ascontiguousarray(B), np.ascontiguousarray(W))
    for x in (short, free):
        ap.ap_destroy(x)
