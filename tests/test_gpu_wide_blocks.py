"""A diagonal block that holds a far point keeps the distances of its near ones: one block,
one step, so W = K_hat^{-1} B by the cached factor alone.  Against the dense float64 solve;
the factor's inverse is stored and applied in FP32: 1e-4 for these condition numbers (about
1e3), as for blocks without a far point."""
import numpy as np
import pytest
import torch

import oracle
import paper_2310_17137_gb300 as ap
import workloads as wl

pytestmark = pytest.mark.gpu


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to("cuda:0")


@pytest.mark.parametrize("far", [0.0, 1e8, 1e12, 1e17], ids=lambda v: f"{v:g}")
@pytest.mark.parametrize("where", [0, 100])
@pytest.mark.parametrize("kern", [wl.RBF, wl.MATERN32, wl.MATERN52])
def test_one_block_solve_with_a_far_point(kern, far, where):
    p = wl.random_problem(256, 3, 256, 2, kern, 0.05, 81)
    X = p.X.copy()
    X[where] += np.float32(far)
    ctx = ap.ap_create(_t(X), ap.Hyper(kern, p.lengthscale, p.outputscale, p.noise),
                       ap.ap_opts_default(block=256, tol=1e-30, min_epochs=0, max_steps=1))
    _, W, info, _ = ap.ap_solve(ctx, _t(p.B))
    assert info["steps"] == 1
    want = oracle.dense_solve(oracle.Hyper.of(p), X.astype(np.float64), p.B.astype(np.float64))
    assert np.abs(W.cpu().numpy() - want).max() <= 1e-4 * np.abs(want).max()
    ap.ap_destroy(ctx)
