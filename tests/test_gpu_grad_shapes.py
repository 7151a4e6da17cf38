"""The gradient quadratic forms over the edges of their work split (row groups of 128 or
256, 64-column chunks, the diagonal inside a chunk) and every padded dimension and width,
against the oracle.  The derivatives' entries are non-negative, so the forms of the
absolute values bound every term; FP32 entries and sums: 1e-5 of that bound (the kernel's
figure in the parity tests)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2310_17137_gb300 as ap
import workloads as wl

pytestmark = pytest.mark.gpu


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to("cuda:0")


@pytest.mark.parametrize("n,d,c,kern", [(1, 2, 1, wl.RBF), (63, 3, 4, wl.MATERN32), (64, 5, 16, wl.MATERN52),
                                        (65, 9, 32, wl.RBF), (129, 13, 2, wl.MATERN32), (255, 17, 16, wl.MATERN52),
                                        (257, 25, 32, wl.RBF), (1000, 8, 31, wl.MATERN32), (1345, 12, 1, wl.MATERN52),
                                        (1500, 32, 9, wl.RBF)])
def test_quadforms_over_shapes(n, d, c, kern):
    p = wl.random_problem(n, d, 128, c, kern, 0.1, 41)
    ctx = ap.ap_create(_t(p.X), ap.Hyper(kern, p.lengthscale, p.outputscale, p.noise), ap.ap_opts_default(block=128))
    rng = np.random.default_rng(9)
    U, V = rng.standard_normal((2, n, c)).astype(np.float32)
    alpha = rng.uniform(-1, 1, c)
    first = ap.ap_grad_quadforms(ctx, _t(U), _t(V), alpha)
    assert np.array_equal(first, ap.ap_grad_quadforms(ctx, _t(U), _t(V), alpha))  # fixed-order sums
    h = oracle.Hyper.of(p)
    X = p.X.astype(np.float64)
    U, V = U.astype(np.float64), V.astype(np.float64)
    ref = oracle.grad_quadforms(h, X, U, V, alpha)
    mag = oracle.grad_quadforms(h, X, np.abs(U), np.abs(V), np.abs(alpha))
    assert np.all(np.abs(first - ref) <= 1e-5 * mag + 1e-12), np.abs(first - ref) / mag
    ap.ap_destroy(ctx)


@pytest.mark.parametrize("c", [1, 4, 16, 32])
def test_static_quadforms_take_arrays_of_any_float_alignment(c):
    """ap_grad_quadforms_static reads the caller's U and V in place: an array that starts
    4 bytes past a 16-byte boundary gives the same bits as an aligned one."""
    n = 300
    p = wl.random_problem(n, 4, 128, c, wl.MATERN32, 0.1, 42)
    ctx = ap.ap_create(_t(p.X), ap.Hyper(p.kernel, p.lengthscale, p.outputscale, p.noise), ap.ap_opts_default(block=128))
    rng = np.random.default_rng(10)
    U, V = _t(rng.standard_normal((n, c))), _t(rng.standard_normal((n, c)))
    alpha = rng.uniform(-1, 1, c)
    want = ap.ap_grad_quadforms_static(ctx, U, V, alpha)

    def shifted(t):
        flat = torch.empty(n * c + 1, device="cuda:0")[1:]
        flat.copy_(t.reshape(-1))
        return flat.view(n, c)

    for a, b in [(shifted(U), V), (U, shifted(V)), (shifted(U), shifted(V))]:
        assert np.array_equal(ap.ap_grad_quadforms_static(ctx, a, b, alpha), want)
    ap.ap_destroy(ctx)
