"""The benchmark's FP32 roofline counts against the FMA pipe only what runs there: with more
than four right-hand sides the contraction is on the tensor cores and reported apart."""
import types

import pytest

import bench
import workloads as wl


@pytest.mark.parametrize("c,kernel,fma,tensor", [(1, "kmv_fp32_kernel", 24 + 2, None), (4, "kmv_fp32_kernel", 24 + 8, None),
                                                 (16, "kmv_x3_kernel", 24 + 4, 192), (32, "kmv_x3_kernel", 24 + 4, 384)])
def test_fp32_roofline_by_width(c, kernel, fma, tensor):
    p = wl.random_problem(64, 8, 32, c, wl.MATERN32, 0.1, 1)
    args = types.SimpleNamespace(precision="fp32", workload="none")
    units, t = 65536.0 * 4096, 302e-6
    r = bench.roofline(p, args, t, units, 2070.0)
    assert r["kernel"].startswith(kernel)
    assert r["achieved"] == pytest.approx(units * fma / t / 1e12)
    assert r["frac"] < 1.0
    assert r.get("tensor_flops_per_entry") == tensor
    if tensor:
        assert r["tensor_tflops"] == pytest.approx(units * tensor / t / 1e12)
