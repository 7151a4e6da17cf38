"""The integer combination of the Cholesky products' levels, as the kernel's own device
functions compute it (compiled here into a small library of their own), against exact sums:

    2^(e_r + e_c - 63) sum_{L=2..9} acc_L 2^(7 (9 - L)),

rounded once to a double.  T = sum_L acc_L 2^(7 (9 - L)) is kept whole below 2^62; from
there on its last five bits are dropped, of which the rounding to 53 bits takes at least
five anyway: half a unit plus 1/32 of the result's last place.  Results outside the normal
doubles go through the library ldexp; a marked row exponent gives NaN."""
import ctypes
import os
import random
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2310_17137_gb300 import build as b

pytestmark = pytest.mark.gpu

SRC = r"""
#include "ozaki.cu"
namespace {
__global__ void level_kernel(const int* p, const int* e, double* out, int rows) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows) return;
    int h1[4], h2[4], l1[4], l2[4], ec[4];
    const int er = e[5 * i];
    bool marked = er == ap::kBadExp;
    for (int c = 0; c < 4; ++c) {
        const int* q = p + 4 * (4 * i + c);
        h1[c] = q[0], h2[c] = q[1], l1[c] = q[2], l2[c] = q[3];
        ec[c] = e[5 * i + 1 + c];
        marked |= ec[c] == ap::kBadExp;
    }
    double t[4];
    ap::level_row(h1, h2, l1, l2, er, ec, marked, t);
    for (int c = 0; c < 4; ++c) out[4 * i + c] = t[c];
}
}  // namespace
extern "C" int bad_exp() { return ap::kBadExp; }
extern "C" int level_rows(const int* p, const int* e, double* out, int rows) {
    int *dp = nullptr, *de = nullptr;
    double* dout = nullptr;
    cudaError_t err = cudaMalloc(&dp, 16 * rows * sizeof(int));
    if (!err) err = cudaMalloc(&de, 5 * rows * sizeof(int));
    if (!err) err = cudaMalloc(&dout, 4 * rows * sizeof(double));
    if (!err) err = cudaMemcpy(dp, p, 16 * rows * sizeof(int), cudaMemcpyHostToDevice);
    if (!err) err = cudaMemcpy(de, e, 5 * rows * sizeof(int), cudaMemcpyHostToDevice);
    if (!err) {
        level_kernel<<<(rows + 127) / 128, 128>>>(dp, de, dout, rows);
        err = cudaMemcpy(out, dout, 4 * rows * sizeof(double), cudaMemcpyDeviceToHost);
    }
    cudaFree(dp);
    cudaFree(de);
    cudaFree(dout);
    return (int)err;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("levels")
    src, so = str(d / "levels.cu"), str(d / "levels.so")
    open(src, "w").write(SRC)
    subprocess.check_call([b.nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", src, "-o", so], cwd=str(d))
    return ctypes.CDLL(so)


def _run(lib, acc, er, ec):
    """acc: rows x 4 x 8 integers acc_2 .. acc_9; er: rows; ec: rows x 4."""
    a = np.asarray(acc, np.int64)
    pairs = np.ascontiguousarray(128 * a[..., 0::2] + a[..., 1::2]).astype(np.int32)
    e = np.ascontiguousarray(np.concatenate([np.asarray(er)[:, None], np.asarray(ec)], 1)).astype(np.int32)
    out = np.empty((len(a), 4))
    rc = lib.level_rows(pairs.ctypes.data_as(ctypes.c_void_p), e.ctypes.data_as(ctypes.c_void_p),
                        out.ctypes.data_as(ctypes.c_void_p), len(a))
    assert rc == 0
    return out


def _accs(rng, rows):
    """Level sums within their bounds |acc_L| <= (L - 1) 2^18, the leading ones often small or
    zero (cancelling products) and the extremes among them."""
    acc = []
    for i in range(rows):
        row = []
        for _ in range(4):
            lead = rng.choice([2, 2, 2, 3, 4, 5, 6, 8, 9])
            size = rng.choice([1, 2 ** 6, 2 ** 12, 2 ** 18])
            v = [0 if L < lead else rng.randint(-min(size, 2 ** 18) * (L - 1), min(size, 2 ** 18) * (L - 1))
                 for L in range(2, 10)]
            if i < 2:
                v = [(1 - 2 * i) * (L - 1) * 2 ** 18 for L in range(2, 10)]
            row.append(v)
        acc.append(row)
    return acc


def _exact(a, e):
    return sum(Fraction(int(x)) * Fraction(2) ** (7 * (9 - L)) for L, x in enumerate(a, 2)) * Fraction(2) ** (e - 63)


def test_rows_are_the_exact_sums_rounded_once(lib):
    rng = random.Random(71)
    rows = 3000
    acc = _accs(rng, rows)
    er = [rng.randint(-400, 400) for _ in range(rows)]
    ec = [[rng.randint(-400, 400) for _ in range(4)] for _ in range(rows)]
    got = _run(lib, acc, er, ec)
    for i in range(rows):
        for c in range(4):
            want = _exact(acc[i][c], er[i] + ec[i][c])
            if want == 0:
                assert got[i, c] == 0.0
                continue
            ulp = Fraction(float(np.spacing(abs(float(want)))))
            assert abs(Fraction(float(got[i, c])) - want) <= ulp * Fraction(17, 32), (i, c, acc[i][c])


def test_results_at_the_ends_of_the_double_range(lib):
    rng = random.Random(72)
    rows = 400
    acc = _accs(rng, rows)
    er = [rng.choice([-1021, -1000, 1000, 1024]) for _ in range(rows)]
    ec = [[rng.choice([-60, -40, -10, 0, 10]) if abs(e) > 900 else 0 for _ in range(4)] for e in er]
    got = _run(lib, acc, er, ec)
    tiny = Fraction(2) ** -1074
    for i in range(rows):
        for c in range(4):
            want = _exact(acc[i][c], er[i] + ec[i][c])
            if abs(want) >= Fraction(2) ** 1024:
                assert np.isinf(got[i, c]) and (got[i, c] > 0) == (want > 0)
                continue
            # (the integer is rounded to a double, then once more where the result is subnormal)
            tol = abs(want) * Fraction(17, 32) / 2 ** 52 + tiny / 2
            if abs(want) < Fraction(2) ** 1023:
                assert abs(Fraction(float(got[i, c])) - want) <= tol, (i, c, acc[i][c], er[i], ec[i][c])


def test_a_marked_exponent_gives_nan(lib):
    bad = lib.bad_exp()
    rng = random.Random(73)
    acc = _accs(rng, 3)
    ec = [[0, 1, bad, 3], [0, 1, 2, 3], [bad, bad, bad, bad]]
    got = _run(lib, acc, [5, bad, bad], ec)
    assert np.array_equal(np.isnan(got), [[False, False, True, False], [True] * 4, [True] * 4])
    for c in (0, 1, 3):
        want = _exact(acc[0][c], 5 + ec[0][c])
        assert abs(Fraction(float(got[0, c])) - want) <= abs(want) * Fraction(17, 32) / 2 ** 52
