// Double-float ("FP32 pair") arithmetic for the compensated residual recompute.
//
// A value is the unevaluated sum hi + lo of two FP32 numbers.  The error-free
// transformations are the classical ones: TwoSum (Knuth, TAOCP vol. 2),
// Fast2Sum (Dekker 1971) and the FMA form of TwoProd; the double-float add and
// multiply follow Dekker's composition.  All arithmetic stays in FP32; nvcc
// does not reassociate additions, and every product whose rounding error is
// needed is taken explicitly through fmaf.
#pragma once

namespace ap {
namespace df {

struct F2 {
    float h, l;
};

__device__ __forceinline__ F2 two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    const float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}

// requires |a| >= |b| (or a == 0)
__device__ __forceinline__ F2 fast_two_sum(float a, float b) {
    const float s = a + b;
    return {s, b - (s - a)};
}

__device__ __forceinline__ F2 two_prod(float a, float b) {
    const float p = a * b;
    return {p, fmaf(a, b, -p)};
}

__device__ __forceinline__ F2 add(F2 a, F2 b) {
    F2 s = two_sum(a.h, b.h);
    const float e = s.l + (a.l + b.l);
    return fast_two_sum(s.h, e);
}

__device__ __forceinline__ F2 add_f(F2 a, float b) {
    F2 s = two_sum(a.h, b);
    return fast_two_sum(s.h, s.l + a.l);
}

__device__ __forceinline__ F2 mul_f(F2 a, float b) {
    F2 p = two_prod(a.h, b);
    return fast_two_sum(p.h, fmaf(a.l, b, p.l));
}

// ln 2 and log2 e as FP32 pairs (hi = nearest float, lo = remainder)
constexpr float kLn2H = 0.693147182464599609375f;
constexpr float kLn2L = -1.9046542121259336e-09f;
constexpr float kLog2eH = 1.44269502162933349609375f;
constexpr float kLog2eL = 1.925963033500011e-08f;
constexpr float kThirdH = 0.3333333432674407958984375f;
constexpr float kThirdL = -9.934107758624577e-09f;
constexpr float kSixthH = 0.16666667163372039794921875f;
constexpr float kSixthL = -4.967053879312289e-09f;

// ------------------------------------------------------------------ two at a time
// The same arithmetic on two independent values, as packed FP32 pairs (one instruction
// for both lanes, each rounded as the scalar operation): the long chains below are bound
// by issue slots, and there is no subtraction or negation of a pair but a multiply-add
// with -1 (exact).
struct P2 {
    float2 h, l;
};

__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }

__device__ __forceinline__ P2 two_sum(float2 a, float2 b) {
    const float2 s = add(a, b), bb = sub(s, a);
    return {s, add(sub(a, sub(s, bb)), sub(b, bb))};
}

// requires |a| >= |b| (or a == 0)
__device__ __forceinline__ P2 fast_two_sum(float2 a, float2 b) {
    const float2 s = add(a, b);
    return {s, sub(b, sub(s, a))};
}

// a b exactly, na = -a
__device__ __forceinline__ P2 two_prod(float2 a, float2 na, float2 b) {
    return {mul(a, b), fma2(a, b, mul(na, b))};
}

__device__ __forceinline__ P2 mul(P2 a, P2 b) {
    const P2 p = two_prod(a.h, sub(make_float2(0.0f, 0.0f), a.h), b.h);
    return fast_two_sum(p.h, fma2(a.h, b.l, fma2(a.l, b.h, p.l)));
}

// a + b for a constant |a| >= |b|
__device__ __forceinline__ P2 const_plus(float ah, float al, P2 b) {
    const P2 s = fast_two_sum(dup(ah), b.h);
    return fast_two_sum(s.h, add(s.l, add(b.l, dup(al))));
}

__device__ __forceinline__ P2 add(P2 a, P2 b) {
    const P2 s = two_sum(a.h, b.h);
    return fast_two_sum(s.h, add(s.l, add(a.l, b.l)));
}

// 2^(-t) for t = t.h + t.l >= 0 with about 2^-40 relative error.
// t = k + r, k = nearest integer, |r| <= 1/2;  2^-r = e^-z, z = r ln 2, |z| < 0.35;
// e^-z = 1 - z + z^2/2 - z^3/6 + z^4 q(z): the leading terms in double-float,
// the tail q (|z^4 q| < 7e-4) in FP32 Horner form (Taylor coefficients).
__device__ __forceinline__ P2 exp2_neg(P2 t) {
    // beyond 125 the result is 0 (set at the end); k by the rounding of a large sum
    const float2 th = make_float2(fminf(t.h.x, 126.0f), fminf(t.h.y, 126.0f));
    // (a large t's low part would overflow the polynomial; a NaN stays in the low part)
    const float2 tl = make_float2(t.h.x > 126.0f ? 0.0f : t.l.x, t.h.y > 126.0f ? 0.0f : t.l.y);
    const float2 big = dup(12582912.0f);  // 1.5 * 2^23
    const float2 kb = add(th, big);
    const float2 k = sub(kb, big);
    const P2 r = fast_two_sum(sub(th, k), tl);
    const P2 z = mul(P2{dup(kLn2H), dup(kLn2L)}, r);
    const float2 zh = z.h, nzh = sub(make_float2(0.0f, 0.0f), z.h);
    float2 q = dup(-1.0f / 362880.0f);
    q = fma2(q, zh, dup(1.0f / 40320.0f));
    q = fma2(q, zh, dup(-1.0f / 5040.0f));
    q = fma2(q, zh, dup(1.0f / 720.0f));
    q = fma2(q, zh, dup(-1.0f / 120.0f));
    q = fma2(q, zh, dup(1.0f / 24.0f));
    // Horner in double-float: ((q z - 1/6) z + 1/2) z - 1) z + 1, every constant larger
    // than what is added to it
    auto times_z = [&](P2 a) {
        const P2 p = two_prod(zh, nzh, a.h);
        return fast_two_sum(p.h, fma2(zh, a.l, fma2(z.l, a.h, p.l)));
    };
    const P2 p0 = two_prod(zh, nzh, q);
    P2 acc = fast_two_sum(p0.h, fma2(z.l, q, p0.l));
    acc = times_z(const_plus(-kSixthH, -kSixthL, acc));
    acc = times_z(const_plus(0.5f, 0.0f, acc));
    acc = times_z(const_plus(-1.0f, 0.0f, acc));
    acc = const_plus(1.0f, 0.0f, acc);
    // scale by 2^-k exactly (k <= 125 keeps the result normal or zero): kb's low mantissa
    // bits are the integer k
    const int kx = __float_as_int(kb.x) & 0x1ff, ky = __float_as_int(kb.y) & 0x1ff;
    const float2 sc = make_float2(kx > 125 ? 0.0f : __int_as_float((127 - kx) << 23),
                                  ky > 125 ? 0.0f : __int_as_float((127 - ky) << 23));
    return {mul(acc.h, sc), mul(acc.l, sc)};
}

// sqrt of double-floats t >= 0: IEEE sqrt of t.h plus one Newton correction.
__device__ __forceinline__ P2 sqrt_df(P2 t) {
    const bool zx = t.h.x <= 0.0f, zy = t.h.y <= 0.0f;
    const float2 s = make_float2(zx ? 1.0f : __fsqrt_rn(t.h.x), zy ? 1.0f : __fsqrt_rn(t.h.y));
    const P2 ss = two_prod(s, sub(make_float2(0.0f, 0.0f), s), s);
    const float2 half = make_float2(0.5f / s.x, 0.5f / s.y);
    const float2 corr = mul(add(sub(sub(t.h, ss.h), ss.l), t.l), half);
    P2 r = fast_two_sum(s, corr);
    if (zx) r.h.x = r.l.x = 0.0f;
    if (zy) r.h.y = r.l.y = 0.0f;
    return r;
}

}  // namespace df
}  // namespace ap
