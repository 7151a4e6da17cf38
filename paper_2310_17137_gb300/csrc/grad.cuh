// Fused backward pass of the stochastic MLL gradient (Eq. loss_grad_unbiased):
// one sweep over the kernel entries that forms G_ij = sum_c alpha_c U_ic V_jc on the
// fly and contracts it with every derivative dK_ij / dtheta at once (d lengthscales,
// outputscale, noise).  No kernel block or G block is stored.
//
// With the pre-scaled inputs xs of the FP32 product (xs = c_K x / l, see
// kernel_input_scale) and t = |xs_i - xs_j|^2:
//   RBF  phi = 2^-t,                     psi = phi
//   M32  u = sqrt(t), phi = (1+u) e^-u,  psi = e^-u
//   M52  u = sqrt(t), phi = (1+u+u^2/3) e^-u, psi = (1+u) e^-u
// and dK/dl_k = s * kappa_K / (c_K^2 l_k) * psi * (xs_ik - xs_jk)^2 with
// kappa_K / c_K^2 = 2/log2(e), 1, 1/3; the host applies those factors.
//
// What bounds it is FP32 work per entry, so the sweep does less of it in two ways.
//   Symmetry: phi, psi and the squared differences are symmetric in (i, j), so only
//   i < j is visited, with S_ij = G_ij + G_ji; the diagonal (phi = 1, no differences)
//   adds sum_i G_ii to the outputscale and noise forms.
//   Contraction on the tensor cores: S = [alpha U | V] [V | alpha U]^T, both operands
//   split into three BF16 parts (exact up to the last rounding), the six products of
//   weight above 2^-24 into two or three FP32 accumulators per entry: hi x hi in chains
//   of at most two steps, the small ones on their own, those of weight 2^-16 first; the
//   parts are added in FP32.  The tensor cores cut their sums off towards zero, a mean
//   error that n^2 entries would not average out: all three parts are rounded to nearest,
//   so that the small products have no preferred sign (with hi cut off, sums of one sign
//   came out 2.8e-9 low at c = 32; now within 2.4e-10 of the exact ones at any width).
// What is left are 4 d multiply-add lanes (as packed pairs) and about 14 instructions
// per visited entry.  Measured (GB300, n = 131,072, d = 8, c = 32, Matern-3/2): 47.0 ->
// 14.35 ms for the n^2 forms, FMA pipe 68 % busy; n = 1024, d = 8, c = 4 a call 62 -> 45 us.
// (With two stages 16.5 ms: the chunk's copy, split and MMAs follow one another.)  Error of the doubles against 64 bits, relative
// to the forms of absolute values, n = 8192, root mean square over 40 inputs, scalar form
// -> this one: RBF d = 8, c = 32 3.25e-9 -> 3.30e-9; Matern-3/2 d = 3, c = 16 6.07e-9 ->
// 6.08e-9; Matern-5/2 d = 20, c = 32 3.47e-9 -> 3.49e-9: that of exp2, sqrt and the inputs.
//
// Work units are (row group, 64-column chunk) pairs of the upper triangle in
// group-major order, cut into equal ranges over a persistent grid; every CTA keeps
// one set of sums whatever groups it meets (FP32 over 128 entries per thread, 64 for
// D = 16, FP64 beyond; folding every 64 takes 5 to 9 % longer at D = 12 and 20 and leaves
// the error as it is), and the CTA that finishes last adds the CTAs' sums in order.
// Warp roles: transform warps (one row, or two rows 128 apart, per thread; 16 columns of
// every chunk, 32 for D > 16), one MMA issuer, one bulk-copy lane for the columns' coordinates, two
// warps that split the chunk's [V | alpha U]; the transform warps split the rows' own
// operand when the group changes.  Every wait is bounded.
#pragma once

#include "kmv_fp32.cuh"
#include "tcgen05.cuh"

namespace ap {

template <int KERN>
__device__ __forceinline__ void phi_psi_fp32(float t, float& phi, float& psi) {
    if constexpr (KERN == AP_RBF) {
        phi = ex2_approx(-t);
        psi = phi;
    } else if constexpr (KERN == AP_MATERN32) {
        const float u = sqrt_approx(t);
        const float e = ex2_approx(-u * kLog2e);
        phi = (1.0f + u) * e;
        psi = e;
    } else {
        const float u = sqrt_approx(t);
        const float e = ex2_approx(-u * kLog2e);
        psi = (1.0f + u) * e;
        phi = fmaf(u * u, (1.0f / 3.0f) * e, psi);
    }
}

namespace gx {

using namespace tc;

constexpr int kChunk = 64;
constexpr int kStages = 4;
constexpr int kConvWarps = 2;
constexpr int kFold = 4;  // chunks between folds of the FP32 sums into FP64

// Rows per thread, one : two (n = 32,768, Matern-3/2, us): D = 8 c = 16 1145 : 925, c = 32 1619 :
// 1030, D = 12 1522 : 1343 and 1740 : 1461; the two-row instances spill 150 to 470 bytes all the
// same.  Transform warps, 8 : 16: D = 12 c = 16 1421 : 1343, D = 16 1922 : 1828.  All of them
// against the scalar form of one pass over n^2: D = 4 1702 : 640, 16 3752 : 1828, 24 5706 : 2591,
// 32 8576 : 3326 (c = 16).
template <int D, int C>
struct Cfg {
    static constexpr int R = D <= 12 ? 2 : 1;                // rows per thread
    static constexpr int kRows = 128 * R;
    static constexpr int kXformWarps = D <= 16 ? 16 : 8;      // (more registers per thread for large D)
    static constexpr int kSlots = kXformWarps / 4;
    static constexpr int kMmaWarp = kXformWarps, kCopyWarp = kXformWarps + 1, kConvWarp = kXformWarps + 2;
    static constexpr int kThreads = (kConvWarp + kConvWarps) * 32;
    static constexpr int KC = 2 * C < 16 ? 16 : 2 * C;        // K of the contraction
    static constexpr int kSteps = KC / 16;
    static constexpr int kHh = (kSteps + 1) / 2;              // hi x hi accumulators
    static constexpr uint32_t kAccCols = (kHh + 1) * kChunk;  // per row tile
    static constexpr uint32_t kTmem = R * kAccCols <= 128 ? 128 : R * kAccCols <= 256 ? 256 : 512;
    static constexpr uint32_t kPlaneA = 128 * KC * 2, kPlaneB = kChunk * KC * 2;
    static constexpr uint32_t kXBytes = kChunk * D * 4;
    static constexpr uint32_t kStageBytes = kXBytes + 3 * kPlaneB;
    static constexpr size_t kSmem = 3 * R * kPlaneA + kStages * kStageBytes + 1024;
    static constexpr int NA = D + 2;
    static_assert(R * kAccCols <= 512, "tensor memory");
    static_assert(kSmem <= 220 * 1024, "shared memory");
};

// Eight consecutive K values k0 .. k0 + 7 of point i's operand into the three planes at
// dst, dst + plane, dst + 2 plane: [first | second | 0], the U half scaled by alpha.
// vec: U and V start on 16-byte boundaries (the caller's own arrays need not).
template <int C>
__device__ __forceinline__ void split_operand(const GradParams& p, int64_t i, int k0, bool u_first, bool vec,
                                              uint8_t* dst, uint32_t plane) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = 0.0f;
    if (i < p.n) {
        if constexpr (C % 8 == 0) {  // the eight values lie in one half
            const bool is_u = (k0 < C) == u_first;
            const int c = k0 < C ? k0 : k0 - C;
            const float* src = (is_u ? p.U : p.V) + i * C + c;
            if (vec) {
                const float4 x = __ldg(reinterpret_cast<const float4*>(src));
                const float4 y = __ldg(reinterpret_cast<const float4*>(src) + 1);
                v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
                v[4] = y.x, v[5] = y.y, v[6] = y.z, v[7] = y.w;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = __ldg(src + j);
            }
            if (is_u) {
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] *= p.alpha[c + j];
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int k = k0 + j, c = k < C ? k : k - C;
                if (k < 2 * C) v[j] = (k < C) == u_first ? p.alpha[c] * __ldg(p.U + i * C + c) : __ldg(p.V + i * C + c);
            }
        }
    }
    uint32_t w[3][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) split3_nearest(v[2 * j], v[2 * j + 1], w[0][j], w[1][j], w[2][j]);
#pragma unroll
    for (int pl = 0; pl < 3; ++pl)
        *reinterpret_cast<uint4*>(dst + pl * plane) = make_uint4(w[pl][0], w[pl][1], w[pl][2], w[pl][3]);
}

// Units before group g: group i has L - i rc chunks (L chunks in all, rc per group's rows).
__host__ __device__ inline int64_t units_before(int64_t g, int64_t L, int rc) { return g * L - rc * (g * (g - 1) / 2); }

template <int KERN, int D, int C>
__global__ void __launch_bounds__(Cfg<D, C>::kThreads, 1) grad_kernel(const GradParams p) {
    using K = Cfg<D, C>;
    constexpr int R = K::R;
    extern __shared__ __align__(1024) uint8_t gx_smem[];
    uint8_t* s_a = gx_smem;                                // 3 planes x R tiles x 128 x KC
    uint8_t* s_stage = gx_smem + 3 * R * K::kPlaneA;
    __shared__ __align__(8) uint64_t bar_full[kStages], bar_ready[kStages], bar_empty[kStages];
    __shared__ __align__(8) uint64_t bar_a, bar_acc, bar_acc_free;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ double s_part[K::kXformWarps][K::NA];
    __shared__ int s_last;

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int64_t n = p.n, L = (n + kChunk - 1) / kChunk, ngroups = (n + K::kRows - 1) / K::kRows;
    constexpr int rc = K::kRows / kChunk;
    const int64_t U = units_before(ngroups, L, rc);
    const int64_t u0 = U * blockIdx.x / gridDim.x, u1 = U * (blockIdx.x + 1) / gridDim.x;
    const int total = (int)(u1 - u0);
    // first group and chunk of the range
    int64_t g0 = 0;
    {
        const double a = 0.5 * rc, b = (double)L + a;
        const double disc = b * b - 4.0 * a * (double)u0;
        g0 = (int64_t)((b - sqrt(disc > 0.0 ? disc : 0.0)) / (2.0 * a));
        g0 = min(max(g0, (int64_t)0), ngroups - 1);
        while (g0 > 0 && units_before(g0, L, rc) > u0) --g0;
        while (g0 + 1 < ngroups && units_before(g0 + 1, L, rc) <= u0) ++g0;
    }
    const int64_t q0 = g0 * rc + (u0 - units_before(g0, L, rc));  // chunk (of all L)

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&bar_full[i], 1);
            mbar_init(&bar_ready[i], kConvWarps);
            mbar_init(&bar_empty[i], 1 + K::kXformWarps);
        }
        mbar_init(&bar_a, K::kXformWarps);
        mbar_init(&bar_acc, 1);
        mbar_init(&bar_acc_free, K::kXformWarps);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == K::kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(K::kTmem)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const bool vec = ((reinterpret_cast<uintptr_t>(p.U) | reinterpret_cast<uintptr_t>(p.V)) & 15) == 0;

    if (warp < K::kXformWarps) {
        // ------------------------------------------------------- transform warps
        const int quarter = warp & 3, slot = warp >> 2, row = quarter * 32 + lane;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        float2 xa[R][D / 2], accf[D / 2];
        double accd[D + 1], diag = 0.0;
        float accp = 0.0f;
#pragma unroll
        for (int k = 0; k < D / 2; ++k) accf[k] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < D + 1; ++k) accd[k] = 0.0;
        auto fold = [&]() {
#pragma unroll
            for (int k = 0; k < D / 2; ++k) {
                accd[2 * k] += (double)accf[k].x;
                accd[2 * k + 1] += (double)accf[k].y;
                accf[k] = make_float2(0.0f, 0.0f);
            }
            accd[D] += (double)accp;
            accp = 0.0f;
        };
        // a group begins: coordinates, this warp's share of the rows' operand planes, and
        // (first chunk of the group) the diagonal sums
        auto begin_group = [&](int64_t g, bool first_chunk) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int64_t i = g * K::kRows + 128 * r + row;
#pragma unroll
                for (int k = 0; k < D / 4; ++k) {
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (i < n) v = __ldg(reinterpret_cast<const float4*>(p.Xs + i * D) + k);
                    xa[r][2 * k] = make_float2(v.x, v.y);
                    xa[r][2 * k + 1] = make_float2(v.z, v.w);
                }
                for (int k8 = slot; k8 < K::KC / 8; k8 += K::kSlots)
                    split_operand<C>(p, i, 8 * k8, true, vec,
                                     s_a + r * K::kPlaneA + ((row >> 3) * (K::KC / 8) + k8) * 128 + (row & 7) * 16,
                                     R * K::kPlaneA);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_a);
            // (the MMAs need not wait for the diagonal)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int64_t i = g * K::kRows + 128 * r + row;
                if (slot == 0 && first_chunk && i < n) {
                    float s = 0.0f;
#pragma unroll 8
                    for (int c = 0; c < C; ++c) s = fmaf(p.alpha[c] * __ldg(p.U + i * C + c), __ldg(p.V + i * C + c), s);
                    diag += (double)s;
                }
            }
        };
        const float2 m1 = make_float2(-1.0f, -1.0f);
        bool ok = true;
        int64_t g = g0, q = q0;
        int stage = 0;
        uint32_t sphase = 0;
        if (total > 0) begin_group(g, q == g * rc);
        for (int c = 0; c < total; ++c) {
            ok = mbar_wait(&bar_full[stage], sphase, &s_abort, p.err) &&
                 mbar_wait(&bar_ready[stage], sphase, &s_abort, p.err) &&
                 mbar_wait(&bar_acc, (uint32_t)(c & 1), &s_abort, p.err);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const float* sx = reinterpret_cast<const float*>(s_stage + (size_t)stage * K::kStageBytes);
            const bool upper = q >= (g + 1) * rc;  // every column is right of every row
            // this warp's columns: eight at 8 slot + 8 kSlots h.  All of S is read first, so
            // that the next chunk's MMAs run under the whole of this one's arithmetic.
            constexpr int kPieces = kChunk / (8 * K::kSlots);
            float sv[kPieces][R][8];
#pragma unroll
            for (int h = 0; h < kPieces; ++h) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t at = tmem + lane_base + (uint32_t)r * K::kAccCols + (uint32_t)(8 * (slot + K::kSlots * h));
                    uint32_t w[8], v[K::kHh][8];
                    tmem_ld8(at + K::kHh * kChunk, w);
#pragma unroll
                    for (int a = 0; a < K::kHh; ++a) tmem_ld8(at + a * kChunk, v[a]);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        sv[h][r][j] = __uint_as_float(w[j]);
#pragma unroll
                        for (int a = 0; a < K::kHh; ++a) sv[h][r][j] += __uint_as_float(v[a][j]);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_acc_free);
#pragma unroll
            for (int h = 0; h < kPieces; ++h) {
                const int h0 = 8 * (slot + K::kSlots * h);
                float(&s)[R][8] = sv[h];
                if (!upper) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int64_t i = g * K::kRows + 128 * r + row, j0 = q * kChunk + h0;
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (j0 + j <= i) s[r][j] = 0.0f;
                    }
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4* xb = reinterpret_cast<const float4*>(sx + (h0 + j) * D);
                    float2 sq[R][D / 2], t2[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) t2[r] = make_float2(0.0f, 0.0f);
#pragma unroll
                    for (int k = 0; k < D / 4; ++k) {
                        const float4 v = xb[k];
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const float2 da = __ffma2_rn(make_float2(v.x, v.y), m1, xa[r][2 * k]);
                            const float2 db = __ffma2_rn(make_float2(v.z, v.w), m1, xa[r][2 * k + 1]);
                            sq[r][2 * k] = __fmul2_rn(da, da);
                            sq[r][2 * k + 1] = __fmul2_rn(db, db);
                            t2[r] = __ffma2_rn(da, da, t2[r]);
                            t2[r] = __ffma2_rn(db, db, t2[r]);
                        }
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        float phi, psi;
                        phi_psi_fp32<KERN>(t2[r].x + t2[r].y, phi, psi);
                        const float gp = s[r][j] * psi;
                        const float2 gp2 = make_float2(gp, gp);
#pragma unroll
                        for (int k = 0; k < D / 2; ++k) accf[k] = __ffma2_rn(gp2, sq[r][k], accf[k]);
                        accp = fmaf(s[r][j], phi, accp);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_empty[stage]);
            if ((c + 1) % kFold == 0) fold();
            if (++stage == kStages) {
                stage = 0;
                sphase ^= 1u;
            }
            if (++q == L) {
                ++g;
                q = g * rc;
                if (c + 1 < total) begin_group(g, true);
            }
        }
        fold();
        // Warp sums in FP64 by halving exchanges: lanes 16, 8, .. apart split the sums
        // between them, NP - 1 additions a lane instead of five per sum (FP64 runs at 2
        // results per clock per SM: 9 us of every call at D = 12 otherwise).
        constexpr int NP = K::NA <= 8 ? 8 : K::NA <= 16 ? 16 : K::NA <= 32 ? 32 : 64;
        double a[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k) a[k] = k < D ? accd[k < D ? k : 0] : k == D ? accd[D] + diag : k == D + 1 ? diag : 0.0;
#pragma unroll
        for (int o = 16, w = NP / 2; o > 0; o >>= 1, w /= 2) {
            const bool up = lane & o;
#pragma unroll
            for (int k = 0; k < (w > 0 ? w : 1); ++k) {
                if (w > 0) {
                    const double keep = up ? a[k + w] : a[k];
                    a[k] = keep + __shfl_xor_sync(0xffffffffu, up ? a[k] : a[k + w], o);
                } else {
                    a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
                }
            }
        }
        // the lane's bits, 16 first, spell the index of what is left
        constexpr int kPerLane = NP > 32 ? NP / 32 : 1, kRepeat = NP < 32 ? 32 / NP : 1;
#pragma unroll
        for (int k = 0; k < kPerLane; ++k) {
            const int idx = lane / kRepeat * kPerLane + k;
            if (lane % kRepeat == 0 && idx < K::NA) s_part[warp][idx] = a[k];
        }
    } else if (warp == K::kMmaWarp) {
        // ------------------------------------------------------------ MMA issuer
        constexpr uint32_t idesc = instr_desc(1, 128, kChunk);
        constexpr uint32_t kSbo = (K::KC / 8) * 128;
        const bool leader = elect_one();
        const uint64_t a0 = smem_desc(smem_u32(s_a), 128, kSbo);
        const uint64_t b0 = smem_desc(smem_u32(s_stage + K::kXBytes), 128, kSbo);
        bool ok = true;
        int stage = 0;
        uint32_t sphase = 0, aphase = 0;
        int64_t g = g0, q = q0;
        bool new_group = true;
        for (int c = 0; c < total && ok; ++c) {
            ok = (!new_group || mbar_wait(&bar_a, aphase, &s_abort, p.err)) &&
                 mbar_wait(&bar_ready[stage], sphase, &s_abort, p.err) &&
                 (c == 0 || mbar_wait(&bar_acc_free, (uint32_t)((c - 1) & 1), &s_abort, p.err));
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            if (new_group) aphase ^= 1u;
            new_group = false;
            tc_fence_after();
            if (leader) {
                const uint64_t b = b0 + (uint64_t)((stage * K::kStageBytes) >> 4);
#pragma unroll 1
                for (int r = 0; r < R; ++r) {
                    const uint64_t a = a0 + (uint64_t)((r * K::kPlaneA) >> 4);
                    const uint32_t d = tmem + (uint32_t)r * K::kAccCols, ds = d + K::kHh * kChunk;
                    constexpr uint64_t pa = (R * K::kPlaneA) >> 4, pb = K::kPlaneB >> 4;
#pragma unroll
                    for (int ks = 0; ks < K::kSteps; ++ks) {
                        // the products of weight 2^-16 of all steps first, while the sum is small
                        const uint64_t ak = a + (uint64_t)(16 * ks), bk = b + (uint64_t)(16 * ks);
                        mma_ss(ds, ak + 2 * pa, bk, idesc, ks > 0 ? 1u : 0u);
                        mma_ss(ds, ak + pa, bk + pb, idesc, 1u);
                        mma_ss(ds, ak, bk + 2 * pb, idesc, 1u);
                    }
#pragma unroll
                    for (int ks = 0; ks < K::kSteps; ++ks) {
                        const uint64_t ak = a + (uint64_t)(16 * ks), bk = b + (uint64_t)(16 * ks);
                        mma_ss(ds, ak + pa, bk, idesc, 1u);
                        mma_ss(ds, ak, bk + pb, idesc, 1u);
                        mma_ss(d + (ks / 2) * kChunk, ak, bk, idesc, (uint32_t)(ks & 1));
                    }
                }
                tc_commit(&bar_acc);
                tc_commit(&bar_empty[stage]);
            }
            __syncwarp();
            if (++stage == kStages) {
                stage = 0;
                sphase ^= 1u;
            }
            if (++q == L) {
                ++g;
                q = g * rc;
                new_group = true;
            }
        }
    } else if (warp == K::kCopyWarp) {
        // ------------------------------------------ bulk copies of the coordinates
        if (lane == 0) {
            bool ok = true;
            int64_t g = g0, q = q0;
            int stage = 0;
            for (int c = 0; c < total && ok; ++c) {
                if (c >= kStages)
                    ok = mbar_wait_issuer(&bar_empty[stage], (uint32_t)((c / kStages - 1) & 1), &s_abort, p.err,
                                          p.wait_cycles);
                if (!ok) break;
                const int cnt = (int)min((int64_t)kChunk, n - q * kChunk);
                const bool in = AP_CHK(q >= 0 && cnt > 0 && q * kChunk + cnt <= n);
                mbar_expect_tx(&bar_full[stage], in ? (uint32_t)(cnt * D * 4) : 0u);
                if (in)
                    bulk_g2s(s_stage + (size_t)stage * K::kStageBytes, p.Xs + q * kChunk * D, (uint32_t)(cnt * D * 4),
                             &bar_full[stage]);
                if (++q == L) {
                    ++g;
                    q = g * rc;
                }
                if (++stage == kStages) stage = 0;
            }
        }
    } else {
        // --------------------------------------- splitters of the chunk's [V | alpha U]
        const int ct = tid - K::kConvWarp * 32;
        int64_t g = g0, q = q0;
        int stage = 0;
        uint32_t sphase = 0;
        for (int c = 0; c < total; ++c) {
            // when the copy into this stage has landed the stage's last users are done (the
            // first chunks find their stages unused)
            auto landed = [&]() { return __all_sync(0xffffffffu, mbar_wait(&bar_full[stage], sphase, &s_abort, p.err)); };
            if (c >= kStages && !landed()) break;
            uint8_t* st = s_stage + (size_t)stage * K::kStageBytes;
            const int cnt = (int)min((int64_t)kChunk, n - q * kChunk);
#pragma unroll 2
            for (int t = ct; t < kChunk * (K::KC / 8); t += 32 * kConvWarps) {
                const int j = t % kChunk, k8 = t / kChunk;  // (neighbouring lanes fill one core matrix)
                split_operand<C>(p, q * kChunk + j, 8 * k8, false, vec,
                                 st + K::kXBytes + ((j >> 3) * (K::KC / 8) + k8) * 128 + (j & 7) * 16, K::kPlaneB);
            }
            if (c < kStages && !landed()) break;
            if (cnt < kChunk)
                for (int t = cnt * D + ct; t < kChunk * D; t += 32 * kConvWarps)
                    reinterpret_cast<float*>(st)[t] = reinterpret_cast<const float*>(st)[(cnt - 1) * D + t % D];
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_ready[stage]);
            if (++q == L) {
                ++g;
                q = g * rc;
            }
            if (++stage == kStages) {
                stage = 0;
                sphase ^= 1u;
            }
        }
    }
    // ---------------------------------------------------------------- teardown
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == K::kMmaWarp) {
        if (s_abort) {
            // a wait gave up: let copies and MMAs still in flight land first
            const long long t0 = clock64();
            while (clock64() - t0 < 4000000LL) {
            }
        }
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(K::kTmem) : "memory");
    }
    if (s_abort) return;
    if (tid < K::NA) {
        double v = 0.0;
        for (int w = 0; w < K::kXformWarps; ++w) v += s_part[w][tid];
        p.part[(int64_t)blockIdx.x * K::NA + tid] = v;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(p.ticket, 1u) == gridDim.x - 1u) ? 1 : 0;
    __syncthreads();
    if (s_last) {
        __threadfence();
        // ranges of CTAs side by side, then the ranges in order
        constexpr int NG = K::kXformWarps;
        const int per = ((int)gridDim.x + NG - 1) / NG;
        for (int t = tid; t < NG * K::NA; t += K::kThreads) {
            const int g = t / K::NA, k = t % K::NA;
            double acc = 0.0;
#pragma unroll 10
            for (int b = g * per; b < min((g + 1) * per, (int)gridDim.x); ++b) acc += __ldcg(p.part + (int64_t)b * K::NA + k);
            s_part[g][k] = acc;
        }
        __syncthreads();
        for (int k = tid; k < K::NA; k += K::kThreads) {
            double acc = 0.0;
            for (int g = 0; g < NG; ++g) acc += s_part[g][k];
            p.out[k] = acc;
        }
        if (tid == 0) *p.ticket = 0u;
    }
}

template <int KERN, int D, int C>
cudaError_t launch_inst(const GradParams& p, cudaStream_t st) {
    using K = Cfg<D, C>;
    auto fn = grad_kernel<KERN, D, C>;
    cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::kSmem);
    if (err != cudaSuccess) return err;
    const int64_t L = (p.n + kChunk - 1) / kChunk, ngroups = (p.n + K::kRows - 1) / K::kRows;
    const int64_t U = units_before(ngroups, L, K::kRows / kChunk);
    const int64_t grid = U < kGradCtas ? U : kGradCtas;
    fn<<<(unsigned)grid, K::kThreads, K::kSmem, st>>>(p);
    return cudaGetLastError();
}

}  // namespace gx

template <int KERN>
cudaError_t dispatch_grad(const GradParams& p, int D, int C, cudaStream_t st) {
#define AP_GRAD_C(DD)                                                    \
    switch (C) {                                                         \
        case 1: return gx::launch_inst<KERN, DD, 1>(p, st);              \
        case 4: return gx::launch_inst<KERN, DD, 4>(p, st);              \
        case 16: return gx::launch_inst<KERN, DD, 16>(p, st);            \
        case 32: return gx::launch_inst<KERN, DD, 32>(p, st);            \
        default: return cudaErrorInvalidValue;                           \
    }
    switch (D) {
        case 4: AP_GRAD_C(4)
        case 8: AP_GRAD_C(8)
        case 12: AP_GRAD_C(12)
        case 16: AP_GRAD_C(16)
        case 24: AP_GRAD_C(24)
        case 32: AP_GRAD_C(32)
        default: return cudaErrorInvalidValue;
    }
#undef AP_GRAD_C
}

}  // namespace ap
