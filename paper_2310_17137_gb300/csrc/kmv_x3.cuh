// FP32 kernel-matrix product for c > 4 right-hand sides (from kX3MinEntries16 / 32
// entries on; kmv_fp32.cuh below): entries in FP32 on the CUDA cores, the contraction with V on the tensor cores in split-precision form.
//
//   out[i,:] = base[i,:] + sgn * (s * sum_j phi(x_i, x_j) V[j,:] + noise V_i (diagonal))
//
// Why: with c = 16..32 right-hand sides 2c of the ~2c + 3d + 6 FP32 operations of an
// entry are the contraction, and the SIMT form of this product ran at half of the FMA
// pipe's rate on them (n = 131,072, d = 3, c = 16: 19.1 ms for n^2 entries; n = 65,536,
// d = 8, c = 32: 665 us per 4096 columns).  Here an entry costs its distance, phi and
// nine integer / packed-FP32 instructions per pair for the split; what bounds it is the
// issue rate of those and the SFU, whatever c is.
//
// Precision: an FP32 value has 24 significant bits, so P = phi is exactly
// P_hi + P_mid + P_lo with three BF16 parts (8 bits each, cut off by masking); V is
// split the same way with rounding.  The six products of weight above 2^-24
// (hh, hm, mh, hl, mm, lh) go to FP32 accumulators by weight (hh | hm + mh |
// hl + mm + lh); ml, lm and ll are below 2^-25 of the product.  The accumulators are
// drained every 64 columns and summed in FP32 registers with rounding to nearest.
// The tensor cores cut their sums off towards zero: each step of 16 columns that is added
// to a running sum takes about half a unit of that sum's last place, always in the same
// sense.  So hh has an accumulator per step (two for the four steps where tensor memory or
// the drain's time do not allow more: 32 columns, and D = 4, where the drain is not hidden)
// and V's parts are rounded to nearest, so that neither the small sums nor the dropped
// products have a preferred sign.
// Measured against 64 bits, root mean square of the error relative to the result, random
// signs in V, SIMT form -> this one: n = 16,384, d = 8, c = 16 Matern-3/2 8.8e-7 -> 2.2e-7;
// n = 65,536, d = 3, c = 16 Matern-5/2 5.6e-7 here; what the error has in common with the
// result (a factor on it): +5e-9 -> +3e-9 there, +2.9e-8 -> +2.9e-8 with V >= 0 (that of
// exp2 and sqrt; -2.9e-8 and -1.9e-8 with one accumulator for hh and V's hi cut off, which
// doubled the error of a training step's gradient).
// Measured time (GB300): n = 131,072, d = 3, c = 16, n^2 entries of Matern-5/2 19.1 ->
// 12.4 ms; n = 65,536, d = 8, c = 32, 4096 columns of Matern-3/2 665 -> 306 us, at
// 71 % of the issue slots and 61 % of the FMA pipe (tensor pipe 15 %).
// Infinities and NaNs in V are taken out of the split, noted per column and chunk, and
// added by the drain to every row of the tile: a row whose kernel entry underflows to 0
// gets the infinity too (the SIMT form: 0 times infinity, NaN).
//
// One persistent CTA per SM.  Work units are (row group, 128-column chunk) pairs in
// group-major order, cut into equal contiguous ranges; a group has 128 R rows (R = 2:
// every column read from shared memory serves two rows of a thread; R = 1 where the
// coordinates of two rows do not fit the registers or a segment is short).  A group
// shared by several CTAs leaves its parts in per-CTA slots; the CTA that arrives last
// adds them in CTA order (deterministic, nobody waits).
//
// Warp roles: 16 transform warps (four per tensor-memory lane quarter) take work items
// of 16 x 2 columns-by-rows-per-thread round-robin and write the three P planes to a
// ring of tensor-memory buffers; the drain warps (tensor-memory lanes as above) empty
// the accumulators and run the epilogue; one warp issues the MMAs, one lane the bulk
// copies of the columns' coordinates and V, two warps split V into its BF16 planes.
// Every wait is bounded.
#pragma once

#include "kmv_fp32.cuh"
#include "tcgen05.cuh"

namespace ap {
namespace x3 {

using namespace tc;

constexpr int kChunk = 128;   // columns per chunk
constexpr int kDrains = 2;    // accumulator drains per chunk
constexpr int kStages = 3;    // shared-memory operand stages
constexpr int kSlots = 4;     // transform warps per lane quarter
constexpr int kXformWarps = 4 * kSlots;
constexpr int kConvWarps = 2;
constexpr int kFlagRing = 8;  // chunks of non-finite flags, half of them being cleared ahead
static_assert(kFlagRing >= 2 * (kStages + 1), "a cleared flag is neither in use nor set yet");
constexpr uint32_t kBufCols = 48;  // tensor-memory columns of one P buffer: 2 units x 3 planes x 8

template <int D, int C, int R>
struct Cfg {
    static constexpr int kRows = 128 * R;
    static constexpr int kTpd = (R == 2 && C == 16) ? 2 : 1;  // tiles per drain warp
    static constexpr int kDrainWarps = 4 * R / kTpd;
    static constexpr int kMmaWarp = kXformWarps + kDrainWarps;
    static constexpr int kCopyWarp = kMmaWarp + 1;
    static constexpr int kConvWarp = kMmaWarp + 2;
    static constexpr int kThreads = (kConvWarp + kConvWarps) * 32;
    static constexpr uint32_t kXBytes = kChunk * D * 4, kVBytes = kChunk * C * 4;
    static constexpr uint32_t kV3Bytes = 3u * C * kChunk * 2u;
    static constexpr uint32_t kStageBytes = kXBytes + kVBytes + kV3Bytes;
    static constexpr int kSteps = kChunk / kDrains / 16;      // steps of 16 columns between drains
    static constexpr int kHh = C == 16 && D >= 8 ? kSteps : 2;  // accumulators of hi x hi
    static constexpr uint32_t kTileCols = (kHh + 2) * C;      // hh_{kHh-1} .. hh_0 | hm + mh | hl + mm + lh
    static constexpr uint32_t kAccCols = R * kTileCols;
    static constexpr int kBufs = (int)((512 - kAccCols) / kBufCols) < 8 ? (int)((512 - kAccCols) / kBufCols) : 8;
    static constexpr int kUnitCols = R == 2 ? 16 : 32;  // columns of a work item
    static constexpr int kItems = kChunk / kUnitCols;   // work items per chunk
    static constexpr size_t kSmem = kStages * kStageBytes + 1024;
    static_assert(kBufs > kSlots, "a free buffer beyond the ones being written");
    static_assert(kItems % kDrains == 0, "drains fall between work items");
    static_assert(kItems >= kSlots && kItems % kSlots == 0, "items go round the slots within a chunk");
    static_assert(kSmem <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&r)[4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3])
                 : "memory");
}

// x0, x1 >= 0 as three exact BF16 parts each, packed (x0 low half, x1 high half): parts cut
// off by masking.  (For D = 4 rounding them by conversions is faster, split3_nearest: the
// masks' pipe is the busier one there, n = 40,000, c = 16 1230 : 1187 us; from D = 8 on it
// takes 1 to 3 % longer.)
__device__ __forceinline__ void split3(float x0, float x1, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    constexpr uint32_t kTop = 0xFFFF0000u;
    const uint32_t b0 = __float_as_uint(x0), b1 = __float_as_uint(x1);
    hi = __byte_perm(b0, b1, 0x7632);
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 r1 = __ffma2_rn(make_float2(__uint_as_float(b0 & kTop), __uint_as_float(b1 & kTop)), m1, make_float2(x0, x1));
    const uint32_t c0 = __float_as_uint(r1.x), c1 = __float_as_uint(r1.y);
    mid = __byte_perm(c0, c1, 0x7632);
    const float2 r2 = __ffma2_rn(make_float2(__uint_as_float(c0 & kTop), __uint_as_float(c1 & kTop)), m1, r1);
    lo = __byte_perm(__float_as_uint(r2.x), __float_as_uint(r2.y), 0x7632);
}

// The CTA whose range [U b / G, U (b + 1) / G) holds unit u.
__device__ __forceinline__ int owner_of(int64_t u, int64_t U, int64_t G) { return (int)(((u + 1) * G - 1) / U); }

template <int KERN, int D, int C, int R>
__global__ void __launch_bounds__(Cfg<D, C, R>::kThreads, 1) kmv_x3_kernel(const KmvParams p) {
    using K = Cfg<D, C, R>;
    extern __shared__ __align__(1024) uint8_t x3_smem[];
    __shared__ __align__(8) uint64_t bar_full[kStages], bar_ready[kStages], bar_empty[kStages];
    __shared__ __align__(8) uint64_t bar_p[K::kBufs], bar_free[K::kBufs], bar_acc, bar_acc_free;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ int s_nf[kFlagRing][C];  // non-finite V per chunk and column: 1 +inf, 2 -inf, 4 NaN
    __shared__ int s_any[kFlagRing];
    __shared__ double s_red[K::kDrainWarps];
    __shared__ double s_col[16 * C];
    __shared__ double red_d[32];
    __shared__ int red_i[32];
    __shared__ int s_fin, s_last;

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const EpiParams& e = p.epi;
    int64_t col0 = p.col0, ncols = p.ncols;
    if (p.sel) {
        col0 = (int64_t)(*p.sel) * p.blk;
        ncols = min(p.blk, p.nb - col0);
    }
    const int nq = (int)((ncols + kChunk - 1) / kChunk);
    const int64_t U = e.ntiles * nq;
    // a short selected block can have fewer units than there are CTAs: the rest idle
    const int64_t grid = min((int64_t)gridDim.x, U), cta = min((int64_t)blockIdx.x, grid);
    const bool share = p.G > 1;  // ranges may cut a group (slots and tickets are there)
    const int64_t u0 = share ? U * cta / grid : e.ntiles * cta / grid * nq;
    const int64_t u1 = cta == grid ? u0 : (share ? U * (cta + 1) / grid : e.ntiles * (cta + 1) / grid * nq);
    const int total = (int)(u1 - u0);  // chunks of this CTA
    const int64_t g0 = u0 / nq;
    const int q0 = (int)(u0 % nq);

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&bar_full[i], 1);
            mbar_init(&bar_ready[i], kConvWarps);
            mbar_init(&bar_empty[i], 1);
        }
        for (int i = 0; i < K::kBufs; ++i) {
            mbar_init(&bar_p[i], 4);
            mbar_init(&bar_free[i], 1);
        }
        mbar_init(&bar_acc, 1);
        mbar_init(&bar_acc_free, K::kDrainWarps);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int t = tid; t < kFlagRing * C; t += K::kThreads) s_nf[t / C][t % C] = 0;
    if (tid < kFlagRing) s_any[tid] = 0;
    if (warp == K::kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t tmem_p = tmem + K::kAccCols;
    pdl_wait();  // V and base (the block index was complete before the block solve began)
    pdl_launch();

    if (warp < kXformWarps) {
        // ------------------------------------------------------- transform warps
        const int quarter = warp & 3, slot = warp >> 2;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        float2 xa[R][D / 2];
        auto load_rows = [&](int64_t g) {
            const int64_t seg_lo = g / e.tiles_per_seg * e.seg, seg_hi = min(seg_lo + e.seg, p.na);
            const int64_t r0 = seg_lo + g % e.tiles_per_seg * K::kRows + quarter * 32 + lane;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int64_t i = r0 + 128 * r;
#pragma unroll
                for (int k = 0; k < D / 4; ++k) {
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (i < seg_hi && AP_CHK(i < p.na)) v = __ldg(reinterpret_cast<const float4*>(p.Xa + i * D) + k);
                    xa[r][2 * k] = make_float2(v.x, v.y);
                    xa[r][2 * k + 1] = make_float2(v.z, v.w);
                }
            }
        };
        const float2 m1 = make_float2(-1.0f, -1.0f);
        bool ok = true;
        int64_t g = g0;
        int q = q0, stage = 0, buf = slot;
        uint32_t sphase = 0, use = 0;
        if (total > 0) load_rows(g);
        for (int c = 0; c < total && ok; ++c) {
            // the copy itself, then the tail of a short chunk (filled by the splitters)
            ok = mbar_wait(&bar_full[stage], sphase, &s_abort, p.err) &&
                 mbar_wait(&bar_ready[stage], sphase, &s_abort, p.err);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const float* sx = reinterpret_cast<const float*>(x3_smem + (size_t)stage * K::kStageBytes);
            for (int it = slot; it < K::kItems; it += kSlots) {
                const uint32_t addr = tmem_p + lane_base + kBufCols * (uint32_t)buf;
                const float* xc = sx + it * K::kUnitCols * D;
#pragma unroll
                for (int sub = 0; sub < K::kUnitCols / 8; ++sub) {
                    uint32_t hi[R][4], mid[R][4], lo[R][4];
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        float kv[R][2];
#pragma unroll
                        for (int jj = 0; jj < 2; ++jj) {
                            const float4* xb = reinterpret_cast<const float4*>(xc + (sub * 8 + 2 * w + jj) * D);
                            float2 tp[R];
#pragma unroll
                            for (int r = 0; r < R; ++r) tp[r] = make_float2(0.0f, 0.0f);
#pragma unroll
                            for (int k = 0; k < D / 4; ++k) {
                                const float4 v = xb[k];
#pragma unroll
                                for (int r = 0; r < R; ++r) {
                                    const float2 da = __ffma2_rn(make_float2(v.x, v.y), m1, xa[r][2 * k]);
                                    tp[r] = __ffma2_rn(da, da, tp[r]);
                                    const float2 db = __ffma2_rn(make_float2(v.z, v.w), m1, xa[r][2 * k + 1]);
                                    tp[r] = __ffma2_rn(db, db, tp[r]);
                                }
                            }
#pragma unroll
                            for (int r = 0; r < R; ++r) kv[r][jj] = phi_fp32<KERN>(tp[r].x + tp[r].y);
                        }
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            if constexpr (D == 4) split3_nearest(kv[r][0], kv[r][1], hi[r][w], mid[r][w], lo[r][w]);
                            else split3(kv[r][0], kv[r][1], hi[r][w], mid[r][w], lo[r][w]);
                        }
                    }
                    if (sub == 0 && use > 0) {
                        ok = __all_sync(0xffffffffu, mbar_wait(&bar_free[buf], (use - 1) & 1u, &s_abort, p.err));
                        if (!ok) break;
                        tc_fence_after();
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        // unit (R = 2: row tile r; R = 1: 16-column half) and 8-column half within it
                        const uint32_t at = addr + 24u * (uint32_t)(R == 2 ? r : sub / 2) +
                                            4u * (uint32_t)(R == 2 ? sub : sub % 2);
                        tmem_st4(at, hi[r]);
                        tmem_st4(at + 8, mid[r]);
                        tmem_st4(at + 16, lo[r]);
                    }
                }
                if (!ok) break;
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bar_p[buf]);
                buf += kSlots;
                if (buf >= K::kBufs) {
                    buf -= K::kBufs;
                    ++use;
                }
            }
            if (++stage == kStages) {
                stage = 0;
                sphase ^= 1u;
            }
            if (++q == nq) {
                q = 0;
                ++g;
                if (c + 1 < total) load_rows(g);
            }
        }
    } else if (warp < K::kMmaWarp) {
        // ----------------------------------------------------------- drain warps
        const int quarter = warp & 3, dw = warp - kXformWarps;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const int tile0 = K::kTpd == 2 ? 0 : dw / 4;
        constexpr int kDrainThreads = K::kDrainWarps * 32;
        const int dtid = tid - kXformWarps * 32;
        float acc[K::kTpd][C];
#pragma unroll
        for (int tt = 0; tt < K::kTpd; ++tt)
#pragma unroll
            for (int k = 0; k < C; ++k) acc[tt][k] = 0.0f;
        bool ok = true;  // after a failed wait the loop runs on through the named barriers only
        int64_t g = g0;
        int q = q0, seg_q = q0;
        for (int n = 0; n < total * kDrains; ++n) {
            const int c = n / kDrains;
            const bool chunk_end = n % kDrains == kDrains - 1;
            if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&bar_acc, (uint32_t)(n & 1), &s_abort, p.err));
            if (ok) {
                tc_fence_after();
#pragma unroll
                for (int tt = 0; tt < K::kTpd; ++tt) {
                    const uint32_t a = tmem + lane_base + (uint32_t)(tile0 + tt) * K::kTileCols;
#pragma unroll
                    for (int k0 = 0; k0 < C; k0 += 8) {
                        float t[8];
#pragma unroll
                        for (int h = K::kHh; h >= 0; h -= 2) {  // the small sums, then hi x hi in pairs
                            uint32_t w0[8], w1[8];
                            tmem_ld8(a + h * C + k0, w0);
                            tmem_ld8(a + (h + 1) * C + k0, w1);
                            tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const float v = __uint_as_float(w0[k]) + __uint_as_float(w1[k]);
                                t[k] = h == K::kHh ? v : t[k] + v;
                            }
                        }
#pragma unroll
                        for (int k = 0; k < 8; ++k) acc[tt][k0 + k] += t[k];
                    }
                }
                tc_fence_before();
                if (chunk_end && s_any[c % kFlagRing]) {
#pragma unroll
                    for (int k = 0; k < C; ++k) {
                        const int f = s_nf[c % kFlagRing][k];
                        float v = 0.0f;
                        if (f & 1) v += __int_as_float(0x7f800000);
                        if (f & 2) v -= __int_as_float(0x7f800000);
                        if (f & 4) v = __int_as_float(0x7fffffff);
#pragma unroll
                        for (int tt = 0; tt < K::kTpd; ++tt) acc[tt][k] += v;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_acc_free);
            if (!chunk_end) continue;
            if (q == nq - 1 || c == total - 1) {
                // ---- the group, or this CTA's part of it, is complete
                const bool whole = seg_q == 0 && q == nq - 1;
                bool apply = whole;
                if (!whole) {
                    const int64_t slot = cta * 2 + (g == g0 ? 0 : 1);
                    float* mine = p.gscr + slot * K::kRows * C;
                    if (ok) {
#pragma unroll
                        for (int tt = 0; tt < K::kTpd; ++tt) {
                            float* row = mine + (int64_t)((tile0 + tt) * 128 + quarter * 32 + lane) * C;
#pragma unroll
                            for (int k = 0; k < C; k += 4)
                                __stcg(reinterpret_cast<float4*>(row + k),
                                       make_float4(acc[tt][k], acc[tt][k + 1], acc[tt][k + 2], acc[tt][k + 3]));
                        }
                    }
                    __threadfence();
                    asm volatile("bar.sync 1, %0;" ::"n"(kDrainThreads) : "memory");
                    const int b0 = owner_of(g * nq, U, grid), b1 = owner_of(g * nq + nq - 1, U, grid);
                    if (dtid == 0) {
                        int fin = 0;
                        if (ok && !s_abort && AP_CHK(g >= 0 && g < e.ntiles)) {
                            fin = atomicAdd(p.gtick + g, 1u) == (unsigned)(b1 - b0);
                            if (fin) p.gtick[g] = 0u;
                            __threadfence();
                        }
                        s_fin = fin;
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(kDrainThreads) : "memory");
                    apply = s_fin != 0;
                    if (apply) {
#pragma unroll
                        for (int tt = 0; tt < K::kTpd; ++tt)
#pragma unroll
                            for (int k = 0; k < C; ++k) acc[tt][k] = 0.0f;
                        for (int b = b0; b <= b1; ++b) {
                            const int64_t sl = (int64_t)b * 2 + (U * b / grid >= g * nq ? 0 : 1);
#pragma unroll
                            for (int tt = 0; tt < K::kTpd; ++tt) {
                                const float* row = p.gscr + sl * K::kRows * C +
                                                   (int64_t)((tile0 + tt) * 128 + quarter * 32 + lane) * C;
#pragma unroll
                                for (int k = 0; k < C; k += 4) {
                                    const float4 v = __ldcg(reinterpret_cast<const float4*>(row + k));
                                    acc[tt][k] += v.x;
                                    acc[tt][k + 1] += v.y;
                                    acc[tt][k + 2] += v.z;
                                    acc[tt][k + 3] += v.w;
                                }
                            }
                        }
                    }
                }
                const int64_t seg_lo = g / e.tiles_per_seg * e.seg, seg_hi = min(seg_lo + e.seg, p.na);
                const int64_t r0 = seg_lo + g % e.tiles_per_seg * K::kRows + quarter * 32 + lane;
                double sq = 0.0;
                double cs[C / 2];  // column squares of this warp's rows, see below
                const bool colnorms = apply && (e.flags & kEpiColNorms);
#pragma unroll
                for (int k = 0; k < C / 2; ++k) cs[k] = 0.0;
#pragma unroll
                for (int tt = 0; tt < K::kTpd; ++tt) {
                    const int64_t i = r0 + 128 * (tile0 + tt);
                    const bool live = ok && apply && i < seg_hi && AP_CHK(i < p.na);
                    const bool diag = live && p.noise_diag && i >= col0 && i < col0 + ncols;
#pragma unroll
                    for (int k = 0; k < C; k += 4) {
                        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (live) {
                            float4 vd = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (diag) vd = __ldg(reinterpret_cast<const float4*>(p.V + (i - col0) * C + k));
                            o = p.base ? *reinterpret_cast<const float4*>(p.base + i * C + k)
                                       : make_float4(p.base_const, p.base_const, p.base_const, p.base_const);
                            auto fin = [&](float a, float v, float b) {
                                float t = p.s * a;
                                if (diag) t = fmaf(p.noise, v, t);
                                return fmaf(p.sgn, t, b);
                            };
                            o.x = fin(acc[tt][k], vd.x, o.x);
                            o.y = fin(acc[tt][k + 1], vd.y, o.y);
                            o.z = fin(acc[tt][k + 2], vd.z, o.z);
                            o.w = fin(acc[tt][k + 3], vd.w, o.w);
                            *reinterpret_cast<float4*>(p.out + i * C + k) = o;
                            sq += (double)o.x * o.x + (double)o.y * o.y + (double)o.z * o.z + (double)o.w * o.w;
                        }
                        acc[tt][k] = o.x;
                        acc[tt][k + 1] = o.y;
                        acc[tt][k + 2] = o.z;
                        acc[tt][k + 3] = o.w;
                    }
                    if (colnorms) {
                        // halving exchange: lanes 16 apart split the C columns between them
                        const bool up = lane & 16;
#pragma unroll
                        for (int k = 0; k < C / 2; ++k) {
                            const float keep = up ? acc[tt][k + C / 2] : acc[tt][k];
                            const float got = __shfl_xor_sync(0xffffffffu, up ? acc[tt][k] : acc[tt][k + C / 2], 16);
                            cs[k] += (double)keep * keep + (double)got * got;
                        }
                    }
                }
                if (e.flags & kEpiBlockNorms) {
                    for (int o = 16; o > 0; o >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, o);
                    if (lane == 0) s_red[dw] = sq;
                }
                if (colnorms) {
                    // the remaining halvings: lanes 8, 4, 2, 1 apart
#pragma unroll
                    for (int o = 8, w = C / 4; o > 0; o >>= 1, w /= 2) {
                        const bool up = lane & o;
#pragma unroll
                        for (int k = 0; k < (w > 0 ? w : 1); ++k) {
                            if (w > 0) {
                                const double keep = up ? cs[k + w] : cs[k];
                                cs[k] = keep + __shfl_xor_sync(0xffffffffu, up ? cs[k] : cs[k + w], o);
                            } else {
                                cs[0] += __shfl_xor_sync(0xffffffffu, cs[0], o);
                            }
                        }
                    }
                    // lane bits 16, 8, 4, 2 (and 1 for C = 32) spell the column from its top bit down
                    const int cc = C == 32 ? lane : lane >> 1;
                    if (C == 32 || !(lane & 1)) s_col[dw * C + cc] = cs[0];
                }
                if (e.flags & (kEpiBlockNorms | kEpiColNorms)) {
                    asm volatile("bar.sync 1, %0;" ::"n"(kDrainThreads) : "memory");
                    if (apply && AP_CHK(g >= 0 && g < e.ntiles)) {
                        if (dtid == 0 && (e.flags & kEpiBlockNorms)) {
                            double t = 0.0;
                            for (int w = 0; w < K::kDrainWarps; ++w) t += s_red[w];
                            e.part_norm[g] = t;
                        }
                        if (dtid < C && (e.flags & kEpiColNorms)) {
                            double t = 0.0;
                            for (int w = 0; w < K::kDrainWarps; ++w) t += s_col[w * C + dtid];
                            e.part_col[g * C + dtid] = t;
                        }
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(kDrainThreads) : "memory");
                }
#pragma unroll
                for (int tt = 0; tt < K::kTpd; ++tt)
#pragma unroll
                    for (int k = 0; k < C; ++k) acc[tt][k] = 0.0f;
            }
            if (++q == nq) {
                q = 0;
                ++g;
                seg_q = 0;
            }
        }
    } else if (warp == K::kMmaWarp) {
        // ------------------------------------------------------------ MMA issuer
        // (whole warp in the loop, warp-uniform descriptors, one elected lane issues)
        constexpr uint32_t i3 = instr_desc(1, 128, 3 * C), i2 = instr_desc(1, 128, 2 * C), i1 = instr_desc(1, 128, C);
        const bool leader = elect_one();
        const uint64_t d0 = smem_desc(smem_u32(x3_smem + K::kXBytes + K::kVBytes), 128, (kChunk / 8) * 128);
        bool ok = true;
        int stage = 0, buf = 0;
        uint32_t sphase = 0, use = 0;
        for (int c = 0; c < total && ok; ++c) {
            ok = __all_sync(0xffffffffu, mbar_wait(&bar_ready[stage], sphase, &s_abort, p.err));
            if (!ok) break;
            const uint64_t dv = d0 + (uint64_t)((stage * K::kStageBytes) >> 4);
            for (int it = 0; it < K::kItems; ++it) {
                constexpr int kPerDrain = K::kItems / kDrains;
                const bool first = it % kPerDrain == 0;
                const int n = c * kDrains + it / kPerDrain;  // drain these items go to
                ok = mbar_wait(&bar_p[buf], use & 1u, &s_abort, p.err) &&
                     (!first || n == 0 || mbar_wait(&bar_acc_free, (uint32_t)((n - 1) & 1), &s_abort, p.err));
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                if (leader) {
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const uint32_t pa = tmem_p + kBufCols * (uint32_t)buf + 24u * (uint32_t)u;
                        const uint32_t acc = tmem + (R == 2 ? (uint32_t)u * K::kTileCols : 0u) + (K::kHh - 1) * C;  // hh_0
                        const uint64_t b = dv + (uint64_t)((R == 2 ? it : 2 * it + u) * 16);
                        const int step = R == 2 ? it % kPerDrain : 2 * (it % kPerDrain) + u, j = step % K::kHh;
                        const uint32_t add = step > 0 ? 1u : 0u, add_hh = step >= K::kHh ? 1u : 0u;
                        if (j == 0) {
                            mma_ts(acc, pa, b, i3, add);  // hi x [hi; mid; lo]
                        } else {
                            mma_ts(acc - (uint32_t)(j * C), pa, b, i1, add_hh);                               // hi x hi
                            mma_ts(acc + C, pa, b + (uint64_t)(C / 8 * (kChunk / 8) * 8), i2, add);  // hi x [mid; lo]
                        }
                        mma_ts(acc + C, pa + 8, b, i2, 1u);       // mid x [hi; mid]
                        mma_ts(acc + 2 * C, pa + 16, b, i1, 1u);  // lo x hi
                    }
                    tc_commit(&bar_free[buf]);
                    if ((it + 1) % kPerDrain == 0) tc_commit(&bar_acc);
                    if (it == K::kItems - 1) tc_commit(&bar_empty[stage]);
                }
                __syncwarp();
                if (++buf == K::kBufs) {
                    buf = 0;
                    ++use;
                }
            }
            if (++stage == kStages) {
                stage = 0;
                sphase ^= 1u;
            }
        }
    } else if (warp == K::kCopyWarp) {
        // ------------------------------------------------------ bulk-copy issuer
        if (lane == 0) {
            bool ok = true;
            int q = q0, stage = 0;
            for (int c = 0; c < total && ok; ++c) {
                if (c >= kStages)
                    ok = mbar_wait_issuer(&bar_empty[stage], (uint32_t)((c / kStages - 1) & 1), &s_abort, p.err, p.wait_cycles);
                if (!ok) break;
                uint8_t* dst = x3_smem + (size_t)stage * K::kStageBytes;
                const int64_t lc = (int64_t)q * kChunk;
                const int cnt = (int)min((int64_t)kChunk, ncols - lc);
                const bool in = AP_CHK(col0 >= 0 && lc >= 0 && cnt > 0 && col0 + lc + cnt <= p.nb);
                mbar_expect_tx(&bar_full[stage], in ? (uint32_t)(cnt * (D + C) * 4) : 0u);
                if (in) {
                    bulk_g2s(dst, p.Xb + (col0 + lc) * D, (uint32_t)(cnt * D * 4), &bar_full[stage]);
                    bulk_g2s(dst + K::kXBytes, p.V + lc * C, (uint32_t)(cnt * C * 4), &bar_full[stage]);
                }
                if (++q == nq) q = 0;
                if (++stage == kStages) stage = 0;
            }
        }
    } else {
        // ------------------------------------------------------------- V splitters
        const int ct = tid - K::kConvWarp * 32;  // 0 .. 63
        bool ok = true;
        int q = q0, stage = 0;
        uint32_t sphase = 0;
        for (int c = 0; c < total && ok; ++c) {
            ok = __all_sync(0xffffffffu, mbar_wait(&bar_full[stage], sphase, &s_abort, p.err));
            if (!ok) break;
            uint8_t* st = x3_smem + (size_t)stage * K::kStageBytes;
            float* sx = reinterpret_cast<float*>(st);
            const float* sv = reinterpret_cast<const float*>(st + K::kXBytes);
            uint8_t* v3 = st + K::kXBytes + K::kVBytes;
            const int cnt = (int)min((int64_t)kChunk, ncols - (int64_t)q * kChunk);
            if (cnt < kChunk)
                for (int t = cnt * D + ct; t < kChunk * D; t += 64) sx[t] = sx[(cnt - 1) * D + t % D];
            int* nf = s_nf[c % kFlagRing];
            // The flags of four chunks ahead: their last user, chunk c - 4, is drained (this
            // stage was free, so the MMAs of chunk c - 3 began, after that drain), and chunk
            // c + 4 is not split before this chunk is complete.
            if (ct < C) s_nf[(c + kFlagRing / 2) % kFlagRing][ct] = 0;
            if (ct == 0) s_any[(c + kFlagRing / 2) % kFlagRing] = 0;
            // item: column k of V and 8 consecutive rows = one 16-byte core row per plane
            for (int t = ct; t < C * (kChunk / 8); t += 64) {
                const int k = t % C, j8 = t / C;
                float v[8];
                unsigned big = 0;  // largest magnitude, as bits
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int row = 8 * j8 + j;
                    v[j] = row < cnt ? sv[row * C + k] : 0.0f;
                    big = max(big, __float_as_uint(v[j]) << 1);
                }
                if (big >= 0xFF000000u) {  // an infinity or NaN among the eight
                    int flags = 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (!(fabsf(v[j]) <= 3.402823466e38f)) {
                            flags |= v[j] > 0.0f ? 1 : (v[j] < 0.0f ? 2 : 4);
                            v[j] = 0.0f;
                        }
                    atomicOr(&nf[k], flags);
                    s_any[c % kFlagRing] = 1;
                }
                uint32_t w[3][4];
#pragma unroll
                for (int j = 0; j < 4; ++j) split3_nearest(v[2 * j], v[2 * j + 1], w[0][j], w[1][j], w[2][j]);
#pragma unroll
                for (int pl = 0; pl < 3; ++pl) {
                    const int vr = pl * C + k;
                    *reinterpret_cast<uint4*>(v3 + ((vr >> 3) * (kChunk / 8) + j8) * 128 + (vr & 7) * 16) =
                        make_uint4(w[pl][0], w[pl][1], w[pl][2], w[pl][3]);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_ready[stage]);
            if (++q == nq) q = 0;
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
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
    if (s_abort || e.flags == 0) return;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(e.ticket, 1u) == gridDim.x - 1u) ? 1 : 0;
    __syncthreads();
    if (s_last) {
        __threadfence();
        epi_finalize<C>(e, red_d, red_i, s_col);
    }
}

template <int KERN, int D, int C, int R>
cudaError_t launch_inst(const KmvParams& p, cudaStream_t st) {
    using K = Cfg<D, C, R>;
    auto fn = kmv_x3_kernel<KERN, D, C, R>;
    cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::kSmem);
    if (err != cudaSuccess) return err;
    return launch_dependent(fn, dim3((unsigned)p.ctas), K::kThreads, K::kSmem, st, p.dependent, p);
}

// (D, C, R) dispatch for one kernel family; rows per thread as kmv_split chose them.
template <int KERN>
cudaError_t dispatch(const KmvParams& p, int D, int C, cudaStream_t st) {
#define AP_X3_R(DD, CC)                                                             \
    if (C == CC && p.rm == 1) return launch_inst<KERN, DD, CC, 1>(p, st);           \
    if constexpr (DD <= kX3MaxD2)                                                   \
        if (C == CC && p.rm == 2) return launch_inst<KERN, DD, CC, 2>(p, st);
#define AP_X3_C(DD)                 \
    {                               \
        AP_X3_R(DD, 16)             \
        AP_X3_R(DD, 32)             \
        return cudaErrorInvalidValue; \
    }
    switch (D) {
        case 4: AP_X3_C(4)
        case 8: AP_X3_C(8)
        case 12: AP_X3_C(12)
        case 16: AP_X3_C(16)
        case 24: AP_X3_C(24)
        case 32: AP_X3_C(32)
        default: return cudaErrorInvalidValue;
    }
#undef AP_X3_C
#undef AP_X3_R
}

}  // namespace x3
}  // namespace ap
