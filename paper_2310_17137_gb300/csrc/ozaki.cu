// Trailing update of the tiled FP64 Cholesky (Sec. 3, "Cached Cholesky
// Factors"; the SYRK/GEMM step carries b^3/3 of the factorisation's flops) and
// its panel solve (TRSM as the product A_ik L_kk^{-T}) on the tensor cores,
// with FP64 results.
//
// A_ij -= A_ik A_jk^T for the trailing tiles k < j <= i is an FP64 dot product
// of length 64 per entry.  GB300 runs FP64 at about 2 FMA per clock per SM, so
// the products are formed as exact integer arithmetic on the BF16 tensor cores
// instead (the splitting scheme of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication", Numer. Algorithms 2012):
//   1. every row r of the 64-wide panel is scaled by a power of two 2^-e_r so
//      that its entries lie in (-1/2, 1/2), and each scaled entry x is written
//      as x = sum_{p=1..8} s_p 2^{-7p} + rest, |rest| < 2^-57, with integer
//      slices |s_p| <= 64 (exact in BF16);
//   2. for every level L = p + q = 2..9 the tensor cores accumulate
//      acc_L = sum_{p+q=L} sum_kk s_p(r, kk) s_q(c, kk) in FP32.  Every partial
//      sum is an integer below 2^22, so the accumulation is exact;
//   3. the levels are combined in integers, T = sum_L acc_L 2^{7(9-L)} (below 2^68; as a
//      64-bit integer, or, from 2^62 on, as one without its last 5 bits), and
//      A_rc -= 2^{e_r+e_c-63} T with two FP64 roundings: T's own to 53 bits, in integer
//      arithmetic, and the sum's.
// The terms left out (levels above 9 and the slice remainders) are below about 2^-50 K max_kk|a_r,kk| max_kk|a_c,kk| per entry, the size of FP64
// rounding when the entries of a panel row have similar magnitudes; the matrix
// itself stays FP64.  On kernel blocks the factor's backward error ||L L^T - K|| / ||K||
// matches the all-FP64 factorisation (6e-16 vs 5e-16 on a Matern-5/2 block
// with condition number 1.6e4, in a NumPy model of these exact steps).
//
// Work item: a 128 x 64 output super-tile (two row tiles i0, i0 + 1 against
// one column tile j) of one block: bulk copies of the 8 slice planes of both
// operands (192 KB of shared memory), 144 MMAs (36 slice products x 4 K-steps
// of 16) into eight 64-column FP32 accumulators (all 512 tensor-memory
// columns), then an epilogue of one row per thread.  One persistent CTA per SM
// walks the work items; the next item's slices are copied in while the
// epilogue of the current one runs.  Every wait is bounded.
//
// The epilogue is what bounds the kernel: FP64 runs at 2 results per clock per SM, so
// an FP64 operation per entry of a super-tile costs 4096 clocks, as much as all its
// MMAs.  It therefore reads and combines the accumulators in 32-bit integers first
// (after which the next item's MMAs start), builds each product's double with integer
// instructions, and spends one FP64 operation per entry, the subtraction itself, under
// those MMAs.  Measured (GB300, b = 4096, mean over the 63 panels): 5 blocks 277 -> 148 us,
// 13 blocks 693 -> 395 us; panel solves of 5 blocks 33 -> 14 us.  Each CTA takes a
// contiguous range of items, whose neighbours share the 128 KB row slab in shared
// memory, and fetches half of the entries to update before it waits for the MMAs:
// 148 -> 120 us and 395 -> 289 us; the 16 x 256 bit reads (see the epilogue) 120 -> 91 us;
// all bits of the level sums kept 98 us (13 blocks 243 us).
#include <cuda_bf16.h>

#include <algorithm>

#include "ap_internal.cuh"
#include "tcgen05.cuh"

namespace ap {
namespace {

using namespace tc;

constexpr int T = kTile;
constexpr int kSlices = 8;
constexpr int kSlabRows = 2 * T;                            // rows of a super-tile
constexpr uint32_t kPlaneA = kSlabRows * T * 2;             // 16 KB of BF16
constexpr uint32_t kPlaneB = T * T * 2;                     // 8 KB
constexpr uint32_t kOzSmem = kSlices * (kPlaneA + kPlaneB); // 192 KB
constexpr int kEpiWarps = 16;                             // four per tensor-memory lane quarter
constexpr int kOzThreads = (kEpiWarps + 1) * 32;          // and one that issues copies and MMAs
constexpr uint32_t kRowBytes = T * 2;                       // one slice row (64 BF16)
constexpr int kBadExp = -(1 << 28);  // row exponent marking a non-finite panel row (two add up without overflow)

// byte offset of (row, kk) in a slice plane: K-major core matrices of 8 rows x
// 8 BF16, 8 K-cores (1 KB) per 8-row group
__device__ __forceinline__ size_t slice_off(int64_t row, int kk) {
    return ((size_t)((row >> 3) * 8 + (kk >> 3)) * 8 + (size_t)(row & 7)) * 16 + (size_t)(kk & 7) * 2;
}

// Slices of the panel (tile column k) for the trailing rows r >= 64 (k + 1),
// in integer arithmetic on the FP64 bit patterns: eight threads per row, each
// owning 8 consecutive K values (one 16-byte core row per slice plane).
//   e_r  = (largest biased exponent of the row) - 1021, so |v| 2^-e_r < 1/2;
//   X    = round(v 2^{56 - e_r}), an integer below 2^55 (values below 2^-1022
//          are taken as 0);
//   s_p  = round(t_p / 2^{56-7p}), t_{p+1} = t_p - s_p 2^{56-7p}, t_1 = X,
// so that X = sum_p s_p 2^{56-7p} exactly with every |s_p| <= 64.
__global__ void __launch_bounds__(256) oz_slice_kernel(const double* src0, int64_t zstride, int64_t sld,
                                                       int64_t nrows, int64_t row0, int64_t rows_pad,
                                                       size_t plane_bytes, uint8_t* S, int* E) {
    const int z = blockIdx.y;
    const int tid = threadIdx.x, grp = tid & 7;  // K values 8 grp .. 8 grp + 7
    const int64_t rr = (int64_t)blockIdx.x * 32 + (tid >> 3);
    const int64_t r = row0 + rr;  // row of the slice planes
    const bool live = rr < nrows;
    long long bits[8];
    if (live) {
        const double2* src = reinterpret_cast<const double2*>(src0 + (int64_t)z * zstride + rr * sld + 8 * grp);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const double2 v = src[h];
            bits[2 * h] = __double_as_longlong(v.x);
            bits[2 * h + 1] = __double_as_longlong(v.y);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) bits[q] = 0;
    }
    int ebmax = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) ebmax = max(ebmax, (int)((bits[q] >> 52) & 0x7ff));
    // the eight threads of a row are eight consecutive lanes
    for (int o = 1; o < 8; o <<= 1) ebmax = max(ebmax, __shfl_xor_sync(0xffffffffu, ebmax, o));
    if (!live) return;
    const bool nonfinite = ebmax == 0x7ff;
    const int e = ebmax - 1021;
    uint32_t w[kSlices][4];  // BF16 pairs of the 8 values, per plane
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int eb = (int)((bits[q] >> 52) & 0x7ff);
        long long X = 0;
        if (eb != 0 && !nonfinite) {
            const long long M = (bits[q] & 0xFFFFFFFFFFFFFLL) | (1LL << 52);
            const int sh = eb - ebmax + 2;  // <= 2
            if (sh >= 0) X = M << sh;
            else if (-sh <= 60) X = (M + (1LL << (-sh - 1))) >> (-sh);
            if (bits[q] < 0) X = -X;
        }
#pragma unroll
        for (int p = 1; p <= kSlices; ++p) {
            const int sft = 56 - 7 * p;
            const long long sp = sft > 0 ? (X + (1LL << (sft - 1))) >> sft : X;
            X -= sp << sft;
            const float f = (float)(int)sp;
            uint32_t hb;
            asm("{\n\t.reg .b16 h;\n\tcvt.rn.bf16.f32 h, %1;\n\tmov.b32 %0, {h, h};\n\t}" : "=r"(hb) : "f"(f));
            if (q & 1) w[p - 1][q >> 1] |= hb & 0xFFFF0000u;
            else w[p - 1][q >> 1] = hb & 0x0000FFFFu;
        }
    }
    uint8_t* Sz = S + (size_t)z * kSlices * plane_bytes + slice_off(r, 8 * grp);
#pragma unroll
    for (int p = 0; p < kSlices; ++p)
        *reinterpret_cast<uint4*>(Sz + (size_t)p * plane_bytes) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
    // a NaN or infinity in the panel must reach the next pivot test as NaN
    if (grp == 0) E[(int64_t)z * rows_pad + r] = nonfinite ? kBadExp : e;
}

// T = 2^42 h1 + 2^28 h2 + 2^14 l1 + l2 for the level pairs h1 .. l2 (h1 below 2^25 + 2^19,
// the others below 2^29) as v 2^drop: all bits below 2^62, otherwise without the last five
// (which the rounding to 53 bits drops anyway).
__device__ __forceinline__ long long level_int(int h1, int h2, int l1, int l2, int& drop) {
    const long long v = (long long)h2 * (1LL << 23) + ((long long)l1 * (1LL << 9) + (l2 >> 5)) + ((long long)h1 << 37);
    const bool whole = (unsigned)((int)(v >> 32) + (1 << 25)) < 1u << 26;  // -2^57 <= v < 2^57
    drop = whole ? 0 : 5;
    return whole ? (v << 5) | (l2 & 31) : v;
}

// 2^e0 v rounded to a double (half away from zero), for results in the normal range:
// normalised and rounded with integer instructions and no branches, so that a thread's
// sixteen chains run side by side.  `extreme` is set when the exponent leaves the
// normal doubles: the result is then not usable.
__device__ __forceinline__ double level_sum(long long v, int e0, bool& extreme) {
    const long long sign = v >> 63;
    const unsigned long long m0 = (unsigned long long)((v ^ sign) - sign);
    const unsigned hi = (unsigned)(m0 >> 32), lo = (unsigned)m0;
    const int lz = hi ? __clz((int)hi) : 32 + __clz((int)lo);
    // m = m0 << lz
    const unsigned a = hi ? hi : lo, b = hi ? lo : 0u;
    const unsigned mh = __funnelshift_l(b, a, lz), ml = b << (lz & 31);
    const int be = 1023 + 63 - lz + e0;  // biased exponent
    extreme |= m0 != 0 && (unsigned)(be - 1) > 2044u;
    // 53 bits, the leading one included; a carry moves on into the exponent
    const unsigned long long r = (((unsigned long long)(mh >> 11) << 32) | __funnelshift_r(ml, mh, 11)) + ((ml >> 10) & 1u);
    const unsigned long long bits = r + ((unsigned long long)(unsigned)(be - 1) << 52);
    const unsigned rh = (unsigned)(bits >> 32) | ((unsigned)(sign >> 32) & 0x80000000u);
    return m0 ? __hiloint2double((int)rh, (int)(unsigned)bits) : 0.0;
}

// The same for any exponents; a NaN or infinity in the panel (marked row exponents) must
// reach the next pivot test as NaN.
__device__ __noinline__ double level_sum_any(int h1, int h2, int l1, int l2, int er, int ec) {
    if (er == kBadExp || ec == kBadExp) return __longlong_as_double(0x7ff8000000000000LL);
    int drop;
    const long long v = level_int(h1, h2, l1, l2, drop);
    return ldexp((double)v, max(-2000, min(2000, er + ec - 63 + drop)));
}

// Four products of a row (exponent er) with four columns from their level pairs; marked:
// one of the exponents is kBadExp.
__device__ __forceinline__ void level_row(const int (&h1)[4], const int (&h2)[4], const int (&l1)[4],
                                          const int (&l2)[4], int er, const int (&ec)[4], bool marked, double (&t)[4]) {
    bool extreme = marked;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        int drop;
        const long long v = level_int(h1[c], h2[c], l1[c], l2[c], drop);
        t[c] = level_sum(v, er + ec[c] - 63 + drop, extreme);
    }
    if (extreme) {
#pragma unroll
        for (int c = 0; c < 4; ++c) t[c] = level_sum_any(h1[c], h2[c], l1[c], l2[c], er, ec[c]);
    }
}

// kFirst, kRest: A_ij -= A_ik A_jk^T over the trailing lower tiles (SYRK/GEMM);
// kPanel: A_ik := A_ik L_kk^{-T} for the panel tiles i > k (TRSM as a
// product with the inverse diagonal tile, whose slices sit in the plane rows
// of tile k), written instead of subtracted.
// The SYRK form runs in two launches: column tile j = k + 1 (kFirst), which the next
// panel's factorisation waits for, and the columns beyond.
enum OzPart { kFirst, kRest, kPanel };

template <OzPart kPart>
__global__ void __launch_bounds__(kOzThreads, 1) oz_gemm_kernel(double* A, int nt, int k, const uint8_t* S,
                                                               size_t plane_bytes, const int* E, int* err,
                                                               int tiles_per_block, int nwork) {
    constexpr bool kTrsm = kPart == kPanel;
    extern __shared__ __align__(1024) uint8_t oz_smem[];
    // slices in shared memory, accumulators complete, accumulators read
    __shared__ __align__(8) uint64_t bar_load, bar_mma, bar_read;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int rem = nt - k - 1;
    const int64_t ld = (int64_t)nt * T, rows_pad = ld + T;
    uint8_t* sA = oz_smem;
    uint8_t* sB = oz_smem + kSlices * kPlaneA;
    // work item w = (block z, super-tile): row tiles i0 = k + 1 + 2u, i0 + 1 and
    // column tile j = k + 1 + jj <= i0 + 1 (SYRK) or j = k (TRSM).  Contiguous items per
    // CTA: neighbours share the row slab (SYRK) or the column tile (TRSM), which then
    // stays in shared memory, and each follows from the one before.
    const int w0 = (int)((int64_t)nwork * blockIdx.x / gridDim.x);
    const int w1 = (int)((int64_t)nwork * (blockIdx.x + 1) / gridDim.x);
    struct Item {
        int z, i0, j;
    };
    auto first_item = [&](int w) {
        const int z = w / tiles_per_block;
        int u = 0, jj = w - z * tiles_per_block;
        if constexpr (kPart == kRest) {
            while (true) {
                const int nc = min(2 * u + 2, rem) - 1;
                if (jj < nc) break;
                jj -= nc;
                ++u;
            }
            ++jj;
        } else {
            u = jj;
            jj = kTrsm ? -1 : 0;
        }
        return Item{z, k + 1 + 2 * u, k + 1 + jj};
    };
    auto next_item = [&](Item t) {
        if constexpr (kPart == kRest) {
            // columns of the row pair: up to its own diagonal (or the last tile)
            if (t.j < min(t.i0 + 1, nt - 1)) return Item{t.z, t.i0, t.j + 1};
            t.j = k + 2;
        }
        t.i0 += 2;
        if (t.i0 >= nt) {
            t.i0 = k + 1;
            ++t.z;
        }
        return t;
    };
    auto issue_loads = [&](Item t, Item prev, bool first) {
        const bool la = first || t.z != prev.z || t.i0 != prev.i0, lb = first || t.z != prev.z || t.j != prev.j;
        const uint8_t* Sz = S + (size_t)t.z * kSlices * plane_bytes;
        mbar_expect_tx(&bar_load, kSlices * ((la ? kPlaneA : 0u) + (lb ? kPlaneB : 0u)));
        if (la)
            for (int p = 0; p < kSlices; ++p)
                bulk_g2s(sA + p * kPlaneA, Sz + (size_t)p * plane_bytes + (size_t)t.i0 * T * kRowBytes, kPlaneA,
                         &bar_load);
        if (lb)
            for (int q = 0; q < kSlices; ++q)
                bulk_g2s(sB + q * kPlaneB, Sz + (size_t)q * plane_bytes + (size_t)t.j * T * kRowBytes, kPlaneB,
                         &bar_load);
    };

    if (tid == 0) {
        mbar_init(&bar_load, 1);
        mbar_init(&bar_mma, 1);
        mbar_init(&bar_read, kEpiWarps);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kEpiWarps) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp == kEpiWarps) {
        // ------------------------------------------------- copy and MMA issuer
        // (whole warp in the loop, warp-uniform descriptors, one elected lane issues)
        constexpr uint32_t idesc = instr_desc(1, kSlabRows, T);  // BF16 x BF16 -> F32, 128 x 64
        const bool leader = elect_one();
        const uint64_t a0 = smem_desc(smem_u32(sA), 128, 1024), b0 = smem_desc(smem_u32(sB), 128, 1024);
        Item item = {}, next = {};
        if (w0 < w1) item = first_item(w0);
        if (leader && w0 < w1) issue_loads(item, item, true);
        __syncwarp();
        bool ok = true;
        int it = 0;
        for (int w = w0; w < w1 && ok; ++w, ++it) {
            ok = mbar_wait(&bar_load, (uint32_t)(it & 1), &s_abort, err) &&
                 (it == 0 || mbar_wait(&bar_read, (uint32_t)((it - 1) & 1), &s_abort, err));
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int L = 2; L <= kSlices + 1; ++L)
#pragma unroll
                    for (int p = 1; p < L; ++p)  // level L <= 9: slices p and L - p, both <= 8
#pragma unroll
                        for (int ks = 0; ks < T / 16; ++ks)
                            mma_ss(tmem + 64u * (uint32_t)(L - 2), a0 + (uint64_t)(((p - 1) * kPlaneA) / 16 + ks * 16),
                                   b0 + (uint64_t)(((L - p - 1) * kPlaneB) / 16 + ks * 16), idesc,
                                   p > 1 || ks > 0 ? 1u : 0u);
                tc_commit(&bar_mma);
            }
            __syncwarp();
            if (w + 1 < w1) {
                next = next_item(item);
                // the MMAs have consumed the slices: fetch the next item's
                ok = __all_sync(0xffffffffu, mbar_wait(&bar_mma, (uint32_t)(it & 1), &s_abort, err));
                if (ok && leader) issue_loads(next, item, false);
                item = next;
                __syncwarp();
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // warp v owns tensor-memory lanes (rows) 32 (v % 4) .. + 31 and columns
        // 16 (v / 4) .. + 15 of the super-tile.  The accumulators are read in the 16 x 256
        // bit form: a thread gets columns 2 (lane % 4), + 1 of two blocks of eight for rows
        // lane / 4 + 8 rr, so that a load or store of the matrix takes 64 bytes of eight
        // rows; with a row per lane it was 16 bytes of 32 rows, and the address path of
        // these accesses alone took 8000 clocks per item.
        const int rl = 32 * (warp & 3) + (lane >> 2), cl = 16 * (warp >> 2) + 2 * (lane & 3);
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16, col_base = 16u * (uint32_t)(warp >> 2);
        int it = 0;
        Item item = {};
        if (w0 < w1) item = first_item(w0);
        for (int w = w0; w < w1; ++w, ++it) {
            const int z = item.z, i0 = item.i0, j = item.j;
            item = next_item(item);
            const int64_t r = (int64_t)i0 * T + rl;
            const int rtile = i0 + (warp & 3) / 2;  // of the warp's 32 rows
            const bool mine = rtile < nt && (kTrsm || j <= rtile);
            int er[4], ec[4];
#pragma unroll
            for (int rr = 0; rr < 4; ++rr) er[rr] = mine ? E[(int64_t)z * rows_pad + r + 8 * rr] : 0;
#pragma unroll
            for (int cb = 0; cb < 2; ++cb) {
                const int2 e2 = *reinterpret_cast<const int2*>(E + (int64_t)z * rows_pad + (int64_t)j * T + cl + 8 * cb);
                ec[2 * cb] = e2.x;
                ec[2 * cb + 1] = e2.y;
            }
            // (the slices of a non-finite row are zero, so its mark is the only sign)
            bool marked = false;
#pragma unroll
            for (int t = 0; t < 4; ++t) marked |= er[t] == kBadExp || ec[t] == kBadExp;
            double* C0 = A + (int64_t)z * ld * ld + r * ld + (int64_t)j * T + cl;
            auto entry = [&](int rr, int cb) { return reinterpret_cast<double2*>(C0 + (int64_t)(8 * rr) * ld + 8 * cb); };
            // half of the entries to update are on their way before the MMAs are waited for
            double2 cv[2][2];  // two rows at a time
            if (!kTrsm && mine) {
#pragma unroll
                for (int rr = 0; rr < 2; ++rr) {
                    cv[rr][0] = *entry(rr, 0);
                    cv[rr][1] = *entry(rr, 1);
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(entry(rr + 2, 0)));
                }
            }
            if (!__all_sync(0xffffffffu, mbar_wait(&bar_mma, (uint32_t)(it & 1), &s_abort, err))) break;
            tc_fence_after();
            // pairs of levels as exact 32-bit integers, acc_L 2^7 + acc_{L+1} (below 2^29):
            // q[pair][rr][2 cb + e]
            int q[4][4][4];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {  // rows 16 hh .. + 15 of the warp's
#pragma unroll
                for (int pr = 0; pr < 4; ++pr) {
                    uint32_t va[8], vb[8];
                    const uint32_t at = tmem + lane_base + ((uint32_t)(16 * hh) << 16) + 128u * (uint32_t)pr + col_base;
                    tmem_ld_16x256b_x2(at, va);
                    tmem_ld_16x256b_x2(at + 64u, vb);
                    tmem_wait_ld();
                    // exact conversion of an FP32 integer below 2^22: its bits after adding
                    // 1.5 * 2^23 are the integer plus those of the constant
                    constexpr float kMagicF = 12582912.0f;
                    constexpr unsigned kMagicBits = 0x4b400000u;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {  // register c: column block c / 4, row c / 2 % 2, column c % 2
                        const unsigned ba = __float_as_uint(__uint_as_float(va[c]) + kMagicF);
                        const unsigned bb = __float_as_uint(__uint_as_float(vb[c]) + kMagicF);
                        q[pr][2 * hh + (c >> 1 & 1)][2 * (c >> 2) + (c & 1)] = (int)(ba * 128u + bb - 129u * kMagicBits);
                    }
                }
            }
            // every accumulator has been read: the next item's MMAs may overwrite them
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_read);
            if (!mine) continue;  // (warp-uniform)
#pragma unroll
            for (int rr = 0; rr < 4; ++rr) {
                double t[4];
                level_row(q[0][rr], q[1][rr], q[2][rr], q[3][rr], er[rr], ec, marked, t);
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) {
                    double2 o = make_double2(t[2 * cb], t[2 * cb + 1]);
                    if constexpr (!kTrsm) o = make_double2(cv[rr & 1][cb].x - o.x, cv[rr & 1][cb].y - o.y);
                    *entry(rr, cb) = o;
                }
                if constexpr (!kTrsm) {
                    if (rr < 2) {
                        cv[rr][0] = *entry(rr + 2, 0);
                        cv[rr][1] = *entry(rr + 2, 1);
                    }
                }
            }
        }
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kEpiWarps) {
        if (s_abort) {
            // a wait gave up: let copies and MMAs still in flight land first
            const long long t0 = clock64();
            while (clock64() - t0 < 4000000LL) {
            }
        }
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// persistent grid: one CTA per SM (the slice planes fill shared memory)
int sm_count() {
    static int sms = 0;
    if (sms <= 0) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            sms = v;
        else
            sms = 148;
        cudaGetLastError();
    }
    return sms;
}

}  // namespace

size_t oz_plane_bytes(int nt) { return (size_t)((int64_t)nt * T + T) * kRowBytes; }
size_t oz_slice_bytes(int nt) { return kSlices * oz_plane_bytes(nt); }
size_t oz_expo_ints(int nt) { return (size_t)((int64_t)nt * T + T); }

cudaError_t launch_oz_update_first(double* A, int nt, int k, int g, uint8_t* S, int* E, int* err, cudaStream_t st,
                                   int64_t* launches) {
    const int rem = nt - k - 1;
    if (rem <= 0) return cudaSuccess;
    static_assert(kOzSmem + 1024 <= 227 * 1024, "shared memory");
    cudaError_t e =
        cudaFuncSetAttribute(oz_gemm_kernel<kFirst>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmem);
    if (e != cudaSuccess) return e;
    const size_t pb = oz_plane_bytes(nt);
    const int64_t ld = (int64_t)nt * T;
    const int64_t rows = (int64_t)rem * T;
    oz_slice_kernel<<<dim3((unsigned)((rows + 31) / 32), (unsigned)g), 256, 0, st>>>(
        A + (int64_t)(k + 1) * T * ld + (int64_t)k * T, ld * ld, ld, rows, (int64_t)(k + 1) * T, ld + T, pb, S, E);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int tiles = (rem + 1) / 2, nwork = tiles * g;
    oz_gemm_kernel<kFirst><<<(unsigned)std::min(nwork, sm_count()), kOzThreads, kOzSmem, st>>>(A, nt, k, S, pb, E, err,
                                                                                             tiles, nwork);
    if (launches) *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_oz_update_rest(double* A, int nt, int k, int g, uint8_t* S, int* E, int* err, int ctas,
                                  cudaStream_t st, int64_t* launches) {
    const int rem = nt - k - 1;
    int tiles = 0;
    for (int u = 0; 2 * u < rem; ++u) tiles += std::min(2 * u + 2, rem) - 1;
    if (tiles <= 0) return cudaSuccess;
    cudaError_t e =
        cudaFuncSetAttribute(oz_gemm_kernel<kRest>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmem);
    if (e != cudaSuccess) return e;
    const int nwork = tiles * g;
    oz_gemm_kernel<kRest><<<(unsigned)std::min(nwork, ctas > 0 ? ctas : sm_count()), kOzThreads, kOzSmem, st>>>(
        A, nt, k, S, oz_plane_bytes(nt), E, err, tiles, nwork);
    if (launches) *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_oz_trsm(double* A, const double* Dinv, int nt, int k, int g, uint8_t* S, int* E, int* err,
                           cudaStream_t st, int64_t* launches) {
    const int rem = nt - k - 1;
    if (rem <= 0) return cudaSuccess;
    cudaError_t e =
        cudaFuncSetAttribute(oz_gemm_kernel<kPanel>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmem);
    if (e != cudaSuccess) return e;
    const size_t pb = oz_plane_bytes(nt);
    const int64_t ld = (int64_t)nt * T;
    const int64_t rows = (int64_t)rem * T;
    // the panel below the diagonal tile, and L_kk^{-1} into the plane rows of tile k
    oz_slice_kernel<<<dim3((unsigned)((rows + 31) / 32), (unsigned)g), 256, 0, st>>>(
        A + (int64_t)(k + 1) * T * ld + (int64_t)k * T, ld * ld, ld, rows, (int64_t)(k + 1) * T, ld + T, pb, S, E);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    oz_slice_kernel<<<dim3(T / 32, (unsigned)g), 256, 0, st>>>(Dinv + (int64_t)k * T * T, (int64_t)nt * T * T, T,
                                                                T, (int64_t)k * T, ld + T, pb, S, E);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int tiles = (rem + 1) / 2, nwork = tiles * g;
    oz_gemm_kernel<kPanel><<<(unsigned)std::min(nwork, sm_count()), kOzThreads, kOzSmem, st>>>(A, nt, k, S, pb, E, err,
                                                                                           tiles, nwork);
    if (launches) *launches += 3;
    return cudaGetLastError();
}

}  // namespace ap
