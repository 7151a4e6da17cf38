// FP32 SIMT form of the fused kernel-matrix product (the AP residual update,
// Eq. text_update_of_r, the residual recompute of the App. B lemma and the
// posterior mean of Sec. 2), with the block-norm / Gauss-Southwell epilogue of
// Eq. approximate_gauss_southwell fused in.  Up to 4 right-hand sides always, more for
// products too small for the tensor cores to pay (kX3MinEntries16 / 32; kmv_x3.cuh).
//
// Work decomposition
//   grid.x = row tiles of ROWS = 128 * RM rows; a tile never straddles an AP
//            block, so its squared norm belongs to exactly one block;
//   grid.y = S column splits, one thread-block cluster per row tile; the S
//            partial products are summed through distributed shared memory in
//            a fixed rank order (deterministic, no atomics on R);
//   grid.z = G groups of S column splits when the row tiles are too few to fill
//            the chip or its last wave: each cluster leaves its sums in global
//            memory, and the group that arrives last at the tile's ticket adds
//            them in group order (kmv_split chooses rm, S and G).
// Each thread keeps RM rows of the scaled inputs and RM x C accumulators in
// registers; the block's columns (scaled inputs and the C right-hand sides of
// Delta) are staged through shared memory and read as warp broadcasts.  The
// n x b kernel block is never stored.
#pragma once

#include <cooperative_groups.h>

#include "ap_internal.cuh"

namespace ap {
namespace cg = cooperative_groups;

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// phi as a function of t = |x_s - x_s'|^2 of the pre-scaled inputs.
template <int KERN>
__device__ __forceinline__ float phi_fp32(float t) {
    if constexpr (KERN == AP_RBF) {
        return ex2_approx(-t);
    } else if constexpr (KERN == AP_MATERN32) {
        float u = sqrt_approx(t);
        return (1.0f + u) * ex2_approx(-u * kLog2e);
    } else {
        float u = sqrt_approx(t);
        return fmaf(u, fmaf(u, 1.0f / 3.0f, 1.0f), 1.0f) * ex2_approx(-u * kLog2e);
    }
}

// SplitMix64 (Steele, Lea, Flood 2014; Vigna's reference constants) of
// (seed, counter): the counter-based stream behind AP_SEL_RANDOM.
__host__ __device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t idx) {
    uint64_t z = seed + (idx + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ int random_block(uint64_t seed, int64_t step, int m) {
    uint64_t z = splitmix64_at(seed, (uint64_t)step);
    return (int)(((z >> 32) * (uint64_t)m) >> 32);
}

// Sum of one double over the CTA; the result is valid in thread 0.
__device__ __forceinline__ double cta_sum_d(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < nw; ++i) r += red[i];
    return r;
}

// Executed by every thread of the CTA that finished last (ticket order):
// reduce the per-tile partials in a fixed order, pick the next block, publish
// the column norms, and leave the ticket at zero for the next launch.
//
// This runs alone on the chip at the end of every step, so it is bound by the
// latency of its loads: the partials of a block (and of a column) are shared out
// over as many threads as the CTA has for it.  With one thread per block and per
// column, the last step of an epoch of a 4096-row solve spent some 20 us in the
// column sums alone.  s_buf: 16 C doubles when the CTA has more than 128 threads,
// 128 otherwise.
template <int C>
__device__ void epi_finalize(const EpiParams& e, double* red_d, int* red_i, double* s_buf) {
    const int tid = threadIdx.x, nth = blockDim.x;
    if (e.flags & kEpiBlockNorms) {
        double best = -1.0;
        int bi = 0x7fffffff;
        int bad = 0;
        const int64_t per = e.tiles_per_seg * e.S;
        // L consecutive lanes per block; whole warps go round together
        int L = 1;
        while (L < 32 && 2 * L * e.m <= nth) L *= 2;
        const int lane = tid % L, stride = nth / L;
        for (int J0 = 0; J0 < e.m; J0 += stride) {
            const int J = J0 + tid / L;
            double acc = 0.0;
            if (J < e.m && tid / L < stride) {
                const double* src = e.part_norm + (int64_t)J * per;
#pragma unroll 8
                for (int64_t t = lane; t < per; t += L) acc += __ldcg(src + t);
            }
            for (int o = L / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (J < e.m && tid / L < stride && AP_CHK((int64_t)(J + 1) * per <= e.ntiles * e.S)) {
                if (lane == 0) e.norms_out[J] = acc;
                if (!isfinite(acc)) bad = 1;
                if (acc > best) { best = acc; bi = J; }
            }
        }
        // argmax over the CTA, ties to the smallest block index
        for (int o = 16; o > 0; o >>= 1) {
            double ov = __shfl_down_sync(0xffffffffu, best, o);
            int oi = __shfl_down_sync(0xffffffffu, bi, o);
            if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
        }
        bad = __syncthreads_or(bad);
        const int w = tid >> 5, nw = nth >> 5;
        if ((tid & 31) == 0) { red_d[w] = best; red_i[w] = bi; }
        __syncthreads();
        if (tid == 0) {
            best = red_d[0];
            bi = red_i[0];
            for (int i = 1; i < nw; ++i)
                if (red_d[i] > best || (red_d[i] == best && red_i[i] < bi)) { best = red_d[i]; bi = red_i[i]; }
            int64_t step = *e.step_ctr + (e.advance ? 1 : 0);
            int next;
            if (e.select == AP_SEL_CYCLIC) next = (int)(step % e.m);
            else if (e.select == AP_SEL_RANDOM) next = random_block(e.seed, step, e.m);
            else next = (bi >= 0 && bi < e.m) ? bi : 0;
            *e.sel_out = next;
            *e.step_ctr = step;
            if (bad) *e.nan_flag = 1;
        }
        __syncthreads();
    }
    if (e.flags & kEpiColNorms) {
        // thread t sums column t % C over the tiles t / C, t / C + groups, ...
        const int64_t tot = e.ntiles * e.S;
        const int nwu = min(nth >> 5, 16), nthu = 32 * nwu;
        double acc = 0.0;
        if (tid < nthu) {
#pragma unroll 8
            for (int64_t t = tid / C; t < tot; t += nthu / C) acc += __ldcg(e.part_col + t * C + tid % C);
        }
        for (int o = 16; o >= C; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        __syncthreads();
        if (tid < nthu && (tid & 31) < C) s_buf[(tid >> 5) * C + (tid & 31)] = acc;
        __syncthreads();
        if (tid < C) {
            acc = 0.0;
            for (int w = 0; w < nwu; ++w) acc += s_buf[w * C + tid];
            e.colnorm_out[tid] = acc;
            if (!isfinite(acc)) *e.nan_flag = 1;
        }
    }
    if (tid == 0) *e.ticket = 0u;
}

// Phase 2 of every product: reduce the S rank partials of this CTA's share of
// rows (fixed rank order), add the base, store, and write the norm partials.
// With G > 1 column groups the sums go to the tile's slots first, and only the
// group that arrives last (returns true) goes on with the slots' sums, added in
// group order.
template <int C, int ROWS>
__device__ __forceinline__ bool epi_store(const KmvParams& p, float* s_part, int S, int rank,
                                          int64_t r0, int64_t r1, int64_t part_idx, double* red_d,
                                          double* s_col, int* s_last) {
    const int tid = threadIdx.x;
    const int rpr = ROWS / S;  // rows reduced by this rank
    const int G = gridDim.z;
    double sq = 0.0, colacc = 0.0;
    auto cluster_sum = [&](int t) {
        const int lc = (rank * rpr + t / C) * C + t % C;
        if (S == 1) return s_part[lc];
        // (all remote loads in flight before the first is added)
        cg::cluster_group cluster = cg::this_cluster();
        float v[kMaxSplit], sum = 0.0f;
#pragma unroll
        for (int src = 0; src < kMaxSplit; ++src) v[src] = src < S ? cluster.map_shared_rank(s_part, src)[lc] : 0.0f;
#pragma unroll
        for (int src = 0; src < kMaxSplit; ++src) sum += v[src];
        return sum;
    };
    // slot of group g: this rank's rpr x C sums of the tile
    float* slots = G > 1 ? p.gscr + (int64_t)blockIdx.x * G * ROWS * C + (int64_t)rank * rpr * C : nullptr;
    if (G > 1) {
        for (int t = tid; t < rpr * C; t += kKmvThreads)
            __stcg(slots + (int64_t)blockIdx.z * ROWS * C + t, cluster_sum(t));
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            unsigned int* tick = p.gtick + (int64_t)blockIdx.x * S + rank;
            *s_last = atomicAdd(tick, 1u) == (unsigned)(G - 1) ? 1 : 0;
            if (*s_last) *tick = 0u;
        }
        __syncthreads();
        if (!*s_last) return false;
        __threadfence();
    }
    auto put = [&](int t, float sum) {
        const int lr = rank * rpr + t / C;
        const int c = t % C;  // == tid % C since kKmvThreads % C == 0
        const int64_t i = r0 + lr;
        if (i < r1 && AP_CHK(i < p.na)) {
            const float bv = p.base ? p.base[i * C + c] : p.base_const;
            const float o = fmaf(p.sgn, sum, bv);
            p.out[i * C + c] = o;
            const double od = (double)o;
            sq += od * od;
            colacc += od * od;
        }
    };
    if (G == 1) {
#pragma unroll 4
        for (int t = tid; t < rpr * C; t += kKmvThreads) put(t, cluster_sum(t));
    } else {
        for (int t = tid; t < rpr * C; t += kKmvThreads) {
            float sum = 0.0f;
#pragma unroll 8
            for (int g = 0; g < G; ++g) sum += __ldcg(slots + (int64_t)g * ROWS * C + t);
            put(t, sum);
        }
    }
    const EpiParams& e = p.epi;
    if (e.flags & kEpiBlockNorms) {
        double tot = cta_sum_d(sq, red_d);
        if (tid == 0 && AP_CHK(part_idx < e.ntiles * e.S)) e.part_norm[part_idx] = tot;
    }
    if (e.flags & kEpiColNorms) {
        __syncthreads();
        s_col[tid] = colacc;
        __syncthreads();
        if (tid < C) {
            double acc = 0.0;
            for (int k = tid; k < kKmvThreads; k += C) acc += s_col[k];
            if (AP_CHK(part_idx < e.ntiles * e.S)) e.part_col[part_idx * C + tid] = acc;
        }
    }
    return true;
}

template <int C>
__device__ __forceinline__ void epi_ticket(const EpiParams& e, double* red_d, int* red_i,
                                           int* s_last, double* s_buf) {
    if (e.flags == 0) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned total = (unsigned)(e.ntiles * e.S);
        *s_last = (atomicAdd(e.ticket, 1u) == total - 1u) ? 1 : 0;
    }
    __syncthreads();
    if (*s_last) {
        __threadfence();
        epi_finalize<C>(e, red_d, red_i, s_buf);
    }
}

// The distance and (for C > 1) the contraction run as packed FP32 pairs
// (fma.rn.f32x2: one instruction for two lanes, each rounded as the scalar
// operation): the squared distance over pairs of coordinates (two partial sums,
// added at the end), the contraction over pairs of right-hand sides.  The FMA pipe
// does the same work either way; the issue slots saved are what the SFU and
// shared-memory instructions need.
template <int D, int C, int RM>
constexpr size_t kmv_smem_floats() {
    return (size_t)kKmvTN * (D + C) + (size_t)kKmvThreads * RM * C;
}

template <int KERN, int D, int C, int RM>
__global__ void __launch_bounds__(kKmvThreads, 4) kmv_fp32_kernel(const KmvParams p) {
    constexpr int ROWS = kKmvThreads * RM;
    extern __shared__ float4 kmv_smem4[];
    float* s_xb = reinterpret_cast<float*>(kmv_smem4);  // kKmvTN * D
    float* s_v = s_xb + kKmvTN * D;                     // kKmvTN * C
    float* s_part = s_v + kKmvTN * C;                   // ROWS * C
    __shared__ double red_d[32];
    __shared__ int red_i[32];
    __shared__ double s_col[kKmvThreads];
    __shared__ int s_last;

    const int tid = threadIdx.x;
    const int S = gridDim.y;
    const int rank = blockIdx.y;
    const EpiParams& e = p.epi;
    const int64_t tile = blockIdx.x;
    const int64_t segi = tile / e.tiles_per_seg;
    const int64_t seg_lo = segi * e.seg;
    const int64_t seg_hi = min(seg_lo + e.seg, p.na);
    const int64_t r0 = seg_lo + (tile % e.tiles_per_seg) * ROWS;
    const int64_t r1 = min(r0 + (int64_t)ROWS, seg_hi);

    int64_t col0 = p.col0, ncols = p.ncols;
    if (p.sel) {
        col0 = (int64_t)(*p.sel) * p.blk;
        ncols = min(p.blk, p.nb - col0);
    }
    const int nsplit = S * gridDim.z, split = (int)blockIdx.z * S + rank;
    const int64_t cs = ((ncols + nsplit - 1) / nsplit + 15) / 16 * 16;
    const int64_t c_lo = col0 + split * cs;
    const int64_t c_hi = min(col0 + ncols, c_lo + cs);

    float xa[RM][D];
#pragma unroll
    for (int q = 0; q < RM; ++q) {
        const int64_t i = r0 + tid + q * kKmvThreads;
#pragma unroll
        for (int k4 = 0; k4 < D / 4; ++k4) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < r1 && AP_CHK(i < p.na)) v = reinterpret_cast<const float4*>(p.Xa + i * D)[k4];
            xa[q][4 * k4 + 0] = v.x;
            xa[q][4 * k4 + 1] = v.y;
            xa[q][4 * k4 + 2] = v.z;
            xa[q][4 * k4 + 3] = v.w;
        }
    }
    pdl_wait();  // V and base (the block index was complete before the block solve began)
    pdl_launch();
    float2 xa2[RM][D / 2], acc2[RM][(C + 1) / 2];
#pragma unroll
    for (int q = 0; q < RM; ++q) {
#pragma unroll
        for (int k = 0; k < D / 2; ++k) xa2[q][k] = make_float2(xa[q][2 * k], xa[q][2 * k + 1]);
#pragma unroll
        for (int c = 0; c < (C + 1) / 2; ++c) acc2[q][c] = make_float2(0.0f, 0.0f);
    }
    const float2 m1 = make_float2(-1.0f, -1.0f);
    for (int64_t cb = c_lo; cb < c_hi; cb += kKmvTN) {
        const int cnt = (int)min((int64_t)kKmvTN, c_hi - cb);
        __syncthreads();
        if (AP_CHK(cb >= 0 && cb + cnt <= p.nb) && AP_CHK(cb - col0 >= 0 && cb - col0 + cnt <= ncols)) {
            const float4* gx = reinterpret_cast<const float4*>(p.Xb + cb * D);
            float4* sx = reinterpret_cast<float4*>(s_xb);
            for (int t = tid; t < cnt * D / 4; t += kKmvThreads) sx[t] = __ldg(gx + t);
            const float* gv = p.V + (cb - col0) * C;
            if constexpr (C % 4 == 0) {
                const float4* gv4 = reinterpret_cast<const float4*>(gv);
                float4* sv4 = reinterpret_cast<float4*>(s_v);
                for (int t = tid; t < cnt * C / 4; t += kKmvThreads) sv4[t] = __ldg(gv4 + t);
            } else {
                for (int t = tid; t < cnt * C; t += kKmvThreads) s_v[t] = __ldg(gv + t);
            }
        }
        __syncthreads();
#pragma unroll 2
        for (int jj = 0; jj < cnt; ++jj) {
            float2 xb2[D / 2];
#pragma unroll
            for (int k4 = 0; k4 < D / 4; ++k4) {
                const float4 v = reinterpret_cast<const float4*>(s_xb + jj * D)[k4];
                xb2[2 * k4] = make_float2(v.x, v.y);
                xb2[2 * k4 + 1] = make_float2(v.z, v.w);
            }
            float kv[RM];
#pragma unroll
            for (int q = 0; q < RM; ++q) {
                float2 tp = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int k = 0; k < D / 2; ++k) {
                    const float2 df = __ffma2_rn(xb2[k], m1, xa2[q][k]);  // xa - xb, exact negation
                    tp = __ffma2_rn(df, df, tp);
                }
                kv[q] = phi_fp32<KERN>(tp.x + tp.y);
            }
            if constexpr (C % 4 == 0) {
#pragma unroll
                for (int c4 = 0; c4 < C / 4; ++c4) {
                    const float4 v = reinterpret_cast<const float4*>(s_v + jj * C)[c4];
#pragma unroll
                    for (int q = 0; q < RM; ++q) {
                        const float2 kd = make_float2(kv[q], kv[q]);
                        acc2[q][2 * c4] = __ffma2_rn(kd, make_float2(v.x, v.y), acc2[q][2 * c4]);
                        acc2[q][2 * c4 + 1] = __ffma2_rn(kd, make_float2(v.z, v.w), acc2[q][2 * c4 + 1]);
                    }
                }
            } else {
                static_assert(C % 4 == 0 || C == 1, "one right-hand side, or quads of them");
                const float v = s_v[jj];
#pragma unroll
                for (int q = 0; q < RM; ++q) acc2[q][0].x = fmaf(kv[q], v, acc2[q][0].x);
            }
        }
    }
    float acc[RM][C];
#pragma unroll
    for (int q = 0; q < RM; ++q)
#pragma unroll
        for (int c = 0; c < C; ++c) acc[q][c] = c % 2 ? acc2[q][c / 2].y : acc2[q][c / 2].x;
    // scale by s, add sigma^2 V_i on the index diagonal, park in shared memory
    __syncthreads();
#pragma unroll
    for (int q = 0; q < RM; ++q) {
        const int lr = tid + q * kKmvThreads;
        const int64_t i = r0 + lr;
        const bool diag = p.noise_diag && i >= c_lo && i < c_hi;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            float v = p.s * acc[q][c];
            if (diag && AP_CHK(i - col0 >= 0 && i - col0 < ncols)) v = fmaf(p.noise, __ldg(p.V + (i - col0) * C + c), v);
            s_part[lr * C + c] = v;
        }
    }
    if (S > 1) cg::this_cluster().sync();
    else __syncthreads();
    const bool done = epi_store<C, ROWS>(p, s_part, S, rank, r0, r1, tile * S + rank, red_d, s_col, &s_last);
    if (S > 1) cg::this_cluster().sync();
    if (done) epi_ticket<C>(e, red_d, red_i, &s_last, s_col);
}

// Norms + selection of R alone (before the first step, after a refinement).
template <int C>
__global__ void __launch_bounds__(kKmvThreads) norms_select_kernel(const float* R, int64_t n,
                                                                   const EpiParams e,
                                                                   int64_t tile_rows) {
    __shared__ double red_d[32];
    __shared__ int red_i[32];
    __shared__ double s_col[kKmvThreads];
    __shared__ int s_last;
    const int tid = threadIdx.x;
    const int64_t tile = blockIdx.x;
    const int64_t seg_lo = (tile / e.tiles_per_seg) * e.seg;
    const int64_t seg_hi = min(seg_lo + e.seg, n);
    const int64_t r0 = seg_lo + (tile % e.tiles_per_seg) * tile_rows;
    const int64_t r1 = min(r0 + tile_rows, seg_hi);
    double sq = 0.0, colacc = 0.0;
    for (int64_t t = tid; t < (r1 - r0) * C && AP_CHK(r1 <= n); t += kKmvThreads) {
        const double v = (double)R[r0 * C + t];
        sq += v * v;
        colacc += v * v;
    }
    if (e.flags & kEpiBlockNorms) {
        double tot = cta_sum_d(sq, red_d);
        if (tid == 0 && AP_CHK(tile < e.ntiles)) e.part_norm[tile] = tot;
    }
    if (e.flags & kEpiColNorms) {
        __syncthreads();
        s_col[tid] = colacc;
        __syncthreads();
        if (tid < C) {
            double acc = 0.0;
            for (int k = tid; k < kKmvThreads; k += C) acc += s_col[k];
            if (AP_CHK(tile < e.ntiles)) e.part_col[tile * C + tid] = acc;
        }
    }
    epi_ticket<C>(e, red_d, red_i, &s_last, s_col);
}

inline int rows_per_thread(int D, int C) {
    const int w = D + C;
    return w <= 20 ? 4 : (w <= 36 ? 2 : 1);
}

template <int KERN, int D, int C, int RM>
cudaError_t launch_kmv_rm(const KmvParams& p, cudaStream_t st) {
    const size_t smem = sizeof(float) * kmv_smem_floats<D, C, RM>();
    auto fn = kmv_fp32_kernel<KERN, D, C, RM>;
    if constexpr (sizeof(float) * kmv_smem_floats<D, C, RM>() > 48 * 1024) {
        cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (err != cudaSuccess) return err;
    }
    return launch_dependent(fn, dim3((unsigned)p.epi.ntiles, (unsigned)p.epi.S, (unsigned)p.G), kKmvThreads, smem, st,
                            p.dependent, p, (unsigned)p.epi.S);
}

// rows per thread as kmv_split chose them, at most what (D, C) leaves registers for
template <int KERN, int D, int C>
cudaError_t launch_kmv_inst(const KmvParams& p, cudaStream_t st) {
    constexpr int kMaxRm = (D + C <= 20) ? 4 : ((D + C <= 36) ? 2 : 1);
    if constexpr (kMaxRm >= 4)
        if (p.rm == 4) return launch_kmv_rm<KERN, D, C, 4>(p, st);
    if constexpr (kMaxRm >= 2)
        if (p.rm == 2) return launch_kmv_rm<KERN, D, C, 2>(p, st);
    return p.rm == 1 ? launch_kmv_rm<KERN, D, C, 1>(p, st) : cudaErrorInvalidValue;
}

// (D, C) dispatch for one kernel family.
template <int KERN>
cudaError_t dispatch_kmv(const KmvParams& p, int D, int C, cudaStream_t st) {
#define AP_KMV_C(DD)                                                      \
    switch (C) {                                                          \
        case 1: return launch_kmv_inst<KERN, DD, 1>(p, st);               \
        case 4: return launch_kmv_inst<KERN, DD, 4>(p, st);               \
        case 16: return launch_kmv_inst<KERN, DD, 16>(p, st);             \
        case 32: return launch_kmv_inst<KERN, DD, 32>(p, st);             \
        default: return cudaErrorInvalidValue;                            \
    }
    switch (D) {
        case 4: AP_KMV_C(4)
        case 8: AP_KMV_C(8)
        case 12: AP_KMV_C(12)
        case 16: AP_KMV_C(16)
        case 24: AP_KMV_C(24)
        case 32: AP_KMV_C(32)
        default: return cudaErrorInvalidValue;
    }
#undef AP_KMV_C
}

}  // namespace ap
