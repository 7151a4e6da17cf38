// Block solve of one AP step.
//
// Delta = K_II^{-1} R_I = L^{-T} (L^{-1} R_I) and W_I += Delta (Alg. 1, the
// weight update Eq. text_update_of_w; Table 6: (b^2 + b) l flops).  I is read
// from device memory, where the previous step's epilogue left the
// Gauss-Southwell choice, so a whole epoch runs without a host round trip.
//
// Both triangular products run over the 64 x 64 tiles of the packed FP32
// inverse factor (nt (nt + 1) / 2 tiles, read once per pass).  The tiles are
// split evenly over the CTAs (tpc consecutive tiles each: row-major order for
// Z = L^{-1} R_I, column-major for Delta = L^{-T} Z), so that every CTA reads
// the same number of bytes whatever the row lengths.  A CTA whose range covers
// part of an output row (of tiles) writes its partial sums to a slot of that
// row; the CTA that arrives last at the row's ticket adds the slots in slot
// order (deterministic) and writes the row; a row inside one CTA's range needs
// neither.
//
// Within a CTA the next tile is copied to shared memory while the current one is used,
// and the eight warps share out the summation index: every warp forms all 64 x C
// outputs of a tile over 8 of its 64 terms, a lane owning two output rows of all
// columns, and the warps' sums are added once per output row of tiles.  A lane then
// reads 2 + 16 vectors of shared memory for 128 multiply-adds (16 columns); with a
// lane owning one row and four columns it was one scalar and one vector for four, and
// both passes were bound by instructions (25 and 26 us at b = 4096, c = 16 against 5 us
// for the bytes).  Measured now (GB300): 21 and 24 us, the second one storing Delta's
// operand layout too (4 us as a kernel of its own); b = 512, c = 1 6.0 and 6.2 -> 4.4 and
// 4.9 us.
//
// Programmatic dependent launch: the second pass reads only the factor and the block
// index before its grid-dependency wait, so its first tiles are on their way while the
// first pass finishes.
#include <algorithm>

#include "ap_internal.cuh"

namespace ap {
namespace {

constexpr int T = kTile;
constexpr int kSolveThreads = 256;
constexpr int kSolveWarps = kSolveThreads / 32;
constexpr int kQ = T / kSolveWarps;  // summation indices of a tile per warp

__device__ __forceinline__ int64_t packed_tile(int i, int k) { return (int64_t)i * (i + 1) / 2 + k; }

// Work split shared by host and device: tiles per CTA and partial slots per
// output row.
__host__ __device__ inline int64_t solve_ntri(int nt) { return (int64_t)nt * (nt + 1) / 2; }

// CTAs that fit an SM: by shared memory up to 4 columns, by registers beyond (2 C
// accumulators per thread)
__host__ __device__ constexpr int solve_ctas_per_sm(int C) { return C <= 4 ? 6 : C <= 16 ? 4 : 2; }

// first tile of column k in column-major order of the lower triangle
__host__ __device__ inline int64_t col_start(int nt, int k) { return (int64_t)k * nt - (int64_t)k * (k - 1) / 2; }

// row i of the lower triangle (row-major) that holds tile t
__device__ __forceinline__ int tri_row(int t) {
    int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((int)packed_tile(i + 1, 0) <= t) ++i;
    while ((int)packed_tile(i, 0) > t) --i;
    return i;
}

template <int C>
constexpr int solve_stage_floats() { return T * T + T * C; }
template <int C>
constexpr size_t solve_smem() { return 2 * sizeof(float) * solve_stage_floats<C>(); }

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool live) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(live ? 16 : 0));
}

__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool live) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(live ? 4 : 0));
}

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A tile of the factor into shared memory: row r's 16-byte granule g at granule
// g ^ (r % 16), so that eight lanes reading one granule of eight consecutive rows, or
// any lanes reading along a row, meet no bank twice.
__device__ __forceinline__ int swz(int r, int g) { return r * T + 4 * (g ^ (r & 15)); }

// (thread tid copies granule tid % 16 of rows tid / 16 + 16 j: one swizzle for all j)
__device__ __forceinline__ void fetch_tile(float* sx, const float* tile, int tid) {
    float* dst = sx + swz(tid / (T / 4), tid % (T / 4));
    const float* src = tile + 4 * tid;
#pragma unroll
    for (int j = 0; j < T * T / 4 / kSolveThreads; ++j)
        cp_async16(dst + j * 4 * kSolveThreads, src + j * 4 * kSolveThreads, true);
}

// 64 rows of a matrix with C columns from M, of which `live` exist (the rest read as zero).
template <int C>
__device__ __forceinline__ void fetch_rhs(float* sv, const float* M, int live, int tid) {
    if constexpr (C % 4 == 0) {
#pragma unroll
        for (int t0 = 0; t0 < T * C / 4; t0 += kSolveThreads) {
            const int t = t0 + tid;
            if (T * C / 4 % kSolveThreads == 0 || t < T * C / 4)
                cp_async16(sv + 4 * t, 4 * t / C < live ? M + 4 * t : M, 4 * t / C < live);
        }
    } else {
        if (tid < T * C) cp_async4(sv + tid, tid / C < live ? M + tid : M, tid / C < live);
    }
}

// acc[h][c] += x[h] * sv[q][c] for one summation index q
template <int C>
__device__ __forceinline__ void rank1(float (&acc)[2][C], float x0, float x1, const float* v) {
    if constexpr (C % 4 == 0) {
#pragma unroll
        for (int c = 0; c < C; c += 4) {
            const float4 w = *reinterpret_cast<const float4*>(v + c);
            acc[0][c] = fmaf(x0, w.x, acc[0][c]);
            acc[0][c + 1] = fmaf(x0, w.y, acc[0][c + 1]);
            acc[0][c + 2] = fmaf(x0, w.z, acc[0][c + 2]);
            acc[0][c + 3] = fmaf(x0, w.w, acc[0][c + 3]);
            acc[1][c] = fmaf(x1, w.x, acc[1][c]);
            acc[1][c + 1] = fmaf(x1, w.y, acc[1][c + 1]);
            acc[1][c + 2] = fmaf(x1, w.z, acc[1][c + 2]);
            acc[1][c + 3] = fmaf(x1, w.w, acc[1][c + 3]);
        }
    } else {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            acc[0][c] = fmaf(x0, v[c], acc[0][c]);
            acc[1][c] = fmaf(x1, v[c], acc[1][c]);
        }
    }
}

// The CTA's sums of one output row (of tiles): add the warps' shares through shared
// memory (red, 16 KB that hold nothing needed any more), then either hand each sum to emit(row-in-tile,
// column, value), or, when `nslots` CTAs contribute to the row, write this CTA's slot
// and let the last of them at the row's ticket add the slots in slot order.  rows:
// which two rows of the tile a lane holds.
template <int C, typename Rows, typename F>
__device__ __forceinline__ void flush_row(const SolveParams& p, int row, int slot, int nslots, float* red,
                                          const float (&acc)[2][C], Rows&& rows, int* s_last, F&& emit) {
    constexpr int CH = C < 8 ? C : 8;  // columns per pass: red holds 8 warps x 64 x CH
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float* dst = p.spart + ((int64_t)row * p.maxj + slot) * T * C;
    const bool slot_ok = AP_CHK(slot >= 0 && slot < p.maxj && nslots <= p.maxj && row < p.nt);
#pragma unroll
    for (int c0 = 0; c0 < C; c0 += CH) {
        __syncthreads();  // the tiles in red's place (or the previous pass) are done with
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float* o = red + (warp * T + rows(lane, h)) * CH;
            if constexpr (CH % 4 == 0) {
#pragma unroll
                for (int c = 0; c < CH; c += 4)
                    *reinterpret_cast<float4*>(o + c) =
                        make_float4(acc[h][c0 + c], acc[h][c0 + c + 1], acc[h][c0 + c + 2], acc[h][c0 + c + 3]);
            } else {
#pragma unroll
                for (int c = 0; c < CH; ++c) o[c] = acc[h][c0 + c];
            }
        }
        __syncthreads();
        for (int t = tid; t < T * CH; t += kSolveThreads) {
            float sum = 0.0f;
#pragma unroll
            for (int w = 0; w < kSolveWarps; ++w) sum += red[w * T * CH + t];
            if (nslots == 1) emit(t / CH, c0 + t % CH, sum);
            else if (slot_ok) __stcg(dst + (t / CH) * C + c0 + t % CH, sum);
        }
    }
    if (nslots == 1) {
        __syncthreads();
        return;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) *s_last = (atomicAdd(p.sticket + row, 1u) == (unsigned)(nslots - 1)) ? 1 : 0;
    __syncthreads();
    if (*s_last) {
        __threadfence();
        const float* src = p.spart + (int64_t)row * p.maxj * T * C;
        // slots in order, several of them and up to four sums per thread at a time, with all
        // their loads in flight: a row of a short block has a slot per tile, and one sum at
        // a time made the last CTA wait for memory C / 4 times over
        constexpr int E = (T * C + kSolveThreads - 1) / kSolveThreads, EB = E < 4 ? E : 4, SB = C == 16 ? 4 : 8;
#pragma unroll 1
        for (int e0 = 0; e0 < E; e0 += EB) {
            float sum[EB];
#pragma unroll
            for (int x = 0; x < EB; ++x) sum[x] = 0.0f;
            const int t0 = tid + e0 * kSolveThreads;
#pragma unroll 1
            for (int j0 = 0; j0 < nslots; j0 += SB) {
                float v[SB][EB];
#pragma unroll
                for (int jj = 0; jj < SB; ++jj)
#pragma unroll
                    for (int x = 0; x < EB; ++x)
                        v[jj][x] = j0 + jj < nslots && (T * C % kSolveThreads == 0 || t0 < T * C)
                                       ? __ldcg(src + (int64_t)(j0 + jj) * T * C + t0 + x * kSolveThreads)
                                       : 0.0f;
#pragma unroll
                for (int jj = 0; jj < SB; ++jj)
#pragma unroll
                    for (int x = 0; x < EB; ++x) sum[x] += v[jj][x];
            }
#pragma unroll
            for (int x = 0; x < EB; ++x) {
                const int t = t0 + x * kSolveThreads;
                if (T * C % kSolveThreads == 0 || t < T * C) emit(t / C, t % C, sum[x]);
            }
        }
        if (tid == 0) p.sticket[row] = 0u;
    }
    __syncthreads();
}

// pass 1: Z_i = sum_{k <= i} X_ik R_I[k]  (X = L^{-1}), tiles in row-major order
template <int C>
__global__ void __launch_bounds__(kSolveThreads, solve_ctas_per_sm(C)) solve_lower_kernel(const SolveParams p) {
    extern __shared__ float4 bs_smem4[];
    float* stage = reinterpret_cast<float*>(bs_smem4);
    __shared__ int s_last;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_wait();  // the block index and R come from the update before
    pdl_launch();
    const int I = *p.sel;
    const int64_t lo = (int64_t)I * p.b;
    if (!AP_CHK(I >= 0 && lo < p.n)) return;
    const int64_t bI = min(p.b, p.n - lo);
    const int ntri = (int)solve_ntri(p.nt);
    const float* Lb = p.Linv + (int64_t)I * ntri * T * T;
    const int t0 = (int)blockIdx.x * p.tpc, t1 = min(t0 + p.tpc, ntri);
    int i = tri_row(t0);
    int k = t0 - (int)packed_tile(i, 0);
    int fk = k, fi = i;  // tile to fetch next
    auto fetch = [&](int t) {
        float* st = stage + (t & 1) * solve_stage_floats<C>();
        if (t < t1) {
            fetch_tile(st, Lb + (int64_t)t * (T * T), tid);
            fetch_rhs<C>(st + T * T, p.R + (lo + fk * T) * C, (int)bI - fk * T, tid);
            if (fk == fi) fk = 0, ++fi;
            else ++fk;
        }
        cp_commit();
    };
    float acc[2][C];
#pragma unroll
    for (int c = 0; c < C; ++c) acc[0][c] = acc[1][c] = 0.0f;
    fetch(t0);
    for (int t = t0; t < t1; ++t) {
        fetch(t + 1);
        cp_wait<1>();
        __syncthreads();
        const float* sx = stage + (t & 1) * solve_stage_floats<C>();
        const float* sv = sx + T * T;
        // rows lane and lane + 32, terms kQ warp .. + kQ - 1
#pragma unroll
        for (int g = 0; g < kQ / 4; ++g) {
            const int q = kQ * warp + 4 * g;
            const float4 x0 = *reinterpret_cast<const float4*>(sx + swz(lane, q / 4));
            const float4 x1 = *reinterpret_cast<const float4*>(sx + swz(lane + 32, q / 4));
            rank1<C>(acc, x0.x, x1.x, sv + q * C);
            rank1<C>(acc, x0.y, x1.y, sv + (q + 1) * C);
            rank1<C>(acc, x0.z, x1.z, sv + (q + 2) * C);
            rank1<C>(acc, x0.w, x1.w, sv + (q + 3) * C);
        }
        if (k == i || t + 1 == t1) {
            const int row0 = (int)packed_tile(i, 0), first = row0 / p.tpc, last = (row0 + i) / p.tpc;
            flush_row<C>(p, i, (int)blockIdx.x - first, last - first + 1,
                         stage + (t & 1) * solve_stage_floats<C>(), acc,
                         [](int l, int h) { return l + 32 * h; }, &s_last,
                         [&](int rr, int c, float sum) { p.Z[((int64_t)i * T + rr) * C + c] = sum; });
#pragma unroll
            for (int c = 0; c < C; ++c) acc[0][c] = acc[1][c] = 0.0f;
        }
        if (k == i) k = 0, ++i;
        else ++k;
        __syncthreads();
    }
}

// pass 2: Delta_k = sum_{i >= k} X_ik^T Z_i, then W_I += Delta; tiles in
// column-major order.  With the tensor-core update Delta also goes to its operand
// layout (BF16 hi and lo, launch_kmv_tc_step), which saves that form a launch.
template <int C>
__global__ void __launch_bounds__(kSolveThreads, solve_ctas_per_sm(C)) solve_upper_kernel(const SolveParams p) {
    extern __shared__ float4 bs_smem4[];
    float* stage = reinterpret_cast<float*>(bs_smem4);
    __shared__ int s_last;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // written by the update before the first pass, which has waited for it
    const int I = *p.sel;
    const int nt = p.nt;
    const int64_t lo = (int64_t)I * p.b;
    if (!AP_CHK(I >= 0 && lo < p.n)) return;
    const int64_t bI = min(p.b, p.n - lo);
    const int ntri = (int)solve_ntri(nt);
    const float* Lb = p.Linv + (int64_t)I * ntri * T * T;
    const int u0 = (int)blockIdx.x * p.tpc, u1 = min(u0 + p.tpc, ntri);
    // counted from the end, columns nt - 1 - k have the lengths of rows
    int k = nt - 1 - tri_row(ntri - 1 - u0);
    int i = k + u0 - (int)col_start(nt, k);
    int fi = i, fk = k, zi = i, zk = k;  // tiles whose factor part / right-hand side to fetch next
    auto step = [&](int& a, int& b) {
        if (a == nt - 1) a = ++b;
        else ++a;
    };
    auto fetch_x = [&](int u) {
        if (u >= u1) return;
        fetch_tile(stage + (u & 1) * solve_stage_floats<C>(), Lb + packed_tile(fi, fk) * T * T, tid);
        step(fi, fk);
    };
    auto fetch_z = [&](int u) {
        if (u >= u1) return;
        fetch_rhs<C>(stage + (u & 1) * solve_stage_floats<C>() + T * T, p.Z + (int64_t)zi * T * C, T, tid);
        step(zi, zk);
    };
    float acc[2][C];
#pragma unroll
    for (int c = 0; c < C; ++c) acc[0][c] = acc[1][c] = 0.0f;
    fetch_x(u0);
    fetch_x(u0 + 1);
    pdl_wait();  // Z
    pdl_launch();
    fetch_z(u0);
    cp_commit();
    for (int u = u0; u < u1; ++u) {
        if (u > u0) fetch_x(u + 1);
        fetch_z(u + 1);
        cp_commit();
        cp_wait<1>();
        __syncthreads();
        const float* sx = stage + (u & 1) * solve_stage_floats<C>();
        const float* sv = sx + T * T;
        // columns 2 lane, 2 lane + 1 of the tile, terms (rows) kQ warp .. + kQ - 1
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const int r = kQ * warp + q;
            const float2 x = *reinterpret_cast<const float2*>(sx + swz(r, lane / 2) + 2 * (lane & 1));
            rank1<C>(acc, x.x, x.y, sv + r * C);
        }
        if (i == nt - 1 || u + 1 == u1) {
            const int col0 = (int)col_start(nt, k), first = col0 / p.tpc, last = (col0 + nt - 1 - k) / p.tpc;
            flush_row<C>(p, k, (int)blockIdx.x - first, last - first + 1, stage + (u & 1) * solve_stage_floats<C>(),
                         acc, [](int l, int h) { return 2 * l + h; }, &s_last, [&](int qq, int c, float sum) {
                             const int64_t li = (int64_t)k * T + qq;
                             const float d = li < bI ? sum : 0.0f;
                             if (li < p.b) p.Delta[li * C + c] = d;
                             if (li < bI && AP_CHK(lo + li < p.n)) p.W[(lo + li) * C + c] += d;
                             if (p.DT) tc_store_delta(p.DT, C, li, c, d);
                         });
#pragma unroll
            for (int c = 0; c < C; ++c) acc[0][c] = acc[1][c] = 0.0f;
        }
        step(i, k);
        __syncthreads();
    }
    if (blockIdx.x == 0 && tid == 0 && p.trace) {
        const int64_t step_no = *p.step_ctr;
        if (step_no < p.trace_cap) p.trace[step_no] = I;
    }
}

template <int C>
cudaError_t launch_solve_inst(const SolveParams& p, cudaStream_t st) {
    const unsigned grid = (unsigned)block_solve_ctas(p.nt, p.tpc);
    constexpr size_t smem = solve_smem<C>();
    cudaError_t err;
    if ((err = cudaFuncSetAttribute(solve_lower_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
        return err;
    if ((err = cudaFuncSetAttribute(solve_upper_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
        return err;
    if ((err = launch_dependent(solve_lower_kernel<C>, grid, kSolveThreads, smem, st, p.dependent, p))) return err;
    return launch_dependent(solve_upper_kernel<C>, grid, kSolveThreads, smem, st, p.dependent, p);
}

}  // namespace

// All CTAs in one wave.
void block_solve_layout(int nt, int C, int num_sms, int* tpc, int* maxj) {
    const int64_t target = (int64_t)solve_ctas_per_sm(C) * std::max(1, num_sms);
    *tpc = (int)std::max<int64_t>(1, (solve_ntri(nt) + target - 1) / target);
    *maxj = (nt + *tpc - 1) / *tpc + 1;
}

int64_t block_solve_ctas(int nt, int tpc) { return (solve_ntri(nt) + tpc - 1) / tpc; }

cudaError_t launch_block_solve(const SolveParams& p, cudaStream_t st, int64_t* launches) {
    if (launches) *launches += 2;
    switch (p.C) {
        case 1: return launch_solve_inst<1>(p, st);
        case 4: return launch_solve_inst<4>(p, st);
        case 16: return launch_solve_inst<16>(p, st);
        case 32: return launch_solve_inst<32>(p, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ap
