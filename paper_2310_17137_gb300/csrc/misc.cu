// Input preparation, padding copies, the stand-alone norm/selection pass and
// the kernel-family dispatch of the FP32 product.
#include <math.h>

#include <algorithm>

#include "kmv_fp32.cuh"

namespace ap {

double kernel_input_scale(int kernel) {
    if (kernel == AP_RBF) return sqrt(0.5 * 1.4426950408889634);  // sqrt(log2(e) / 2)
    if (kernel == AP_MATERN32) return sqrt(3.0);
    return sqrt(5.0);
}

// The split of one product of `nseg` segments of `seg` rows with `ncols` columns.
//
// Rows per thread: more rows share each staged column (the shared-memory reads per
// entry fall as 1 / rm), but a tile of 128 rm rows may be mostly padding (a segment of
// 600 rows is 60 % of two 512-row tiles) and leaves fewer tiles.  The modelled issue
// slots per useful entry, times the shortfall of work when the whole product cannot
// fill the chip, decide (2894 x 2894, d = 6, 16 columns: 96 CTAs of two rows a thread 67 us
// a call, 184 of one 59).
//
// Columns, SIMT form: S splits inside a cluster until 4 CTAs per SM exist, then G groups
// through global memory: enough of them for about 8 waves of CTAs while every CTA keeps
// at least 512 columns (a last wave that is nearly empty costs at most an eighth), and
// for 8 CTAs per SM with at least 64 columns when the clusters alone leave places free.
// Measured on GB300: n = 100,003, d = 11, 1024 test points, 16 CTAs (cluster only)
// 1102 us per ap_predict_mean call, with the groups 135 us; n = 20,600, d = 8, one
// column, ap_residual 500 -> 377 us.
// With 16 and 32 right-hand sides a group needs 64 columns per right-hand side: the sums
// that pass through global memory grow with them (3000 x 3000, c = 32: 91 us with groups of
// 75 columns, 80 us without).
// Tensor-core form: one CTA per SM over equal ranges of (tile, 128-column chunk) units.
KmvSplit kmv_split(int D, int C, int64_t seg, int64_t nseg, int64_t ncols) {
    constexpr int64_t kSms = 152, kMaxScratch = (int64_t)8 << 20;
    const bool x3 = C >= kX3MinC && (double)(seg * nseg) * (double)ncols >= (C == 16 ? kX3MinEntries16 : kX3MinEntries32);
    const int64_t chunk = x3 ? kX3Chunk : kKmvTN;
    const double places = x3 ? kSms : 2.0 * kSms;
    const double instr = x3 ? D + 16.0 : D + C + 8.0, lds = x3 ? D / 4.0 : (D + C) / 4.0;
    const int64_t wide = C >= kX3MinC ? 64 * C : 0;  // columns of a group
    KmvSplit best = {};
    double best_cost = 0.0;
    for (int rm = x3 ? (D <= kX3MaxD2 ? 2 : 1) : rows_per_thread(D, C); rm >= 1; rm /= 2) {
        KmvSplit sp = {};
        sp.rm = rm;
        sp.rows = (int64_t)kKmvThreads * rm;
        sp.tps = (seg + sp.rows - 1) / sp.rows;
        sp.ntiles = nseg * sp.tps;
        const double pad = (double)(sp.tps * sp.rows) / (double)seg;
        // (many right-hand sides in the SIMT form: only as many column ranges as it is cut into)
        int64_t ranges = (ncols + chunk - 1) / chunk;
        if (!x3 && C >= kX3MinC) ranges = std::min(ranges, kMaxSplit * std::max<int64_t>(1, ncols / (kMaxSplit * wide)));
        const double units = (double)sp.ntiles * (double)ranges;
        const double idle = units < places ? places / units : 1.0;
        const double cost = pad * idle * (instr + lds / rm);
        if (!best.rm || cost < best_cost) best = sp, best_cost = cost;
    }
    best.S = 1;
    best.x3 = x3;
    if (x3) {
        best.ctas = (int)std::min<int64_t>(kSms, best.ntiles * ((ncols + chunk - 1) / chunk));
        best.G = 2;
        best.scratch = 2 * (int64_t)best.ctas * best.rows * C;
        best.tickets = best.ntiles;
        return best;
    }
    while (best.S < kMaxSplit && best.ntiles * best.S < 4 * kSms && ncols / (2 * best.S) >= chunk) best.S *= 2;
    const int64_t ctas = best.ntiles * best.S;
    auto groups = [&](int64_t want, int64_t min_cols) {
        return std::min<int64_t>((want + ctas - 1) / ctas, ncols / (best.S * min_cols));
    };
    int64_t G = groups(64 * kSms, std::max<int64_t>(512, wide));
    if (ctas < 4 * kSms) G = std::max(G, groups(8 * kSms, std::max(chunk, wide)));
    G = std::min<int64_t>(G, kMaxScratch / (best.ntiles * best.rows * C));
    best.G = (int)std::max<int64_t>(1, std::min<int64_t>(G, 1024));
    if (best.G > 1) {
        best.scratch = best.ntiles * best.G * best.rows * C;
        best.tickets = best.ntiles * best.S;
    }
    return best;
}

cudaError_t launch_kmv(int kernel, const KmvParams& p, int D, int C, cudaStream_t st) {
    const bool x3 = p.x3;
    switch (kernel) {
        case AP_RBF: return x3 ? launch_x3_rbf(p, D, C, st) : launch_kmv_rbf(p, D, C, st);
        case AP_MATERN32: return x3 ? launch_x3_m32(p, D, C, st) : launch_kmv_m32(p, D, C, st);
        case AP_MATERN52: return x3 ? launch_x3_m52(p, D, C, st) : launch_kmv_m52(p, D, C, st);
        default: return cudaErrorInvalidValue;
    }
}

namespace {

struct ScaleVec {
    float v[AP_MAX_DIM];
};

// Xs[i, k] = fl(X[i, k] * sc_k) for k < d, 0 for the padding k in [d, D);
// sc_k = hi_k + lo_k, and Xs_lo gets X * sc_k - Xs (TwoProd remainder plus
// the lo part of the scale) when requested.  A NaN or Inf input sets *bad.
__global__ void prep_inputs_kernel(const float* __restrict__ X, int64_t n, int d, int D, const ScaleVec sh,
                                   const ScaleVec sl, float* __restrict__ Xs, float* __restrict__ Xs_lo,
                                   int* __restrict__ bad) {
    const int64_t total = n * D;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / D;
        const int k = (int)(t % D);
        float hi = 0.0f, lo = 0.0f;
        if (k < d && AP_CHK(i < n)) {
            const float x = X[i * d + k];
            if (!isfinite(x) && bad) *bad = 1;
            hi = x * sh.v[k];
            lo = fmaf(x, sh.v[k], -hi) + x * sl.v[k];
        }
        Xs[t] = hi;
        if (Xs_lo) Xs_lo[t] = lo;
    }
}

__global__ void pad_copy_kernel(const float* __restrict__ src, int64_t n, int c, float* __restrict__ dst, int C) {
    const int64_t total = n * C;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / C;
        const int k = (int)(t % C);
        dst[t] = k < c ? src[i * c + k] : 0.0f;
    }
}

__global__ void unpad_copy_kernel(const float* __restrict__ src, int64_t n, int C, float* __restrict__ dst, int c) {
    const int64_t total = n * c;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / c;
        const int k = (int)(t % c);
        dst[t] = src[i * C + k];
    }
}

// Start of a solve in one pass over n x C: Bp = B padded, R = Bp (when the start is
// zero), W = W0 padded or 0, W_ckpt = W.
__global__ void init_solve_kernel(const float* __restrict__ B, const float* __restrict__ W0, int64_t n, int c, int C,
                                  float* __restrict__ Bp, float* __restrict__ R, float* __restrict__ W,
                                  float* __restrict__ W_ckpt) {
    const int64_t total = n * C;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / C;
        const int k = (int)(t % C);
        const float b = k < c ? B[i * c + k] : 0.0f, w = W0 && k < c ? W0[i * c + k] : 0.0f;
        Bp[t] = b;
        if (R) R[t] = b;
        W[t] = w;
        if (W_ckpt) W_ckpt[t] = w;
    }
}

unsigned grid_for(int64_t total) {
    int64_t g = (total + 255) / 256;
    if (g > 152 * 32) g = 152 * 32;
    if (g < 1) g = 1;
    return (unsigned)g;
}

}  // namespace

cudaError_t launch_prep_inputs(const float* X, int64_t n, int d, int D, const float* sc_hi, const float* sc_lo,
                               float* Xs, float* Xs_lo, int* bad, cudaStream_t st) {
    ScaleVec sh = {}, sl = {};
    for (int k = 0; k < d && k < AP_MAX_DIM; ++k) {
        sh.v[k] = sc_hi[k];
        sl.v[k] = sc_lo ? sc_lo[k] : 0.0f;
    }
    prep_inputs_kernel<<<grid_for(n * D), 256, 0, st>>>(X, n, d, D, sh, sl, Xs, Xs_lo, bad);
    return cudaGetLastError();
}

cudaError_t launch_init_solve(const float* B, const float* W0, int64_t n, int c, int C, float* Bp, float* R, float* W,
                              float* W_ckpt, cudaStream_t st) {
    init_solve_kernel<<<grid_for(n * C), 256, 0, st>>>(B, W0, n, c, C, Bp, R, W, W_ckpt);
    return cudaGetLastError();
}

cudaError_t launch_pad_copy(const float* src, int64_t n, int c, float* dst, int C, cudaStream_t st) {
    pad_copy_kernel<<<grid_for(n * C), 256, 0, st>>>(src, n, c, dst, C);
    return cudaGetLastError();
}

cudaError_t launch_unpad_copy(const float* src, int64_t n, int C, float* dst, int c, cudaStream_t st) {
    unpad_copy_kernel<<<grid_for(n * c), 256, 0, st>>>(src, n, C, dst, c);
    return cudaGetLastError();
}

cudaError_t launch_norms_select(const float* R, int64_t n, int C, const EpiParams& e, int64_t tile_rows,
                                cudaStream_t st) {
    const dim3 grid((unsigned)e.ntiles, 1, 1);
    switch (C) {
        case 1: norms_select_kernel<1><<<grid, kKmvThreads, 0, st>>>(R, n, e, tile_rows); break;
        case 4: norms_select_kernel<4><<<grid, kKmvThreads, 0, st>>>(R, n, e, tile_rows); break;
        case 16: norms_select_kernel<16><<<grid, kKmvThreads, 0, st>>>(R, n, e, tile_rows); break;
        case 32: norms_select_kernel<32><<<grid, kKmvThreads, 0, st>>>(R, n, e, tile_rows); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace ap

namespace ap {

cudaError_t launch_kmv_comp(int kernel, const KmvParams& p, int D, int C, cudaStream_t st) {
    switch (kernel) {
        case AP_RBF: return launch_kmv_comp_rbf(p, D, C, st);
        case AP_MATERN32: return launch_kmv_comp_m32(p, D, C, st);
        case AP_MATERN52: return launch_kmv_comp_m52(p, D, C, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_grad(int kernel, const GradParams& p, int D, int C, cudaStream_t st) {
    switch (kernel) {
        case AP_RBF: return launch_grad_rbf(p, D, C, st);
        case AP_MATERN32: return launch_grad_m32(p, D, C, st);
        case AP_MATERN52: return launch_grad_m52(p, D, C, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ap

namespace ap {
namespace {

__device__ __forceinline__ float rademacher_at(uint64_t seed, uint64_t idx) {
    return (splitmix64_at(seed, idx) >> 63) ? 1.0f : -1.0f;
}

// B = [y - mu, z_1..z_l] (n x c); Z == nullptr draws z from SplitMix64(seed).
__global__ void assemble_rhs_kernel(const float* __restrict__ y, float mu, const float* __restrict__ Z, int l,
                                    uint64_t seed, int64_t n, float* __restrict__ B, float* __restrict__ Zout) {
    const int c = l + 1;
    const int64_t total = n * c;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / c;
        const int k = (int)(t % c);
        float v;
        if (k == 0) {
            v = y[i] - mu;
        } else {
            const int64_t zi = i * l + (k - 1);
            v = Z ? Z[zi] : rademacher_at(seed, (uint64_t)zi);
            if (Zout) Zout[zi] = v;
        }
        B[t] = v;
    }
}

// V = [u, z_1..z_l] from the solved W (n x C, column 0 = u) and B (n x c).
__global__ void assemble_v_kernel(const float* __restrict__ W, int C, const float* __restrict__ B, int c, int64_t n,
                                  float* __restrict__ V) {
    const int64_t total = n * C;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / C;
        const int k = (int)(t % C);
        V[t] = k == 0 ? W[i * C] : (k < c ? B[i * c + k] : 0.0f);
    }
}

// out[0] = sum_i W[i * C] * (Y ? Y[i * cy] : 1) in FP64 (the ticketed last CTA
// adds the per-CTA partials in order).
__global__ void dot0_kernel(const float* __restrict__ W, int C, const float* __restrict__ Y, int cy, int64_t n,
                            double* part, unsigned* ticket, double* out) {
    __shared__ double red[32];
    __shared__ int s_last;
    double v = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        v += (double)W[i * C] * (Y ? (double)Y[i * cy] : 1.0);
    double t = cta_sum_d(v, red);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(ticket, 1u) == gridDim.x - 1u) ? 1 : 0;
    __syncthreads();
    if (s_last && threadIdx.x == 0) {
        __threadfence();
        double acc = 0.0;
        for (unsigned b = 0; b < gridDim.x; ++b) acc += __ldcg(part + b);
        *out = acc;
        *ticket = 0u;
    }
}

}  // namespace

cudaError_t launch_assemble_rhs(const float* y, float mu, const float* Z, int l, uint64_t seed, int64_t n, float* B,
                                float* Zout, cudaStream_t st) {
    assemble_rhs_kernel<<<grid_for(n * (l + 1)), 256, 0, st>>>(y, mu, Z, l, seed, n, B, Zout);
    return cudaGetLastError();
}

cudaError_t launch_assemble_v(const float* W, int C, const float* B, int c, int64_t n, float* V, cudaStream_t st) {
    assemble_v_kernel<<<grid_for(n * C), 256, 0, st>>>(W, C, B, c, n, V);
    return cudaGetLastError();
}

constexpr unsigned kColsumGrid = 256;

cudaError_t launch_dot0(const float* W, int C, const float* Y, int cy, int64_t n, double* part, unsigned* ticket,
                       double* out, cudaStream_t st) {
    dot0_kernel<<<kColsumGrid, kKmvThreads, 0, st>>>(W, C, Y, cy, n, part, ticket, out);
    return cudaGetLastError();
}

}  // namespace ap

// ---------------------------------------------------- bounds-check self-test
namespace ap {
namespace {

// One thread reads element `index` of an 8-element buffer through AP_CHK: in
// the checked build an index outside [0, 8) is recorded and the read skipped.
__global__ void bounds_selftest_kernel(const float* __restrict__ buf, int index, float* __restrict__ out) {
    float v = 0.0f;
    if (AP_CHK(index >= 0 && index < 8)) v = buf[index];
    *out = v;
}

}  // namespace
}  // namespace ap

extern "C" ap_status ap_bounds_selftest(int32_t index) {
#ifdef AP_CHECKED
    float* d = nullptr;
    if (cudaMalloc(&d, 9 * sizeof(float)) != cudaSuccess) return AP_ERR_NOMEM;
    cudaMemset(d, 0, 9 * sizeof(float));
    ap::bounds_selftest_kernel<<<1, 1>>>(d, index, d + 8);
    const cudaError_t err = cudaDeviceSynchronize();
    cudaFree(d);
    return err == cudaSuccess ? AP_OK : AP_ERR_CUDA;
#else
    (void)index;
    return AP_ERR_UNSUPPORTED;
#endif
}
