// Cached block-Cholesky factors (Sec. 3, "Cached Cholesky Factors"; Table 6:
// (1/3) n b^2 flops, n b memory).
//
// For every diagonal block K_hat_II (b x b, the last one possibly short and
// padded with the identity to a whole number of 64 x 64 tiles):
//   1. build K_hat_II in FP64 directly from the FP32 inputs;
//   2. factor it in FP64 by a right-looking tiled Cholesky: POTRF of the
//      diagonal tile (which also inverts L_kk), TRSM of the panel below it as
//      a product with L_kk^{-T}, SYRK/GEMM update of the trailing tiles (the
//      products as FP64 FMAs here, or as exact integer slice products on the
//      tensor cores in ozaki.cu); all blocks of a group advance together, one
//      launch per phase;
//   3. form the inverse factor L^{-1} tile by tile (diagonal tiles from the
//      FP64 tile inverses, off-diagonal blocks by halves,
//      [A 0; B C]^{-1} = [A^{-1} 0; -C^{-1} B A^{-1} C^{-1}]) and store it packed in FP32.
// The per-step block solve Delta = L^{-T} (L^{-1} R_I) then becomes two
// parallel triangular products instead of two sequential substitutions.
#include <math.h>

#include <algorithm>

#include "ap_internal.cuh"

namespace ap {
namespace {

constexpr int T = kTile;
constexpr int TP = kTile + 1;  // padded shared-memory row stride
constexpr int kSms = 152;

// ---------------------------------------------------------------- FP64 phi
// The kernel profile phi(r^2) in FP64 for K_II, built from a handful of FP64
// FMAs instead of the library exp and sqrt.  FP64 arithmetic (2 results per clock per
// SM) is all that bounds the K_II build, and comparisons, conversions and rounding count
// as much as a multiply-add, so ranges are tested and integers taken on the bits
// (GB300, 5 blocks of 4096, d = 8: 4.28 -> 3.79 ms).
//
// exp(x), x <= 0: Tang's table-driven method (P. T. P. Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point
// arithmetic", ACM TOMS 15(2), 1989): x = (64 k + j) ln2/64 + r with
// |r| <= ln2/128, e^x = 2^k 2^(j/64) e^r.  ln2/64 is split into the double
// nearest to it and the double nearest to the remainder, so r is exact to a
// rounding; e^r - 1 is its Taylor polynomial to degree 6 (truncation below
// r^7/7! < 2^-62 relative).  The integer 64 k + j is the low word of the product plus
// 1.5 * 2^52, and k is added to the exponent bits.  Below x = -708 the result is 0
// (e^-708 ~ 3e-308, far below any kernel value that matters next to sigma^2; above it
// 2^k 2^(j/64) stays normal).
// sqrt(x): from the hardware's approximate reciprocal square root (relative error
// below 2^-20) one coupled Newton step for sqrt(x) and 1/(2 sqrt(x)) (Goldschmidt's
// form; error 3/2 e^2 < 2^-39), then one Newton correction with the exact residual
// (error ~e^2, below the last bit).
constexpr double kLn2By64Hi = 0x1.62e42fefa39efp-7;   // double nearest to ln2 / 64
constexpr double kLn2By64Lo = 0x1.abc9e3b39803fp-62;  // ln2 / 64 - kLn2By64Hi, rounded
constexpr double k64ByLn2 = 92.33248261689366;        // 64 / ln2
constexpr double kRound = 6755399441055744.0;         // 1.5 * 2^52

__device__ __forceinline__ double exp_nonpos(double x, const double* tab2) {
    if ((__double2hiint(x) & 0x7fffffff) > __double2hiint(708.0)) return 0.0;  // (also a NaN; callers pass finite x)
    const double nb = fma(x, k64ByLn2, kRound);
    const int n = __double2loint(nb);
    const double nf = nb - kRound;
    const double r = fma(-nf, kLn2By64Lo, fma(-nf, kLn2By64Hi, x));
    double q = 1.0 / 720.0;
    q = fma(q, r, 1.0 / 120.0);
    q = fma(q, r, 1.0 / 24.0);
    q = fma(q, r, 1.0 / 6.0);
    q = fma(q, r, 0.5);
    q = fma(q, r, 1.0);
    const double t = tab2[n & 63];
    const double y = fma(t, q * r, t);
    // k = floor(n / 64) in [-1022, 0]
    return __hiloint2double(__double2hiint(y) + ((n >> 6) << 20), __double2loint(y));
}

__device__ __forceinline__ double sqrt_nonneg(double x) {
    const int hi = __double2hiint(x);
    const bool nan = (hi & 0x7fffffff) > 0x7ff00000;  // (stays one)
    if (hi < __double2hiint(1e-36)) return nan ? x : 0.0;  // phi is flat at 0: the error is below the last bit
    if (hi > __double2hiint(1e12)) return nan ? x : 1e6;   // e^-sqrt(x) underflows either way
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double g = x * y, h = 0.5 * y;
    const double e = fma(-g, h, 0.5);
    g = fma(g, e, g);
    h = fma(h, e, h);
    return fma(fma(-g, g, x), h, g);
}

// phi from t = r^2 / 2 (RBF), 3 r^2 (Matern-3/2) or 5 r^2 (Matern-5/2)
__device__ __forceinline__ double phi_of(int kernel, double t, const double* tab2) {
    if (kernel == AP_RBF) return exp_nonpos(-t, tab2);
    const double u = sqrt_nonneg(t);
    const double poly = kernel == AP_MATERN32 ? 1.0 + u : fma(u, fma(u, 1.0 / 3.0, 1.0), 1.0);
    return poly * exp_nonpos(-u, tab2);
}

__host__ __device__ inline double phi_scale(int kernel) {
    return kernel == AP_RBF ? 0.5 : (kernel == AP_MATERN32 ? 3.0 : 5.0);
}

// 2^(j/64), j = 0..63, into shared memory (first 64 threads; caller syncs)
__device__ __forceinline__ void fill_exp2_table(double* tab2) {
    if (threadIdx.x < 64) tab2[threadIdx.x] = exp2((double)threadIdx.x / 64.0);
}

// lower-triangular tile index t -> (i, j), j <= i
__device__ __forceinline__ void tri_index(int64_t t, int& i, int& j) {
    int ii = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while ((int64_t)(ii + 1) * (ii + 2) / 2 <= t) ++ii;
    while ((int64_t)ii * (ii + 1) / 2 > t) --ii;
    i = ii;
    j = (int)(t - (int64_t)ii * (ii + 1) / 2);
}

__device__ __forceinline__ int64_t packed_tile(int i, int k) { return (int64_t)i * (i + 1) / 2 + k; }

__global__ void __launch_bounds__(256) build_kii_kernel(const CacheParams cp, int64_t blk0, double* A) {
    __shared__ double s_tab[64];
    __shared__ double s_unit[AP_MAX_DIM];
    __shared__ double s_xi[AP_MAX_DIM * T], s_xj[AP_MAX_DIM * T];  // dimension-major
    const int z = blockIdx.y;
    const int64_t blk = blk0 + z;
    const int64_t ld = (int64_t)cp.nt * T;
    const int d = cp.d;
    int ti, tj;
    tri_index(blockIdx.x, ti, tj);
    const int64_t lo = blk * cp.b;
    const int64_t bJ = min(cp.b, cp.n - lo);
    double* Ab = A + (int64_t)z * ld * ld;
    fill_exp2_table(s_tab);
    if (threadIdx.x < d) s_unit[threadIdx.x] = cp.unit[threadIdx.x];
    // the tile's row and column points (rows past the block are never read)
    for (int t = threadIdx.x; t < T * d; t += blockDim.x) {
        const int r = t / d, k = t % d;
        const int64_t li = (int64_t)ti * T + r, lj = (int64_t)tj * T + r;
        s_xi[k * T + r] = li < bJ ? (double)cp.X[(lo + li) * d + k] : 0.0;
        s_xj[k * T + r] = lj < bJ ? (double)cp.X[(lo + lj) * d + k] : 0.0;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < T * T; t += blockDim.x) {
        const int r = t / T, q = t % T;
        const int64_t li = (int64_t)ti * T + r, lj = (int64_t)tj * T + q;
        double v;
        if (li < bJ && lj < bJ) {
            // the difference of two FP32 values is exact in FP64 (29 binades apart at most,
            // otherwise rounded once); its unit makes the squared distance phi's argument.
            // (Points scaled ahead, relative to the block's first one, would save a
            // multiplication per entry and dimension but lose near points of a block that
            // holds a far one.)
            double r2 = 0.0;
            for (int k = 0; k < d; ++k) {
                const double df = (s_xi[k * T + r] - s_xj[k * T + q]) * s_unit[k];
                r2 = fma(df, df, r2);
            }
            v = cp.s * phi_of(cp.kernel, r2, s_tab);
            if (li == lj) v += cp.noise;
        } else {
            v = (li == lj) ? 1.0 : 0.0;
        }
        Ab[li * ld + lj] = v;
    }
}

// FP64 phi at given squared distances (verification of the cache's kernel values)
__global__ void __launch_bounds__(256) phi_fp64_eval_kernel(int kernel, const double* r2, int64_t count,
                                                            double* out) {
    __shared__ double s_tab[64];
    fill_exp2_table(s_tab);
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = phi_of(kernel, phi_scale(kernel) * r2[i], s_tab);
}

// 1/sqrt(p) for a pivot: the reciprocal square root approximation (relative error
// below 2^-21) refined by one third-order step, y + y e (1/2 + 3/8 e) with
// e = 1 - p y^2 (error 5/16 e^3 < 2^-60, below the last bit); outside the FP32 range
// the library square root and division.
__device__ __forceinline__ double rsqrt_pivot(double p) {
    if (!(p > 1e-30 && p < 1e30)) return 1.0 / sqrt(p);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(p));
    const double e = fma(-p * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// Factor the diagonal tile (k, k) in place and write its inverse to Dinv.
//
// One CTA per block, on the critical path of every panel.  FP64 runs at 2 results per
// clock per SM, whoever asks: a warp instruction holds the pipe for 16 clocks, so the
// 2 x 64^3 / 6 multiply-adds of the factor and the inverse cost 21 us however they are
// arranged, and work done for all threads (or by threads with nothing to do) counts in
// full.  The tile is factored in 16-column panels: the diagonal 16 x 16 in one warp's
// registers (the pivot chain: shuffles and about six dependent FP64 operations per
// column, no CTA barrier), the rows below by one thread each, the rest as a rank-16
// update on all warps.  While warp 0 is on a diagonal block, the other warps form the
// inverse's block row above it, X_ik = -X_ii sum_j L_ij X_jk.
// Measured (GB300, 5 blocks): 206 us per launch with a barrier round per column and
// every thread deriving every pivot, 101 us now (FP64 pipe 46 % busy).
constexpr int NB = 16;

__device__ __forceinline__ void bar_sync_n(int id, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Block row bi of the inverse by threads t = 0 .. nthr - 1 (whole warps, named barrier id).
__device__ __forceinline__ void inverse_block_row(const double* a, double* x, const double* s_rd, int bi, int t,
                                                  int nthr, int bar) {
    const int r0 = NB * bi;
    if (t < 32) {
        // X_ii: lane c forward-substitutes the unit vector c (lanes 16 .. 31 repeat 0 .. 15)
        const int c = t & (NB - 1);
        double v[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) v[i] = i == c ? 1.0 : 0.0;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            v[i] *= s_rd[r0 + i];
#pragma unroll
            for (int l = i + 1; l < NB; ++l) v[l] = fma(-a[(r0 + l) * TP + r0 + i], v[i], v[l]);
        }
        if (t < NB) {
#pragma unroll
            for (int i = 0; i < NB; ++i) x[(r0 + i) * TP + r0 + c] = v[i];
        }
    } else {
        // E_ik = sum_j L_ij X_jk (j = k .. i - 1) into the place of X_ik
        for (int o = t - 32; o < bi * NB * NB; o += nthr - 32) {
            const int c = o % (bi * NB), r = r0 + o / (bi * NB);
            double s0 = 0.0, s1 = 0.0;
            for (int q = c & ~(NB - 1); q < r0; q += 2) {
                s0 = fma(a[r * TP + q], x[q * TP + c], s0);
                s1 = fma(a[r * TP + q + 1], x[(q + 1) * TP + c], s1);
            }
            x[r * TP + c] = s0 + s1;
        }
    }
    bar_sync_n(bar, nthr);
    double out[4];
    int n = 0;
    for (int o = t; o < bi * NB * NB; o += nthr, ++n) {
        const int c = o % (bi * NB), rl = o / (bi * NB);
        double s = 0.0;
        for (int q = 0; q <= rl; ++q) s = fma(x[(r0 + rl) * TP + r0 + q], x[(r0 + q) * TP + c], s);
        out[n & 3] = -s;
    }
    bar_sync_n(bar, nthr);
    n = 0;
    for (int o = t; o < bi * NB * NB; o += nthr, ++n) x[(r0 + o / (bi * NB)) * TP + o % (bi * NB)] = out[n & 3];
    bar_sync_n(bar, nthr);
}

__global__ void __launch_bounds__(256) potrf_diag_kernel(double* A, int nt, int k, double* Dinv, int* bad) {
    extern __shared__ double pd_sm[];
    double* a = pd_sm;
    double* x = pd_sm + T * TP;
    __shared__ double s_rd[T];  // 1 / L_jj
    __shared__ int s_bad;
    const int z = blockIdx.x, tid = threadIdx.x, nth = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int64_t ld = (int64_t)nt * T;
    double* Ab = A + (int64_t)z * ld * ld + (int64_t)k * T * ld + (int64_t)k * T;
    for (int t = tid; t < T * T; t += nth) {
        const int r = t / T, q = t % T;
        a[r * TP + q] = (q <= r) ? Ab[r * ld + q] : 0.0;
        x[r * TP + q] = 0.0;
    }
    if (tid == 0) s_bad = 0;
    for (int kb = 0; kb < T / NB; ++kb) {
        const int c0 = NB * kb;
        __syncthreads();
        if (warp == 0) {
            // the diagonal block: lane i holds row c0 + i (lanes 16 .. 31 repeat 0 .. 15)
            const int i = lane & (NB - 1);
            double p[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) p[j] = a[(c0 + i) * TP + c0 + j];
            bool anybad = false;
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                double pv = __shfl_sync(0xffffffffu, p[j], j);
                const bool badp = !(pv > 0.0) || !isfinite(pv);
                if (badp) pv = 1.0;
                anybad |= badp;
                const double rj = rsqrt_pivot(pv);
                if (lane == j) s_rd[c0 + j] = rj;
                p[j] *= rj;
                if (i == j) {
                    const double l = pv * rj;
                    p[j] = fma(0.5 * rj, fma(-l, l, pv), l);  // sqrt(pv), Newton-corrected
                }
#pragma unroll
                for (int l = j + 1; l < NB; ++l) p[l] = fma(-p[j], __shfl_sync(0xffffffffu, p[j], l), p[l]);
            }
            if (lane < NB) {
#pragma unroll
                for (int j = 0; j < NB; ++j)
                    if (j <= i) a[(c0 + i) * TP + c0 + j] = p[j];
            }
            if (lane == 0 && anybad) s_bad = 1;
        } else if (kb > 0) {
            inverse_block_row(a, x, s_rd, kb - 1, tid - 32, nth - 32, 1);
        }
        __syncthreads();
        const int M = T - NB - c0;  // rows below
        if (tid < M) {
            const int r = c0 + NB + tid;
            double p[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) p[j] = a[r * TP + c0 + j];
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                p[j] *= s_rd[c0 + j];
#pragma unroll
                for (int l = j + 1; l < NB; ++l) p[l] = fma(-p[j], a[(c0 + l) * TP + c0 + j], p[l]);
            }
#pragma unroll
            for (int j = 0; j < NB; ++j) a[r * TP + c0 + j] = p[j];
        }
        __syncthreads();
        // rank-16 update of the lower 16 x 16 tiles below and right of the panel
        const int ty = tid / NB, tx = tid % NB;
        for (int ta = 0; ta < M / NB; ++ta) {
            const int r = c0 + NB + ta * NB + ty;
            double row[NB];
#pragma unroll
            for (int q = 0; q < NB; ++q) row[q] = a[r * TP + c0 + q];
            for (int tb = 0; tb <= ta; ++tb) {
                const int c = c0 + NB + tb * NB + tx;
                double s = a[r * TP + c];
#pragma unroll
                for (int q = 0; q < NB; ++q) s = fma(-row[q], a[c * TP + c0 + q], s);
                if (c <= r) a[r * TP + c] = s;
            }
        }
    }
    __syncthreads();
    inverse_block_row(a, x, s_rd, T / NB - 1, tid, nth, 1);
    double* Db = Dinv + ((int64_t)z * nt + k) * T * T;
    for (int t = tid; t < T * T; t += nth) {
        const int r = t / T, q = t % T;
        if (q <= r) Ab[r * ld + q] = a[r * TP + q];
        Db[t] = x[r * TP + q];
    }
    if (tid == 0 && s_bad) bad[z] = 1;
}

// A_ik <- A_ik L_kk^{-T} for the tiles i > k of the panel.
__global__ void __launch_bounds__(256) trsm_kernel(double* A, int nt, int k, const double* Dinv) {
    extern __shared__ double ts_sm[];
    double* sa = ts_sm;
    double* sd = ts_sm + T * TP;
    const int z = blockIdx.y, tid = threadIdx.x;
    const int i = k + 1 + blockIdx.x;
    const int64_t ld = (int64_t)nt * T;
    double* Aik = A + (int64_t)z * ld * ld + (int64_t)i * T * ld + (int64_t)k * T;
    const double* Db = Dinv + ((int64_t)z * nt + k) * T * T;
    for (int t = tid; t < T * T; t += 256) {
        const int r = t / T, q = t % T;
        sa[r * TP + q] = Aik[r * ld + q];
        sd[r * TP + q] = Db[t];
    }
    __syncthreads();
    const int tr = tid / 16, tc = tid % 16;
    double acc[4][4] = {};
    for (int p = 0; p < T; ++p) {
        double av[4], dv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) av[u] = sa[(tr + 16 * u) * TP + p];
#pragma unroll
        for (int v = 0; v < 4; ++v) dv[v] = sd[(tc + 16 * v) * TP + p];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = fma(av[u], dv[v], acc[u][v]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) Aik[(int64_t)(tr + 16 * u) * ld + tc + 16 * v] = acc[u][v];
}

// A_ij -= A_ik A_jk^T for the trailing lower tiles k < j <= i.
__global__ void __launch_bounds__(256) syrk_kernel(double* A, int nt, int k) {
    extern __shared__ double sy_sm[];
    double* sa = sy_sm;
    double* sb = sy_sm + T * TP;
    const int z = blockIdx.y, tid = threadIdx.x;
    int ii, jj;
    tri_index(blockIdx.x, ii, jj);
    const int i = k + 1 + ii, j = k + 1 + jj;
    const int64_t ld = (int64_t)nt * T;
    double* Ab = A + (int64_t)z * ld * ld;
    const double* Aik = Ab + (int64_t)i * T * ld + (int64_t)k * T;
    const double* Ajk = Ab + (int64_t)j * T * ld + (int64_t)k * T;
    double* Aij = Ab + (int64_t)i * T * ld + (int64_t)j * T;
    for (int t = tid; t < T * T; t += 256) {
        const int r = t / T, q = t % T;
        sa[r * TP + q] = Aik[r * ld + q];
        sb[r * TP + q] = Ajk[r * ld + q];
    }
    __syncthreads();
    const int tr = tid / 16, tc = tid % 16;
    double acc[4][4] = {};
    for (int p = 0; p < T; ++p) {
        double av[4], bv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) av[u] = sa[(tr + 16 * u) * TP + p];
#pragma unroll
        for (int v = 0; v < 4; ++v) bv[v] = sb[(tc + 16 * v) * TP + p];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = fma(av[u], bv[v], acc[u][v]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            double* dst = Aij + (int64_t)(tr + 16 * u) * ld + tc + 16 * v;
            *dst -= acc[u][v];
        }
}

// Diagonal tiles of the packed FP32 inverse factor.
__global__ void __launch_bounds__(256) pack_diag_kernel(const double* Dinv, int nt, int64_t blk0,
                                                        int64_t ntri, float* Linv) {
    const int z = blockIdx.y, k = blockIdx.x;
    const double* Db = Dinv + ((int64_t)z * nt + k) * T * T;
    float* dst = Linv + ((blk0 + z) * ntri + packed_tile(k, k)) * T * T;
    for (int t = threadIdx.x; t < T * T; t += 256) dst[t] = (float)Db[t];
}

// FP32 copies of the off-diagonal factor tiles L_ij (i > j) for the inverse
// recurrence, converted once and kept in the unused upper triangle of the FP64
// workspace: L_ij as a row-major 64 x 64 float tile in the first half of the
// rows of tile (j, i).
__device__ __forceinline__ float* lf32_tile(double* Ab, int64_t ld, int i, int j) {
    return reinterpret_cast<float*>(Ab + (int64_t)j * T * ld + (int64_t)i * T);
}

__global__ void __launch_bounds__(256) lower_to_f32_kernel(double* A, int nt) {
    const int z = blockIdx.y;
    int i, j;
    tri_index(blockIdx.x, i, j);  // i >= j; the diagonal tiles are not needed
    if (i == j) return;
    const int64_t ld = (int64_t)nt * T;
    double* Ab = A + (int64_t)z * ld * ld;
    const double* src = Ab + (int64_t)i * T * ld + (int64_t)j * T;
    float* dst = lf32_tile(Ab, ld, i, j);
    for (int t = threadIdx.x; t < T * T; t += 256) {
        const int r = t / T, q = t % T;
        dst[(int64_t)r * 2 * ld + q] = (float)src[(int64_t)r * ld + q];
    }
}

// Off-diagonal tiles of the inverse, by halves: for a lower-triangular matrix
// [A 0; B C] with A^{-1} and C^{-1} known, the block below is -C^{-1} (B A^{-1}).  Level h
// joins neighbouring diagonal blocks of h tiles (all pairs, all blocks of the group in
// one launch): T = B A^{-1}, then X = -C^{-1} T, both triangular times dense.
// log2(nt) levels of two launches replace nt row-by-row launches, whose later ones
// were a few hundred CTAs with up to nt dependent tile products each (GB300, b = 4096:
// 5 blocks 10.5 -> 2.4 ms in all, 13 blocks 15.6 -> 5.9 ms).  T is kept in FP32 in the place of the FP64 factor tiles, which
// nothing reads any more (the inverse uses the FP32 copies).
//
// One CTA of 128 threads per 64 x 64 output tile; K in slices of 32, copied
// asynchronously one slice ahead.  Thread (tr, tc) owns rows tr + 8 u and columns
// 4 tc .. + 3: per four K values 8 + 4 shared 16-byte loads (the first eight are
// broadcasts) for 128 multiply-adds, as packed pairs.
constexpr int kTriK = 32;
constexpr int kTriThreads = 128;
constexpr int kTriLda = kTriK + 4;  // padded rows: 16-byte aligned

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}

template <bool kSecond>
__global__ void __launch_bounds__(kTriThreads) tri_join_kernel(double* A, int nt, int h, int64_t blk0, int64_t ntri,
                                                               float* Linv) {
    __shared__ __align__(16) float sa[2][T * kTriLda];  // left operand, row-major 64 x 32
    __shared__ __align__(16) float sb[2][kTriK * T];    // right operand, 32 x 64
    const int tid = threadIdx.x;
    // the tiles with the longest sums first
    const int npair = (nt + 2 * h - 1) / (2 * h);
    const int pair = (int)blockIdx.x % npair, rest = (int)blockIdx.x / npair;
    const int mid = pair * 2 * h + h;
    const int i = kSecond ? mid + h - 1 - rest / h : mid + rest % h;
    const int k = mid - h + (kSecond ? rest % h : rest / h);
    if (i >= nt) return;
    const int64_t ld = (int64_t)nt * T;
    double* Ab = A + (int64_t)blockIdx.y * ld * ld;
    float* Lb = Linv + (blk0 + blockIdx.y) * ntri * T * T;
    const int j0 = kSecond ? mid : k, j1 = kSecond ? i : mid - 1;  // tiles of the sum
    const int nslice = (j1 - j0 + 1) * (T / kTriK);
    auto fetch = [&](int sl, int buf) {
        const int j = j0 + sl / (T / kTriK), off = (sl % (T / kTriK)) * kTriK;
        // left: L_ij (FP32 copy) or X_ij (packed); right: X_jk (packed) or T_jk
        const float* la = kSecond ? Lb + packed_tile(i, j) * T * T : lf32_tile(Ab, ld, i, j);
        const int64_t lda = kSecond ? T : 2 * ld;
        const float* rb = kSecond ? lf32_tile(Ab, ld, k, j) : Lb + packed_tile(j, k) * T * T;
        const int64_t ldb = kSecond ? 2 * ld : T;
        for (int t = tid; t < T * kTriK / 4; t += kTriThreads) {
            const int r = t / (kTriK / 4), q = 4 * (t % (kTriK / 4));
            cp_async16(&sa[buf][r * kTriLda + q], la + r * lda + off + q);
            const int rr = t / (T / 4), qq = 4 * (t % (T / 4));
            cp_async16(&sb[buf][rr * T + qq], rb + (int64_t)(off + rr) * ldb + qq);
        }
        asm volatile("cp.async.commit_group;");
    };
    const int tr = tid / 16, tc = tid % 16;
    float2 acc[8][2];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc[u][0] = acc[u][1] = make_float2(0.0f, 0.0f);
    fetch(0, 0);
    for (int sl = 0; sl < nslice; ++sl) {
        const int buf = sl & 1;
        if (sl + 1 < nslice) {
            fetch(sl + 1, buf ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
#pragma unroll 2
        for (int p = 0; p < kTriK; p += 4) {
            float4 av[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) av[u] = *reinterpret_cast<const float4*>(&sa[buf][(tr + 8 * u) * kTriLda + p]);
#pragma unroll
            for (int pp = 0; pp < 4; ++pp) {
                const float4 bv = *reinterpret_cast<const float4*>(&sb[buf][(p + pp) * T + 4 * tc]);
                const float2 b0 = make_float2(bv.x, bv.y), b1 = make_float2(bv.z, bv.w);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float a = pp == 0 ? av[u].x : pp == 1 ? av[u].y : pp == 2 ? av[u].z : av[u].w;
                    acc[u][0] = __ffma2_rn(make_float2(a, a), b0, acc[u][0]);
                    acc[u][1] = __ffma2_rn(make_float2(a, a), b1, acc[u][1]);
                }
            }
        }
        __syncthreads();
    }
    float* dst = kSecond ? Lb + packed_tile(i, k) * T * T : lf32_tile(Ab, ld, k, i);
    const int64_t ldd = kSecond ? T : 2 * ld;
    const float sg = kSecond ? -1.0f : 1.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u)
        *reinterpret_cast<float4*>(dst + (int64_t)(tr + 8 * u) * ldd + 4 * tc) =
            make_float4(sg * acc[u][0].x, sg * acc[u][0].y, sg * acc[u][1].x, sg * acc[u][1].y);
}

}  // namespace

cudaError_t launch_phi_fp64_eval(int kernel, const double* r2, int64_t count, double* out, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((count + 255) / 256, 4096);
    phi_fp64_eval_kernel<<<(unsigned)blocks, 256, 0, st>>>(kernel, r2, count, out);
    return cudaGetLastError();
}

double cache_unit(int kernel, double ell) { return sqrt(phi_scale(kernel)) / ell; }

cudaError_t cache_factor_group(const CacheParams& cp, int64_t blk0, int g, double* A, double* Dinv,
                               float* Linv, int* bad, const OzWork* oz, cudaStream_t st, int64_t* launches) {
    const int nt = cp.nt;
    const int64_t ntri = (int64_t)nt * (nt + 1) / 2;
    const size_t smem2 = 2 * sizeof(double) * T * TP;
    cudaError_t err;
    if ((err = cudaFuncSetAttribute(potrf_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2)))
        return err;
    if ((err = cudaFuncSetAttribute(trsm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2)))
        return err;
    if ((err = cudaFuncSetAttribute(syrk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2)))
        return err;
    int64_t nl = 0;
    build_kii_kernel<<<dim3((unsigned)ntri, g), 256, 0, st>>>(cp, blk0, A);
    ++nl;
    // Look-ahead: the factorisation of the next panel's diagonal tiles (g CTAs, a serial
    // chain of 100 us) needs only the first trailing column of this panel's update.  That
    // column is updated in a launch of its own, and the diagonal tiles run on a second
    // stream beside the rest, which leaves them g SMs.  The rest takes about 10.5 us per
    // super-tile and SM; a share g / 152 of that is lost, which must stay below the chain.
    // Measured (GB300): training step on 5 blocks of 4096 34.3 -> 31.2 ms, host solve on 13
    // blocks 59.8 -> 57.3 ms; ap_set_hyper, never ahead : by this rule : always, ms: 64 blocks
    // of 256 1.11 : 1.07 : 1.09, 16 of 2048 12.5 : 10.9 : 10.9, 64 of 2048 34.3 : 33.8 : 37.0,
    // 1 of 4096 12.8 : 11.3 : 11.3, 32 of 4096 90.1 : 88.8 : 92.3, 8 of 8192 144 : 137 : 137.
    auto ahead_of = [&](int k) {
        const int64_t rem = nt - k - 1, tiles = rem * rem / 4;
        return oz && oz->side && g <= kSms / 2 && tiles * g * g < 170000;
    };
    bool factored = false;  // diagonal tiles of column k
    for (int k = 0; k < nt; ++k) {
        if (!factored) {
            potrf_diag_kernel<<<g, 256, smem2, st>>>(A, nt, k, Dinv, bad);
            ++nl;
        }
        factored = false;
        if (k + 1 == nt) break;
        if (oz) {
            const bool ahead = ahead_of(k);
            if ((err = launch_oz_trsm(A, Dinv, nt, k, g, oz->S, oz->E, oz->err, st, &nl)) != cudaSuccess) return err;
            if ((err = launch_oz_update_first(A, nt, k, g, oz->S, oz->E, oz->err, st, &nl)) != cudaSuccess) return err;
            if (ahead) {
                if ((err = cudaEventRecord(oz->ev_col, st)) != cudaSuccess) return err;
                if ((err = cudaStreamWaitEvent(oz->side, oz->ev_col, 0)) != cudaSuccess) return err;
                potrf_diag_kernel<<<g, 256, smem2, oz->side>>>(A, nt, k + 1, Dinv, bad);
                ++nl;
                if ((err = cudaEventRecord(oz->ev_diag, oz->side)) != cudaSuccess) return err;
                factored = true;
            }
            err = launch_oz_update_rest(A, nt, k, g, oz->S, oz->E, oz->err, ahead ? kSms - g : 0, st, &nl);
            // (the side stream is joined whatever happened)
            if (ahead) {
                const cudaError_t e2 = cudaStreamWaitEvent(st, oz->ev_diag, 0);
                if (err == cudaSuccess) err = e2;
            }
            if (err != cudaSuccess) return err;
        } else {
            const int rem = nt - k - 1;
            trsm_kernel<<<dim3(rem, g), 256, smem2, st>>>(A, nt, k, Dinv);
            ++nl;
            syrk_kernel<<<dim3((unsigned)((int64_t)rem * (rem + 1) / 2), g), 256, smem2, st>>>(A, nt, k);
            ++nl;
        }
    }
    pack_diag_kernel<<<dim3(nt, g), 256, 0, st>>>(Dinv, nt, blk0, ntri, Linv);
    ++nl;
    lower_to_f32_kernel<<<dim3((unsigned)ntri, g), 256, 0, st>>>(A, nt);
    ++nl;
    for (int h = 1; h < nt; h *= 2) {
        const dim3 grid((unsigned)((nt + 2 * h - 1) / (2 * h) * h * h), g);
        tri_join_kernel<false><<<grid, kTriThreads, 0, st>>>(A, nt, h, blk0, ntri, Linv);
        tri_join_kernel<true><<<grid, kTriThreads, 0, st>>>(A, nt, h, blk0, ntri, Linv);
        nl += 2;
    }
    if (launches) *launches += nl;
    return cudaGetLastError();
}

}  // namespace ap
