// Internal declarations shared by the CUDA translation units of libap.so.
// Nothing here is part of the public ABI (include/ap.h is).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/ap.h"

namespace ap {

// Bounds-checked build (compiled with -DAP_CHECKED into a separate library):
// AP_CHK(cond) guards an index before the access it protects.  A failing check
// records its source line in a device word of its translation unit (the first
// one wins) and yields false, so that the caller skips the access instead of
// faulting; ap_bounds_violations reads and clears the words of every unit.  In
// the product build AP_CHK(cond) is `true` and compiles away.
#ifdef AP_CHECKED
namespace {
__device__ unsigned int g_chk_line;  // one per translation unit
}
#define AP_CHK(cond) ((cond) ? true : (atomicCAS(&g_chk_line, 0u, (unsigned int)__LINE__), false))
// Host registry of the per-unit words (defined in ap_api.cu).
int chk_register(const char* unit, unsigned int (*read_and_clear)());
namespace {
unsigned int chk_read_and_clear() {
    unsigned int v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_chk_line, sizeof v) != cudaSuccess) return 0;
    cudaMemcpyToSymbol(g_chk_line, &zero, sizeof zero);
    return v;
}
const int g_chk_registered = chk_register(__BASE_FILE__, &chk_read_and_clear);
}  // namespace
#else
#define AP_CHK(cond) true
#endif

constexpr int kTile = 64;           // tile edge of the block-Cholesky cache
constexpr int kKmvThreads = 128;    // threads per CTA of the kernel-matrix products
constexpr int kKmvTN = 64;          // columns staged per shared-memory chunk
constexpr int kMaxSplit = 8;        // portable thread-block-cluster size

// Programmatic dependent launch between the kernels of an AP step: a kernel launched
// with launch_dependent may start once every CTA of the kernel before has passed its
// pdl_launch (or ended); what that kernel writes is read after pdl_wait.  Every kernel
// of the chain waits before it lets its successor go, so that anything a kernel two
// places back wrote is complete and visible from the start.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename P>
cudaError_t launch_dependent(void (*fn)(P), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, bool dependent,
                             const P& p, unsigned cluster_y = 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (dependent) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster_y > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = 1;
        attr[n].val.clusterDim.y = cluster_y;
        attr[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, fn, p);
}

// flags of the kernel-matrix product epilogue
constexpr int kEpiBlockNorms = 1;   // per-block ||R_J||_F^2 partials + block selection
constexpr int kEpiColNorms = 2;     // per-column ||R_:,c||^2 partials

// Scale applied to x / l so that the FP32 kernels evaluate phi with one ex2:
//   RBF:  |x_s - x_s'|^2 = r^2 log2(e) / 2          -> phi = 2^(-|.|^2)
//   M32:  |x_s - x_s'|   = sqrt(3) r = u             -> phi = (1 + u) 2^(-u log2 e)
//   M52:  |x_s - x_s'|   = sqrt(5) r = u             -> phi = (1 + u + u^2/3) 2^(-u log2 e)
double kernel_input_scale(int kernel);

// Epilogue bookkeeping of one AP step (block norms, selection, column norms).
struct EpiParams {
    int flags;
    int advance;            // 1: a step finished (step_ctr += 1) before selecting
    int64_t seg;            // rows per AP block b (tiles never straddle a block)
    int64_t tiles_per_seg;  // CTA row tiles per block
    int64_t ntiles;         // row tiles in the grid (y dimension)
    int S;                  // CTAs per row tile (cluster size, x dimension)
    int m;                  // number of blocks
    double* part_norm;      // [ntiles * S]
    double* part_col;       // [ntiles * S * C]
    unsigned int* ticket;   // last-CTA counter, left at 0 after each launch
    double* norms_out;      // [m]   block norms after the step
    double* colnorm_out;    // [C]   column norms (when kEpiColNorms)
    int select;             // ap_select
    uint64_t seed;
    int64_t* step_ctr;      // steps completed (device)
    int* sel_out;           // block chosen for the next step (device)
    int* nan_flag;          // set to 1 when a norm is not finite
};

// out[i,:] = base[i,:] + sgn * s * sum_j phi(xa_i, xb_j) V[j - col0, :]
//            + sgn * noise * V[i - col0, :]   (if noise_diag and col0 <= i < col0 + ncols)
struct KmvParams {
    const float* Xa;       // na x D scaled rows
    int64_t na;
    const float* Xb;       // nb x D scaled columns
    int64_t nb;
    const float* V;        // ncols x C
    const float* base;     // na x C or nullptr (then base_const)
    float base_const;
    float* out;            // na x C (may alias base)
    float sgn;
    float s;
    float noise;
    int noise_diag;
    int64_t col0, ncols;   // column range when sel == nullptr
    const int* sel;        // device block index: col0 = sel*blk, ncols = min(blk, nb - col0)
    int64_t blk;
    const float* Xa_lo;    // compensated form only: low parts of the scaled inputs
    const float* Xb_lo;
    bool x3;               // the tensor-core form (KmvSplit)
    int rm;                // rows per thread (KmvSplit)
    int G;                 // > 1: row tiles are shared between CTAs through gscr (KmvSplit)
    int ctas;              // CTAs of the tensor-core form's persistent grid (KmvSplit)
    float* gscr;           // G > 1: partial sums (KmvSplit::scratch floats)
    unsigned int* gtick;   // G > 1: arrival tickets (KmvSplit::tickets), zero between launches
    int* err;              // wait-timeout flag of the tensor-core form
    long long wait_cycles; // bound of its copy issuer's waits (<= 0: the default, about 2 s)
    bool dependent;        // launch without waiting for the kernel before (launch_dependent)
    EpiParams epi;
};

// How one FP32 product is cut into CTAs: row tiles of 128 * rm rows (never across a
// segment).  SIMT form (C <= 4): S column splits per tile summed inside a cluster, G
// groups of S splits summed through global memory by the last group to arrive.
// Tensor-core form: a persistent grid over (tile, column chunk) units; G > 1 lets a
// range of units end inside a tile.
struct KmvSplit {
    bool x3;  // the tensor-core form
    int rm, S, G, ctas;
    int64_t rows, tps, ntiles;
    int64_t scratch;  // floats of partial sums when G > 1
    int64_t tickets;  // arrival tickets when G > 1
};
KmvSplit kmv_split(int D, int C, int64_t seg, int64_t nseg, int64_t ncols);
constexpr int kX3MinC = 16;  // right-hand sides (padded) from which the tensor-core form exists
// Entries of a product from which the tensor-core form runs, 16 and 32 right-hand sides: it
// has some 12 us more of start-up (tensor memory, splitting and draining the first chunk,
// the hand-over of shared row groups), the SIMT form the slope of its FP32 contraction.
// Measured at d = 8, Matern-3/2 (GB300, us per ap_residual call R or step, SIMT : tensor
// cores; rows x columns).  16: R 3000^2 60 : 69, 4096^2 68 : 75, 4500^2 73 : 80; 8000 x 1000
// 46 : 52, 8000 x 2000 66 : 68, 6000 x 3000 82 : 81, 24,000 x 1000 75 : 67, 12,000 x 2000 79 :
// 75.  32: R 2048^2 65 : 68, 2500^2 72 : 80, 3300^2 82 : 82, 3600^2 88 : 81; 6000 x 1000 58 : 64,
// 8000 x 1000 67 : 65, 12,000 x 512 66 : 69, 16,000 x 512 73 : 57, 12,000 x 1000 83 : 67.
constexpr double kX3MinEntries16 = 2.2e7, kX3MinEntries32 = 8e6;
// Largest D with two rows per thread (beyond, their coordinates do not fit the registers).
// One row : two, n = 32,768, Matern-3/2, c = 16, us: D = 4 890 : 808, 8 1143 : 1033, 12 1434 :
// 1315, 16 1687 : 1518, although the two-row instances spill some registers; one row against
// the SIMT form: D = 24 2305 : 2968, 32 3004 : 3517 (c = 32 2430 : 3937, 3130 : 4500).
constexpr int kX3MaxD2 = 16;
constexpr int kX3Chunk = 128;

// FP32 SIMT kernel-matrix product with the AP epilogue (one per kernel family TU).
cudaError_t launch_kmv_rbf(const KmvParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_kmv_m32(const KmvParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_kmv_m52(const KmvParams& p, int D, int C, cudaStream_t st);
// The same product for C >= kX3MinC with the contraction on the tensor cores (kmv_x3.cuh).
cudaError_t launch_x3_rbf(const KmvParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_x3_m32(const KmvParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_x3_m52(const KmvParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_kmv(int kernel, const KmvParams& p, int D, int C, cudaStream_t st);
// Compensated (double-float FP32) form of the same product, for refinement.
cudaError_t launch_kmv_comp_rbf(const KmvParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_kmv_comp_m32(const KmvParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_kmv_comp_m52(const KmvParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_kmv_comp(int kernel, const KmvParams& p, int D, int C, cudaStream_t st);
constexpr int kCompRows = 128;  // rows per CTA of the compensated product

// Norms of R alone (n x C) + selection: used before the first step and after refinement.
cudaError_t launch_norms_select(const float* R, int64_t n, int C, const EpiParams& e,
                                int64_t tile_rows, cudaStream_t st);

// ---- block-Cholesky cache (FP64 factorisation, FP32 inverse factor) --------
struct CacheParams {
    const float* X;        // n x d, original inputs
    int64_t n;
    int d;
    int kernel;
    double unit[AP_MAX_DIM];  // cache_unit per dimension
    double s, noise;
    int64_t b;             // block size
    int nt;                // tiles per block edge = ceil(b / kTile)
};

// Factor blocks [blk0, blk0 + g) into the packed FP32 inverse factors Linv.
// A (g * (nt*64)^2 doubles) and Dinv (g * nt * 64^2 doubles) are work buffers.
// bad (g ints) gets 1 for a block whose factorisation met a non-positive pivot.
// Tensor-core panel solves and trailing updates with FP64 results (ozaki.cu): slice planes of
// oz_slice_bytes(nt) bytes and oz_expo_ints(nt) row exponents per block.
size_t oz_slice_bytes(int nt);
size_t oz_expo_ints(int nt);
// The trailing update of panel k in two parts: the panel's slices and the first trailing
// column of tiles, then the remaining columns on `ctas` CTAs (0: one per SM).
cudaError_t launch_oz_update_first(double* A, int nt, int k, int g, uint8_t* S, int* E, int* err, cudaStream_t st,
                                   int64_t* launches);
cudaError_t launch_oz_update_rest(double* A, int nt, int k, int g, uint8_t* S, int* E, int* err, int ctas,
                                  cudaStream_t st, int64_t* launches);
// The panel solve A_ik := A_ik L_kk^{-T} (i > k) the same way, L_kk^{-1} from Dinv.
cudaError_t launch_oz_trsm(double* A, const double* Dinv, int nt, int k, int g, uint8_t* S, int* E, int* err,
                           cudaStream_t st, int64_t* launches);
// Work buffers of the tensor-core panel solves and trailing updates; null = FP64 FMA.
struct OzWork {
    uint8_t* S;  // g * oz_slice_bytes(nt)
    int* E;      // g * oz_expo_ints(nt)
    int* err;    // wait-timeout flag
    cudaStream_t side;           // the next diagonal tiles are factored here meanwhile
    cudaEvent_t ev_col, ev_diag; // first trailing column updated; next diagonal tiles factored
};
// FP64 phi of the cache build at count squared distances (device arrays).
cudaError_t launch_phi_fp64_eval(int kernel, const double* r2, int64_t count, double* out, cudaStream_t st);
// Scale of a coordinate such that the squared distance is phi's argument in the cache.
double cache_unit(int kernel, double ell);
cudaError_t cache_factor_group(const CacheParams& cp, int64_t blk0, int g, double* A, double* Dinv,
                               float* Linv, int* bad, const OzWork* oz, cudaStream_t st, int64_t* launches);

// ---- block solve: Delta = L^-T L^-1 R_I, W_I += Delta -----------------------
struct SolveParams {
    const float* Linv;     // packed inverse factors of all blocks
    int64_t n, b;
    int nt;
    int C;
    const float* R;        // n x C
    float* W;              // n x C
    float* Z;              // nt*64 x C work
    float* Delta;          // b x C (rows >= b_I are written as 0)
    const int* sel;
    const int64_t* step_ctr;
    int* trace;            // device trace or nullptr
    int64_t trace_cap;
    int tpc;               // tiles per CTA (block_solve_layout)
    int maxj;              // partial slots per output row of tiles
    float* spart;          // nt * maxj * 64 * C floats of partial sums
    unsigned* sticket;     // nt tickets, zero between launches
    uint8_t* DT;           // tensor-core form: operand layout of Delta to fill too, or nullptr
    bool dependent;        // launch without waiting for the kernel before (launch_dependent)
};
// Work split of the block solve for nt tiles per block edge and C right-hand sides.
void block_solve_layout(int nt, int C, int num_sms, int* tpc, int* maxj);
int64_t block_solve_ctas(int nt, int tpc);
cudaError_t launch_block_solve(const SolveParams& p, cudaStream_t st, int64_t* launches);

// ---- small helpers ----------------------------------------------------------
// Xs = fl(X * sc) with sc = sc_hi + sc_lo per dimension; Xs_lo (may be null)
// gets the remainder X * sc - Xs to FP32 precision.
cudaError_t launch_prep_inputs(const float* X, int64_t n, int d, int D, const float* sc_hi, const float* sc_lo,
                               float* Xs, float* Xs_lo, int* bad, cudaStream_t st);
cudaError_t launch_init_solve(const float* B, const float* W0, int64_t n, int c, int C, float* Bp, float* R, float* W,
                              float* W_ckpt, cudaStream_t st);
cudaError_t launch_pad_copy(const float* src, int64_t n, int c, float* dst, int C, cudaStream_t st);
cudaError_t launch_unpad_copy(const float* src, int64_t n, int C, float* dst, int c, cudaStream_t st);

// ---- derivative quadratic forms (Eq. loss_grad_unbiased) ------------------
// Accumulates, over all pairs (i, j), G_ij = sum_c alpha_c U_ic V_jc times
//   out[k]     (k < D): G_ij psi(t_ij) (xs_ik - xs_jk)^2   (lengthscale terms)
//   out[D]:            G_ij phi(t_ij)                      (outputscale term)
//   out[D + 1]:        G_ii                                 (noise term)
// with the pre-scaled inputs xs of the FP32 product; the host turns these
// into dK/dtheta quadratic forms.
struct GradParams {
    const float* Xs;       // n x D scaled inputs
    int64_t n;
    const float* U;        // n x C
    const float* V;        // n x C
    float alpha[AP_MAX_RHS];
    double* part;          // [kGradCtas * (D + 2)]
    unsigned int* ticket;  // zero between launches
    double* out;           // D + 2
    int* err;              // wait-timeout flag
    long long wait_cycles; // bound of the copy issuer's waits (<= 0: the default, about 2 s)
};
constexpr int kGradCtas = 152;  // persistent grid: one CTA per SM
cudaError_t launch_grad(int kernel, const GradParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_grad_rbf(const GradParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_grad_m32(const GradParams& p, int D, int C, cudaStream_t st);
cudaError_t launch_grad_m52(const GradParams& p, int D, int C, cudaStream_t st);

// B = [y - mu, z_1..z_l]; Z == nullptr draws Rademacher z from SplitMix64(seed);
// Zout (may be nullptr) receives the z actually used.
cudaError_t launch_assemble_rhs(const float* y, float mu, const float* Z, int l, uint64_t seed, int64_t n,
                                float* B, float* Zout, cudaStream_t st);
// V = [W[:,0], B[:,1..c)] padded to C columns.
cudaError_t launch_assemble_v(const float* W, int C, const float* B, int c, int64_t n, float* V, cudaStream_t st);
// out = sum_i W[i*C] * (Y ? Y[i*cy] : 1) in FP64; part needs 256 doubles.
cudaError_t launch_dot0(const float* W, int C, const float* Y, int cy, int64_t n, double* part, unsigned* ticket,
                       double* out, cudaStream_t st);

// ---- tensor-core form of the residual update (kmv_tc.cu) -------------------
constexpr int kTcChunk = 128;  // columns of the block per chunk
// One value of Delta^T in the contraction's operand layout: per 128-column chunk C rows
// (right-hand sides) x 128 columns (block-local points) as BF16 hi, then lo, K-major core
// matrices of 8 rows x 8 halves (16 K-cores per row group).
__device__ __forceinline__ void tc_store_delta(uint8_t* DT, int C, int64_t li, int c, float v) {
    const int k = (int)(li % kTcChunk);
    const size_t half_bytes = (size_t)C * kTcChunk * 2;
    uint8_t* dst = DT + (size_t)(li / kTcChunk) * 2 * half_bytes +
                   ((size_t)((c >> 3) * (kTcChunk / 8) + (k >> 3)) * 8 + (c & 7)) * 16 + (size_t)(k & 7) * 2;
    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
    *reinterpret_cast<__nv_bfloat16*>(dst) = hi;
    *reinterpret_cast<__nv_bfloat16*>(dst + half_bytes) = __float2bfloat16_rn(v - __bfloat162float(hi));
}
struct TcParams;
int tc_kd(int d);
int tc_chunks_per_block(int64_t b);
size_t tc_rows_bytes(int64_t ntiles, int kd);
size_t tc_cols_bytes(int64_t m, int cpb, int kd);
size_t tc_delta_bytes(int cpb, int C);
cudaError_t launch_tc_pack_inputs(int kernel, const float* Xs, int64_t n, int d, int D, int64_t b, int64_t m,
                                  int64_t tps, int cpb, int kd, uint8_t* XA, uint8_t* XB, cudaStream_t st);
struct TcLaunch {
    const uint8_t* XA;
    const uint8_t* XB;
    const uint8_t* DT;
    const float* Delta;
    float* R;
    int64_t n, b;
    int cpb;
    float s, noise;
    const int* sel;
    int* err;
    long long wait_cycles;  // bound of the kernel's waits (<= 0: the default, about 2 s)
    float* scr;  // grid x 2 x 128 x C floats (tc_share_bytes)
    int* tick;   // grid ints, zero
    EpiParams epi;
};
// Boundary slots of the tensor-core update for a grid of CTAs and C right-hand sides.
size_t tc_share_bytes(int grid, int C);
cudaError_t launch_kmv_tc_step(int kernel, const TcLaunch& l, int kd, int C, int grid, cudaStream_t st);

// Makes the context's device current for one call and restores the caller's.
class DeviceGuard {
   public:
    explicit DeviceGuard(int dev) {
        ok_ = cudaGetDevice(&prev_) == cudaSuccess;
        if (ok_ && prev_ != dev) ok_ = cudaSetDevice(dev) == cudaSuccess, switched_ = ok_;
        if (!ok_) cudaGetLastError();
    }
    ~DeviceGuard() {
        if (switched_) cudaSetDevice(prev_);
    }
    bool ok() const { return ok_; }

   private:
    int prev_ = 0;
    bool ok_ = false, switched_ = false;
};

// Read-only view of what the gradient kernel needs from a context.
struct GradView {
    int device;           // the context's device
    const float* Xs;
    int64_t n;
    int d, D, kernel;
    float s;
    const float* ell;
    cudaStream_t stream;  // the caller's stream of the context
    long long wait_cycles;
};
void ctx_grad_view(const ap_ctx* ctx, GradView* v);
// Turn the raw D + 2 sums of the gradient kernel into the d + 2 quadratic forms.
void grad_finish(const GradView& v, const double* raw, double* out_host);

}  // namespace ap
