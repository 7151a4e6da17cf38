// Compensated FP32 form of the kernel-matrix product, used to recompute the
// residual R = B - K_hat W for refinement when the requested tolerance is
// below what plain FP32 kernel entries can certify.
//
// Every quantity is a double-float (FP32 pair): the scaled inputs carry their
// rounding remainders (x_s = hi + lo), the squared distance is summed exactly
// enough (TwoSum of the coordinate differences, TwoProd of the squares), phi
// is evaluated with the double-float exp2 / sqrt of dfloat.cuh, and the
// products with V are accumulated with TwoProd + double-float additions.  The
// entries then carry ~1e-11 relative error instead of ~3e-7.  Same grid, same
// fixed-order cluster reduction and the same epilogue as the plain form.
//
// About 22 FP32 operations per coordinate, 90 per exp2 and 15 per right-hand side bound
// it: FMA-pipe and issue slots, nothing else.  A thread works on one row and two columns
// at a time as packed FP32 pairs, which halves the instructions (the pipe does the same
// work), coordinates staged dimension by dimension so that a pair is one 8-byte read;
// squares of unnormalised differences (s + e)^2 = s^2 + e (2 s + e) and one
// renormalisation of the sum spare a quarter of the distance.  Measured (GB300,
// n = 16,384, d = 8, one column, RBF): 3.42 -> 2.61 ms for the n^2 entries,
// the same results.  A coordinate is kept twice, which takes up to 50 registers more (D = 32,
// C = 32: one CTA per SM fewer); n = 8192, RBF, us: D = 24 c = 1 2162 -> 1499, c = 32 3903 ->
// 3168; D = 32 c = 1 2519 -> 1961, c = 16 3072 -> 2999, c = 32 4569 -> 3913.
#pragma once

#include "dfloat.cuh"
#include "kmv_fp32.cuh"

namespace ap {

template <int KERN>
__device__ __forceinline__ df::P2 phi_df(df::P2 t) {
    if constexpr (KERN == AP_RBF) {
        return df::exp2_neg(t);
    } else {
        const df::P2 u = df::sqrt_df(t);
        const df::P2 e = df::exp2_neg(df::mul(u, df::P2{df::dup(df::kLog2eH), df::dup(df::kLog2eL)}));
        df::P2 poly = df::two_sum(u.h, df::dup(1.0f));
        poly = df::fast_two_sum(poly.h, df::add(poly.l, u.l));
        if constexpr (KERN == AP_MATERN52) {
            const df::P2 u2 = df::mul(u, u);
            poly = df::add(poly, df::mul(u2, df::P2{df::dup(df::kThirdH), df::dup(df::kThirdL)}));
        }
        return df::mul(poly, e);
    }
}

template <int KERN, int D, int C>
__global__ void __launch_bounds__(kKmvThreads) kmv_comp_kernel(const KmvParams p) {
    constexpr int ROWS = kCompRows;
    extern __shared__ float4 kc_smem4[];
    float* s_xh = reinterpret_cast<float*>(kc_smem4);  // kKmvTN * D
    float* s_xl = s_xh + kKmvTN * D;                  // kKmvTN * D
    float* s_v = s_xl + kKmvTN * D;                   // kKmvTN * C
    float* s_ph = s_v + kKmvTN * C;                   // ROWS * C
    float* s_pl = s_ph + ROWS * C;                    // ROWS * C
    __shared__ double red_d[32];
    __shared__ int red_i[32];
    __shared__ double s_col[kKmvThreads];
    __shared__ int s_last;

    const int tid = threadIdx.x;
    const int S = gridDim.y;
    const int rank = blockIdx.y;
    const EpiParams& e = p.epi;
    const int64_t tile = blockIdx.x;
    const int64_t seg_lo = (tile / e.tiles_per_seg) * e.seg;
    const int64_t seg_hi = min(seg_lo + e.seg, p.na);
    const int64_t r0 = seg_lo + (tile % e.tiles_per_seg) * ROWS;
    const int64_t r1 = min(r0 + (int64_t)ROWS, seg_hi);
    int64_t col0 = p.col0, ncols = p.ncols;
    if (p.sel) {
        col0 = (int64_t)(*p.sel) * p.blk;
        ncols = min(p.blk, p.nb - col0);
    }
    const int64_t cs = ((ncols + S - 1) / S + kKmvTN - 1) / kKmvTN * kKmvTN;
    const int64_t c_lo = col0 + rank * cs;
    const int64_t c_hi = min(col0 + ncols, c_lo + cs);

    const int64_t i = r0 + tid;
    const bool live = i < r1 && AP_CHK(i < p.na);
    float2 xh[D], xl[D];  // both lanes the row's coordinate
#pragma unroll
    for (int k = 0; k < D; ++k) {
        xh[k] = df::dup(live ? p.Xa[i * D + k] : 0.0f);
        xl[k] = df::dup(live ? p.Xa_lo[i * D + k] : 0.0f);
    }
    // sums over the column pairs: per right-hand side pair (C > 1), or per lane (C = 1)
    constexpr int NP = C > 1 ? C / 2 : 1;
    df::P2 acc[NP];
#pragma unroll
    for (int c = 0; c < NP; ++c) acc[c] = {df::dup(0.0f), df::dup(0.0f)};
    // acc += kv v: the product's error and the sums' go to the low part
    auto accumulate = [](df::P2& a, float2 kh, float2 nkh, float2 kl, float2 v) {
        const df::P2 pr = df::two_prod(kh, nkh, v);
        const df::P2 s2 = df::two_sum(a.h, pr.h);
        a = df::fast_two_sum(s2.h, df::add(df::add(s2.l, a.l), df::fma2(kl, v, pr.l)));
    };

    for (int64_t cb = c_lo; cb < c_hi; cb += kKmvTN) {
        const int cnt = (int)min((int64_t)kKmvTN, c_hi - cb);
        __syncthreads();
        if (AP_CHK(cb >= 0 && cb + cnt <= p.nb) && AP_CHK(cb - col0 >= 0 && cb - col0 + cnt <= ncols)) {
            for (int t = tid; t < kKmvTN * D; t += kKmvThreads) {
                const int j = t / D, k = t % D;  // dimension-major, the last column repeated
                const int64_t src = (cb + min(j, cnt - 1)) * D + k;
                s_xh[k * kKmvTN + j] = p.Xb[src];
                s_xl[k * kKmvTN + j] = p.Xb_lo[src];
            }
            for (int t = tid; t < kKmvTN * C; t += kKmvThreads) s_v[t] = t < cnt * C ? p.V[(cb - col0) * C + t] : 0.0f;
        }
        __syncthreads();
        for (int jj = 0; jj < cnt; jj += 2) {
            float2 th = df::dup(0.0f), tl = df::dup(0.0f);
#pragma unroll
            for (int k = 0; k < D; ++k) {
                const float2 bh = *reinterpret_cast<const float2*>(&s_xh[k * kKmvTN + jj]);
                const float2 bl = *reinterpret_cast<const float2*>(&s_xl[k * kKmvTN + jj]);
                // x - y = s + e exactly for the high parts, the low parts' difference added to e
                const float2 s = df::sub(xh[k], bh), ns = df::sub(bh, xh[k]);
                const float2 bb = df::sub(s, xh[k]);
                const float2 e1 = df::sub(xh[k], df::sub(s, bb));
                const float2 e = df::add(df::sub(e1, df::add(bh, bb)), df::sub(xl[k], bl));
                const df::P2 sq = df::two_prod(s, ns, s);
                const float2 r = df::fma2(e, df::fma2(df::dup(2.0f), s, e), sq.l);
                const df::P2 sum = df::two_sum(th, sq.h);
                th = sum.h;
                tl = df::add(tl, df::add(sum.l, r));
            }
            const df::P2 kv = phi_df<KERN>(df::fast_two_sum(th, tl));
            if constexpr (C == 1) {
                const float2 v = *reinterpret_cast<const float2*>(&s_v[jj]);
                accumulate(acc[0], kv.h, df::sub(df::dup(0.0f), kv.h), kv.l, v);
            } else {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const float kh1 = half ? kv.h.y : kv.h.x, kl1 = half ? kv.l.y : kv.l.x;
                    const float* vr = &s_v[(jj + half) * C];
#pragma unroll
                    for (int c = 0; c < NP; ++c)
                        accumulate(acc[c], df::dup(kh1), df::dup(-kh1), df::dup(kl1),
                                   *reinterpret_cast<const float2*>(vr + 2 * c));
                }
            }
        }
    }
    df::F2 tot[C];
    if constexpr (C == 1) {
        tot[0] = df::add(df::F2{acc[0].h.x, acc[0].l.x}, df::F2{acc[0].h.y, acc[0].l.y});
    } else {
#pragma unroll
        for (int c = 0; c < NP; ++c) {
            tot[2 * c] = {acc[c].h.x, acc[c].l.x};
            tot[2 * c + 1] = {acc[c].h.y, acc[c].l.y};
        }
    }
    __syncthreads();
    const bool diag = live && p.noise_diag && i >= c_lo && i < c_hi;
#pragma unroll
    for (int c = 0; c < C; ++c) {
        df::F2 v = df::mul_f(tot[c], p.s);
        if (diag && AP_CHK(i - col0 >= 0 && i - col0 < ncols)) v = df::add(v, df::two_prod(p.noise, p.V[(i - col0) * C + c]));
        s_ph[tid * C + c] = v.h;
        s_pl[tid * C + c] = v.l;
    }
    if (S > 1) cg::this_cluster().sync();
    else __syncthreads();
    // fixed-order reduction of the S double-float partials, then the common epilogue
    const int rpr = ROWS / S;
    double sq = 0.0, colacc = 0.0;
    for (int t = tid; t < rpr * C; t += kKmvThreads) {
        const int lr = rank * rpr + t / C;
        const int c = t % C;
        const int64_t ii = r0 + lr;
        df::F2 sum = {s_ph[lr * C + c], s_pl[lr * C + c]};
        if (S > 1) {
            cg::cluster_group cluster = cg::this_cluster();
            sum = {0.0f, 0.0f};
            for (int src = 0; src < S; ++src)
                sum = df::add(sum, df::F2{cluster.map_shared_rank(s_ph, src)[lr * C + c],
                                          cluster.map_shared_rank(s_pl, src)[lr * C + c]});
        }
        if (ii < r1 && AP_CHK(ii < p.na)) {
            const float bv = p.base ? p.base[ii * C + c] : p.base_const;
            const df::F2 o2 = df::add_f(df::F2{p.sgn * sum.h, p.sgn * sum.l}, bv);
            const float o = o2.h + o2.l;
            p.out[ii * C + c] = o;
            const double od = (double)o;
            sq += od * od;
            colacc += od * od;
        }
    }
    if (e.flags & kEpiBlockNorms) {
        double tot = cta_sum_d(sq, red_d);
        if (tid == 0 && AP_CHK(tile * S + rank < e.ntiles * e.S)) e.part_norm[tile * S + rank] = tot;
    }
    if (e.flags & kEpiColNorms) {
        __syncthreads();
        s_col[tid] = colacc;
        __syncthreads();
        if (tid < C) {
            double a = 0.0;
            for (int k = tid; k < kKmvThreads; k += C) a += s_col[k];
            if (AP_CHK(tile * S + rank < e.ntiles * e.S)) e.part_col[(tile * S + rank) * C + tid] = a;
        }
    }
    if (S > 1) cg::this_cluster().sync();
    epi_ticket<C>(e, red_d, red_i, &s_last, s_col);
}

template <int KERN, int D, int C>
cudaError_t launch_kmv_comp_inst(const KmvParams& p, cudaStream_t st) {
    const size_t smem = sizeof(float) * ((size_t)kKmvTN * (2 * D + C) + (size_t)2 * kCompRows * C);
    auto fn = kmv_comp_kernel<KERN, D, C>;
    cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    const int S = p.epi.S;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.epi.ntiles, (unsigned)S, 1);
    cfg.blockDim = dim3(kKmvThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (S > 1) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = (unsigned)S;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelEx(&cfg, fn, p);
}

template <int KERN>
cudaError_t dispatch_kmv_comp(const KmvParams& p, int D, int C, cudaStream_t st) {
#define AP_KMVC_C(DD)                                                       \
    switch (C) {                                                            \
        case 1: return launch_kmv_comp_inst<KERN, DD, 1>(p, st);            \
        case 4: return launch_kmv_comp_inst<KERN, DD, 4>(p, st);            \
        case 16: return launch_kmv_comp_inst<KERN, DD, 16>(p, st);          \
        case 32: return launch_kmv_comp_inst<KERN, DD, 32>(p, st);          \
        default: return cudaErrorInvalidValue;                              \
    }
    switch (D) {
        case 4: AP_KMVC_C(4)
        case 8: AP_KMVC_C(8)
        case 12: AP_KMVC_C(12)
        case 16: AP_KMVC_C(16)
        case 24: AP_KMVC_C(24)
        case 32: AP_KMVC_C(32)
        default: return cudaErrorInvalidValue;
    }
#undef AP_KMVC_C
}

}  // namespace ap
