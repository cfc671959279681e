// gwns_slice.cuh -- the per-candidate likelihood and the slice-sampling
// update (paper Sec. 2) as templates over precision and detector count. Each
// gwns_inst_p<P>_d<D>.cu translation unit instantiates one (precision,
// detectors) pair, so the kernels compile in parallel.
#pragma once
#include "gwns_kernels.cuh"

namespace gwns {

// The warp sums of one candidate's double-float sums zh/zl[d][re, im] by the
// transposing butterfly (warp_sum_df_many; lanes 2v hold value v = 2 d + re/im),
// written as doubles to out[v] (2 NDET entries), times the detector's data scale
// where there is one.
template <int NDET>
__device__ __forceinline__ void warp_sums_df_to(const float (&zh)[NDET][2], const float (&zl)[NDET][2],
                                                double *out, const double *scale = nullptr) {
    const int lane = threadIdx.x & 31;
    float vh[16], vl[16];
#pragma unroll
    for (int d = 0; d < NDET; d++)
#pragma unroll
        for (int ri = 0; ri < 2; ri++) { vh[2 * d + ri] = zh[d][ri]; vl[2 * d + ri] = zl[d][ri]; }
    float rh, rl;
    warp_sum_df_many<2 * NDET>(vh, vl, rh, rl);
    const int v = lane >> 1;
    if ((lane & 1) == 0 && v < 2 * NDET) {
        const double z = (double)rh + (double)rl;
        out[v] = scale ? z * __ldg(scale + (v >> 1)) : z;
    }
}

// The same sums combined with G_d: returns sum_d (Re G_d Re Z_d - gim_d Im Z_d)
// on lane 0 (the detector terms of log L), from the transposed warp sums: the
// lane holding value v multiplies it by its factor, then lanes 0, 2, .., 14 add.
template <int NDET>
__device__ __forceinline__ double warp_detector_terms_df(const float (&zh)[NDET][2], const float (&zl)[NDET][2],
                                                         const Coef &c, const double *scale = nullptr) {
    const int lane = threadIdx.x & 31;
    float vh[16], vl[16];
#pragma unroll
    for (int d = 0; d < NDET; d++)
#pragma unroll
        for (int ri = 0; ri < 2; ri++) { vh[2 * d + ri] = zh[d][ri]; vl[2 * d + ri] = zl[d][ri]; }
    float rh, rl;
    warp_sum_df_many<2 * NDET>(vh, vl, rh, rl);
    const int v = lane >> 1, dd = v >> 1;
    double t = 0.0;
    if ((lane & 1) == 0 && v < 2 * NDET) {
        double z = (double)rh + (double)rl;
        if (scale) z *= __ldg(scale + dd);
        t = (v & 1) ? -c.gim[dd] * z : c.gre[dd] * z;
    }
#pragma unroll
    for (int o = 2; o < 16; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Coefficients of one point from warp 0 (shared), then all warps run the bin
// loop and the CTA reduces Z_d. Returns log L in *lval (shared) after the
// second barrier; every thread of the CTA must call it.
template <int PREC, int NDET, int W>
__device__ __forceinline__ void cta_loglike_bins(const Model &M, const Tables &T, Coef &coef, CoefMixed &cm,
                                                 const FxPoint &fx, const float4 *sc, double (*red)[2 * MAXDET],
                                                 double *lval) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (M.model == M_TOY) {
        if (threadIdx.x == 0) *lval = coef.toy;
        return;
    }
    if (PREC == 0) {
        float zh[NDET][2], zl[NDET][2];
        bins_fx<NDET>(T, fx, sc, threadIdx.x, W * 32, zh, zl);
        warp_sums_df_to<NDET>(zh, zl, red[warp], T.fxs);
    } else if (M.tlg) {
        // tiled form: warp w takes tile groups w, w + W, ...
        float zh[NDET][2], zl[NDET][2];
        if (M.tlg >= 5)
            tile_bins<NDET, true, true, true>(T, M.tlg, M.np, cm, coef.jcut, warp, W, zh, zl);
        else
            tile_bins<NDET, false>(T, M.tlg, M.np, cm, coef.jcut, warp, W, zh, zl);
        warp_sums_df_to<NDET>(zh, zl, red[warp]);
    } else {
        float zh[NDET][2], zl[NDET][2];
        bins_mixed<NDET>(T, M.N, cm, coef.jcut, threadIdx.x, W * 32, zh, zl);
        warp_sums_df_to<NDET>(zh, zl, red[warp]);
    }
    __syncthreads();
    if (warp == 0) {
        double v = 0.0;
        if (lane < NDET) {
            double ZR = 0.0, ZI = 0.0;
            for (int w = 0; w < W; w++) { ZR += red[w][2 * lane]; ZI += red[w][2 * lane + 1]; }
            v = coef.gre[lane] * ZR - coef.gim[lane] * ZI;
        }
        v = warp_sum(v);
        if (lane == 0) *lval = v - 0.5 * coef.hh;
    }
}

// Warp 0 computes the coefficients of the point with unit-cube coordinates u
// (or physical parameters theta when in_is_theta).
__device__ __forceinline__ void warp_point_coef(const Model &M, const Tables &T, const double *in,
                                                int in_is_theta, int precision, Coef *coef,
                                                CoefMixed *cm, FxPoint *fx) {
    if (M.model == M_TOY) {
        point_coef_warp(M, T, in, coef);
        return;
    }
    if (precision == 1 && M.cdf && !in_is_theta) {
        point_coef_group_mx(M, T, in, 0, coef, cm, 1, M.tlg >= 5);
        return;
    }
    if (in_is_theta) {
        // a model whose parameters are all FIXED at theta
        Model Mt = M;
#pragma unroll
        for (int p = 0; p < NPARAM; p++) { Mt.kind[p] = K_FIXED; Mt.lo[p] = in[p]; }
        point_coef_warp(Mt, T, in, coef);
    } else {
        point_coef_warp(M, T, in, coef);
    }
    __syncwarp();
    if (precision == 1) coef_to_mixed_warp(*coef, M.n_det, M.df, cm, M.rb ? T.rb.fid : nullptr, M.tlg >= 5);
    else coef_to_fx_group(T, M.n_det, coef, fx, 1, M.rb ? T.rb.fid : nullptr);
}

// Points per CTA of the batched likelihood: the coefficient stage packs up to
// four points into one warp pass (8 lanes each), so the per-point FP64 work that
// binds the mixed form on grids of a few thousand bins is shared. GB300, 8192
// prior draws of the 64,897-bin workload: 4.0e7 -> 5.9e7 evals/s. Where the
// bins bind (the FP64 form; 519,169 bins) the coarser grid of CTAs cost 4-9%,
// and there, as for physical-parameter and toy inputs, a CTA takes one point.
constexpr int EVAL_PPC = 4;

// CTAs per SM that the batched likelihood's kernels are compiled for. Left alone,
// the compiler settled on 56 to 106 registers, by whatever else the kernel held, and
// kept too few of the tile loop's loads and chains in flight; 16 warps an SM at 128
// registers (fewer registers with one detector, whose tile loop needs less) is
// faster on every grid in tiles of 32 bins or more. GB300, 100 / 8192 draws, before ->
// now: 3 detectors, 104,000 bins 656 / 1633 -> 478 / 1558 us, 519,169 bins 232 / 4056 ->
// 200 / 3991; 2 detectors, 31,489 bins 250 / 604 -> 162 / 500; 1 detector, 129,793
// bins 487 / 1256 -> 387 / 1147. The kernels' other calls, left alone -> so, 8192 draws,
// 3 detectors: shorter tiles (16,225 / 32,449 bins) 97 / 132 -> 78 / 99 us, bin by bin
// (4017) 74 -> 62, physical parameters (4017 / 32,449 bins) 326 / 718 -> 207 / 406,
// relative binning 525 -> 327; 64 draws of any of them lose up to 2 us. One detector in
// CTAs of 4 warps: 5 of them, 4017 bins 8192 draws 55.7 us (4: 58.5, 6: 56.9, left alone
// 61.2). Four detectors' tile loop on tiles of 32 bins or
// more wants 3 CTAs of 4 warps (EVAL_BATCH4_BLOCKS): at 4 its registers spill, 32 s
// (64,897 bins) 64 / 8192 draws 56 / 121 -> 49 / 118 us, 64 s of low masses 720 / 2124 ->
// 486 / 1927; on shorter tiles 4 stay better (4017 bins, 8192 draws 71 -> 66).
#define EVAL_BATCH4_BLOCKS 3
#define EVAL_BATCH_BLOCKS(NDET, W) ((NDET) == 1 ? ((W) == 4 ? 5 : 32 / (W)) : 16 / (W))
#define EVAL_BLOCKS(PREC, NDET, W) ((PREC) == 0 ? 16 / (W) : (NDET) == 1 ? 32 / (W) : (NDET) == 2 ? 20 / (W) : 16 / (W))

template <int PREC, int NDET, int W>
__global__ void __launch_bounds__(W * 32, EVAL_BLOCKS(PREC, NDET, W)) k_eval(Model M, Tables T, const double *in, int in_is_theta,
                                                 int m, int ppc, double *logl, RunState *st) {
    __shared__ Coef coef[EVAL_PPC];
    __shared__ CoefMixed cm[EVAL_PPC];
    __shared__ double red[W][2 * MAXDET];
    __shared__ double lval;
    __shared__ double pt[EVAL_PPC][NPARAM + MAXD];
    __shared__ FxPoint fx;
    __shared__ float4 sc[PREC == 0 ? FX_SC : 1];
    const int i0 = blockIdx.x * ppc;
    if (i0 >= m) return;
    if (PREC == 0 && M.model == M_GW) load_sc(T, sc);
    const int np = m - i0 < ppc ? m - i0 : ppc;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int stride_in = in_is_theta ? NPARAM : M.dim;
    for (int t = threadIdx.x; t < np * stride_in; t += W * 32)
        pt[t / stride_in][t % stride_in] = in[(size_t)i0 * stride_in + t];
    __syncthreads();
    if (warp == 0) {
        if (ppc == 1) {
            warp_point_coef(M, T, pt[0], in_is_theta, PREC, &coef[0], &cm[0], &fx);
        } else {
            point_coef_group(M, T, pt[0], NPARAM + MAXD, coef, np);
            __syncwarp();
            if (PREC == 1)
                for (int p = 0; p < np; p++)
                    coef_to_mixed_warp(coef[p], M.n_det, M.df, &cm[p], M.rb ? T.rb.fid : nullptr, M.tlg >= 5);
        }
    }
    __syncthreads();
    for (int p = 0; p < np; p++) {
        if (M.rb) {
            // relative-binning sums: one warp
            if (warp == 0) {
                const double v = PREC == 0 ? rb_loglike_fx<NDET>(M, T, coef[p], fx, sc)
                                           : rb_loglike_mixed<NDET>(M, T.rb, coef[p], cm[p], lane);
                if (lane == 0) {
                    logl[i0 + p] = v;
                    if (st) atomicAdd(&st->eval_points, 1ull);
                }
            }
            continue;
        }
        cta_loglike_bins<PREC, NDET, W>(M, T, coef[p], cm[p], fx, sc, red, &lval);
        if (threadIdx.x == 0) {
            logl[i0 + p] = lval;
            if (st) {
                atomicAdd(&st->eval_points, 1ull);
                if (M.model != M_TOY) {
                    atomicAdd(&st->eval_point_bins, (unsigned long long)(coef[p].jcut + 1));
                    // the rotation form here sums the groups from T.g_lo at the low Taylor degree
                    if (PREC == 1 && M.tlg >= 5) {
                        const long long lo = (long long)coef[p].jcut + 1 - ((long long)T.g_lo << (M.tlg + 5));
                        if (lo > 0) atomicAdd(&st->eval_point_bins_lo, (unsigned long long)lo);
                    }
                }
            }
        }
        __syncthreads();    // red and lval serve the next point
    }
}

// Batched likelihood, mixed precision, unit-cube points on grids of up to
// 262,144 bins (where the per-point FP64 work weighs most): 4 max(1, W/2)
// points per CTA. The coefficient stage runs as its two halves on two warps per
// group of four points (mass and phase on one, sky and detectors on the other,
// independent FP64 chains on two SM sub-partitions), joined by the first; then
// each point's bins are summed by one warp (points dealt to the warps in turn),
// reduced in double-float, and only the final log L is formed in FP64. GB300,
// 8192 prior draws of the 64,897-bin workload: the previous kernel (coefficients
// of four points on one warp, the other warp waiting, every point's tile groups
// shared by both warps and reduced in FP64) reached 5.75e7 evals/s.
template <int NDET, int W, int BLOCKS = EVAL_BATCH_BLOCKS(NDET, W)>
__global__ void __launch_bounds__(W * 32, BLOCKS) k_eval_batch(Model M, Tables T, const double *in, int m, double *logl,
                                                               RunState *st) {
    constexpr int NG = W >= 2 ? W / 2 : 1;
    constexpr int PPC = 4 * NG;
    __shared__ Coef coef[PPC];
    __shared__ CoefMixed cm[PPC];
    __shared__ double pt[PPC][MAXD];
    const int i0 = blockIdx.x * PPC;
    if (i0 >= m) return;
    const int np = m - i0 < PPC ? m - i0 : PPC;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int d = M.dim;
    for (int t = threadIdx.x; t < np * d; t += W * 32) pt[t / d][t % d] = in[(size_t)i0 * d + t];
    __syncthreads();
    const int grp = W >= 2 ? warp >> 1 : warp;
    const bool lead = W >= 2 ? (warp & 1) == 0 : true;
    const int cnt = (grp < NG && 4 * grp < np) ? min(4, np - 4 * grp) : 0;
    if (cnt > 0) {
        if (M.cdf)
            point_coef_group_mx(M, T, pt[4 * grp], MAXD, &coef[4 * grp], &cm[4 * grp], cnt, M.tlg >= 5,
                                W >= 2 ? 1 + (warp & 1) : 0);
        else
            point_coef_group(M, T, pt[4 * grp], MAXD, &coef[4 * grp], cnt, W >= 2 ? 1 + (warp & 1) : 0);
    }
    __syncthreads();
    if (cnt > 0 && lead) {
        if (W >= 2) point_coef_join(M, T, &coef[4 * grp], cnt);
        __syncwarp();
        if (!M.cdf)
            for (int p = 4 * grp; p < 4 * grp + cnt; p++)
                coef_to_mixed_warp(coef[p], M.n_det, M.df, &cm[p], nullptr, M.tlg >= 5);
    }
    __syncthreads();
    unsigned long long n_pts = 0, n_pb = 0;     // this warp's counts, added once at the end
    for (int p = warp; p < np; p += W) {
        double t;       // on lane 0: sum over detectors of Re(G_d Z_d)
        if (M.tlg) {
            float zh[NDET][2], zl[NDET][2];
            if (M.tlg >= 5)
                tile_bins<NDET, true, true>(T, M.tlg, M.np, cm[p], coef[p].jcut, 0, 1, zh, zl);
            else
                tile_bins<NDET, false>(T, M.tlg, M.np, cm[p], coef[p].jcut, 0, 1, zh, zl);
            t = warp_detector_terms_df<NDET>(zh, zl, coef[p]);
        } else {
            float zh[NDET][2], zl[NDET][2];
            bins_mixed<NDET>(T, M.N, cm[p], coef[p].jcut, lane, 32, zh, zl);
            t = warp_detector_terms_df<NDET>(zh, zl, coef[p]);
        }
        if (lane == 0) {
            const double v = t - 0.5 * coef[p].hh;
            logl[i0 + p] = v;
            n_pts++;
            n_pb += (unsigned long long)(coef[p].jcut + 1);
        }
    }
    if (st && lane == 0 && n_pts) {
        atomicAdd(&st->eval_points, n_pts);
        atomicAdd(&st->eval_point_bins, n_pb);
    }
}

// Batched likelihood, FP64, unit-cube points: the CTA's warps take as many points
// at most. The coefficient stage, bound by the FP64 pipe and its latency (about 250 dependent
// instructions for up to four points in a warp's lane groups), runs as its two
// halves on two warps per four points; then the warps share the P C items
// (point, C-th part of its bin rows), reduced in double-float, and one lane per
// (point, detector) adds the parts in order. C depends on the grid alone, so a
// point's log L does not depend on the batch it comes in. GB300, one point per CTA
// with its coefficients on one warp -> this kernel: 1000 draws of 4017 bins 55.7 ->
// 47.2 us, 64 draws of 512 bins 36.6 -> 32.5 us (8 warps a CTA: 50.5 and 38.1).
constexpr int EVAL_FX_W = 4;                // warps
constexpr int EVAL_FX_P = EVAL_FX_W;        // points at most

// Relative binning (RB): one warp sums a point's coarse bins (C = 1). Four CTAs an
// SM; three for four detectors' rows, whose arithmetic wants more registers (64 / 1000
// draws of 519,169 bins 112 / 407 -> 103 / 385 us; coarse bins 297 -> 317 us of 8192, so not
// there).
#define EVAL_FX_BLOCKS(NDET, RB) ((NDET) == 4 && !(RB) ? 3 : 16 / EVAL_FX_W)
template <int NDET, bool RB>
__global__ void __launch_bounds__(EVAL_FX_W * 32, EVAL_FX_BLOCKS(NDET, RB)) k_eval_fx(Model M, Tables T, const double *in,
                                                                            int m, int P, int C, double *logl,
                                                                            RunState *st) {
    __shared__ Coef coef[EVAL_FX_P];
    __shared__ FxPoint fx[EVAL_FX_P];
    __shared__ float4 sc[FX_SC];
    __shared__ double pt[EVAL_FX_P][MAXD];
    __shared__ double red[EVAL_FX_P][8][2 * NDET];
    const int i0 = blockIdx.x * P;
    if (i0 >= m) return;
    const int np = m - i0 < P ? m - i0 : P;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, d = M.dim;
    for (int t = threadIdx.x; t < np * d; t += EVAL_FX_W * 32) pt[t / d][t % d] = in[(size_t)i0 * d + t];
    load_sc(T, sc);
    __syncthreads();
    const int grp = warp >> 1, cnt = 4 * grp < np ? min(4, np - 4 * grp) : 0;
    if (cnt > 0) point_coef_group(M, T, pt[4 * grp], MAXD, &coef[4 * grp], cnt, 1 + (warp & 1));
    __syncthreads();
    if (cnt > 0) {
        if (warp & 1) coef_to_fx_group(T, M.n_det, &coef[4 * grp], &fx[4 * grp], cnt, RB ? T.rb.fid : nullptr);
        else point_coef_join(M, T, &coef[4 * grp], cnt);
    }
    __syncthreads();
    if constexpr (RB) {
        for (int p = warp; p < np; p += EVAL_FX_W) {
            const double v = rb_loglike_fx<NDET>(M, T, coef[p], fx[p], sc);
            if (lane == 0) logl[i0 + p] = v;
        }
        if (st && threadIdx.x == 0) atomicAdd(&st->eval_points, (unsigned long long)np);
        return;
    }
    for (int it = warp; it < np * C; it += EVAL_FX_W) {
        const int p = it / C, c = it - p * C;
        float zh[NDET][2], zl[NDET][2];
        bins_fx<NDET>(T, fx[p], sc, c * 32 + lane, C * 32, zh, zl);
        warp_sums_df_to<NDET>(zh, zl, red[p][c], T.fxs);
    }
    __syncthreads();
    if (warp == 0) {
        const int p = lane / NDET, dd = lane - p * NDET;
        double v = 0.0;
        if (p < np) {
            double zr = red[p][0][2 * dd], zi = red[p][0][2 * dd + 1];
            for (int c = 1; c < C; c++) { zr += red[p][c][2 * dd]; zi += red[p][c][2 * dd + 1]; }
            v = coef[p].gre[dd] * zr - coef[p].gim[dd] * zi;
        }
        const double t = group_sum_down<NDET>(v);
        if (p < np && dd == 0) logl[i0 + p] = t - 0.5 * coef[p].hh;
        if (st && lane == 0) {
            unsigned long long n = 0;
            for (int q = 0; q < np; q++) n += (unsigned long long)(coef[q].jcut + 1);
            atomicAdd(&st->eval_points, (unsigned long long)np);
            atomicAdd(&st->eval_point_bins, n);
        }
    }
}

template <int PREC, int NDET>
cudaError_t eval_launch(const Model &M, const Tables &T, int warps, int n_sm, const double *in, int th, int m,
                        double *logl, RunState *st, cudaStream_t s) {
    const int nbins = M.rb ? T.rb.nb : M.N;
    if constexpr (PREC == 1) {
        if (M.model == M_GW && !th && !M.rb && nbins <= 262144) {
            const int ppc = 4 * (warps >= 2 ? warps / 2 : 1);
            const int gb = (m + ppc - 1) / ppc;
            switch (warps) {
                case 1: k_eval_batch<NDET, 1><<<gb, 32, 0, s>>>(M, T, in, m, logl, st); break;
                case 2: k_eval_batch<NDET, 2><<<gb, 64, 0, s>>>(M, T, in, m, logl, st); break;
                case 4:
                    if (NDET == 4 && M.tlg >= 5)
                        k_eval_batch<NDET, 4, NDET == 4 ? EVAL_BATCH4_BLOCKS : EVAL_BATCH_BLOCKS(NDET, 4)>
                            <<<gb, 128, 0, s>>>(M, T, in, m, logl, st);
                    else
                        k_eval_batch<NDET, 4><<<gb, 128, 0, s>>>(M, T, in, m, logl, st);
                    break;
                default: k_eval_batch<NDET, 8><<<gb, 256, 0, s>>>(M, T, in, m, logl, st); break;
            }
            return cudaGetLastError();
        }
    }
    if constexpr (PREC == 0) {
        if (M.model == M_GW && !th) {
            // as many points a CTA as leave a CTA for every SM
            int P = 1;
            while (P < EVAL_FX_P && m >= 2 * P * n_sm) P *= 2;
            if (M.rb) k_eval_fx<NDET, true><<<(m + P - 1) / P, EVAL_FX_W * 32, 0, s>>>(M, T, in, m, P, 1, logl, st);
            else k_eval_fx<NDET, false><<<(m + P - 1) / P, EVAL_FX_W * 32, 0, s>>>(M, T, in, m, P, warps, logl, st);
            return cudaGetLastError();
        }
    }
    const int ppc = (PREC == 1 && M.model == M_GW && !th && nbins <= 262144) ? EVAL_PPC : 1;
    const int g = (m + ppc - 1) / ppc;
    switch (warps) {
        case 1: k_eval<PREC, NDET, 1><<<g, 32, 0, s>>>(M, T, in, th, m, ppc, logl, st); break;
        case 2: k_eval<PREC, NDET, 2><<<g, 64, 0, s>>>(M, T, in, th, m, ppc, logl, st); break;
        case 4: k_eval<PREC, NDET, 4><<<g, 128, 0, s>>>(M, T, in, th, m, ppc, logl, st); break;
        default: k_eval<PREC, NDET, 8><<<g, 256, 0, s>>>(M, T, in, th, m, ppc, logl, st); break;
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------ slice update
// One CTA per chain, S warps ("slots"). Warp 0 owns the chain: the point x,
// the direction e and the bracket (lane i < d holds coordinate i). Every slice
// step draws a direction and a bracket offset, steps out to the left and to the
// right, then shrinks (Neal 2003, Sec. 4, along a hit-and-run direction).
//
// The candidates of each stage form sequences fixed by the draws alone:
// stepping out to the left visits x + (a - q) e, to the right x + (b + q) e,
// and the q-th shrink draw is determined once the earlier draws are known to be
// rejected. Each round, warp 0 plans the next S candidates of these sequences
// that lie inside the prior box and are not yet evaluated; every slot warp
// computes one candidate's coefficients and bins; warp 0 then consumes the
// results strictly in the sequential order (left stepping out, right stepping
// out, shrinkage) and keeps results it could not consume yet in a small cache.
// Evaluations the sequential order never reaches are discarded. The trajectory,
// the evaluation count and every draw are those of the sequential algorithm;
// the slots only shorten the chain's critical path.
enum { PH_NEWSTEP = 0, PH_OUT = 1, PH_SHRINK = 2, PH_DONE = 3, PH_WALK = 4 };
enum { KIND_L = 0, KIND_R = 1, KIND_SH = 2, KIND_W = 3 };
constexpr int CACHE_MAX = 16;

// Planned candidates and evaluated, not yet consumed ones, in shared memory: a
// plan writes its entries behind the n kept ones, the coefficient stage reads the
// points there, and the results join them. One copy per lane in local memory, 900
// bytes a thread, took up to 110 KB of each SM's L1 and its latency at every
// transition; with it here, found by one ballot, and the positions and points kept
// instead of computed again when a result is consumed (24 FP64 instructions a
// candidate), GB300: slice update of 512 bins FP64 755 -> 674 us, 4017 bins FP64
// 4.06 -> 3.70 ms, 64,897 bins mixed 10.9 -> 10.4 ms; four served analyses 286 -> 241 ms.
struct CandCache {
    double y[CACHE_MAX][MAXD];     // the point
    double val[CACHE_MAX];         // log L
    double t[CACHE_MAX];           // slice sampling: the position on the line
    int key[CACHE_MAX];            // kind << 16 | index
    int bins[CACHE_MAX];
};

__device__ __forceinline__ int cand_key(int kind, int idx) { return (kind << 16) | idx; }

struct Chain {
    double x, e;
    double lx, a, b;
    int s, phase, nl, nr, nsh, caps, left_done, right_done;
    long long evals;
    unsigned long long bins, bins_lo;   // bins read by the consumed evaluations; of those, in low-degree groups
    int ncache;
    // the candidate that chain_run stopped at, for the plan
    double next_t, next_y;
};

// A chain between its rounds, in shared memory, so that its state takes no
// registers of the bin sums.
struct ChainStore {
    double x[MAXD], e[MAXD];
    Chain c;        // with x and e of lane 0
};
__device__ __forceinline__ void chain_load(const ChainStore &q, Chain &c, int lane, int d) {
    c = q.c;
    c.x = lane < d ? q.x[lane] : 0.0;
    c.e = lane < d ? q.e[lane] : 0.0;
}
__device__ __forceinline__ void chain_save(ChainStore &q, const Chain &c, int lane, int d) {
    __syncwarp();
    if (lane < d) {
        q.x[lane] = c.x;
        q.e[lane] = c.e;
    }
    if (lane == 0) q.c = c;
    __syncwarp();
}

// A consumed evaluation's bins (jcut + 1 of them): all, and those at or past lo_bin.
__device__ __forceinline__ void count_bins(Chain &c, int bins, long long lo_bin) {
    c.bins += (unsigned long long)bins;
    if ((long long)bins > lo_bin) c.bins_lo += (unsigned long long)((long long)bins - lo_bin);
}

// Lane i's coordinate of the candidate x + t e (lanes >= d: 0.5, inside the
// box); periodic coordinates wrap into [0, 1).
__device__ __forceinline__ double line_y(const Model &M, const Chain &c, double t, int lane, int d) {
    if (lane >= d) return 0.5;
    double y = __dadd_rn(c.x, __dmul_rn(t, c.e));
    if ((M.periodic >> lane) & 1u) y = __dsub_rn(y, floor(y));
    return y;
}

__device__ __forceinline__ bool warp_inbox(double y, int lane, int d) {
    // 0 <= y <= 1 by the bits (and -0): an FP64 comparison costs 64 cycles
    const unsigned long long b = (unsigned long long)__double_as_longlong(y);
    return __all_sync(0xffffffffu, lane >= d || b <= 0x3ff0000000000000ull || b == 0x8000000000000000ull);
}

// Index of an entry (all lanes), -1 if absent: one key per lane.
__device__ __forceinline__ int cache_find(const Chain &c, const CandCache &q, int kind, int idx) {
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, lane < c.ncache && q.key[lane & (CACHE_MAX - 1)] == cand_key(kind, idx));
    return (int)__ffs(m) - 1;
}

// Drop entry i: the last one takes its place.
__device__ __forceinline__ void cache_drop(Chain &c, CandCache &q, int i) {
    const int lane = threadIdx.x & 31;
    const int l = --c.ncache;
    __syncwarp();
    if (i != l) {
        if (lane < MAXD) q.y[i][lane] = q.y[l][lane];
        if (lane == 0) {
            q.val[i] = q.val[l];
            q.t[i] = q.t[l];
            q.key[i] = q.key[l];
            q.bins[i] = q.bins[l];
        }
    }
    __syncwarp();
}

// Drop every cached result of one kind (once a stepping-out side has ended, its
// later candidates are never consumed).
__device__ __forceinline__ void cache_purge(Chain &c, CandCache &q, int kind) {
    for (int i = c.ncache - 1; i >= 0; i--)
        if ((q.key[i] >> 16) == kind) cache_drop(c, q, i);
}

__device__ __forceinline__ void end_side(Chain &c, CandCache &q, bool left) {
    if (left) c.left_done = 1;
    else c.right_done = 1;
    cache_purge(c, q, left ? KIND_L : KIND_R);
}

__device__ __forceinline__ double shrink_t(const StepArgs &A, double a, double b, int nsh, int step,
                                           int chain, uint32_t iter) {
    const uint4 w = draw(A.seed, SLOT_SHRINK0 + (uint32_t)nsh, (uint32_t)step, (uint32_t)chain, iter);
    return __dadd_rn(a, __dmul_rn(__dsub_rn(b, a), u01(w.x, w.y)));
}

// Hit-and-run direction of slice step s: lane i < d gets coordinate i of
// L z / |z|, z ~ N(0, I) by Box-Muller (two normals per draw), L the Cholesky factor.
static __device__ __noinline__ double slice_direction(const StepArgs &A, int chain, uint32_t iter, int s, int lane, int d) {
    double z = 0.0;
    if (lane < d) {
        const uint4 w = draw(A.seed, (uint32_t)(lane >> 1), (uint32_t)s, (uint32_t)chain, iter);
        const double u1 = u01(w.x, w.y), u2 = u01(w.z, w.w);
        const double r = sqrt(-2.0 * log(u1));
        double sn, cs;
        sincos(TWO_PI_D * u2, &sn, &cs);
        z = (lane & 1) ? r * sn : r * cs;
    }
    const double nz = sqrt(warp_sum(z * z));
    double acc = 0.0;
    for (int j = 0; j < d; j++) {
        const double zj = __shfl_sync(0xffffffffu, z, j);
        if (j <= lane && lane < d) acc = __dadd_rn(acc, __dmul_rn(A.chol[lane * d + j], zj));
    }
    return (lane < d) ? acc / nz : 0.0;
}

// Apply every transition that needs no new evaluation: new steps (direction and
// bracket draws), cap and prior-box outcomes, and results already in the cache.
// Returns when the next transition needs an evaluation not in the cache, or the
// chain is done.
static __device__ void chain_run(const Model &M, const StepArgs &A, Chain &c, CandCache &q, int chain, uint32_t iter,
                                 double lstar, const double *e_pre, int e_pre_step) {
    const int lane = threadIdx.x & 31, d = M.dim;
    for (int guard = 0; guard < (1 << 22); guard++) {
        if (c.phase == PH_DONE) return;
        if (c.phase == PH_NEWSTEP) {
            if (c.s >= A.steps) { c.phase = PH_DONE; return; }
            // direction (computed ahead by a spare warp when it could be)
            if (e_pre_step == c.s) c.e = (lane < d) ? e_pre[lane] : 0.0;
            else c.e = slice_direction(A, chain, iter, c.s, lane, d);
            const uint4 w = draw(A.seed, SLOT_OFFSET, (uint32_t)c.s, (uint32_t)chain, iter);
            const double r = u01(w.x, w.y);
            c.a = -r;
            c.b = 1.0 - r;
            c.nl = c.nr = c.nsh = 0;
            c.left_done = c.right_done = 0;
            c.ncache = 0;
            c.phase = PH_OUT;
            continue;
        }
        if (c.phase == PH_OUT) {
            const bool left = !c.left_done;
            if (!left && c.right_done) { c.phase = PH_SHRINK; continue; }
            const int n = left ? c.nl : c.nr;
            if (n >= A.max_stepout) {
                end_side(c, q, left);
                continue;
            }
            const int ci = cache_find(c, q, left ? KIND_L : KIND_R, n);
            if (ci < 0) {
                c.next_t = left ? c.a : c.b;
                c.next_y = line_y(M, c, c.next_t, lane, d);
                if (warp_inbox(c.next_y, lane, d)) return;
                end_side(c, q, left);
                continue;
            }
            const bool in = q.val[ci] > lstar;
            c.evals++;
            count_bins(c, q.bins[ci], A.lo_bin);
            cache_drop(c, q, ci);
            if (left) { if (in) { c.a -= 1.0; c.nl++; } else end_side(c, q, true); }
            else { if (in) { c.b += 1.0; c.nr++; } else end_side(c, q, false); }
            continue;
        }
        // PH_SHRINK
        if (c.nsh >= A.max_shrink) {
            c.caps++;
            c.s++;
            c.phase = PH_NEWSTEP;
            continue;
        }
        // an evaluated candidate comes with its position and point: planned as the
        // next draw after rejections, which is how it is reached
        const int ci = cache_find(c, q, KIND_SH, c.nsh);
        double t;
        if (ci < 0) {
            t = shrink_t(A, c.a, c.b, c.nsh, c.s, chain, iter);
            const double y = line_y(M, c, t, lane, d);
            if (warp_inbox(y, lane, d)) {
                c.next_t = t;
                c.next_y = y;
                return;
            }
        } else {
            t = q.t[ci];
            const double val = q.val[ci], y = (lane < d) ? q.y[ci][lane] : 0.5;
            c.evals++;
            count_bins(c, q.bins[ci], A.lo_bin);
            cache_drop(c, q, ci);
            if (val > lstar) {
                c.x = y;
                c.lx = val;
                c.s++;
                c.phase = PH_NEWSTEP;
                continue;
            }
        }
        if (t < 0.0) c.a = t; else c.b = t;
        c.nsh++;
    }
    c.phase = PH_DONE;   // unreachable with finite caps; keeps the loop bounded
}

// Candidate ns of a plan: its point, position and key behind the cache's entries.
__device__ __forceinline__ void plan_put(const Chain &c, CandCache &q, int ns, int key, double t, double y, int lane, int d) {
    const int i = c.ncache + ns;
    if (lane < d) q.y[i][lane] = y;
    if (lane == 0) {
        q.t[i] = t;
        q.key[i] = key;
    }
}

// Plan up to S candidates to evaluate in the next round (in-box, not cached),
// continuing the current stage's sequences; returns their number.
template <int S>
__device__ int chain_plan(const Model &M, const StepArgs &A, const Chain &c, CandCache &q, int chain, uint32_t iter,
                          int depth) {
    const int lane = threadIdx.x & 31, d = M.dim;
    int ns = 0;
    const int room = CACHE_MAX - c.ncache;
    const int lim = depth < S ? depth : S;
    const int cap = lim < room ? lim : room;
    if (c.phase == PH_OUT) {
        // the side in progress first (half the slots if the other side is
        // still open), then the other side; each looks at most S candidates
        // ahead of its consumed position, so the cache holds at most 2S entries
        for (int side = 0; side < 2 && ns < cap; side++) {
            const bool left = (side == 0);
            if (left ? c.left_done : c.right_done) continue;
            const int limit = (left && !c.right_done) ? (cap + 1) / 2 : cap;
            const int kind = left ? KIND_L : KIND_R;
            double t = left ? c.a : c.b;
            const int n0 = left ? c.nl : c.nr;
            for (int n = n0; n < n0 + S && n < A.max_stepout && ns < limit; n++) {
                if (cache_find(c, q, kind, n) < 0) {
                    // the side in progress stopped at its first candidate
                    const bool next = n == n0 && (left || c.left_done);
                    const double y = next ? c.next_y : line_y(M, c, t, lane, d);
                    if (!next && !warp_inbox(y, lane, d)) break;
                    plan_put(c, q, ns++, cand_key(kind, n), t, y, lane, d);
                }
                if (left) t -= 1.0; else t += 1.0;
            }
        }
    } else if (c.phase == PH_SHRINK) {
        double a = c.a, b = c.b;
        for (int n = c.nsh; n < c.nsh + S && n < A.max_shrink && ns < cap; n++) {
            double t;
            const int ci = n == c.nsh ? -1 : cache_find(c, q, KIND_SH, n);
            if (ci >= 0) {
                t = q.t[ci];
            } else {
                const bool next = n == c.nsh;
                t = next ? c.next_t : shrink_t(A, a, b, n, c.s, chain, iter);
                const double y = next ? c.next_y : line_y(M, c, t, lane, d);
                if (next || warp_inbox(y, lane, d)) plan_put(c, q, ns++, cand_key(KIND_SH, n), t, y, lane, d);
            }
            if (t < 0.0) a = t; else b = t;     // as if rejected
        }
    }
    return ns;
}

// ------------------------------------------------------------ random walk
// The random-walk inner kernel (acceptance walk): from the chain's start point,
// walk_len proposals y = x + scale L z_p, z_p ~ N(0, I) from the draws of
// proposal p (the slice directions' slots with p in place of the step); a
// proposal inside the prior box (periodic coordinates wrapped) and above L*
// is accepted. The walk length is fixed within an iteration and rescaled
// between iterations (k_finish). Speculation: the proposals after the current
// one are evaluated from the current point, as if it were rejected; an
// acceptance discards them. c.s counts accepted moves, c.nsh the proposal.
static __device__ __noinline__ double walk_disp(const StepArgs &A, int chain, uint32_t iter, int p, int lane, int d) {
    double z = 0.0;
    if (lane < d) {
        const uint4 w = draw(A.seed, (uint32_t)(lane >> 1), (uint32_t)p, (uint32_t)chain, iter);
        const double u1 = u01(w.x, w.y), u2 = u01(w.z, w.w);
        const double r = sqrt(-2.0 * log(u1));
        double sn, cs;
        sincos(TWO_PI_D * u2, &sn, &cs);
        z = (lane & 1) ? r * sn : r * cs;
    }
    double acc = 0.0;
    for (int j = 0; j < d; j++) {
        const double zj = __shfl_sync(0xffffffffu, z, j);
        if (j <= lane && lane < d) acc = __dadd_rn(acc, __dmul_rn(A.chol[lane * d + j], zj));
    }
    return __dmul_rn(acc, A.walk_scale);
}

__device__ __forceinline__ double walk_y(const Model &M, const Chain &c, double disp, int lane, int d) {
    if (lane >= d) return 0.5;
    double y = __dadd_rn(c.x, disp);
    if ((M.periodic >> lane) & 1u) y = __dsub_rn(y, floor(y));
    return y;
}

static __device__ void walk_run(const Model &M, const StepArgs &A, Chain &c, CandCache &q, int chain, uint32_t iter,
                                double lstar, int walk_len) {
    const int lane = threadIdx.x & 31, d = M.dim;
    for (int guard = 0; guard < (1 << 22); guard++) {
        if (c.phase == PH_DONE) return;
        if (c.nsh >= walk_len) { c.phase = PH_DONE; return; }
        // an evaluated proposal comes with its point (planned from the current
        // point: the cache is emptied at every acceptance); otherwise compute
        // it, skip it outside the box, or wait for its evaluation
        const int ci = cache_find(c, q, KIND_W, c.nsh);
        double y;
        if (ci >= 0) {
            y = (lane < d) ? q.y[ci][lane] : 0.5;
        } else {
            y = walk_y(M, c, walk_disp(A, chain, iter, c.nsh, lane, d), lane, d);
            if (!warp_inbox(y, lane, d)) { c.nsh++; continue; }
            return;
        }
        const double val = q.val[ci];
        c.evals++;
        count_bins(c, q.bins[ci], A.lo_bin);
        cache_drop(c, q, ci);
        if (val > lstar) {
            c.x = y;
            c.lx = val;
            c.s++;
            cache_purge(c, q, KIND_W);
        }
        c.nsh++;
    }
    c.phase = PH_DONE;
}

template <int S>
__device__ int walk_plan(const Model &M, const StepArgs &A, const Chain &c, CandCache &q, int chain, uint32_t iter,
                         int depth, int walk_len) {
    const int lane = threadIdx.x & 31, d = M.dim;
    const int room = CACHE_MAX - c.ncache;
    const int lim = depth < S ? depth : S;
    const int cap = lim < room ? lim : room;
    int ns = 0;
    for (int p = c.nsh; p < c.nsh + S && p < walk_len && ns < cap; p++) {
        if (cache_find(c, q, KIND_W, p) >= 0) continue;
        const double y = walk_y(M, c, walk_disp(A, chain, iter, p, lane, d), lane, d);
        if (warp_inbox(y, lane, d)) plan_put(c, q, ns++, cand_key(KIND_W, p), 0.0, y, lane, d);
    }
    return ns;
}

// ------------------------------------------------- work-shared slice update
// Mixed precision on fine tiled grids (the 519,169-bin workload): when fewer
// chains remain than CTA slots, the update's last chains would run alone on
// otherwise idle SMs. Instead, persistent CTAs take chains from a counter, and
// each round's candidates are evaluated in fixed chunks of ws_gchunk tile
// groups. The owner publishes the round in its slot (coefficients, then the
// claim word); its own warps and the warps of CTAs without a chain claim
// chunks through the word, each chunk's sums are computed by one warp and
// written to the slot's partials, and the owner adds them in chunk order. The
// decomposition does not depend on who computes a chunk, so results do not
// depend on timing. No warp waits on a CTA that has not claimed work: the
// owner waits only for chunks already claimed (their warps are running), and
// helpers stop once no chain is running. Both waits are bounded; on a timeout
// the run state's status gets bit 1 and the host reports NS_ERR_TIMEOUT.
constexpr long long WS_WAIT_LIMIT = 1ll << 24;   // owner polls of the done count (~100 ns apart)
constexpr long long WS_IDLE_LIMIT = 1ll << 22;   // consecutive helper polls without work (~1 us each)

__device__ __forceinline__ unsigned long long ws_word(unsigned long long seq, int n, int next) {
    return (seq << 40) | ((unsigned long long)n << 20) | (unsigned long long)next;
}

// Lane 0: claim the next chunk of a slot's round; -1 if none is left. A stale
// view of the word is harmless: the atomic's return value names the round and
// chunk actually claimed, and a round's data stay in place until all its
// claimed chunks are done.
__device__ __forceinline__ int ws_claim(WsSlot *s) {
    const unsigned long long w = *((volatile unsigned long long *)&s->word);
    if ((w & 0xFFFFFull) >= ((w >> 20) & 0xFFFFFull)) return -1;
    const unsigned long long old = atomicAdd(&s->word, 1ull);
    const int n = (int)((old >> 20) & 0xFFFFFull), nx = (int)(old & 0xFFFFFull);
    return nx < n ? nx : -1;
}

// One warp: the sums of chunk c (tile groups c G .. c G + G - 1) for the ns
// candidates, reduced over the warp; lane 0 writes out[candidate][detector][re, im].
template <int NDET>
__device__ __forceinline__ void ws_chunk(const Model &M, const Tables &T, const CoefMixed *cm, const int *jc,
                                         int ns, int c, int G, double *out) {
    const int lane = threadIdx.x & 31;
    const int g0 = c * G, g1 = g0 + G;
    for (int c0 = 0; c0 < ns; c0++) {
        float zh[NDET][2], zl[NDET][2];
        tile_bins<NDET, true, true, true>(T, M.tlg, M.np, cm[c0], jc[c0], g0, 1, zh, zl, g1);
        // value v = (detector, re/im), summed over the warp at once
        float vh[16], vl[16];
#pragma unroll
        for (int dd = 0; dd < NDET; dd++)
#pragma unroll
            for (int ri = 0; ri < 2; ri++) {
                vh[dd * 2 + ri] = zh[dd][ri];
                vl[dd * 2 + ri] = zl[dd][ri];
            }
        float rh, rl;
        warp_sum_df_many<2 * NDET>(vh, vl, rh, rl);
        const int v = lane >> 1, dd = v >> 1, ri = v & 1;
        if ((lane & 1) == 0 && v < 2 * NDET)
            out[(c0 * MAXDET + dd) * 2 + ri] = (double)rh + (double)rl;
    }
}

// One warp: find a slot (other than skip) with an unclaimed chunk, claim it
// and compute it into that slot's partials. Returns 1 if it did a chunk. The
// round's coefficients are staged in this warp's shared buffer.
template <int NDET, int W>
__device__ int ws_take_any(const Model &M, const Tables &T, const StepArgs &A, int skip) {
    __shared__ CoefMixed hcm[W][4];
    __shared__ int hjc[W][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nslot = A.ws_nslot;
    const int start = (int)(((unsigned)blockIdx.x * 37u + (unsigned)warp * 11u) % (unsigned)nslot);
    int found = -1;
    for (int base = 0; base < nslot && found < 0; base += 32) {
        const int j = base + lane;
        int s = start + j;
        if (s >= nslot) s -= nslot;
        bool open = false;
        if (j < nslot && s != skip) {
            const unsigned long long w = *((volatile unsigned long long *)&A.ws[s].word);
            open = (w & 0xFFFFFull) < ((w >> 20) & 0xFFFFFull);
        }
        const unsigned b = __ballot_sync(0xffffffffu, open);
        if (b) found = __shfl_sync(0xffffffffu, s, __ffs(b) - 1);
    }
    int c = -1;
    if (found >= 0 && lane == 0) c = ws_claim(A.ws + found);
    c = __shfl_sync(0xffffffffu, c, 0);
    if (c < 0) return 0;
    __threadfence();
    WsSlot *sl = A.ws + found;
    const int ns = __ldcg(&sl->ns);
    const int nwords = ns * (int)(sizeof(CoefMixed) / sizeof(int));
    for (int i = lane; i < nwords; i += 32) ((int *)hcm[warp])[i] = __ldcg(((const int *)sl->cm) + i);
    if (lane < ns) hjc[warp][lane] = __ldcg(&sl->jc[lane]);
    __syncwarp();
    ws_chunk<NDET>(M, T, hcm[warp], hjc[warp], ns, c, A.ws_gchunk,
                   A.ws_part + ((size_t)found * A.ws_maxchunk + c) * WS_PART_PER_CHUNK);
    __threadfence();
    if (lane == 0) atomicAdd(&sl->done, 1);
    __syncwarp();
    return 1;
}

// Owner CTA (all threads): publish the round's ns candidates (coefficients cm,
// last bins jc, in shared memory), take part in its chunks, then warp 0 waits
// for the chunks helpers took and writes the sums over chunks, in chunk order,
// to zs[candidate][detector][re, im] (shared).
template <int NDET, int W>
__device__ void ws_owner_round(const Model &M, const Tables &T, const StepArgs &A, const CoefMixed *cm,
                               const int *jc, int ns, double (*zs)[NDET][2]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    WsSlot *slot = A.ws + blockIdx.x;
    double *part = A.ws_part + (size_t)blockIdx.x * A.ws_maxchunk * WS_PART_PER_CHUNK;
    int jmax = -1;
    for (int c = 0; c < ns; c++) jmax = max(jmax, jc[c]);
    const int G = A.ws_gchunk;
    const int ng = jmax < 0 ? 0 : (jmax >> (M.tlg + 5)) + 1;
    const int nch = min((ng + G - 1) / G, A.ws_maxchunk);
    const int nwords = ns * (int)(sizeof(CoefMixed) / sizeof(int));
    for (int i = threadIdx.x; i < nwords; i += W * 32) ((int *)slot->cm)[i] = ((const int *)cm)[i];
    if (threadIdx.x < ns) slot->jc[threadIdx.x] = jc[threadIdx.x];
    if (threadIdx.x == 0) {
        slot->ns = ns;
        slot->done = 0;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long w = *((volatile unsigned long long *)&slot->word);
        atomicExch(&slot->word, ws_word((w >> 40) + 1, nch, 0));
    }
    __syncthreads();
    // every warp claims the round's chunks; warp 0 then waits for the chunks
    // other CTAs took (GB300, 519,169 bins: letting the other warps take other
    // rounds' chunks meanwhile was slower, 264 -> 297 ms per update, as a
    // chain's next round then waits for its warps to come back)
    for (int guard = 0; guard < (1 << 20); guard++) {
        int c = -1;
        if (lane == 0) c = ws_claim(slot);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c < 0) break;
        ws_chunk<NDET>(M, T, cm, jc, ns, c, G, part + (size_t)c * WS_PART_PER_CHUNK);
        __threadfence();
        if (lane == 0) atomicAdd(&slot->done, 1);
    }
    if (warp == 0 && lane == 0) {
        // ws_test_extra (a test hook, 0 in use) makes the owner wait for chunks
        // nobody computes, so that the bounded wait runs out
        for (long long it = 0; *((volatile int *)&slot->done) < nch + A.ws_test_extra; it++) {
            if (it > WS_WAIT_LIMIT) {
                atomicOr(&A.state->status, 2);
                break;
            }
            __nanosleep(100);
        }
    }
    __syncthreads();
    if (warp == 0) {
        __threadfence();
        const int sc = lane / NDET, dd = lane - sc * NDET;
        if (lane < ns * NDET) {
            double zr = 0.0, zi = 0.0;
            for (int c = 0; c < nch; c++) {
                const double *p = part + (size_t)c * WS_PART_PER_CHUNK + (sc * MAXDET + dd) * 2;
                zr += __ldcg(p);
                zi += __ldcg(p + 1);
            }
            zs[sc][dd][0] = zr;
            zs[sc][dd][1] = zi;
        }
    }
}

// A CTA without a chain left: each warp takes chunks of any running chain's
// round until no chain is running.
template <int NDET, int W>
__device__ void ws_help(const Model &M, const Tables &T, const StepArgs &A) {
    const int lane = threadIdx.x & 31;
    long long idle = 0;
    for (;;) {
        if (*((volatile int *)A.active) <= 0) break;
        if (ws_take_any<NDET, W>(M, T, A, -1)) {
            idle = 0;
            continue;
        }
        if (++idle > WS_IDLE_LIMIT) {
            if (lane == 0) atomicOr(&A.state->status, 2);
            break;
        }
        __nanosleep(200);
    }
}

// Form of the tiled mixed sums a kernel compiles: FORM_ROT, rotation
// (tile_bins_rot), for grids with tiles of 32 bins or more only; FORM_DIRECT for
// all others (shorter tiles, per-bin grids, FP64).
enum { FORM_DIRECT = 0, FORM_ROT = 2 };

template <int NDET, int FORM>
__device__ __forceinline__ void tile_bins_form(const Model &M, const Tables &T, const CoefMixed &cm, const int &jc,
                                               int g0, int gstride, float (&zh)[NDET][2], float (&zl)[NDET][2]) {
    tile_bins<NDET, FORM == FORM_ROT>(T, M.tlg, M.np, cm, jc, g0, gstride, zh, zl);
}

template <int PREC, int NDET, int S, int W, int FORM, bool WS = false>
__device__ void slice_body(const Model &M, const Tables &T, const StepArgs &A, const int chain) {
    __shared__ Coef coef[S];
    __shared__ CoefMixed cm[S];
    __shared__ CandCache cq;
    __shared__ ChainStore cs;
    __shared__ double lval[S];
    __shared__ int nslot, nbase, tailmode;
    __shared__ double e_next[MAXD];         // direction of slice step e_next_step, computed ahead
    __shared__ int e_next_step, cur_step;
    __shared__ int jc[S];
    __shared__ double part[W][S][NDET][2];
    __shared__ FxPoint fx[PREC == 0 ? S : 1];
    __shared__ float4 sct[PREC == 0 ? FX_SC : 1];
    if (chain >= A.k) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, d = M.dim;
    const bool use_fx = PREC == 0 && M.model == M_GW;
    const Coef *fid = M.rb ? T.rb.fid : nullptr;
    if (use_fx) load_sc(T, sct);    // used after the first round's barriers
    const uint32_t iter = (uint32_t)A.state->iter;
    const double lstar = A.state->lstar;
    const int walk_len = A.state->walk_len;
    if (warp == 0) {
        Chain c;
        const int m = A.n - A.k;
        const uint4 w = draw(A.seed, 0u, STEP_START, (uint32_t)chain, iter);
        int idx = (int)(u01(w.x, w.y) * m);
        if (idx >= m) idx = m - 1;
        const int src = A.order[A.k + idx];
        c.x = (lane < d) ? A.live_u[(size_t)src * d + lane] : 0.0;
        c.lx = A.live_logl[src];
        c.e = 0.0; c.a = 0.0; c.b = 0.0;
        c.s = 0; c.phase = A.kernel == 1 ? PH_WALK : PH_NEWSTEP; c.nl = c.nr = c.nsh = 0; c.caps = 0;
        c.evals = 0; c.bins = 0; c.bins_lo = 0;
        c.left_done = c.right_done = 0; c.ncache = 0;
        c.next_t = c.next_y = 0.0;
        chain_save(cs, c, lane, d);
        if (lane == 0) e_next_step = -1;
        __syncwarp();
    }
    for (;;) {
        if (warp == 0) {
            Chain c;
            chain_load(cs, c, lane, d);
            // a bounded wait of the work-shared update gave up (status bit 1):
            // every chain ends at its current point, so that the launch ends
            if (WS && (*((volatile int *)&A.state->status) & 2)) c.phase = PH_DONE;
            if (A.kernel == 1) walk_run(M, A, c, cq, chain, iter, lstar, walk_len);
            else chain_run(M, A, c, cq, chain, iter, lstar, e_next, e_next_step);
            // plan the base depth while many chains run; the stragglers of the
            // update (fewer running chains than the tail threshold) use every warp.
            // FP64 above 1024 bins splits every candidate's bins over two warps in
            // every round instead (FP64 branch below), with at most W/2 candidates.
            int depth = S, tail = 1;
            if (A.active) {
                const int running = *((volatile int *)A.active);
                if (running > A.tail) { depth = A.depth; tail = 0; }
            }
            if (PREC == 0 && A.fp64_split == 2 && W >= 2) {
                depth = A.depth < W / 2 ? A.depth : W / 2;
                tail = 2;
            }
            int ns = (c.phase == PH_DONE) ? 0
                   : A.kernel == 1 ? walk_plan<S>(M, A, c, cq, chain, iter, depth, walk_len)
                                   : chain_plan<S>(M, A, c, cq, chain, iter, depth);
            if (ns == 0 && c.phase != PH_DONE) {
                // cannot happen with the bounds above; end the chain at its
                // current (in-slice) point and flag the run state
                c.phase = PH_DONE;
                if (lane == 0) atomicOr(&A.state->status, 1);
            }
            if (lane == 0) { nslot = ns; nbase = c.ncache; tailmode = tail; cur_step = c.s; }
            chain_save(cs, c, lane, d);
        }
        __syncthreads();
        const int ns = nslot;
        if (ns == 0) break;
        const double (*ysh)[MAXD] = cq.y + nbase;       // the round's points
        // coefficients: candidates 4j .. 4j+3 (8 lanes each) by one warp, or,
        // with two warps per group of four, the mass/phase half on warp 2j and
        // the sky/detector half on warp 2j + 1 (independent FP64 chains on two
        // sub-partitions), joined after the barrier
        if (M.model == M_TOY) {
            if (warp < ns) point_coef_warp(M, T, ysh[warp], &coef[warp]);
            __syncthreads();
        } else if (S >= 2) {
            const int grp = warp >> 1;
            if (4 * grp < ns && 2 * grp + 1 < W) {
                const int cnt = ns - 4 * grp < 4 ? ns - 4 * grp : 4;
                if (PREC == 1 && M.cdf)
                    point_coef_group_mx(M, T, ysh[4 * grp], MAXD, &coef[4 * grp], &cm[4 * grp], cnt,
                                        FORM == FORM_ROT, 1 + (warp & 1));
                else
                    point_coef_group(M, T, ysh[4 * grp], MAXD, &coef[4 * grp], cnt, 1 + (warp & 1));
            } else if (warp == W - 1 && A.kernel == 0) {
                // a warp without coefficients computes the next slice step's direction
                const int s1 = cur_step + 1;
                if (s1 < A.steps && e_next_step != s1) {
                    const double e1 = slice_direction(A, chain, iter, s1, lane, d);
                    if (lane < d) e_next[lane] = e1;
                    __syncwarp();
                    if (lane == 0) e_next_step = s1;
                }
            }
            __syncthreads();
            if (warp == 0) point_coef_join(M, T, coef, ns);
            // meanwhile the odd warp of each group of four: the fixed-point coefficients
            if (use_fx && (warp & 1) && 4 * grp < ns)
                coef_to_fx_group(T, M.n_det, &coef[4 * grp], &fx[4 * grp], min(4, ns - 4 * grp), fid);
            __syncthreads();
        } else {
            if (4 * warp < ns) {
                const int cnt = ns - 4 * warp < 4 ? ns - 4 * warp : 4;
                if (PREC == 1 && M.cdf)
                    point_coef_group_mx(M, T, ysh[4 * warp], MAXD, &coef[4 * warp], &cm[4 * warp], cnt,
                                        FORM == FORM_ROT);
                else
                    point_coef_group(M, T, ysh[4 * warp], MAXD, &coef[4 * warp], cnt);
                if (use_fx) {
                    __syncwarp();
                    coef_to_fx_group(T, M.n_det, &coef[4 * warp], &fx[4 * warp], cnt, fid);
                }
            }
            __syncthreads();
        }
        if (warp < ns && M.rb) {
            // relative-binning likelihood of the slot's candidate
            double v;
            if (PREC == 1) {
                coef_to_mixed_warp(coef[warp], M.n_det, M.df, &cm[warp], T.rb.fid);
                __syncwarp();
                v = rb_loglike_mixed<NDET>(M, T.rb, coef[warp], cm[warp], lane);
            } else {
                v = rb_loglike_fx<NDET>(M, T, coef[warp], fx[warp], sct);
            }
            if (lane == 0) {
                lval[warp] = v;
                coef[warp].jcut = T.rb.nb - 1;     // bins counted for the work statistics
            }
        } else if (PREC == 1 && S > 1 && S <= 4 && M.model == M_GW && !M.rb && M.coop) {
            // mixed, every warp on every candidate of the round: the tiled form
            // shares out the tile groups, the per-bin form strides the bins
            if (warp < ns && !M.cdf) coef_to_mixed_warp(coef[warp], M.n_det, M.df, &cm[warp], nullptr, FORM == FORM_ROT);
            if (lane == 0 && warp < ns) jc[warp] = coef[warp].jcut;
            __syncthreads();
            if (WS) {
                // work-shared: fixed chunks of tile groups, computed by this CTA's
                // warps and by helper CTAs, summed in chunk order into part[0]
                ws_owner_round<NDET, W>(M, T, A, cm, jc, ns, part[0]);
            } else if (FORM == FORM_ROT || M.tlg) {
                // items (candidate, r): the candidate's tile groups r, r + W, .., dealt to
                // the warps in turn, candidate after candidate; a candidate's sums
                // and their order do not depend on the round's other candidates.
                // (Candidate pairs by group, one after the other on the same warp, left
                // the warps past a pair's last group idle: most candidates of 64,897
                // bins end in their first or second group. GB300: 64,897 bins 8.9 -> 8.4 ms
                // per update, four served analyses 210 -> 181 ms; no spills left.)
                int it = 0;
                for (int c0 = 0; c0 < ns; c0++) {
                    const int ng = jc[c0] < 0 ? 0 : (jc[c0] >> (M.tlg + 5)) + 1;
                    for (int r = 0; r < min(ng, W); r++, it++) {
                        if ((it & (W - 1)) != warp) continue;
                        float zh[NDET][2], zl[NDET][2];
                        tile_bins_form<NDET, FORM>(M, T, cm[c0], jc[c0], r, W, zh, zl);
                        warp_sums_df_to<NDET>(zh, zl, &part[r][c0][0][0]);
                    }
                }
            } else {
                float zrh[S][NDET], zrl[S][NDET], zih[S][NDET], zil[S][NDET];
                bins_mixed_multi<NDET, S>(T, M.N, cm, jc, ns, threadIdx.x, W * 32, zrh, zrl, zih, zil);
#pragma unroll
                for (int sc = 0; sc < S; sc++)
#pragma unroll
                    for (int dd = 0; dd < NDET; dd++) {
                        warp_sum_df(zrh[sc][dd], zrl[sc][dd]);
                        warp_sum_df(zih[sc][dd], zil[sc][dd]);
                        if (lane == 0) {
                            part[warp][sc][dd][0] = (double)zrh[sc][dd] + (double)zrl[sc][dd];
                            part[warp][sc][dd][1] = (double)zih[sc][dd] + (double)zil[sc][dd];
                        }
                    }
            }
            __syncthreads();
            if (warp == 0) {
                // lane = (candidate, detector): sum over warps, then log L per candidate
                double v = 0.0;
                const int sc = lane / NDET, dd = lane % NDET;
                if (sc < ns && lane < S * NDET) {
                    double ZR = 0.0, ZI = 0.0;
                    // the parts: work-shared 1, tiled one per warp's groups (none beyond the last), per bin W
                    const int np = WS ? 1 : M.tlg ? min(W, (jc[sc] >> (M.tlg + 5)) + 1) : W;
                    for (int w2 = 0; w2 < np; w2++) { ZR += part[w2][sc][dd][0]; ZI += part[w2][sc][dd][1]; }
                    v = coef[sc].gre[dd] * ZR - coef[sc].gim[dd] * ZI;
                }
                const double t = group_sum_down<NDET>(v);
                if (dd == 0 && sc < ns && lane < S * NDET) lval[sc] = t - 0.5 * coef[sc].hh;
            }
        } else if (PREC == 0 && W > 1 && M.model == M_GW && !M.rb && tailmode == 2) {
            // FP64 above 1024 bins: each candidate's bins on two warps (on different
            // SM sub-partitions, each with its own FP32 and integer issue), row r on
            // lane r mod 32 of warp (r / 32) mod 2; the two warp sums meet in
            // shared memory in a fixed order, whatever the round.
            const int lg = 1;
            const int wpc = 1 << lg, cand = warp >> lg, sub = warp & (wpc - 1);
            if (cand < ns) {
                float zh[NDET][2], zl[NDET][2];
                bins_fx<NDET>(T, fx[cand], sct, sub * 32 + lane, wpc * 32, zh, zl);
                warp_sums_df_to<NDET>(zh, zl, &part[warp][0][0][0], T.fxs);
            }
            __syncthreads();
            if (warp == 0) {
                // lane = (candidate, detector): sum over the candidate's warps
                double v = 0.0;
                const int sc = lane / NDET, dd = lane % NDET;
                if (sc < ns && lane < S * NDET) {
                    double ZR = 0.0, ZI = 0.0;
                    for (int w2 = 0; w2 < wpc; w2++) {
                        ZR += part[sc * wpc + w2][0][dd][0];
                        ZI += part[sc * wpc + w2][0][dd][1];
                    }
                    v = coef[sc].gre[dd] * ZR - coef[sc].gim[dd] * ZI;
                }
                const double t = group_sum_down<NDET>(v);
                if (dd == 0 && sc < ns && lane < S * NDET) lval[sc] = t - 0.5 * coef[sc].hh;
            }
        } else if (warp < ns) {
            // one candidate per slot warp: bins and warp reduction
            double v = 0.0;
            if (PREC == 0) {
                if (M.model == M_GW) {
                    float zh[NDET][2], zl[NDET][2];
                    bins_fx<NDET>(T, fx[warp], sct, lane, 32, zh, zl);
                    v = warp_detector_terms_df<NDET>(zh, zl, coef[warp], T.fxs);
                }
            } else if (FORM == FORM_ROT || M.tlg) {
                if (!M.cdf) coef_to_mixed_warp(coef[warp], M.n_det, M.df, &cm[warp], nullptr, FORM == FORM_ROT);
                if (lane == 0) jc[warp] = coef[warp].jcut;
                __syncwarp();
                float zh[NDET][2], zl[NDET][2];
                tile_bins_form<NDET, FORM>(M, T, cm[warp], jc[warp], 0, 1, zh, zl);
                v = warp_detector_terms_df<NDET>(zh, zl, coef[warp]);
            } else {
                if (!M.cdf) coef_to_mixed_warp(coef[warp], M.n_det, M.df, &cm[warp], nullptr, FORM == FORM_ROT);
                __syncwarp();
                float zh[NDET][2], zl[NDET][2];
                bins_mixed<NDET>(T, M.N, cm[warp], coef[warp].jcut, lane, 32, zh, zl);
                v = warp_detector_terms_df<NDET>(zh, zl, coef[warp]);
            }
            if (lane == 0) lval[warp] = (M.model == M_TOY) ? coef[warp].toy : v - 0.5 * coef[warp].hh;
        }
        __syncthreads();
        if (warp == 0) {
            if (lane < ns) {
                cq.val[nbase + lane] = lval[lane];
                cq.bins[nbase + lane] = coef[lane].jcut + 1;
            }
            if (lane == 0) cs.c.ncache = nbase + ns;
            __syncwarp();
        }
        // coef/lval are rewritten only after the next barrier's plan
    }
    if (warp == 0) {
        Chain c;
        chain_load(cs, c, lane, d);
        const int dst = A.order[chain];
        if (lane < d) A.live_u[(size_t)dst * d + lane] = c.x;
        if (lane == 0) {
            A.live_logl[dst] = c.lx;
            if (A.active) atomicSub(A.active, 1);
            atomicAdd(&A.state->evals, (unsigned long long)c.evals);
            atomicAdd(&A.state->caps, (unsigned long long)c.caps);
            atomicAdd(&A.state->point_bins, c.bins);
            atomicAdd(&A.state->point_bins_lo, c.bins_lo);
            if (A.kernel == 1) atomicAdd(&A.state->walk_acc, (unsigned long long)c.s);
        }
    }
}

// At most 128 registers, so that 512 threads of chains fit on an SM: measured
// on GB300 against the uncapped 168 (3 CTAs of 4 warps per SM), c1 FP64 10.9 ->
// 9.8 ms, c1 mixed 4.7 -> 3.4 ms, c4 mixed 631 -> 550 ms per slice update, in
// spite of ~100 bytes of spills in the mixed tile loop.
#define SLICE_MIN_BLOCKS(PREC, S) (16 / (S))

template <int PREC, int NDET, int S, int W, int FORM>
__global__ void __launch_bounds__(W * 32, SLICE_MIN_BLOCKS(PREC, W)) k_slice(Model M, Tables T, StepArgs A) {
    slice_body<PREC, NDET, S, W, FORM>(M, T, A, blockIdx.x);
}

// One form of the tiled mixed sums per kernel, as in the serving kernels: with
// both, a chain's hot code is longer and its registers spill (GB300, 64,897 bins,
// slice update of 1000 chains: 10.4 -> 9.6 ms; ncu: instruction fetch is the largest stall).
template <int PREC, int NDET, int FORM>
cudaError_t slice_launch_form(const Model &M, const Tables &T, int slots, const StepArgs &A, cudaStream_t s) {
    switch (slots) {
        case 1: k_slice<PREC, NDET, 1, 1, FORM><<<A.k, 32, 0, s>>>(M, T, A); break;
        case 2: k_slice<PREC, NDET, 2, 2, FORM><<<A.k, 64, 0, s>>>(M, T, A); break;
        case 4: k_slice<PREC, NDET, 4, 4, FORM><<<A.k, 128, 0, s>>>(M, T, A); break;
        default: k_slice<PREC, NDET, 8, 8, FORM><<<A.k, 256, 0, s>>>(M, T, A); break;
    }
    return cudaGetLastError();
}

// The work-shared slice update: persistent CTAs (as many as fit on the GPU at
// once) take chains until none is left, then help the running ones.
template <int NDET>
__global__ void __launch_bounds__(256, SLICE_MIN_BLOCKS(1, 8)) k_slice_ws(Model M, Tables T, StepArgs A) {
    __shared__ int s_chain;
    for (int guard = 0; guard < (1 << 20); guard++) {
        if (threadIdx.x == 0) s_chain = atomicAdd(A.chain_ctr, 1);
        __syncthreads();
        const int chain = s_chain;
        __syncthreads();
        if (chain >= A.k) break;
        slice_body<1, NDET, 4, 8, FORM_ROT, true>(M, T, A, chain);
        __syncthreads();
    }
    ws_help<NDET, 8>(M, T, A);
}

// CTAs of the work-shared slice update that fit on one SM (0: not used for
// this precision).
template <int PREC, int NDET>
int slice_ws_blocks_per_sm() {
    if constexpr (PREC == 1) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_slice_ws<NDET>, 256, 0) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return nb;
    } else {
        return 0;
    }
}

template <int PREC, int NDET>
cudaError_t slice_launch(const Model &M, const Tables &T, int slots, const StepArgs &A, cudaStream_t s) {
    // on grids of 262,144 bins or more in tiles of 32 bins or more the tiled
    // mixed form with cooperative bins takes 8 warps for 4 slots: as many warps
    // per SM as 4-warp CTAs, twice as many per chain, so the update's last chains
    // finish sooner (GB300, 519,169 bins: 536 -> 467 ms per slice update; on
    // 64,897 bins, where an evaluation has a few tile groups, 15.2 -> 17.5 ms,
    // hence the threshold)
    if constexpr (PREC == 1) {
        if (slots == 4 && M.model == M_GW && M.coop && M.tlg >= 5 && !M.rb && M.N >= 262144) {
            if (A.ws) k_slice_ws<NDET><<<A.ws_nslot, 256, 0, s>>>(M, T, A);
            else k_slice<PREC, NDET, 4, 8, FORM_ROT><<<A.k, 256, 0, s>>>(M, T, A);
            return cudaGetLastError();
        }
        if (M.tlg >= 5) return slice_launch_form<PREC, NDET, FORM_ROT>(M, T, slots, A, s);
    }
    return slice_launch_form<PREC, NDET, FORM_DIRECT>(M, T, slots, A, s);
}

// Many analyses in one launch (serving), one form of the tiled mixed sums per
// kernel: the direct form for every analysis (FP64, per-bin and short-tile
// grids) or the rotation form for mixed grids with tiles of 32 bins or more.
// A kernel with both forms spilled registers (serving stream p50 4.0 -> 5.8 s).
template <int PREC, int NDET, int S, int FORM>
__global__ void __launch_bounds__(S * 32, SLICE_MIN_BLOCKS(PREC, S)) k_slice_multi(const Desc *D, const int2 *map) {
    __shared__ Desc d;
    const int2 ac = map[blockIdx.x];
    load_desc(D + ac.x, d);
    slice_body<PREC, NDET, S, S, FORM>(d.M, d.T, d.A, ac.y);
}

template <int PREC, int NDET, int FORM>
cudaError_t slice_multi_launch_form(const Desc *D, const int2 *map, int nblocks, int slots, cudaStream_t s) {
    switch (slots) {
        case 1: k_slice_multi<PREC, NDET, 1, FORM><<<nblocks, 32, 0, s>>>(D, map); break;
        case 2: k_slice_multi<PREC, NDET, 2, FORM><<<nblocks, 64, 0, s>>>(D, map); break;
        case 4: k_slice_multi<PREC, NDET, 4, FORM><<<nblocks, 128, 0, s>>>(D, map); break;
        default: k_slice_multi<PREC, NDET, 8, FORM><<<nblocks, 256, 0, s>>>(D, map); break;
    }
    return cudaGetLastError();
}

template <int PREC, int NDET>
cudaError_t slice_multi_launch(const Desc *D, const int2 *map, int nblocks, int slots, int rot, cudaStream_t s) {
    if constexpr (PREC == 1) {
        if (rot) return slice_multi_launch_form<PREC, NDET, FORM_ROT>(D, map, nblocks, slots, s);
    }
    return slice_multi_launch_form<PREC, NDET, FORM_DIRECT>(D, map, nblocks, slots, s);
}

// Explicit instantiation of the launchers of one (precision, detectors) pair.
#define GWNS_INSTANTIATE(P, D)                                                                       \
    template int slice_ws_blocks_per_sm<P, D>();                                                     \
    template cudaError_t eval_launch<P, D>(const Model &, const Tables &, int, int, const double *, int, int, \
                                           double *, RunState *, cudaStream_t);                     \
    template cudaError_t slice_launch<P, D>(const Model &, const Tables &, int, const StepArgs &,     \
                                            cudaStream_t);                                          \
    template cudaError_t slice_multi_launch<P, D>(const Desc *, const int2 *, int, int, int, cudaStream_t);

}  // namespace gwns
