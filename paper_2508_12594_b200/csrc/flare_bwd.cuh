// Backward of the FLARE mixer for float32 and float16 inputs (and the bfloat16 shapes the tensor-core kernels do not take);
// bfloat16 inputs otherwise take the tensor-core kernels with the same formulas.
//
// The paper times a backward pass without writing it out; these kernels apply the chain rule to its encode and
// decode equations (Section 3.2).  With S[m,n] = scale * q_m . k_n,
//   W_dec[n,m] = exp(S[m,n] - lse_dec[n]),   W_enc[m,n] = valid(n) ? exp(S[m,n] - lse_enc[m]) : 0,
// both softmax matrices are recomputed from the saved log-sum-exp rows, one score at a time:
//   pass A   dZ[m]  = sum_n W_dec[n,m] dY_n                      (the dZ form of encode_simt_kernel; split over N)
//   pass B   dd[n]  = dY_n . Y_n = sum_m W_dec[n,m] (dY_n . Z_m),   de[m] = dZ_m . Z_m
//            dS[m,n] = W_dec[n,m] (dY_n . Z_m - dd[n]) + W_enc[m,n] (dZ_m . V_n - de[m])
//            dV_n   = sum_m W_enc[m,n] dZ_m        dK_n = scale * sum_m dS[m,n] q_m       (rows are tokens)
//            dQ_m   = scale * sum_b sum_n dS[m,n] k_n                                     (rows are latents; split over N, then summed)
// dd[n] is formed from the dot products dY_n . Z_m rather than from the stored Y: Y has been rounded to
// the output type, and where the rows Z_m that a token mixes are nearly equal that rounding would dominate dS.
// Reductions add their partial results in a fixed order, so the gradients are bitwise reproducible.
//
// dd enters linearly, so the token side takes one sweep: dK_n = scale (T_n - dd[n] U_n), T without dd, U_n = sum_m W_dec[n,m] q_m, all products and
// sums in double, and dd[n] over the sum of the weights as they were rounded: where a token follows one latent, T and dd U agree to many digits, and
// what is left, (1 - W_dec) A q, takes 1 - W_dec from the other latents' weights instead of from the last digits of this one's.  (Two sweeps, dd first, took 5 D score products and three exponentials per pair instead of 3 D and two.)
//
// The kernels have the shape of the forward ones: row operands as A fragments in registers, column operands in
// shared memory, all products of a pair (q.k, dY.Z, dZ.V, and the contractions of dS and the weights) on the double-precision MMA, which is
// busy 55 to 65 % of the time: 6 D double multiply-adds per pair on the token side, 4 D in the dQ pass.  Neither a second tile buffer, nor
// twice the warps, nor the wider MMA shapes (m16n8k16) moved that.  us per training step, before (contractions as float32 FMAs, expf) -> now: float16
// 4 x 10007 tokens, M = 64, D = 16, 8 heads 487 -> 470; float32 2 x 9973 272 -> 249; 16384, M = 64, D = 32, 4 heads 236 -> 217; 10000, D = 64 389 -> 295.
// (Of these 12, 5, 3 and 1 are exp_diff's second term, and as much the products of dd and T in double.)
#pragma once

#include "flare_ptx.cuh"
#include "flare_common.cuh"
#include "flare_simt.cuh"

namespace flare {

// Row blocks of 8 per warp: three operands of a row and its accumulators are in registers.
template <int D> struct BwdSimtGeom {
    static constexpr int RB = D <= 16 ? 2 : 1;
    // token side: as many warps as the registers of three operands and three accumulators leave room for
    static constexpr int kTokThreads = D <= 32 ? 384 : 256, kTokRows = kTokThreads / 32 * 8 * RB;
};

// Pass B, token side.  Rows are tokens (8 RB per warp, the block's warps side by side).  grid = (ceil(N / kTokRows), H, B).
template <typename T, int D>
__global__ void __launch_bounds__(BwdSimtGeom<D>::kTokThreads, 1)
bwd_token_simt_kernel(const T *Q, const T *K, const T *V,
                      const uint8_t *key_mask, const T *dY, const float *Z,
                      const float *dZ, const float *de, const float *lse_enc,
                      const float *lse_dec, T *dK, T *dV,
                      float *dd_out, int B, int H, int N, int M, float scale) {
    ptx::grid_launch();
    ptx::grid_wait();
    using SG = SimtGeom<D>;
    constexpr int CT = SG::CT, RB = BwdSimtGeom<D>::RB, TH = BwdSimtGeom<D>::kTokThreads;
    extern __shared__ __align__(16) unsigned char simt_smem[];
    double *sQ = reinterpret_cast<double *>(simt_smem), *sZ = sQ + CT * SG::DK, *sDZ = sZ + CT * SG::DK;
    float *sLe = reinterpret_cast<float *>(sDZ + CT * SG::DK), *sDe = sLe + CT;   // (in the order of the MMA's indices)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, h = blockIdx.y, b = blockIdx.z;
    const int r0 = (blockIdx.x * (TH / 32) + warp) * 8 * RB;
    const size_t stride = (size_t)H * D, base = ((size_t)b * N * H + h) * D;
    const T *Qh = Q + (size_t)h * M * D;
    const size_t lat = ((size_t)b * H + h) * M;
    double ak[RB][D / 4], ag[RB][D / 4];
    load_rows<T, D, RB>(ak, K + base, stride, r0, N, (double)scale);
    load_rows<T, D, RB>(ag, dY + base, stride, r0, N, 1.0);
    float ld[RB];
    double dd[RB], sum[RB];
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        const int n = r0 + 8 * rb + (lane >> 2);
        ld[rb] = n < N ? lse_dec[((size_t)b * N + n) * H + h] : INFINITY;
        dd[rb] = sum[rb] = 0.0;
    }
    float *sC = sDe + CT;
    unsigned char *raw = reinterpret_cast<unsigned char *>(sC + D);
    TileFetch<T, D, TH> fq(raw);
    TileFetch<float, D, TH> fz(raw + fq.kBytes), fdz(raw + fq.kBytes + fz.kBytes);
    double av[RB][D / 4];
    load_rows<T, D, RB>(av, V + base, stride, r0, N, 1.0);
    bool valid[RB];
    double2 dk[RB][SG::NB], dv[RB][SG::NB], un[RB][SG::NB];         // T, dV, U
    clear_rows<D, RB>(dk);
    clear_rows<D, RB>(dv);
    clear_rows<D, RB>(un);
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        const int n = r0 + 8 * rb + (lane >> 2);
        valid[rb] = n < N && (key_mask == nullptr || key_mask[(size_t)b * N + n] != 0);
    }
    z_centre<D>(sC, Z + lat * D, M);
    fq.load(Qh, D, M);
    fz.load(Z + lat * D, D, M);
    fdz.load(dZ + lat * D, D, M);
    for (int m0 = 0; m0 < M; m0 += CT) {
        const int mc = min(CT, M - m0);
        fq.wait();
        __syncthreads();
        fq.put_double(sQ);
        fz.template put_double<true>(sZ, sC);
        fdz.put_double(sDZ);
        if (threadIdx.x < CT) {
            const int m = m0 + threadIdx.x;
            const float le = m < M ? lse_enc[lat + m] : -INFINITY;
            sLe[column_slot(threadIdx.x)] = le == -INFINITY ? -INFINITY : -le;   // added to the scores: weight 0 for a latent without valid tokens
            sDe[column_slot(threadIdx.x)] = m < M ? de[lat + m] : 0.f;
        }
        __syncthreads();
        if (m0 + CT < M) {
            fq.load(Qh + (size_t)(m0 + CT) * D, D, M - m0 - CT);
            fz.load(Z + (lat + m0 + CT) * D, D, M - m0 - CT);
            fdz.load(dZ + (lat + m0 + CT) * D, D, M - m0 - CT);
        }
        if (r0 < N)
            for (int nb = 0; nb < (mc + 7) / 8; ++nb) {
                double2 s[RB], a[RB], c[RB];
                mma_block<D, RB>(s, ak, sQ, nb);
                mma_block<D, RB>(a, ag, sZ, nb);
                mma_block<D, RB>(c, av, sDZ, nb);
                const int at = nb * 8 + 2 * (lane & 3);
                const float2 le = *reinterpret_cast<const float2 *>(sLe + at), dem = *reinterpret_cast<const float2 *>(sDe + at);
                const bool in0 = nb * 8 + column_slot(2 * (lane & 3)) < mc, in1 = nb * 8 + column_slot(2 * (lane & 3) + 1) < mc;
                double2 t[RB], wd[RB], we[RB];
#pragma unroll
                for (int rb = 0; rb < RB; ++rb) {
                    const float s0 = (float)s[rb].x, s1 = (float)s[rb].y;
                    wd[rb] = make_double2(in0 ? exp_diff(s0 - ld[rb]) : 0.f, in1 ? exp_diff(s1 - ld[rb]) : 0.f);
                    we[rb] = make_double2(in0 && valid[rb] ? exp_diff(s0 + le.x) : 0.f, in1 && valid[rb] ? exp_diff(s1 + le.y) : 0.f);
                    const double wa0 = wd[rb].x * a[rb].x, wa1 = wd[rb].y * a[rb].y;
                    dd[rb] += wa0 + wa1;
                    sum[rb] += wd[rb].x + wd[rb].y;
                    // (de is a rounded sum: rounded alike, the two cancel where a latent follows a single token)
                    t[rb] = make_double2(fma(we[rb].x, (double)((float)c[rb].x - dem.x), wa0), fma(we[rb].y, (double)((float)c[rb].y - dem.y), wa1));
                }
                double v[2][SG::NB];
                load_values<D>(v, sQ, nb);
                add_values<D, RB>(dk, t, v);
                add_values<D, RB>(un, wd, v);
                load_values<D>(v, sDZ, nb);
                add_values<D, RB>(dv, we, v);
            }
    }
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        const int n = r0 + 8 * rb + (lane >> 2);
        dd[rb] = quad_sum(dd[rb]);
        sum[rb] = quad_sum(sum[rb]);
        if (fabs(sum[rb] - 1.0) < 1e-3) dd[rb] /= sum[rb];          // (0 where a caller has switched the stage off)
#pragma unroll
        for (int j = 0; j < SG::NB; ++j)
            dk[rb][j] = make_double2(dk[rb][j].x - dd[rb] * un[rb][j].x, dk[rb][j].y - dd[rb] * un[rb][j].y);
        if (n < N) {
            if ((lane & 3) == 0) dd_out[((size_t)b * H + h) * N + n] = (float)dd[rb];
            write_row<T, D>(dK + base + (size_t)n * stride, dk[rb], scale);
            write_row<T, D>(dV + base + (size_t)n * stride, dv[rb], 1.0);
        }
    }
}
template <typename T, int D> inline size_t bwd_token_simt_smem() {
    using SG = SimtGeom<D>;
    return sizeof(double) * 3 * SG::CT * SG::DK + sizeof(float) * (2 * SG::CT + D) + (sizeof(T) + 2 * sizeof(float)) * SG::CT * D;
}

// Pass B, latent side: partial dQ rows.  Rows are latents, columns tokens; grid and warps as in encode_simt_kernel.
template <typename T, int D>
__global__ void __launch_bounds__(kBwdThreads, D <= 32 ? 2 : 1)
bwd_dq_simt_kernel(const T *Q, const T *K, const T *V,
                   const uint8_t *key_mask, const T *dY, const float *Z,
                   const float *dZ, const float *de, const float *dd,
                   const float *lse_enc, const float *lse_dec, float *part,
                   int B, int H, int N, int M, int WM, int mblocks, int chunk, float scale) {
    ptx::grid_launch();
    ptx::grid_wait();
    using SG = SimtGeom<D>;
    constexpr int CT = SG::CT, RB = BwdSimtGeom<D>::RB, RW = 8 * RB;
    extern __shared__ __align__(16) unsigned char simt_smem[];
    double *sK = reinterpret_cast<double *>(simt_smem), *sG = sK + CT * SG::DK, *sV = sG + CT * SG::DK;
    float *sLd = reinterpret_cast<float *>(sV + CT * SG::DK), *sDd = sLd + CT, *sMask = sDd + CT;   // (in the order of the MMA's indices)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = blockIdx.x, h = blockIdx.y / mblocks, mb = blockIdx.y % mblocks, b = blockIdx.z;
    const int WT = kBwdThreads / 32 / WM, wm = warp % WM, wt = warp / WM;
    const int rbase = mb * WM * RW, r0 = rbase + wm * RW;
    const int n0 = split * chunk, n1 = min(N, n0 + chunk);
    const size_t stride = (size_t)H * D, base = ((size_t)b * N * H + h) * D;
    const size_t lat = ((size_t)b * H + h) * M;
    double aq[RB][D / 4], az[RB][D / 4], adz[RB][D / 4];
    load_rows<T, D, RB>(aq, Q + (size_t)h * M * D, D, r0, M, (double)scale);
    float *sC = sMask + CT;
    z_centre<D>(sC, Z + lat * D, M);
    __syncthreads();
    load_rows<float, D, RB>(az, Z + lat * D, D, r0, M, 1.0, sC);
    load_rows<float, D, RB>(adz, dZ + lat * D, D, r0, M, 1.0);
    float nle[RB], dem[RB];
    double2 acc[RB][SG::NB];
    clear_rows<D, RB>(acc);
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        const int m = r0 + 8 * rb + (lane >> 2);
        const float le = m < M ? lse_enc[lat + m] : -INFINITY;
        nle[rb] = le == -INFINITY ? -INFINITY : -le;
        dem[rb] = m < M ? de[lat + m] : 0.f;
    }
    using Fetch = TileFetch<T, D, kBwdThreads>;
    unsigned char *raw = reinterpret_cast<unsigned char *>(sC + D);
    Fetch fk(raw), fg(raw + Fetch::kBytes), fv(raw + 2 * Fetch::kBytes);
    auto fetch = [&](int t0) {
        const size_t at = base + (size_t)t0 * stride;
        fk.load(K + at, stride, n1 - t0);
        fg.load(dY + at, stride, n1 - t0);
        fv.load(V + at, stride, n1 - t0);
    };
    fetch(n0);
    for (int t0 = n0; t0 < n1; t0 += CT) {
        Fetch::wait();
        __syncthreads();
        fk.put_double(sK);
        fg.put_double(sG);
        fv.put_double(sV);
        if (threadIdx.x < CT) {
            const int n = t0 + threadIdx.x;
            const bool in = n < n1;
            sLd[column_slot(threadIdx.x)] = in ? -lse_dec[((size_t)b * N + n) * H + h] : -INFINITY;
            sDd[column_slot(threadIdx.x)] = in ? dd[((size_t)b * H + h) * N + n] : 0.f;
            sMask[column_slot(threadIdx.x)] = in && (key_mask == nullptr || key_mask[(size_t)b * N + n] != 0) ? 0.f : -INFINITY;
        }
        __syncthreads();
        if (t0 + CT < n1) fetch(t0 + CT);
        const int blocks = (min(CT, n1 - t0) + 7) / 8;
        if (r0 < M)
            for (int nb = wt; nb < blocks; nb += WT) {
                double2 s[RB], a[RB], c[RB];
                mma_block<D, RB>(s, aq, sK, nb);
                mma_block<D, RB>(a, az, sG, nb);
                mma_block<D, RB>(c, adz, sV, nb);
                const int at = nb * 8 + 2 * (lane & 3);
                const float2 nld = *reinterpret_cast<const float2 *>(sLd + at), ddn = *reinterpret_cast<const float2 *>(sDd + at);
                const float2 msk = *reinterpret_cast<const float2 *>(sMask + at);
                float2 ds[RB];
#pragma unroll
                for (int rb = 0; rb < RB; ++rb) {
                    const float s0 = (float)s[rb].x, s1 = (float)s[rb].y;
                    const float we0 = exp_diff((s0 + nle[rb]) + msk.x), we1 = exp_diff((s1 + nle[rb]) + msk.y);
                    ds[rb] = make_float2(exp_diff(s0 + nld.x) * ((float)a[rb].x - ddn.x) + we0 * ((float)c[rb].x - dem[rb]),
                                         exp_diff(s1 + nld.y) * ((float)a[rb].y - ddn.y) + we1 * ((float)c[rb].y - dem[rb]));
                }
                double v[2][SG::NB];
                load_values<D>(v, sK, nb);
                add_values<D, RB>(acc, ds, v);
            }
    }
    __syncthreads();
    // the shares of the columns meet
    constexpr int ROW = D + 4;
    float *sR = reinterpret_cast<float *>(simt_smem);
    const int rows_here = WM * RW;
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        write_row<float, D>(sR + ((size_t)wt * rows_here + wm * RW + 8 * rb + (lane >> 2)) * ROW, acc[rb], 1.0);
    }
    __syncthreads();
    const long rows = (long)B * H * M;
    for (int i = threadIdx.x; i < rows_here * D; i += kBwdThreads) {
        const int r = i / D, d = i % D, m = rbase + r;
        if (m >= M) continue;
        float z = 0.f;
        for (int w = 0; w < WT; ++w) z += sR[((size_t)w * rows_here + r) * ROW + d];
        part[((size_t)split * rows + lat + m) * D + d] = z;
    }
}
template <typename T, int D> inline size_t bwd_dq_simt_smem() {
    using SG = SimtGeom<D>;
    const size_t tiles = sizeof(double) * 3 * SG::CT * SG::DK + sizeof(float) * (3 * SG::CT + D) + 3 * sizeof(T) * SG::CT * D;
    const size_t join = sizeof(float) * (kBwdThreads / 32) * 8 * BwdSimtGeom<D>::RB * (D + 4);
    return tiles > join ? tiles : join;
}

}  // namespace flare
