// Linear-time spectral analysis of the induced mixing matrix (paper: spectral-analysis appendix, Algorithm 1).
//
// With A = exp(S), S = scale * Q K^T, L_M = diag(1 / row sums of A) and L_N = diag(1 / column sums of A), the mixing
// matrix W = W_dec W_enc = L_N A^T L_M A has the non-zero eigenvalues of the M x M matrix G = J J^T,
// J = L_M^{1/2} A L_N^{1/2}.  With the log-sum-exp rows the forward already produces,
//     J[m,n] = exp(S[m,n] - lse_enc[m] / 2 - lse_dec[n] / 2),        G[m,m'] = sum_n J[m,n] J[m',n],
// so G is one more reduction over the tokens in which every (latent, token) pair costs one exponential (as in
// encode) and every pair of latents one multiply-add per token: 2 N M^2 FLOP per head, O(M^2) memory.  Nothing
// of size M x N or N x N is written.  The M x M symmetric eigenproblem is O(M^3), off the hot path.
//
//   spectral_gram_tc_kernel    bfloat16, M <= 128, D in {16, 32}: tcgen05.  A CTA takes one head and a range of
//                              tokens; the head's latents sit on the 128 TMEM lanes.  Per 32 tokens: S = Q K^T; 128
//                              threads form J as two bf16 halves (hi + lo): hi back over the scores (the A operand of the
//                              next MMAs), hi and 2 lo into shared memory (their B operands); X += hi hi^T + 2 hi lo^T with
//                              the accumulator in TMEM.  G = (X + X^T) / 2 = hi hi^T + hi lo^T + lo hi^T, taken when the
//                              splits are summed: two products instead of three (eight heads of 131072 tokens, M = 128,
//                              D = 32: 113 -> 106 us).  (The diagonal of G is a sum of squares: with single
//                              bf16 factors nothing cancels and G is off by 4e-3 of its largest entries.)
//   spectral_gram_simt_kernel  everything else (float32 inputs, other shapes): CUDA cores, a 16 x 16 tile of G per block.
//   spectral_gram_reduce_kernel sums the token splits and writes the symmetric G.
//   spectral_jacobi_kernel     eigenvalues and eigenvectors of G by cyclic two-sided Jacobi rotations.
//   spectral_tridiag_*kernel, spectral_bisect_kernel   eigenvalues alone: Householder tridiagonalisation, then bisection.
#pragma once

#include "flare_common.cuh"
#include "flare_ptx.cuh"
#include "flare_tc.cuh"

namespace flare {

struct SpectralArgs {
    const __nv_bfloat16 *Q;   // [H,M,D]
    const float *lse_enc;     // [B,H,M]
    const float *lse_dec;     // [B,N,H]
    float *part;              // [splits * kSpectralGroups][B*H][128][128] float32 partial sums of G
    uint32_t *status;
    int B, H, N, M;
    float sl2;                // scale * log2(e)
    int tiles, splits;
};

// Groups of 128 threads at work in a CTA of the tensor-core Gram kernel: each takes every third token tile with its own
// score buffer, accumulator (160 of the 512 tensor-memory columns) and partial sum.
constexpr int kSpectralGroups = 3;

template <int D>
struct SpectralSmem {
    using G = TileGeom<D>;
    static constexpr int kStages = 6;
    static constexpr size_t k_off = 0;                                      // K tiles
    static constexpr size_t q_off = (size_t)kStages * G::TILE_BYTES;        // Q rows
    static constexpr size_t pb_off = q_off + (size_t)kTile * G::RB;         // J (hi, lo) as B operands: [128 latents, 32 tokens] bf16 each
    static constexpr size_t kPbBytes = (size_t)kTile * 64;
    static constexpr size_t col_off = pb_off + kSpectralGroups * 2 * kPbBytes;   // (a hi and a lo tile per group); per softmax warp 32 column addends
    static constexpr size_t bar_off = (col_off + kSpectralGroups * 4 * 32 * sizeof(float) + 1023) & ~(size_t)1023;
    static constexpr size_t total = bar_off + 512 + 1024 < kTcMinSmem ? kTcMinSmem : bar_off + 512 + 1024;
};

// grid = (splits, H, B).  Warp 0: TMA; warps 1-3: MMA issue, one per group; warps 5-16: three groups of 128 threads, the
// latent rows on their lanes.  Group g works on the tiles g, g + 3, ... of the CTA's range and leaves its own partial sum.
template <int D>
__global__ void __launch_bounds__(kTcThreads, 1)
spectral_gram_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ, SpectralArgs a) {
    using G = TileGeom<D>;
    using GP = TileGeom<32>;                                    // the J tiles in shared memory: 32 tokens = 64 bytes per latent row
    using SM = SpectralSmem<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = ptx::align_1024(smem_raw);
    uint8_t *sK = smem + SM::k_off, *sQ = smem + SM::q_off, *sPB = smem + SM::pb_off;
    float *colneg = reinterpret_cast<float *>(smem + SM::col_off);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + SM::bar_off);
    constexpr int kStages = SM::kStages, UNIT = 32;
    constexpr int NGS = kSpectralGroups;
    enum { K_FULL = 0, K_EMPTY = K_FULL + kStages, Q_FULL = K_EMPTY + kStages, S_FULL, P_FULL = S_FULL + NGS,
           G_DONE = P_FULL + NGS, NBARS = G_DONE + NGS };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + NBARS);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    // tensor memory, per group 160 columns: G [0,128)  S [128,160)
    constexpr uint32_t G_AA = 0, S_A = 128, GROUP_COLS = 160, NCOLS = 512;

    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const int split = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int M = a.M;
    const int t_begin = (int)((long)a.tiles * split / a.splits), t_end = (int)((long)a.tiles * (split + 1) / a.splits);
    const int nt = t_end - t_begin;
    auto bar = [&](int i) { return ptx::smem_u32(bars + i); };

    if (threadIdx.x == 0) {
        for (int i = 0; i < NBARS; ++i) ptx::mbar_init(bar(i), (i >= P_FULL && i < P_FULL + NGS) ? 4u : 1u);   // P_FULL: one arrival per warp
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmK);
        ptx::prefetch_tensormap(&tmQ);
    }
    if (warp == kFirstIssuerWarp) ptx::tmem_alloc(ptx::smem_u32(tmem_slot), NCOLS);
    ptx::grid_launch();
    ptx::grid_wait();
    for (int i = threadIdx.x; i < kTile * (G::RB / 16); i += kTcThreads)          // latent rows beyond M stay zero
        reinterpret_cast<uint4 *>(sQ)[i] = make_uint4(0, 0, 0, 0);
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = *tmem_slot;

    if (warp == 0) {
        if (ptx::elect_one()) {
            ptx::mbar_arrive_expect_tx(bar(Q_FULL), (uint32_t)(M * G::RB));
            for (int r = 0; r < M; r += 16) ptx::tma_load_2d(ptx::smem_u32(sQ + (size_t)r * G::RB), &tmQ, bar(Q_FULL), 0, h * M + r);
            for (int i = 0; i < nt; ++i) {
                const int s = i % kStages;
                if (!ptx::mbar_wait(bar(K_EMPTY + s), ((i / kStages) & 1) ^ 1, abort_flag, kErrSpectral | 1)) break;
                ptx::mbar_arrive_expect_tx(bar(K_FULL + s), G::TILE_BYTES);
                ptx::tma_load_3d(ptx::smem_u32(sK + (size_t)s * G::TILE_BYTES), &tmK, bar(K_FULL + s), h * D, (t_begin + i) * kTile, b);
            }
        }
    } else if (warp >= kFirstIssuerWarp && warp < kFirstIssuerWarp + NGS) {
        const int g = warp - kFirstIssuerWarp;
        const int mytiles = (nt - g + NGS - 1) / NGS;
        const uint32_t gtm = tm + g * GROUP_COLS;
        if (ptx::elect_one()) {
            const uint32_t idescS = ptx::instr_desc_bf16(128, UNIT, 0, 0), idescG = ptx::instr_desc_bf16(128, 128, 0, 0);
            const uint64_t qdesc = ptx::smem_desc(ptx::smem_u32(sQ), 16, G::SBO, G::SWZ);
            const uint64_t pbdesc = ptx::smem_desc(ptx::smem_u32(sPB + (size_t)g * 2 * SM::kPbBytes), 16, GP::SBO, GP::SWZ);
            bool ok = ptx::mbar_wait(bar(Q_FULL), 0, abort_flag, kErrSpectral | 2);
            const int units = 4 * mytiles;
            auto issue_scores = [&](int u) -> bool {              // unit u: the group's tile u / 4, tokens 32 (u % 4) ... of it
                const int i = g + NGS * (u >> 2), s = i % kStages;
                if ((u & 3) == 0 && !ptx::mbar_wait(bar(K_FULL + s), (i / kStages) & 1, abort_flag, kErrSpectral | 3)) return false;
                ptx::tc_fence_after();
                const uint64_t kdesc = ptx::smem_desc(ptx::smem_u32(sK + (size_t)s * G::TILE_BYTES), 16, G::SBO, G::SWZ) +
                                       (uint64_t)(((u & 3) * UNIT * G::RB) >> 4);
#pragma unroll
                for (int k = 0; k < D / 16; ++k) ptx::mma_ss(gtm + S_A, qdesc + 2 * k, kdesc + 2 * k, idescS, k > 0);
                ptx::mma_commit(bar(S_FULL + g));
                if ((u & 3) == 3) ptx::mma_commit(bar(K_EMPTY + s));
                return true;
            };
            if (ok && units > 0) ok = issue_scores(0);
            for (int u = 0; ok && u < units; ++u) {
                if (!ptx::mbar_wait(bar(P_FULL + g), u & 1, abort_flag, kErrSpectral | 4)) break;
                ptx::tc_fence_after();
                // X += hi (hi + 2 lo)^T over the unit's 32 tokens (two k-steps of 16): A = hi in tensor memory (the first 16 columns
                // of the score buffer), B in shared memory (hi tile, then 2 lo tile)
                constexpr uint64_t LO = (uint64_t)(SM::kPbBytes >> 4);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const uint32_t acc = (u > 0 || k > 0 || t > 0) ? 1u : 0u;
                        ptx::mma_ts(gtm + G_AA, gtm + S_A + 8 * k, pbdesc + (t == 1 ? LO : 0) + 2 * k, idescG, acc);
                    }
                }
                // the next unit's scores overwrite J in tensor memory after those MMAs (a thread's MMAs run in order); the
                // commit behind them also tells the threads that J in shared memory has been read
                if (u + 1 < units) ok = issue_scores(u + 1);
                else ptx::mma_commit(bar(G_DONE + g));
            }
        }
    } else if (warp >= kFirstSoftmaxWarp && warp < kFirstSoftmaxWarp + 4 * NGS) {
        const int g = (warp - kFirstSoftmaxWarp) >> 2;
        const int mytiles = (nt - g + NGS - 1) / NGS;
        const int row = ((warp & 3) << 5) + lane;               // TMEM lane = latent
        const int m = row;
        const uint32_t lane_addr = (uint32_t)((warp & 3) << 5) << 16;
        const uint32_t scol = tm + lane_addr + g * GROUP_COLS + S_A;
        float *cn = colneg + (warp - kFirstSoftmaxWarp) * 32;
        const float rowneg = m < M ? -0.5f * 1.4426950408889634f * a.lse_enc[((size_t)b * a.H + h) * M + m] : -INFINITY;
        const float2 sl2p = make_float2(a.sl2, a.sl2);
        uint8_t *pb = sPB + (size_t)g * 2 * SM::kPbBytes + (size_t)row * GP::RB;   // this latent's row of the group's hi tile; 2 lo: kPbBytes on
        bool ok = true;
        const int units = 4 * mytiles;
        auto column = [&](int u) {                              // lse_dec of this lane's token of unit u
            const int n = (t_begin + g + NGS * (u >> 2)) * kTile + (u & 3) * UNIT + lane;
            return u < units && n < a.N ? a.lse_dec[((size_t)b * a.N + n) * a.H + h] : INFINITY;
        };
        float ld = column(0);                                   // (fetched a unit ahead)
        for (int u = 0; ok && u < units; ++u) {
            __syncwarp();
            cn[lane] = -0.5f * 1.4426950408889634f * ld;
            ld = column(u + 1);
            __syncwarp();
            if (!(ok = warp_wait(bar(S_FULL + g), u & 1, abort_flag, kErrSpectral | 5))) break;
            ptx::tc_fence_after();
            uint32_t r[32], hi[16], lo[16];
            ptx::tmem_ld32(scol, r);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 8; ++k) {                       // J = 2^(s sl2 + rowneg + colneg[n]); -inf rows and columns give 0
                const float4 ng = *reinterpret_cast<const float4 *>(cn + 4 * k);
                const float2 x0 = __ffma2_rn(make_float2(__uint_as_float(r[4 * k]), __uint_as_float(r[4 * k + 1])), sl2p,
                                             make_float2(ng.x + rowneg, ng.y + rowneg));
                const float2 x1 = __ffma2_rn(make_float2(__uint_as_float(r[4 * k + 2]), __uint_as_float(r[4 * k + 3])), sl2p,
                                             make_float2(ng.z + rowneg, ng.w + rowneg));
                const float p0 = ptx::ex2(x0.x), p1 = ptx::ex2(x0.y), p2 = ptx::ex2(x1.x), p3 = ptx::ex2(x1.y);
                const uint32_t h0 = ptx::pack_bf16(p0, p1), h1 = ptx::pack_bf16(p2, p3);
                hi[2 * k] = h0;
                hi[2 * k + 1] = h1;
                const float2 l0 = ptx::rest_of(make_float2(p0, p1), h0), l1 = ptx::rest_of(make_float2(p2, p3), h1);
                lo[2 * k] = ptx::pack_bf16(__fadd2_rn(l0, l0));
                lo[2 * k + 1] = ptx::pack_bf16(__fadd2_rn(l1, l1));
            }
            ptx::tmem_st16(scol, hi);                           // A operand: back over the scores
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {                    // B operand: this latent's 64-byte rows, 16-byte chunks swizzled
                *reinterpret_cast<uint4 *>(pb + ((ch ^ GP::swz(row)) << 4)) = make_uint4(hi[4 * ch], hi[4 * ch + 1], hi[4 * ch + 2], hi[4 * ch + 3]);
                *reinterpret_cast<uint4 *>(pb + SM::kPbBytes + ((ch ^ GP::swz(row)) << 4)) =
                    make_uint4(lo[4 * ch], lo[4 * ch + 1], lo[4 * ch + 2], lo[4 * ch + 3]);
            }
            ptx::fence_proxy_async_smem();
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(P_FULL + g));
        }
        // the partial sum X: this thread's lane holds row m
        if (ok && units > 0) ok = warp_wait(bar(G_DONE + g), 0, abort_flag, kErrSpectral | 6);
        ptx::tc_fence_after();
        if (ok) {
            float *dst = a.part + ((((size_t)split * NGS + g) * a.B + b) * a.H + h) * (size_t)kTile * kTile + (size_t)row * kTile;
#pragma unroll 1
            for (int c0 = 0; c0 < kTile; c0 += 32) {
                uint32_t v[32];
                if (units > 0) {
                    ptx::tmem_ld32(tm + lane_addr + g * GROUP_COLS + G_AA + c0, v);
                    ptx::tmem_wait_ld();
                } else {
#pragma unroll
                    for (int k = 0; k < 32; ++k) v[k] = 0u;
                }
#pragma unroll
                for (int k = 0; k < 32; k += 4)
                    *reinterpret_cast<float4 *>(dst + c0 + k) = make_float4(__uint_as_float(v[k]), __uint_as_float(v[k + 1]),
                                                                            __uint_as_float(v[k + 2]), __uint_as_float(v[k + 3]));
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kFirstIssuerWarp) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tm, NCOLS);
    }
    if (threadIdx.x == 0 && *abort_flag != 0 && a.status != nullptr) atomicCAS(a.status, 0u, *abort_flag);
}

// Sum of the token splits X into G [B,H,M,M] = (X + X^T) / 2.  grid = (heads, pairs of 16 x 16 blocks (i, j), i <= j): both blocks of X are
// read by rows and meet in shared memory.
constexpr int kGramTile = 16;
__host__ __device__ constexpr int gram_tile_pairs(int M) { return ((M + kGramTile - 1) / kGramTile) * ((M + kGramTile - 1) / kGramTile + 1) / 2; }
static __global__ void __launch_bounds__(kGramTile *kGramTile)
spectral_gram_reduce_kernel(const float *part, float *Gout, int splits, long heads, int M) {
    ptx::grid_launch();
    ptx::grid_wait();
    __shared__ float lower[kGramTile][kGramTile + 1], upper[kGramTile][kGramTile + 1];
    int ti = 0, tj = blockIdx.y;                                // pair number -> (ti, tj), tj >= ti
    for (int row = (M + kGramTile - 1) / kGramTile; tj >= row; --row) {
        tj -= row;
        ++ti;
    }
    tj += ti;
    const int r = threadIdx.x / kGramTile, c = threadIdx.x % kGramTile;
    const float *x = part + (size_t)blockIdx.x * kTile * kTile;
    const size_t up = (size_t)(ti * kGramTile + r) * kTile + tj * kGramTile + c, low = (size_t)(tj * kGramTile + r) * kTile + ti * kGramTile + c;
    float u = 0.f, l = 0.f;
#pragma unroll 6
    for (int p = 0; p < splits; ++p) {
        const float *xp = x + (size_t)p * heads * kTile * kTile;
        u += xp[up];
        l += xp[low];
    }
    upper[r][c] = u;
    lower[r][c] = l;
    __syncthreads();
    float *g = Gout + (size_t)blockIdx.x * M * M;
    const int i = ti * kGramTile + r, j = tj * kGramTile + c, i2 = tj * kGramTile + r, j2 = ti * kGramTile + c;
    if (i < M && j < M) g[(size_t)i * M + j] = 0.5f * (u + lower[c][r]);
    if (ti != tj && i2 < M && j2 < M) g[(size_t)i2 * M + j2] = 0.5f * (upper[c][r] + l);
}

// Score q.k of one (latent, token) pair.  For float32 and float16 inputs the products are summed in double so that
// the score, which is exponentiated, carries no float32 summation error; bfloat16 inputs sum in float.
template <typename T, int D>
__device__ __forceinline__ float score_dot(const float (&a)[D], const float *b) {
    if constexpr (!std::is_same<T, __nv_bfloat16>::value) {   // float32 and float16 inputs
        double s = 0.0;
#pragma unroll
        for (int d = 0; d < D; ++d) s = fma((double)a[d], (double)b[d], s);
        return (float)s;
    } else {
        float s = 0.f;
#pragma unroll
        for (int d = 0; d < D; ++d) s = fmaf(a[d], b[d], s);
        return s;
    }
}

// G on the CUDA cores, for everything the tensor-core kernel does not take: one block per 16 x 16 tile of G of
// one (b, h); the tokens are walked in chunks of 64 whose J rows for the tile's 16 + 16 latents sit in shared memory.
template <typename T, int D>
__global__ void __launch_bounds__(256)
spectral_gram_simt_kernel(const T *__restrict__ Q, const T *__restrict__ K, const float *__restrict__ lse_enc,
                          const float *__restrict__ lse_dec, float *__restrict__ Gout, int B, int H, int N, int M, float scale) {
    constexpr int TN = 64;
    __shared__ float sQ[32][D];
    __shared__ float sK[TN][D];
    __shared__ float sJ[32][TN + 1];
    __shared__ float sLe[32];
    const int tiles_m = (M + 15) / 16;
    const int ti = blockIdx.x / tiles_m, tj = blockIdx.x % tiles_m, h = blockIdx.y, b = blockIdx.z;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    for (int i = threadIdx.x; i < 32 * D; i += 256) {
        const int rr = i / D, d = i % D, m = (rr < 16 ? ti * 16 + rr : tj * 16 + rr - 16);
        sQ[rr][d] = m < M ? to_f32(Q[((size_t)h * M + m) * D + d]) * scale : 0.f;
        if (d == 0) sLe[rr] = m < M ? lse_enc[((size_t)b * H + h) * M + m] : INFINITY;
    }
    float acc = 0.f;
    for (int n0 = 0; n0 < N; n0 += TN) {
        __syncthreads();
        for (int i = threadIdx.x; i < TN * D; i += 256) {
            const int jn = i / D, d = i % D, n = n0 + jn;
            sK[jn][d] = n < N ? to_f32(K[(((size_t)b * N + n) * H + h) * D + d]) : 0.f;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 32 * TN; i += 256) {
            const int rr = i / TN, jn = i % TN, n = n0 + jn;
            float q[D];
#pragma unroll
            for (int d = 0; d < D; ++d) q[d] = sQ[rr][d];
            const float s = score_dot<T, D>(q, sK[jn]);
            sJ[rr][jn] = n < N ? expf(s - 0.5f * sLe[rr] - 0.5f * lse_dec[((size_t)b * N + n) * H + h]) : 0.f;
        }
        __syncthreads();
#pragma unroll 8
        for (int jn = 0; jn < TN; ++jn) acc = fmaf(sJ[ty][jn], sJ[16 + tx][jn], acc);
    }
    const int mi = ti * 16 + ty, mj = tj * 16 + tx;
    if (mi < M && mj < M) Gout[(((size_t)b * H + h) * M + mi) * M + mj] = acc;
}

// A matrix that holds a NaN or an infinity has no eigenvalues: every output for it is NaN.  (Maxima, comparisons and rotations
// drop a NaN: left to them, a matrix of NaN comes out with eigenvalues 0, as if of rank 0.)
constexpr float kEigNan = __builtin_nanf("");
// All threads of the block call it.
__device__ __forceinline__ bool eig_broken(const float *G, int M) {
    bool bad = false;
    for (int i = threadIdx.x; i < M * M; i += blockDim.x) bad |= !isfinite(G[i]);
    return __syncthreads_or(bad);
}

// Eigenvalues (descending) and eigenvectors (columns of U) of the symmetric matrices G [heads, M, M], by cyclic two-sided Jacobi
// rotations on disjoint index pairs (round-robin ordering: M - 1 steps of M / 2 rotations per sweep).  One block per matrix; G is overwritten.  Off the hot path: O(M^3) per sweep, about ten sweeps.
static __global__ void __launch_bounds__(1024)
spectral_jacobi_kernel(float *__restrict__ Gall, float *__restrict__ evals, float *__restrict__ Uall, int M, int sweeps) {
    extern __shared__ float sh[];
    float *cs = sh;                         // [M/2 pairs] cosines, then sines
    int *pp = reinterpret_cast<int *>(sh + 2 * ((M + 1) / 2));   // [pairs] p, then q; then [M] ranks
    float *G = Gall + (size_t)blockIdx.x * M * M;
    float *U = Uall + (size_t)blockIdx.x * M * M;
    const int Me = (M + 1) & ~1, pairs = Me / 2, t = threadIdx.x, T = blockDim.x;
    if (eig_broken(G, M)) {
        for (int i = t; i < M; i += T) evals[(size_t)blockIdx.x * M + i] = kEigNan;
        for (int i = t; i < M * M; i += T) U[i] = kEigNan;
        return;
    }
    for (int i = t; i < M * M; i += T) U[i] = (i / M == i % M) ? 1.f : 0.f;
    __syncthreads();
    // A sweep that met no off-diagonal element above 2^-22 of the largest diagonal one (float32 rotations change nothing
    // below that) was the last: six to eight sweeps in practice instead of the twelve allowed.
    __shared__ unsigned off_max, diag_max;                      // bit patterns of non-negative floats order like the floats
    for (int sweep = 0; sweep < sweeps; ++sweep) {
        if (t == 0) { off_max = 0u; diag_max = 0u; }
        __syncthreads();
        for (int i = t; i < M; i += T) atomicMax(&diag_max, __float_as_uint(fabsf(G[(size_t)i * M + i])));
        for (int step = 0; step < Me - 1; ++step) {
            // round-robin pairing of 0 .. Me-1 (index Me-1 fixed); an index >= M is a bye
            for (int k = t; k < pairs; k += T) {
                int p = k == 0 ? Me - 1 : (step + k) % (Me - 1);
                int q = (step + Me - 1 - k) % (Me - 1);
                if (p > q) { const int tmp = p; p = q; q = tmp; }
                float c = 1.f, s = 0.f;
                if (q < M) {
                    const float gpq = G[(size_t)p * M + q];
                    atomicMax(&off_max, __float_as_uint(fabsf(gpq)));
                    if (fabsf(gpq) > 1e-30f) {
                        const float tau = (G[(size_t)q * M + q] - G[(size_t)p * M + p]) / (2.f * gpq);
                        const float tt = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
                        c = rsqrtf(1.f + tt * tt);
                        s = tt * c;
                    }
                }
                cs[k] = c; cs[pairs + k] = s; pp[k] = p; pp[pairs + k] = q;
            }
            __syncthreads();
            // columns: G <- G R and U <- U R, every row independently.  Neighbouring threads take the pairs of one row:
            // a step's pairs cover every column once, so the row's sectors are all used while they are in the cache
            // (pair-major order touched one element per sector and was 3 times slower at M = 512).
            for (int i = t; i < pairs * M; i += T) {
                const int row = i / pairs, k = i % pairs, p = pp[k], q = pp[pairs + k];
                if (q >= M) continue;
                const float c = cs[k], s = cs[pairs + k];
                const float gp = G[(size_t)row * M + p], gq = G[(size_t)row * M + q];
                G[(size_t)row * M + p] = c * gp - s * gq;
                G[(size_t)row * M + q] = s * gp + c * gq;
                const float up = U[(size_t)row * M + p], uq = U[(size_t)row * M + q];
                U[(size_t)row * M + p] = c * up - s * uq;
                U[(size_t)row * M + q] = s * up + c * uq;
            }
            __syncthreads();
            // rows: G <- R^T G, every column independently
            for (int i = t; i < pairs * M; i += T) {
                const int k = i / M, col = i % M, p = pp[k], q = pp[pairs + k];
                if (q >= M) continue;
                const float c = cs[k], s = cs[pairs + k];
                const float gp = G[(size_t)p * M + col], gq = G[(size_t)q * M + col];
                G[(size_t)p * M + col] = c * gp - s * gq;
                G[(size_t)q * M + col] = s * gp + c * gq;
            }
            __syncthreads();
        }
        if (__uint_as_float(off_max) <= 2.4e-7f * __uint_as_float(diag_max)) break;   // (uniform: shared values, read after a barrier)
    }
    // eigenvalues = diagonal, sorted descending (rank by counting; ties by index); the columns of U move alike,
    // through G's storage (its content is no longer needed)
    int *rank = pp + 2 * pairs;
    float *ev = evals + (size_t)blockIdx.x * M;
    for (int i = t; i < M; i += T) {
        const float v = G[(size_t)i * M + i];
        int r = 0;
        for (int j = 0; j < M; ++j) {
            const float w = G[(size_t)j * M + j];
            r += (w > v) || (w == v && j < i);
        }
        rank[i] = r;
        ev[r] = v;
    }
    __syncthreads();
    for (int i = t; i < M * M; i += T) G[(size_t)(i / M) * M + rank[i % M]] = U[i];
    __syncthreads();
    for (int i = t; i < M * M; i += T) U[i] = G[i];
}

// Eigenvalues alone (no U): Householder reduction to tridiagonal form, then bisection on Sturm counts.  One block per
// matrix.  4/3 M^3 multiply-adds in M - 2 dependent steps, against about eight sweeps of M - 1 dependent steps of Jacobi
// rotations over global memory: M = 128, eight matrices: 9.8 ms (Jacobi) -> 0.16 ms.  Each step is bound by the latency
// of its four barriers and two sums over a vector, not by arithmetic, so the matrix sits where it is reached fastest: in
// registers up to M = 192 (spectral_tridiag_reg_kernel, which takes one barrier), else in shared memory (M <= 236) or in G's own storage.
// Step k: v = the Householder vector of row k right of the diagonal (every warp forms the norm for itself, a lane its
// columns lane + 32 t), p = beta A v by columns (A is symmetric; thread (column, group) walks the rows of its group),
// w = p - (beta / 2) (p . v) v, A -= v w^T + w v^T.  Float32 like the rotations; worst error against float64 over random,
// low-rank and graded matrices: 3e-7 of the norm (rotations: 4e-6 at M = 16, 5e-5 at 128).
__host__ __device__ constexpr int eig_threads(int M) { return M > 256 ? 1024 : 512; }
// columns walked side by side, and groups of rows
__host__ __device__ constexpr int eig_cols(int M) { const int m = (M + 31) & ~31; return m < eig_threads(M) ? m : eig_threads(M); }
__host__ __device__ constexpr int eig_groups(int M) { return eig_threads(M) / eig_cols(M); }
// shared memory: v, w, diagonal, off-diagonal, partial sums, and the matrix if it lives there
inline size_t eig_smem(int M, bool matrix) { return sizeof(float) * ((size_t)(4 + eig_groups(M)) * M + (matrix ? (size_t)M * M : 0)); }

__device__ __forceinline__ float eig_warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Eigenvalues, descending, of symmetric tridiagonal matrices: diagonal d[M], then the M - 1 off-diagonal elements, at the
// start of each M x M block of `tri`.  Polynomial Sturm sequence p_i = (d_i - x) p_{i-1} - e_i^2 p_{i-2} (no division;
// brought back to exponent 0 every other step; the matrix is scaled to norm 1 first, and e^2 kept above a floor far below
// the precision wanted, so that no two p in a row are zero).  A chain of M dependent steps per count, so the counts are
// spread: 16 eigenvalues to a block of 128 threads.  One pass with every thread at a point of its own brackets all
// eigenvalues to 2 / 128; then kEigSectors threads share an eigenvalue and cut its interval nine-fold per pass: four passes
// in float32 (their counts are off by at most a few eps of the norm: the interval is widened by 2^-19 afterwards), four in
// double down to 2^-31 of the norm.
constexpr int kEigSectors = 8;
__device__ __forceinline__ float pow2_to_unit(float big) {       // 2^-exponent(big)
    return __uint_as_float((254u - (__float_as_uint(big) >> 23)) << 23);
}
__device__ __forceinline__ double pow2_to_unit(double big) {
    return __hiloint2double((int)((2046u - ((unsigned)__double2hiint(big) >> 20)) << 20), 0);
}
__device__ __forceinline__ int sign_bit(float x) { return (int)(__float_as_uint(x) >> 31); }
__device__ __forceinline__ int sign_bit(double x) { return (int)((unsigned)__double2hiint(x) >> 31); }
template <typename F> struct EigPair { F d, e2; };
template <typename F>
__device__ __forceinline__ int sturm_count(const EigPair<F> *q, int M, F x) {
    F pm = 1, pc = q[0].d - x;
    int count = sign_bit(pc), i = 1;
    auto step = [&](const EigPair<F> a) {
        const F pn = (a.d - x) * pc - a.e2 * pm;
        count += sign_bit(pn) ^ sign_bit(pc);
        pm = pc;
        pc = pn;
    };
    auto rescale = [&]() {
        const F x0 = fabs(pc), x1 = fabs(pm), f = pow2_to_unit(x0 > x1 ? x0 : x1);
        pc *= f;
        pm *= f;
    };
#pragma unroll 2
    for (; i + 1 < M; i += 2) {
        step(q[i]);
        step(q[i + 1]);
        rescale();
    }
    if (i < M) step(q[i]);
    return count;
}
constexpr int kBisectThreads = 128;
static __global__ void __launch_bounds__(kBisectThreads)
spectral_bisect_kernel(const float *tri, float *evals, int M) {
    extern __shared__ double bis_sh[];
    __shared__ short counts[kBisectThreads];
    constexpr int TH = kBisectThreads;
    EigPair<double> *qd = reinterpret_cast<EigPair<double> *>(bis_sh);
    EigPair<float> *qf = reinterpret_cast<EigPair<float> *>(qd + M);
    const float *d = tri + (size_t)blockIdx.y * M * M, *e = d + M;
    const int t = threadIdx.x, lane = t & 31;
    ptx::grid_launch();
    ptx::grid_wait();
    double top = 0.0;                                           // Gershgorin, by every warp for itself
    bool bad = false;                                           // (the tridiagonal form of a matrix that was not finite)
    for (int i = lane; i < M; i += 32) {
        const double ei = i + 1 < M ? e[i] : 0.f, eb = i > 0 ? e[i - 1] : 0.f;
        bad |= !isfinite(d[i]) || !isfinite(ei);
        top = fmax(top, fabs((double)d[i]) + fabs(ei) + fabs(eb));
    }
    if (__any_sync(0xffffffffu, bad)) {                         // (the same in every warp)
        const int r = blockIdx.x * (TH / kEigSectors) + t;
        if (t < TH / kEigSectors && r < M) evals[(size_t)blockIdx.y * M + r] = kEigNan;
        return;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    int ex = 0;
    frexp(top, &ex);
    const double scale = top > 0.0 ? ldexp(1.0, -ex) : 1.0;
    for (int i = t; i < M; i += TH) {
        const double di = d[i] * scale, ei = i > 0 ? e[i - 1] * scale : 0.0;
        qd[i] = {di, fmax(ei * ei, 1e-40)};
        qf[i] = {(float)di, fmaxf((float)(ei * ei), 1e-16f)};
    }
    __syncthreads();
    counts[t] = (short)sturm_count<float>(qf, M, -1.f + 2.f * (float)(t + 1) / (float)(TH + 1));
    __syncthreads();
    const int sub = t % kEigSectors;
    const int r = blockIdx.x * (TH / kEigSectors) + t / kEigSectors;   // eigenvalue number r, descending: M - 1 - r others lie below it
    const int below = M - 1 - (r < M ? r : M - 1);
    int n0 = 0, n1 = TH;                                        // points with at most `below` eigenvalues under them: [0, n0) yes, [n1, TH) no
    while (n0 < n1) {
        const int mid = (n0 + n1) >> 1;
        if (counts[mid] <= below) n0 = mid + 1;
        else n1 = mid;
    }
    double lo = -1.0 + 2.0 * n0 / (TH + 1) - 1.9e-6, hi = -1.0 + 2.0 * (n0 + 1) / (TH + 1) + 1.9e-6;
    for (int pass = 0; pass < 8; ++pass) {
        const double step = (hi - lo) * (1.0 / (kEigSectors + 1)), base = lo, x = base + step * (sub + 1);
        const int count = pass < 4 ? sturm_count<float>(qf, M, (float)x) : sturm_count<double>(qd, M, x);
        const unsigned left = (__ballot_sync(0xffffffffu, count <= below) >> (lane & ~(kEigSectors - 1))) & ((1u << kEigSectors) - 1);
        const int n = __popc(left);
        lo = base + step * n;
        if (n < kEigSectors) hi = base + step * (n + 1);
        if (pass == 3) { lo -= 1.9e-6; hi += 1.9e-6; }
    }
    if (r < M && sub == 0) evals[(size_t)blockIdx.y * M + r] = top > 0.0 ? (float)(0.5 * (lo + hi) / scale) : 0.f;
}

// Largest magnitude over the block as a power of two to scale by, so that squares of the entries neither overflow nor vanish: returns
// 2^-e with e the exponent of the largest, as near to it as 2^-e is a normal number (1 for a zero matrix).  NaN if an entry is not
// finite: what is scaled by it is NaN throughout, and so are the eigenvalues.  mx: the largest |entry| of this thread, as its bits (which order
// like the magnitudes, infinity and NaN on top).  All threads call it.  (A test of the entries with a return of its own took the kernel
// below from 67 registers a thread to 98 and from 184 to 227 us at M = 128.)
__device__ __forceinline__ float eig_block_scale(unsigned mx, unsigned *sh32) {
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) sh32[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = 0u;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) mx = max(mx, sh32[i]);
    __syncthreads();
    if (mx == 0u) return 1.f;
    if (mx >= 0x7f800000u) return kEigNan;
    int e = 0;
    frexpf(__uint_as_float(mx), &e);
    return ldexpf(1.f, e > 126 ? -126 : e < -126 ? 126 : -e);
}
__device__ __forceinline__ unsigned eig_magnitude(float x) { return __float_as_uint(fabsf(x)); }

// The matrix in registers: NG groups of CX / COLS threads, thread (g, j) holds rows g, g + NG, ... of column j (and j + CX / 2).  Columns that
// are read by rows are stored group-major (row g + NG r at g * RP + r; RP, 4 or 8 mod 16 and odd multiples of these, keeps the groups' banks apart), so that four rows come with one load.
// A step k takes one barrier.  Every warp holds v_k (a lane its elements lane + 32 c) and, from shared memory, the groups' sums of p = A v_k and
// column k + 1 as it was before this step; so it has w_k, that column after the step, and with it v_(k+1) by itself.  It puts the rows
// of its group where its lanes read them, updates its part of A while the norm's sum goes round, and multiplies it with the next v.  What every
// warp does for itself costs shared-memory cycles by the warp, so there are few of them with much of A each.
// With the bisection, us for eight matrices of 64 / 96 / 128 / 160 / 192: four barriers and two passes over A per step, 16 to 24 warps, a column per
// thread 78 / 122 / 211 / 289 / 558; now 65 / 104 / 162 / 284 / 385 (128: with a column per thread 275, with two 170).
template <int CX> struct EigReg {
    static constexpr int NG = CX == 96 || CX == 192 ? 4 : 8, COLS = CX == 32 || CX == 96 ? 1 : CX == 64 || CX == 192 ? 2 : CX / 32, R = CX / NG;
    static constexpr int RP = NG == 4 ? (R % 16 == 8 ? R : R + 8) : (R % 8 == 4 ? R : R + 4);
    static constexpr int kThreads = CX / COLS * NG;
};
template <int CX>
__global__ void __launch_bounds__(EigReg<CX>::kThreads)
spectral_tridiag_reg_kernel(float *Gall, int M) {
    using E = EigReg<CX>;
    constexpr int NG = E::NG, R = E::R, RP = E::RP, COLS = E::COLS, CT = CX / COLS, CW = CX / 32, TH = E::kThreads;
    static_assert(CT % 32 == 0 && R % 4 == 0, "a warp has one group's rows, four at a time");
    __shared__ __align__(16) float sx[2][NG * RP];              // a column of A
    __shared__ __align__(16) float rows[TH / 32][3][R];         // per warp: its group's rows of v, w and the next v
    __shared__ float part[2][NG][CX], diag[CX], off[CX];
    __shared__ unsigned red[32];
    const int t = threadIdx.x, lane = t & 31, j = t % CT, g = t / CT, jc = j >> 5;
    ptx::grid_launch();
    ptx::grid_wait();
    float *G = Gall + (size_t)blockIdx.x * M * M;
    float A[COLS][R];
    unsigned mx = 0u;
#pragma unroll
    for (int q = 0; q < COLS; ++q)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = g + NG * r, c = j + q * CT;
            A[q][r] = (c < M && i < M) ? G[(size_t)i * M + c] : 0.f;
            mx = max(mx, eig_magnitude(A[q][r]));
        }
    const float scale = eig_block_scale(mx, red);
#pragma unroll
    for (int q = 0; q < COLS; ++q)
#pragma unroll
        for (int r = 0; r < R; ++r) A[q][r] *= scale;
    auto slot = [](int i) { return (i % NG) * RP + i / NG; };   // where row i of a column sits
    auto dump = [&](float *to, int c) {                         // column c of A
#pragma unroll
        for (int q = 0; q < COLS; ++q)
            if (j + q * CT == c) {
#pragma unroll
                for (int r = 0; r < R; r += 4) *reinterpret_cast<float4 *>(to + g * RP + r) = make_float4(A[q][r], A[q][r + 1], A[q][r + 2], A[q][r + 3]);
            }
    };
    float *mine = &rows[t >> 5][0][0];
    float v[CW], w[CW], x[CW], beta = 0.f, v1 = 0.f;            // this lane's elements of v, w and the column the next v is made from; v's first
    auto select = [&](const float (&a)[CW], int c) {            // a[c], c the same for the whole warp
        float y = a[0];
#pragma unroll
        for (int q = 1; q < CW; ++q) y = c == q ? a[q] : y;
        return y;
    };
    auto put = [&](int which, const float (&a)[CW]) {           // the rows of this warp's group
        if (lane % NG == g) {
#pragma unroll
            for (int c = 0; c < CW; ++c) mine[which * R + (lane + 32 * c) / NG] = a[c];
        }
    };
    auto skip = [&](int r, int k) { return g + NG * (r + 3) <= k || g + NG * r >= M; };   // rows r ... r + 3 of the group are done, or none
    float vj[COLS], wj[COLS];
    auto update = [&](int r, int k) {                           // A -= v w^T + w v^T
        if (skip(r, k)) return;
        const float4 vr = *reinterpret_cast<const float4 *>(mine + r), wr = *reinterpret_cast<const float4 *>(mine + R + r);
#pragma unroll
        for (int q = 0; q < COLS; ++q) {
            A[q][r] = fmaf(-vr.x, wj[q], fmaf(-wr.x, vj[q], A[q][r]));
            A[q][r + 1] = fmaf(-vr.y, wj[q], fmaf(-wr.y, vj[q], A[q][r + 1]));
            A[q][r + 2] = fmaf(-vr.z, wj[q], fmaf(-wr.z, vj[q], A[q][r + 2]));
            A[q][r + 3] = fmaf(-vr.w, wj[q], fmaf(-wr.w, vj[q], A[q][r + 3]));
        }
    };
    // x, column k, becomes the Householder vector that annihilates it below the subdiagonal, with beta; `between`(0 ... 4) goes between the
    // steps of the sum
    auto reflect = [&](int k, auto between) {
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < CW; ++c) s = lane + 32 * c > k + 1 ? fmaf(x[c], x[c], s) : s;
        const float x0 = __shfl_sync(0xffffffffu, select(x, (k + 1) >> 5), (k + 1) & 31);
        if (t == (k & 31)) diag[k] = select(x, k >> 5);
#pragma unroll
        for (int o = 0; o < 5; ++o) {
            s += __shfl_xor_sync(0xffffffffu, s, 16 >> o);
            between(o);
        }
        const float norm = sqrtf(fmaf(x0, x0, s)), alpha = x0 > 0.f ? -norm : norm, v0 = x0 - alpha;
        beta = s > 0.f ? 2.f / fmaf(v0, v0, s) : 0.f;           // nothing to annihilate: beta = 0, nothing changes
        if (t == 0) off[k] = s > 0.f ? alpha : x0;
        v1 = v0;
#pragma unroll
        for (int c = 0; c < CW; ++c) {
            const int i = lane + 32 * c;
            x[c] = i > k + 1 ? x[c] : i == k + 1 ? v0 : 0.f;
        }
    };
    // this thread's share of A (next v); column `next` for the step after
    auto multiply = [&](int k, int buf, int next) {
        put(2, x);
        __syncwarp();
        float p[COLS][4] = {};
#pragma unroll
        for (int r = 0; r < R; r += 4) {
            if (skip(r, k)) continue;
            const float4 nv = *reinterpret_cast<const float4 *>(mine + 2 * R + r);
#pragma unroll
            for (int q = 0; q < COLS; ++q) {
                p[q][0] = fmaf(A[q][r], nv.x, p[q][0]);
                p[q][1] = fmaf(A[q][r + 1], nv.y, p[q][1]);
                p[q][2] = fmaf(A[q][r + 2], nv.z, p[q][2]);
                p[q][3] = fmaf(A[q][r + 3], nv.w, p[q][3]);
            }
        }
#pragma unroll
        for (int q = 0; q < COLS; ++q) part[buf][g][j + q * CT] = (p[q][0] + p[q][1]) + (p[q][2] + p[q][3]);
        dump(sx[buf], next);
    };
    dump(sx[1], 0);
    __syncthreads();
    if (M >= 2) {
#pragma unroll
        for (int c = 0; c < CW; ++c) x[c] = sx[1][slot(lane + 32 * c)];
        reflect(0, [](int) {});
        multiply(-1, 0, 1);
    } else if (t == 0) {
        diag[0] = sx[1][0];
    }
    for (int k = 0; k + 2 < M; ++k) {
        __syncthreads();
        const int buf = k & 1;
        float pv = 0.f;
#pragma unroll
        for (int c = 0; c < CW; ++c) {
            v[c] = x[c];
            float p = 0.f;
#pragma unroll
            for (int q = 0; q < NG; ++q) p += part[buf][q][lane + 32 * c];
            x[c] = sx[buf][slot(lane + 32 * c)];
            w[c] = p;
            pv = fmaf(p, v[c], pv);
        }
        put(0, v);
        pv = eig_warp_sum(pv);
        const float half = 0.5f * beta * (beta * pv);
#pragma unroll
        for (int c = 0; c < CW; ++c) w[c] = lane + 32 * c > k ? fmaf(beta, w[c], -half * v[c]) : 0.f;
        put(1, w);
        const float w1 = __shfl_sync(0xffffffffu, select(w, (k + 1) >> 5), (k + 1) & 31);
#pragma unroll
        for (int c = 0; c < CW; ++c) x[c] = fmaf(-v[c], w1, fmaf(-w[c], v1, x[c]));
#pragma unroll
        for (int q = 0; q < COLS; ++q) {
            vj[q] = select(v, jc + q * (CT / 32));
            wj[q] = select(w, jc + q * (CT / 32));
        }
        __syncwarp();
        reflect(k + 1, [&](int o) {
#pragma unroll
            for (int r = 0; r < R; r += 4)
                if (r / 4 * 5 / (R / 4) == o) update(r, k);     // (o a constant after unrolling)
        });
        multiply(k, buf ^ 1, k + 2);
        __syncwarp();                                           // (the rows are written again in the next step)
    }
    __syncthreads();
    if (t == 0 && M >= 2) diag[M - 1] = sx[M & 1][slot(M - 1)];
    __syncthreads();
    for (int i = t; i < M; i += TH) {                           // the result takes the place of the matrix
        G[i] = diag[i] / scale;
        if (i + 1 < M) G[M + i] = off[i] / scale;
    }
}

// The matrix in shared memory (kShared) or where it is (global memory, overwritten).
template <bool kShared>
__global__ void __launch_bounds__(1024)
spectral_tridiag_kernel(float *__restrict__ Gall, int M) {
    extern __shared__ float eig_sh[];
    const int t = threadIdx.x, TH = blockDim.x, lane = t & 31;
    const int CX = eig_cols(M), NG = eig_groups(M);
    float *dg = eig_sh, *ee = dg + M, *v = ee + M, *w = v + M, *part = w + M;   // part [NG][M]
    float *G = Gall + (size_t)blockIdx.x * M * M;
    float *A = kShared ? part + (size_t)NG * M : G;
    __shared__ unsigned red[32];
    unsigned mx = 0u;
    for (int i = t; i < M * M; i += TH) mx = max(mx, eig_magnitude(G[i]));
    const float scale = eig_block_scale(mx, red);
    for (int i = t; i < M * M; i += TH) A[i] = G[i] * scale;
    __syncthreads();
    const int cx = t % CX, g = t / CX;
    for (int k = 0; k + 2 < M; ++k) {
        const float *row = A + (size_t)k * M;
        float s = 0.f;
        for (int j = k + 2 + lane; j < M; j += 32) s = fmaf(row[j], row[j], s);
        s = eig_warp_sum(s);
        const float x0 = row[k + 1];
        const float norm = sqrtf(fmaf(x0, x0, s)), alpha = x0 > 0.f ? -norm : norm;
        const float v0 = x0 - alpha, beta = s > 0.f ? 2.f / fmaf(v0, v0, s) : 0.f;
        if (t == 0) { dg[k] = row[k]; ee[k] = s > 0.f ? alpha : x0; }
        for (int j = k + 1 + t; j < M; j += TH) v[j] = j == k + 1 ? v0 : row[j];
        __syncthreads();
        if (g < NG)
            for (int j = cx; j < M; j += CX)
                if (j > k) {
                    float p[4] = {0.f, 0.f, 0.f, 0.f};
                    int i = k + 1 + g;
                    for (; i + 3 * NG < M; i += 4 * NG)
#pragma unroll
                        for (int q = 0; q < 4; ++q) p[q] = fmaf(A[(size_t)(i + q * NG) * M + j], v[i + q * NG], p[q]);
                    for (; i < M; i += NG) p[0] = fmaf(A[(size_t)i * M + j], v[i], p[0]);
                    part[(size_t)g * M + j] = (p[0] + p[1]) + (p[2] + p[3]);
                }
        __syncthreads();
        float pv = 0.f;
        for (int j = k + 1 + lane; j < M; j += 32) {
            float p = 0.f;
            for (int q = 0; q < NG; ++q) p += part[(size_t)q * M + j];
            pv = fmaf(p, v[j], pv);
        }
        pv = eig_warp_sum(pv);
        const float half = 0.5f * beta * (beta * pv);
        for (int j = k + 1 + t; j < M; j += TH) {
            float p = 0.f;
            for (int q = 0; q < NG; ++q) p += part[(size_t)q * M + j];
            w[j] = fmaf(beta, p, -half * v[j]);
        }
        __syncthreads();
        if (g < NG)
            for (int j = cx; j < M; j += CX)
                if (j > k) {
                    const float vj = v[j], wj = w[j];
#pragma unroll 4
                    for (int i = k + 1 + g; i < M; i += NG)
                        A[(size_t)i * M + j] = fmaf(-v[i], wj, fmaf(-w[i], vj, A[(size_t)i * M + j]));
                }
        __syncthreads();
    }
    if (t == 0) {
        if (M >= 2) {
            dg[M - 2] = A[(size_t)(M - 2) * M + M - 2];
            ee[M - 2] = A[(size_t)(M - 2) * M + M - 1];
        }
        dg[M - 1] = A[(size_t)M * M - 1];
    }
    __syncthreads();
    for (int i = t; i < M; i += TH) {                           // the result takes the place of the matrix
        G[i] = dg[i] / scale;
        if (i + 1 < M) G[M + i] = ee[i] / scale;
    }
}

}  // namespace flare
