// Tensor-core kernels of the backward for bfloat16 inputs on sm_100a, heads up to 32 wide: two sweeps over the tokens.
//
//   bwd_dz_sweep_kernel     dZ_m = sum_n W_dec[n,m] dY_n,   dd[n] = sum_m W_dec[n,m] A[n,m]
//   bwd_grad_sweep_kernel   dK_n = scale sum_m dS[n,m] q_m,   dV_n = sum_m W_enc[m,n] dZ_m,   dQ_m = scale sum_n dS[n,m] k_n   with
//                           dS[n,m] = W_dec (A - dd[n]) + W_enc (C - de[m]),   A = dY_n . Z_m,   C = V_n . dZ_m
//
// Tokens on the 128 lanes, latents on the columns, in units of 64, in both.  Sums over latents take their weights as the A operand in tensor memory, or
// in shared memory; sums over tokens (dZ, dQ) contract over the lanes, which tensor memory cannot: their weights go to shared memory, [token][64 latents] as
// two bf16 halves, and are read as a transposed A operand whose 128 rows are the hi halves of the unit's 64 latents and the lo halves, so that one
// instruction per 16 tokens serves both and hi and lo have sums of their own (they meet where the partial results are added up).
//
// Three kernels before (dZ with latents on the lanes; dK, dV and dd with tokens; dQ with latents) exponentiated every score three times and formed A and C
// twice; here it is twice and once, and since dd is known when dS is formed, no first guess of it is needed (a pass over Y and dY) and nothing is put right
// afterwards.  us per training step, before -> now, both timed in turn: 16384 tokens, M = 32, D = 32, 8 heads 86 -> 68; 32 x 4096, M = 128, D = 32, 4 heads 288 -> 238; 131072
// tokens, 8 heads, D = 32: M = 32 327 -> 237, 64 375 -> 305, 256 771 -> 663, 320 1026 -> 830; D = 16: M = 16 238 -> 214, 32 239 -> 218, 256 705 -> 604, 1024 2616 -> 2312; D = 8: M = 64 285 -> 248,
// 1024 2524 -> 2220, 2048 5129 -> 4373; D = 4, 16 heads, M = 64 596 -> 499.  At D = 32 two ranges of latents, with float32 rows to read and write between
// them, are no faster (M = 400 1312 : 1309, 512 1391 : 1414): more than 320 latents take the kernels of flare_bwd_tc.cuh, and so do heads 64 wide.
//
// What bounds them: issue slots (54 to 64 % in use; some 210 warp instructions per 16 columns of a unit in the first, 340 in the second at D = 16, M = 256, of which
// 84 and 144 are the arithmetic) and, lane by lane, latency: a unit takes a warp of the second 1250 cycles of work, 160 of finding its scores ready and 130 around.  All
// forms of the second spill a few registers (8 to 24 bytes at 96 registers; taking them out by chance of code changed no time by more than 2 %).  Tensor core,
// cycles per unit of 64 latents: S 48, A and C 96 each (D = 32: twice that), dV 100, dK and dZ or dQ 320 each (an instruction with both operands in shared memory takes 40,
// whichever way its rows lie).  What the loop over a kernel's units should not hold is anything done once per tile: see the second kernel's.
#pragma once

#include "flare_bwd_tc.cuh"

namespace flare {

constexpr int kSwThreads = 640, kSwFirstMathWarp = 4, kSwUnit = 64, kSwGroups = kSwUnit / 16;
constexpr uint32_t kSwHalf = kTile * kSwUnit * 2, kSwBuf = 2 * kSwHalf;     // bytes of a unit's hi (lo) halves, of both
constexpr int kSwRing = 4, kSwMaxStages = 6;
// Sums over tokens that take a CTA's tiles in turn, up to four where tensor memory has the columns (as a logarithm; `each`: columns of one).  The tensor core
// truncates: n parts in a row lose n 2^-24 / 3 of their sum on average, all in one direction.  Distance of dQ from float64, of its norm, one sum : in turn : the
// three kernels before, 65536 tokens, 8 heads: D = 32, M = 32 5.8e-6 : 4.8e-6 : 5.4e-6, M = 64 5.7e-6 : 4.8e-6 : 5.3e-6; D = 16, M = 32 5.6e-6 : 4.6e-6 : 4.9e-6, M = 128 9.1e-6 : 8.2e-6 : 8.5e-6.
__host__ __device__ constexpr int sweep_log2_sums(int columns, int each) { return columns >= 4 * each ? 2 : columns >= 2 * each ? 1 : 0; }
// Tiles (eight parts of 16 tokens each) after which these sums are added to the float32 partial results, which stops the pipeline for some 4000 cycles: a power
// of two, by units of a tile.  64 to 128 parts in a row up to two units; with more units, whose tiles take longer and are fewer to a CTA at the same time, up
// to 256 and 512, which leave dQ no further from float64 than the three kernels before (100000 tokens, M = 1024, D = 16 8.9e-6, before 10.7e-6).
__host__ __device__ constexpr int sweep_flush_tiles(int nu, int sums) { return nu <= 2 && sums < 4 ? 16 : nu <= 4 ? 32 : 64; }

// Descriptors of a unit's weights in shared memory: rows of 128 bytes (64 latents of a token), swizzled.
constexpr uint32_t kSwDescHi = ptx::desc_hi(1024, 2);
constexpr uint32_t kSwDescMn = ptx::desc_lo(0, kSwHalf), kSwDescK = ptx::desc_lo(0, 16);   // transposed: the lo halves follow as rows 64 on; as they lie

// The sums over tokens that a CTA has in tensor memory (`sums` of them, columns base + (s nu + u) D of unit u; lanes 0-63 hi, 64-127 lo) to partial results 2 part
// and 2 part + 1, or added to them.  By the warps that worked on the last unit: `mine` of `cps` column groups.
template <int D, int DR>
__device__ __forceinline__ void sweep_flush(uint32_t base, float *part, size_t rows, int cta, size_t row0, int M, int nu, int sums, int mine, int cps, int row, int off, bool add) {
    float *dst0 = part + ((size_t)(2 * cta + (row >> 6)) * rows + row0) * DR;
    constexpr int PIECES = DR <= 8 ? 1 : DR / 8;                // of eight columns, in turn to the warps that share the tokens
    for (int p = mine; p < nu * PIECES; p += cps) {
        const int u = p / PIECES, c0 = p % PIECES * 8, m = u * kSwUnit + (row & 63);
        uint32_t x[8];
        ptx::tmem_ld8(base + u * D + c0, x);
        ptx::tmem_wait_ld();
#pragma unroll
        for (int s = 1; s < 4; ++s) {
            if (s >= sums) break;
            uint32_t y[8];
            ptx::tmem_ld8(base + (s * nu + u) * D + c0, y);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 8; ++c) x[c] = __float_as_uint(__uint_as_float(x[c]) + __uint_as_float(y[c]));
        }
        float4 *dst = reinterpret_cast<float4 *>(dst0 + (size_t)m * DR + c0);
        if (m < M) {
#pragma unroll
            for (int c = 0; c < (DR == 4 ? 1 : 2); ++c) {
                float4 v;
                if (DR == 4 && off != 0) v = make_float4(__uint_as_float(x[4]), __uint_as_float(x[5]), __uint_as_float(x[6]), __uint_as_float(x[7]));
                else v = make_float4(__uint_as_float(x[4 * c]), __uint_as_float(x[4 * c + 1]), __uint_as_float(x[4 * c + 2]), __uint_as_float(x[4 * c + 3]));
                if (add) {
                    const float4 o = dst[c];
                    v = make_float4(v.x + o.x, v.y + o.y, v.z + o.z, v.w + o.w);
                }
                dst[c] = v;
            }
        }
        __syncwarp();
    }
}

// Wait of an issuing warp, inline; the same for all lanes.
__device__ __forceinline__ bool issue_wait(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t code) {
    if (__all_sync(0xffffffffu, ptx::mbar_try_wait(bar, parity))) return true;
    return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity, abort_flag, code));
}

// The sum of two floats and what its rounding lost, added to `lost`.
__device__ __forceinline__ void add_exactly(float &sum, float &lost, float x) {
    const float t = sum + x, b = t - sum;
    lost += (sum - (t - b)) + (x - b);
    sum = t;
}

// sum_m W A and sum_m W of a token over some of a row's latents, each as a float and what that lost.  Where one latent has most of the weight, dS is what is
// left of A - dd there, down to 2^-40 of A, so dd has to be known beyond a float: the columns are then summed once more about their own mean.
struct RowSums {
    float sum, lost, wsum, wlost;
    __device__ __forceinline__ void clear() { sum = lost = wsum = wlost = 0.f; }
    __device__ __forceinline__ float4 get() const { return make_float4(sum, lost, wsum, wlost); }
    __device__ __forceinline__ void set(float4 x) { sum = x.x; lost = x.y; wsum = x.z; wlost = x.w; }
    __device__ __forceinline__ void join(float4 x) {
        add_exactly(sum, lost, x.x);
        add_exactly(wsum, wlost, x.z);
        lost += x.y;
        wlost += x.w;
    }
    // their quotient, as a float and what is left of it
    __device__ __forceinline__ float2 mean() const {
        if (wsum == 0.f) return make_float2(0.f, 0.f);
        const float inv = 1.f / wsum, q = sum * inv, q2 = (fmaf(-q, wsum, sum) + fmaf(-q, wlost, lost)) * inv, hi = q + q2;
        return make_float2(hi, fabsf(hi) <= 3.0e38f ? q2 - (hi - q) : 0.f);
    }
    // sixteen columns: their weights, A (raw bits), and plain sums of both
    __device__ __forceinline__ void add(const float2 (&pd)[8], const uint32_t *av, float2 s2, float2 w2) {
        const float w = w2.x + w2.y;
        float s = s2.x + s2.y;
        add_exactly(wsum, wlost, w);
        if (__any_sync(0xffffffffu, w > 0.7f)) {
            const float e = w > 0.f ? __fdividef(s, w) : 0.f;
            const float2 ne = make_float2(-e, -e);
            float2 r2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 8; ++k) r2 = __ffma2_rn(pd[k], __fadd2_rn(make_float2(__uint_as_float(av[2 * k]), __uint_as_float(av[2 * k + 1])), ne), r2);
            s = w * e;
            lost += fmaf(w, e, -s) + (r2.x + r2.y);
        }
        add_exactly(sum, lost, s);
    }
};

// ---------------------------------------------------------------------------------------------------------- first sweep: dZ, dd
struct BwdDzArgs {
    const __nv_bfloat16 *Q;    // [H,M,D]
    const float *Z;            // [B,H,M,D]
    const float *lse_dec;      // [B,N,H]
    float *part;               // [2 * CTAs per head][B*H*M][D] partial dZ rows
    float *dd;                 // [2][B,H,N]: dd as a float and what is left of it
    uint32_t *status;
    int B, H, N, M;            // M: latents this launch works on (all of them, or a range; the last of several side by side may be shorter)
    int mtot, m0;              // latents per head in memory, and the first one of this launch's range
    int first, last;           // range of latents (without ranges both; side by side the first only)
    float4 *sums;              // [range of those side by side][B,H][tile of this launch][token of the tile]: RowSums of the earlier ranges
    float sl2;                 // scale * log2(e)
    int tiles, stages;         // tiles of tokens this launch works on
    int t0;                    // the first of them (without ranges 0)
    int side;                  // ranges side by side, in neighbouring blocks (else 1)
};

template <int D>
struct BwdDzSmem {
    using G = TileGeom<D>;
    enum { QR = 0, ZH = 1, ZL = 2 };                            // latent operands: Q, Z hi, lo
    static constexpr int kBufs = 3;                             // of weights
    // sums over tokens beside S and A twice
    __host__ __device__ static int log2_sums(int M) {
        const int ucols = (M + 31) / 32 * 32 < kSwUnit ? (M + 31) / 32 * 32 : kSwUnit;
        return sweep_log2_sums(512 - 4 * ucols, (M + kSwUnit - 1) / kSwUnit * D);
    }
    static constexpr size_t tile_off = (size_t)kBufs * kSwBuf;
    __host__ __device__ static size_t lat_off(int stages, int M, int which) { return tile_off + (size_t)stages * 2 * G::TILE_BYTES + (size_t)which * M * G::RB; }
    __host__ __device__ static size_t ring_off(int stages, int M) { return lat_off(stages, M, 3); }         // [ring][token] -lse_dec
    __host__ __device__ static size_t dds_off(int stages, int M) { return ring_off(stages, M) + kSwRing * kTile * sizeof(float); }   // [2][group][token], see RowSums
    __host__ __device__ static size_t bar_off(int stages, int M) { return dds_off(stages, M) + 2 * kSwGroups * kTile * sizeof(float4); }
    __host__ __device__ static size_t total(int stages, int M) {
        const size_t t = bar_off(stages, M) + 512 + D * sizeof(float) + 1024;
        return t < kTcMinSmem ? kTcMinSmem : t;
    }
    __host__ static int stages(int M) {
        int s = kSwMaxStages;
        while (s > 0 && total(s, M) > (size_t)227 * 1024) --s;
        return s;
    }
};

template <int D, int DRT, bool kRanges>
__global__ void __launch_bounds__(kSwThreads, 1)
bwd_dz_sweep_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmG, BwdDzArgs a) {
    using G = TileGeom<D>;
    using SM = BwdDzSmem<D>;
    constexpr int UNIT = kSwUnit, RING = kSwRing, DR = DRT ? DRT : D;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = ptx::align_1024(smem_raw);
    const int side = kRanges ? a.side : 1, which_range = kRanges ? (int)blockIdx.x % side : 0, cta = (int)blockIdx.x / side, ctas = (int)gridDim.x / side;
    const int m0 = a.m0 + which_range * a.M, M = kRanges ? min(a.M, a.mtot - m0) : a.M, stages = a.stages;
    uint8_t *tiles_s = smem + SM::tile_off;
    float *ring = reinterpret_cast<float *>(smem + SM::ring_off(stages, M));
    float4 *dds = reinterpret_cast<float4 *>(smem + SM::dds_off(stages, M));
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + SM::bar_off(stages, M));
    enum { T_FULL = 0, T_EMPTY = T_FULL + kSwMaxStages, S_FULL = T_EMPTY + kSwMaxStages, S_READ = S_FULL + 2, P_FULL = S_READ + 2, C_FULL = P_FULL + 4,
           C_EMPTY = C_FULL + RING, DD_FULL = C_EMPTY + RING, DD_EMPTY = DD_FULL + 2, FL_FULL = DD_EMPTY + 2, FL_DONE, NBARS };
    static_assert(NBARS * 8 + 8 <= 512, "barrier area too small");
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + NBARS);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    float *centre = reinterpret_cast<float *>(reinterpret_cast<uint8_t *>(bars) + 512);

    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const int h = blockIdx.y, b = blockIdx.z;
    const int nt = (a.tiles - cta + ctas - 1) / ctas;   // tiles of this CTA
    auto tile_at = [&](int i) { return cta + i * ctas + (kRanges ? a.t0 : 0); };   // the i-th of them
    const int nu = (M + UNIT - 1) / UNIT, wlast = M - (nu - 1) * UNIT;                 // latent units of a tile; columns of the last
    const int ucols = min(UNIT, (M + 31) & ~31);                // columns of a region S or A
    const int sets = M <= 32 ? 2 : 1, cps = sets == 2 ? 2 : kSwGroups;                 // sets of warps that take the tiles in turn, column groups of each
    const int off = DRT ? narrow_offset(h, DR) : 0;
    const int units = nu * nt, sums_in_turn = 1 << SM::log2_sums(M), flush = sweep_flush_tiles(nu, sums_in_turn);
    // (opaque: an address that can be formed again from the kernel's arguments is, at every use, by a dozen instructions)
    uint32_t bars0 = ptx::smem_u32(bars);
    ptx::opaque(bars0);
    auto bar = [&](int i) { return bars0 + 8u * i; };

    if (threadIdx.x == 0) {
        const uint32_t math = 4 * cps;                          // warps that work on a unit
        for (int i = 0; i < NBARS; ++i)
            ptx::mbar_init(bar(i), (i >= S_READ && i < C_FULL) || (i >= C_EMPTY && i < DD_EMPTY) || i == FL_DONE ? math : 1u);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmK);
        ptx::prefetch_tensormap(&tmG);
    }
    if (warp == 1) ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
    ptx::grid_launch();
    ptx::grid_wait();
    const size_t bh = (size_t)b * a.H + h, q0 = (size_t)h * a.mtot + m0, r0 = bh * a.mtot + m0;
    z_centre<DR>(centre, a.Z + bh * a.mtot * DR, a.mtot);
    if (DRT != 0)                                               // narrow form: the other columns of every row stay zero
        for (int i = threadIdx.x; i < 3 * M * (G::RB / 16); i += kSwThreads) reinterpret_cast<uint4 *>(smem + SM::lat_off(stages, M, 0))[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    {
        uint8_t *q = smem + SM::lat_off(stages, M, SM::QR), *zh = smem + SM::lat_off(stages, M, SM::ZH), *zl = smem + SM::lat_off(stages, M, SM::ZL);
        if constexpr (DR == 4) {
            stage_rows4<D>(q, a.Q + q0 * DR, M, off);
            stage_rows4_hilo<D>(zh, zl, a.Z + r0 * DR, M, off, centre);
        } else {
            stage_bf16<D, DR>(q, a.Q + q0 * DR, M, 0, 0, threadIdx.x, kSwThreads);
            stage_hilo<D, DR>(zh, zl, a.Z + r0 * DR, M, 0, 0, threadIdx.x, kSwThreads, centre);
        }
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = *tmem_slot;
    const uint32_t acc0 = tm + 4 * ucols;                       // two buffers S | A, then the sums over tokens

    if (warp == 0) {
        if (ptx::elect_one()) {
            for (int i = 0; i < nt; ++i) {
                const int s = i % stages, t = tile_at(i);
                if (!ptx::mbar_wait(bar(T_EMPTY + s), ((i / stages) & 1) ^ 1, abort_flag, kErrBwdDz | 1)) break;
                ptx::mbar_arrive_expect_tx(bar(T_FULL + s), 2 * G::TILE_BYTES);
                uint8_t *dst = tiles_s + (size_t)s * 2 * G::TILE_BYTES;
                ptx::tma_load_3d(ptx::smem_u32(dst), &tmK, bar(T_FULL + s), h * DR - off, t * kTile, b);
                ptx::tma_load_3d(ptx::smem_u32(dst + G::TILE_BYTES), &tmG, bar(T_FULL + s), h * DR - off, t * kTile, b);
            }
        }
    } else if (warp == 2) {
        // -lse_dec (log2 units) of every tile, fetched by asynchronous copies three tiles ahead.
        constexpr int AH = RING - 1;
        auto fetch = [&](int i) {
            float *at = ring + (i % RING) * kTile;
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) {
                const int r = e * 32 + lane, n = min(tile_at(i) * kTile + r, a.N - 1);
                ptx::copy_async4(ptx::smem_u32(at + r), a.lse_dec + ((size_t)b * a.N + n) * a.H + h);
            }
        };
        for (int k = 0; k < AH; ++k) {
            if (k < nt) fetch(k);
            ptx::copy_async_commit();
        }
        for (int i = 0; i < nt; ++i) {
            ptx::copy_async_wait<AH - 1>();
            __syncwarp();
            float *at = ring + (i % RING) * kTile;
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) {
                const int r = e * 32 + lane, n = tile_at(i) * kTile + r;
                at[r] = n < a.N ? -at[r] * kBwdLog2e : -INFINITY;
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(C_FULL + i % RING));
            const int next = i + AH;
            if (next < nt) {
                if (!warp_wait(bar(C_EMPTY + next % RING), ((next / RING) & 1) ^ 1, abort_flag, kErrBwdDz | 3)) break;
                fetch(next);
            }
            ptx::copy_async_commit();
        }
        ptx::copy_async_wait<0>();
    } else if (warp == 3) {
        // dd of every tile, from the column groups' shares: over the sum of the weights as they are (they add up to 1 to some 2^-20, and the weighed mean
        // of A is what makes a row of dS add up to 0).
        for (int i = 0; i < nt; ++i) {
            if (!warp_wait(bar(DD_FULL + (i & 1)), (i >> 1) & 1, abort_flag, kErrBwdDz | 2)) break;
            RowSums all[kTile / 32];
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) all[e].set(dds[(i & 1) * kSwGroups * kTile + e * 32 + lane]);
            for (int g = 1; g < cps; ++g)
#pragma unroll
                for (int e = 0; e < kTile / 32; ++e) all[e].join(dds[((i & 1) * kSwGroups + g) * kTile + e * 32 + lane]);
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(DD_EMPTY + (i & 1)));
            const size_t plane = (size_t)a.B * a.H * a.N;
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) {
                const int n = tile_at(i) * kTile + e * 32 + lane;
                if (n >= a.N) continue;
                const size_t at = bh * a.N + n;
                const size_t so_far = ((((size_t)which_range * a.B * a.H + bh) * a.tiles + (tile_at(i) - (kRanges ? a.t0 : 0))) * kTile) + e * 32 + lane;
                if (kRanges && !a.first) all[e].join(a.sums[so_far]);
                if (!kRanges || a.last) {
                    const float2 d = all[e].mean();
                    a.dd[at] = d.x;
                    a.dd[plane + at] = d.y;
                } else {
                    a.sums[so_far] = all[e].get();
                }
            }
        }
    } else if (warp == 1) {
        {
            const uint32_t lead = ptx::elect_one() ? 1u : 0u;
            constexpr uint32_t HI = ptx::desc_hi(G::SBO, G::SWZ), TILE = G::TILE_BYTES >> 4, STEP16 = (16 * G::RB) >> 4;
            const uint32_t LAT = (uint32_t)(M * G::RB) >> 4;
            const uint32_t lat0 = ptx::desc_lo(ptx::smem_u32(smem + SM::lat_off(stages, M, 0)), 16), td0 = ptx::desc_lo(ptx::smem_u32(tiles_s), 16);
            constexpr uint32_t MN = ptx::desc_lo(0, G::SBO) - ptx::desc_lo(0, 16);          // K-major to MN-major
            const uint32_t w0 = ptx::desc_lo(ptx::smem_u32(smem), 0) + kSwDescMn;
            int s_stage = 0, s_wrap = 0, s_u = 0, o_stage = 0, o_u = 0, o_tile = 0, o_buf = 0, window = 0;
            // S = K Q^T | A = dY (Z_lo + Z_hi)^T of unit n
            auto tiles = [&](int n) -> bool {
                if (s_u == 0) {
                    if (!issue_wait(bar(T_FULL + s_stage), (uint32_t)s_wrap, abort_flag, kErrBwdDz | 4)) return false;
                    ptx::tc_fence_after();
                }
                const uint32_t idescS = ptx::instr_desc_bf16(128, 0, 0, 0) | (uint32_t)((s_u == nu - 1 ? wlast : UNIT) >> 3) << 17;
                uint32_t td = td0 + (uint32_t)s_stage * 2 * TILE, ld = lat0 + (uint32_t)s_u * (UNIT / 16) * STEP16;
                const uint32_t col = tm + (n & 1) * 2 * ucols;
#pragma unroll
                for (int k = 0; k < D / 16; ++k) ptx::mma_ss_by(lead, col, ptx::desc(td + 2 * k, HI), ptx::desc(ld + SM::QR * LAT + 2 * k, HI), idescS, k > 0);
#pragma unroll
                for (int k = 0; k < D / 16; ++k) ptx::mma_ss_by(lead, col + ucols, ptx::desc(td + TILE + 2 * k, HI), ptx::desc(ld + SM::ZL * LAT + 2 * k, HI), idescS, k > 0);
#pragma unroll
                for (int k = 0; k < D / 16; ++k) ptx::mma_ss_by(lead, col + ucols, ptx::desc(td + TILE + 2 * k, HI), ptx::desc(ld + SM::ZH * LAT + 2 * k, HI), idescS, 1u);
                ptx::mma_commit_by(lead, bar(S_FULL + (n & 1)));
                if (++s_u == nu) {
                    s_u = 0;
                    if (++s_stage == stages) { s_stage = 0; s_wrap ^= 1; }
                }
                return true;
            };
            // Scores are formed two units ahead: what says that those of a unit are there says as well that the sums that read its buffer of weights
            // before, three units earlier, are formed.
            bool ok = true;
            for (int n = 0; ok && n < 2 && n < units; ++n) ok = tiles(n);
            for (int n = 0; ok && n < units; ++n) {
                if (n + 2 < units) {
                    if (!issue_wait(bar(S_READ + (n & 1)), (n >> 1) & 1, abort_flag, kErrBwdDz | 5)) break;
                    ptx::tc_fence_after();
                    if (!tiles(n + 2)) break;
                }
                // (four barriers in turn: scores two units on are there before all warps are done with this one, and one that is may arrive for that unit first)
                if (!issue_wait(bar(P_FULL + (n & 3)), (n >> 2) & 1, abort_flag, kErrBwdDz | 6)) break;
                if (o_u == 0 && o_tile == 0 && window > 0 && !issue_wait(bar(FL_DONE), (window - 1) & 1, abort_flag, kErrBwdDz | 7)) break;
                ptx::tc_fence_after();
                // dZ += W^T dY: 16 tokens per step
                constexpr uint32_t idescO = ptx::instr_desc_bf16(128, D, 1, 1);
                uint32_t wd = w0 + (uint32_t)o_buf * (kSwBuf >> 4), gd = td0 + MN + (uint32_t)o_stage * 2 * TILE + TILE;
                const uint32_t to = acc0 + ((o_tile & (sums_in_turn - 1)) * nu + o_u) * D;
#pragma unroll
                for (int k = 0; k < kTile / 16; ++k)
                    ptx::mma_ss_by(lead, to, ptx::desc(wd + k * (2048 >> 4), kSwDescHi), ptx::desc(gd + k * STEP16, HI), idescO, (o_tile >= sums_in_turn || k > 0) ? 1u : 0u);
                if (++o_buf == SM::kBufs) o_buf = 0;
                if (++o_u == nu) {
                    o_u = 0;
                    ptx::mma_commit_by(lead, bar(T_EMPTY + o_stage));
                    if (++o_stage == stages) o_stage = 0;
                    if (++o_tile == flush || n + 1 == units) {
                        ptx::mma_commit_by(lead, bar(FL_FULL));
                        o_tile = 0;
                        ++window;
                    }
                }
            }
        }
    } else if (warp >= kSwFirstMathWarp) {
        const int cg = (warp - kSwFirstMathWarp) >> 2, set = sets == 2 ? cg >> 1 : 0, mine = sets == 2 ? cg & 1 : cg;   // columns: 16 from 16 mine on
        const int row = ((warp & 3) << 5) + lane;               // TMEM lane = token within the tile
        const uint32_t gcol = tm + ((uint32_t)((warp & 3) << 5) << 16), lead = lane == 0;
        const float2 sl2p = make_float2(a.sl2, a.sl2);
        // this thread's first 16 bytes (8 latents) of the hi halves in its next buffer of weights; the next 8 latents are at `w ^ 16`
        const uint32_t w_first = ptx::smem_u32(smem) + (uint32_t)row * 128 + ((uint32_t)((2 * mine) ^ (row & 7)) << 4);
        uint32_t w = w_first + (uint32_t)set * kSwBuf, w_end = w_first + SM::kBufs * kSwBuf;
        ptx::opaque(w);
        ptx::opaque(w_end);
        RowSums sums;
        int n = set;
        bool ok = true;
        for (int i = set; ok && i < nt; i += sets) {
            const int c = i % RING;
            if (!(ok = warp_wait(bar(C_FULL + c), (i / RING) & 1, abort_flag, kErrBwdDz | 8))) break;
            const float nld = ring[c * kTile + row];
            __syncwarp();
            ptx::mbar_arrive_if(bar(C_EMPTY + c), lead);
            sums.clear();
            const float2 nldp = make_float2(nld, nld);
#pragma unroll 1
            for (int u = 0; u < nu; ++u, n += sets) {
                const uint32_t col = gcol + (n & 1) * 2 * ucols + 16 * mine, read = bar(S_READ + (n & 1));
                if (!(ok = warp_wait(read - 8 * (S_READ - S_FULL), (n >> 1) & 1, abort_flag, kErrBwdDz | 9))) break;
                ptx::tc_fence_after();
                if (u * UNIT + 16 * mine < M) {
                    uint32_t s[16], av[16];
                    ptx::tmem_ld16(col, s);
                    ptx::tmem_ld16(col + ucols, av);
                    ptx::tmem_wait_ld();
                    ptx::tc_fence_before();
                    __syncwarp();
                    ptx::mbar_arrive_if(read, lead);
                    float2 s2 = make_float2(0.f, 0.f), w2 = s2, pd[8];
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int j = 8 * p + 2 * q;
                            const float2 x = __ffma2_rn(make_float2(__uint_as_float(s[j]), __uint_as_float(s[j + 1])), sl2p, nldp);
                            const float2 e = pd[4 * p + q] = make_float2(ptx::ex2(x.x), ptx::ex2(x.y));
                            s2 = __ffma2_rn(e, make_float2(__uint_as_float(av[j]), __uint_as_float(av[j + 1])), s2);
                            w2 = __fadd2_rn(w2, e);
                            hi[q] = ptx::pack_bf16(e);
                            lo[q] = ptx::pack_bf16(ptx::rest_of(e, hi[q]));
                        }
                        ptx::sts128(w ^ (p ? 16u : 0u), hi);
                        ptx::sts128((w ^ (p ? 16u : 0u)) + kSwHalf, lo);
                    }
                    sums.add(pd, av, s2, w2);
                } else {
                    ptx::mbar_arrive_if(read, lead);
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                ptx::mbar_arrive_if(bar(P_FULL + (n & 3)), lead);
                w += (uint32_t)sets * kSwBuf;
                if (w >= w_end) w -= SM::kBufs * kSwBuf;
            }
            if (!ok || !(ok = warp_wait(bar(DD_EMPTY + (i & 1)), ((i >> 1) & 1) ^ 1, abort_flag, kErrBwdDz | 12))) break;
            dds[((i & 1) * kSwGroups + mine) * kTile + row] = sums.get();
            __syncwarp();
            ptx::mbar_arrive_if(bar(DD_FULL + (i & 1)), lead);
            if (((i + 1) & (flush - 1)) == 0 || i + 1 == nt) {
                const int window = i / flush;                // (after the window before, which the other set of warps may be about)
                if (window > 0 && !warp_wait(bar(FL_DONE), (window - 1) & 1, abort_flag, kErrBwdDz | 11)) break;
                if (!warp_wait(bar(FL_FULL), window & 1, abort_flag, kErrBwdDz | 10)) break;
                ptx::tc_fence_after();
                sweep_flush<D, DR>(acc0 - tm + gcol, a.part, (size_t)a.B * a.H * a.mtot, cta, r0, M, nu, min(sums_in_turn, i + 1 - window * flush), mine, cps, row, off, window > 0 || (kRanges && a.t0 > 0));
                ptx::tc_fence_before();
                __syncwarp();
                ptx::mbar_arrive_if(bar(FL_DONE), lead);
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tm, 512);
    }
    if (threadIdx.x == 0 && *abort_flag != 0 && a.status != nullptr) atomicCAS(a.status, 0u, *abort_flag);
}

// ---------------------------------------------------------------------------------------------------------- second sweep: dK, dV, dQ
// W_enc = W_dec r[n] c[m] with r = 2^(lse_dec[n] - K), c = 2^(K - lse_enc[m]) and K in the middle of the latents' lse_enc, so that with c dZ in the
// place of dZ one exponential and one split of a weight serve both:
//     dS = W_dec (A - dd + r (C' - c de)),   C' = V (c dZ)^T,     dV_n = r sum_m W_dec (c dZ)_m.
// What the factors may lose: W_dec below 2^-126 is flushed, which is a W_enc below 2^-126 r c = 2^(lse_dec[n] - lse_enc[m] - 126) (log2 units): below 2^-86 in
// tiles whose tokens have an lse_dec within kOneExpLog2 of the least lse_enc.  (A bound by the range of lse_enc alone would not
// do: of a range of latents lse_dec may lie far above all, and weights it flushes may then be all there is of a row of dV.)  Tiles beyond that
// (an infinite lse_dec is how the two-query variant switches a stage off) take a form of the body with an exponential of its own for W_enc,
// 2^(S - K) against c dZ, c at most 2^(kFoldLog2 / 2); for wider ranges of lse_enc all tiles do, and c is 1.
constexpr float kSwFoldLog2 = 80.f;

struct BwdGradArgs {
    const __nv_bfloat16 *Q;    // [H,M,D]
    const float *Z, *dZ;       // [B,H,M,D]
    const float *lse_enc, *de; // [B,H,M]
    const float *lse_dec;      // [B,N,H]
    const float *dd;           // [2][B,H,N], see BwdDzArgs
    const uint8_t *key_mask;   // [B,N] or null
    __nv_bfloat16 *dK, *dV;    // [B,N,H,D]
    float *part;               // [2 * CTAs per head][B*H*M][D] partial dQ rows (un-scaled)
    uint32_t *status;
    int B, H, N, M, mtot, m0, first, last;   // as in BwdDzArgs
    float *kvacc;              // float32 dK and dV so far, where there are ranges; the last writes the rows.  [range of those side by side][2][B,H][tile of this launch][D / 4][token of the tile][4]
    float scale, sl2;
    int tiles, stages, bufs, t0, side;   // as in BwdDzArgs
};

template <int D>
struct BwdGradSmem {
    using G = TileGeom<D>;
    enum { ZH = 0, ZL = 1, DH = 2, DL = 3, QR = 4 };            // latent operands: Z hi, lo, c dZ hi, lo, Q
    static constexpr int kAccStride = 3 * D;                    // columns of an accumulator: dK | dV | dV's share of c dZ lo
    // accumulators beside S twice, A, C and the sums over tokens: a power of two up to four (as a logarithm); negative if there is none
    __host__ __device__ static int log2_accs(int M) {
        const int ucols = (M + 31) / 32 * 32 < kSwUnit ? (M + 31) / 32 * 32 : kSwUnit, fit = (512 - 4 * ucols - (M + kSwUnit - 1) / kSwUnit * D) / kAccStride;
        return fit >= 4 ? 2 : fit >= 2 ? 1 : fit >= 1 ? 0 : -1;
    }
    // sums over tokens in what is left
    __host__ __device__ static int log2_sums(int M) {
        const int ucols = (M + 31) / 32 * 32 < kSwUnit ? (M + 31) / 32 * 32 : kSwUnit;
        return sweep_log2_sums(512 - 4 * ucols - (kAccStride << log2_accs(M)), (M + kSwUnit - 1) / kSwUnit * D);
    }
    __host__ __device__ static size_t tile_off(int bufs) { return (size_t)bufs * kSwBuf; }
    __host__ __device__ static size_t lat_off(int bufs, int stages, int M, int which) { return tile_off(bufs) + (size_t)stages * 3 * G::TILE_BYTES + (size_t)which * M * G::RB; }
    __host__ __device__ static size_t cst_off(int bufs, int stages, int M) { return lat_off(bufs, stages, M, 5); }     // per latent the exponent's addend and -c de
    __host__ __device__ static size_t ring_off(int bufs, int stages, int M) { return cst_off(bufs, stages, M) + 2 * sizeof(float) * M; }   // [ring][-lse_dec | -dd | what is left of it | r][token]
    __host__ __device__ static size_t bar_off(int bufs, int stages, int M) { return ring_off(bufs, stages, M) + kSwRing * 4 * kTile * sizeof(float); }
    __host__ __device__ static size_t total(int bufs, int stages, int M) {
        const size_t t = bar_off(bufs, stages, M) + 768 + 1024;
        return t < kTcMinSmem ? kTcMinSmem : t;
    }
    __host__ static int stages(int bufs, int M) {
        int s = kSwMaxStages;
        while (s > 0 && total(bufs, s, M) > (size_t)227 * 1024) --s;
        return s;
    }
};

template <int D, int DRT, bool kRanges>
__global__ void __launch_bounds__(kSwThreads, 1)
bwd_grad_sweep_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmG,
                      const __grid_constant__ CUtensorMap tmDK, const __grid_constant__ CUtensorMap tmDV, BwdGradArgs a) {
    using G = TileGeom<D>;
    using SM = BwdGradSmem<D>;
    constexpr int UNIT = kSwUnit, RING = kSwRing, DR = DRT ? DRT : D;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = ptx::align_1024(smem_raw);
    const int side = kRanges ? a.side : 1, which_range = kRanges ? (int)blockIdx.x % side : 0, cta = (int)blockIdx.x / side, ctas = (int)gridDim.x / side;
    const int m0 = a.m0 + which_range * a.M, M = kRanges ? min(a.M, a.mtot - m0) : a.M, stages = a.stages, bufs = a.bufs;
    uint8_t *tiles_s = smem + SM::tile_off(bufs);
    float *cst = reinterpret_cast<float *>(smem + SM::cst_off(bufs, stages, M));
    float *ring = reinterpret_cast<float *>(smem + SM::ring_off(bufs, stages, M));
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + SM::bar_off(bufs, stages, M));
    enum { T_FULL = 0, T_DONE = T_FULL + kSwMaxStages, T_OUT = T_DONE + kSwMaxStages, S_FULL = T_OUT + kSwMaxStages, S_READ = S_FULL + 2, P_FULL = S_READ + 2, C_FULL = P_FULL + 2,
           C_EMPTY = C_FULL + RING, ACC_FULL = C_EMPTY + RING, ACC_EMPTY = ACC_FULL + 4, FL_FULL = ACC_EMPTY + 4, FL_DONE, NBARS };
    static_assert(NBARS * 8 + 8 + 4 * RING + 8 * kSwThreads / 32 <= 768, "barrier area too small");
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + NBARS);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    volatile uint32_t *two_exp = tmem_slot + 2;                 // [RING]: the tile takes the form with two exponentials
    float *extremes = reinterpret_cast<float *>(tmem_slot + 2 + RING);          // [warp][least, greatest lse_enc]

    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const int h = blockIdx.y, b = blockIdx.z;
    const int nt = (a.tiles - cta + ctas - 1) / ctas;
    auto tile_at = [&](int i) { return cta + i * ctas + (kRanges ? a.t0 : 0); };   // the i-th of them
    const int nu = (M + UNIT - 1) / UNIT, wlast = M - (nu - 1) * UNIT;
    const int sets = M <= 32 ? 2 : 1, cps = sets == 2 ? 2 : kSwGroups;
    const int ucols = min(UNIT, (M + 31) & ~31);                // columns of a region S, A or C
    const int log_accs = SM::log2_accs(M);
    const int off = DRT ? narrow_offset(h, DR) : 0;
    const int units = nu * nt, sums_in_turn = 1 << SM::log2_sums(M), flush = sweep_flush_tiles(nu, sums_in_turn);
    // (opaque: an address that can be formed again from the kernel's arguments is, at every use, by a dozen instructions)
    uint32_t bars0 = ptx::smem_u32(bars);
    ptx::opaque(bars0);
    auto bar = [&](int i) { return bars0 + 8u * i; };

    if (threadIdx.x == 0) {
        const uint32_t math = 4 * cps;
        for (int i = 0; i < NBARS; ++i)
            ptx::mbar_init(bar(i), (i >= T_OUT && i < S_FULL) || (i >= S_READ && i < C_FULL) || (i >= C_EMPTY && i < ACC_FULL) || (i >= ACC_EMPTY && i < FL_FULL) || i == FL_DONE ? math
                                   : (i >= S_FULL && i < S_READ) || (i >= ACC_FULL && i < ACC_EMPTY) ? 2u : 1u);   // (two issuing warps)
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmK);
        ptx::prefetch_tensormap(&tmV);
        ptx::prefetch_tensormap(&tmG);
    }
    if (warp == 1) ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
    ptx::grid_launch();
    ptx::grid_wait();
    const size_t bh = (size_t)b * a.H + h, q0 = (size_t)h * a.mtot + m0, r0 = bh * a.mtot + m0;
    float K, least, unfolded;                                   // (unfolded != 0: c is 1)
    {
        // K: the middle of the latents' lse_enc (log2 units), leaving out those that saw no valid token and those whose encode is switched off
        float lo = INFINITY, hi = -INFINITY;
        for (int m = threadIdx.x; m < M; m += kSwThreads) {
            const float le = a.lse_enc[r0 + m] * kBwdLog2e;
            if (le != -INFINITY && le != INFINITY) {
                lo = fminf(lo, le);
                hi = fmaxf(hi, le);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if (lane == 0) {
            extremes[2 * warp] = lo;
            extremes[2 * warp + 1] = hi;
        }
        z_centre<DR>(ring, a.Z + bh * a.mtot * DR, a.mtot);     // (over the ring, which is not in use yet)
        if (DRT != 0)                                           // narrow form: the other columns of every row stay zero
            for (int i = threadIdx.x; i < 5 * M * (G::RB / 16); i += kSwThreads) reinterpret_cast<uint4 *>(smem + SM::lat_off(bufs, stages, M, 0))[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        for (int w = 0; w < kSwThreads / 32; ++w) {
            lo = fminf(lo, extremes[2 * w]);
            hi = fmaxf(hi, extremes[2 * w + 1]);
        }
        K = lo <= hi ? 0.5f * (lo + hi) : 0.f;
        least = lo <= hi ? lo : 0.f;
        unfolded = lo > hi || hi - lo <= kSwFoldLog2 ? 0.f : 1.f;
    }
    auto factor = [&](int m) {                                  // c of latent m; 0 for those left out
        const float le = a.lse_enc[r0 + m] * kBwdLog2e;
        return le == -INFINITY || le == INFINITY ? 0.f : unfolded != 0.f ? 1.f : ptx::ex2(K - le);
    };
    {
        uint8_t *lat[5];
#pragma unroll
        for (int w = 0; w < 5; ++w) lat[w] = smem + SM::lat_off(bufs, stages, M, w);
        if constexpr (DR == 4) {
            stage_rows4<D>(lat[SM::QR], a.Q + q0 * DR, M, off);
            stage_rows4_hilo<D>(lat[SM::ZH], lat[SM::ZL], a.Z + r0 * DR, M, off, ring);
            stage_rows4_hilo<D>(lat[SM::DH], lat[SM::DL], a.dZ + r0 * DR, M, off, nullptr, factor);
        } else {
            stage_bf16<D, DR>(lat[SM::QR], a.Q + q0 * DR, M, 0, 0, threadIdx.x, kSwThreads);
            stage_hilo<D, DR>(lat[SM::ZH], lat[SM::ZL], a.Z + r0 * DR, M, 0, 0, threadIdx.x, kSwThreads, ring);
            stage_hilo<D, DR>(lat[SM::DH], lat[SM::DL], a.dZ + r0 * DR, M, 0, 0, threadIdx.x, kSwThreads, nullptr, factor);
        }
        for (int m = threadIdx.x; m < M; m += kSwThreads) {
            const float c = factor(m);
            cst[m] = c == 0.f ? -INFINITY : unfolded != 0.f ? -a.lse_enc[r0 + m] * kBwdLog2e : -K;
            cst[M + m] = -c * a.de[r0 + m];
        }
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = *tmem_slot;
    // columns: S twice, A, C, the accumulators, the sums over tokens
    const uint32_t a_col = 2 * ucols, acc0 = 4 * ucols, dq0 = acc0 + ((uint32_t)SM::kAccStride << log_accs);

    if (warp == 0) {
        if (ptx::elect_one()) {
            // Rows of dK and dV leave from where K and V of their tile were.
            auto store = [&](int i) -> bool {
                const int s = i % stages, t = tile_at(i);
                if (!ptx::mbar_wait(bar(T_OUT + s), (i / stages) & 1, abort_flag, kErrBwdTok | 16)) return false;
                if (DR >= 8 && (!kRanges || a.last)) {
                    const uint32_t src = ptx::smem_u32(tiles_s + (size_t)s * 3 * G::TILE_BYTES);
                    ptx::tma_store_3d(&tmDK, src, h * DR, t * kTile, b);
                    ptx::tma_store_3d(&tmDV, src + G::TILE_BYTES, h * DR, t * kTile, b);
                    ptx::tma_store_commit();
                }
                return true;
            };
            int i = 0;
            for (; i < nt; ++i) {
                const int s = i % stages, t = tile_at(i);
                if (i >= stages) {
                    if (!store(i - stages)) break;
                    ptx::tma_store_wait<true>();
                }
                ptx::mbar_arrive_expect_tx(bar(T_FULL + s), 3 * G::TILE_BYTES);
                uint8_t *dst = tiles_s + (size_t)s * 3 * G::TILE_BYTES;
                ptx::tma_load_3d(ptx::smem_u32(dst), &tmK, bar(T_FULL + s), h * DR - off, t * kTile, b);
                ptx::tma_load_3d(ptx::smem_u32(dst + G::TILE_BYTES), &tmV, bar(T_FULL + s), h * DR - off, t * kTile, b);
                ptx::tma_load_3d(ptx::smem_u32(dst + 2 * G::TILE_BYTES), &tmG, bar(T_FULL + s), h * DR - off, t * kTile, b);
            }
            if (i == nt)
                for (int j = max(0, nt - stages); j < nt && store(j); ++j) {}
            ptx::tma_store_wait<false>();
        }
    } else if (warp == 2) {
        // Token constants of every tile: -lse_dec, -dd and r (0 for a token that takes no part in the encode softmax), or, in a tile that takes
        // two exponentials, 0 or -inf in the place of r.  Fetched by asynchronous copies three tiles ahead.
        constexpr int AH = RING - 1;
        auto fetch = [&](int i) {
            float *at = ring + (i % RING) * 4 * kTile;
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) {
                const int r = e * 32 + lane, n = min(tile_at(i) * kTile + r, a.N - 1);
                ptx::copy_async4(ptx::smem_u32(at + r), a.lse_dec + ((size_t)b * a.N + n) * a.H + h);
                ptx::copy_async4(ptx::smem_u32(at + kTile + r), a.dd + bh * a.N + n);
                ptx::copy_async4(ptx::smem_u32(at + 2 * kTile + r), a.dd + ((size_t)a.B * a.H + bh) * a.N + n);
            }
        };
        for (int k = 0; k < AH; ++k) {
            if (k < nt) fetch(k);
            ptx::copy_async_commit();
        }
        for (int i = 0; i < nt; ++i) {
            ptx::copy_async_wait<AH - 1>();
            __syncwarp();
            float *at = ring + (i % RING) * 4 * kTile;
            float ld[kTile / 32];
            bool part[kTile / 32], far = unfolded != 0.f;
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) {
                const int r = e * 32 + lane, n = tile_at(i) * kTile + r;
                const bool in = n < a.N;
                ld[e] = in ? at[r] * kBwdLog2e : INFINITY;
                part[e] = in && (a.key_mask == nullptr || a.key_mask[(size_t)b * a.N + n] != 0);
                at[r] = -ld[e];
                at[kTile + r] = in ? -at[kTile + r] : 0.f;
                at[2 * kTile + r] = in ? -at[2 * kTile + r] : 0.f;
                far = far || (part[e] && !(ld[e] - least <= kOneExpLog2));
            }
            far = __any_sync(0xffffffffu, far);
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e)
                at[3 * kTile + e * 32 + lane] = far ? (part[e] ? 0.f : -INFINITY) : (part[e] ? ptx::ex2(ld[e] - K) : 0.f);
            if (lane == 0) two_exp[i % RING] = far ? 1u : 0u;
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(C_FULL + i % RING));
            const int next = i + AH;
            if (next < nt) {
                if (!warp_wait(bar(C_EMPTY + next % RING), ((next / RING) & 1) ^ 1, abort_flag, kErrBwdTok | 2)) break;
                fetch(next);
            }
            ptx::copy_async_commit();
        }
        ptx::copy_async_wait<0>();
    } else if (warp == 1) {
        // Forms A and C and adds up dK and dQ, whose operand dS lies in shared memory.
        {
            const uint32_t lead = ptx::elect_one() ? 1u : 0u;
            constexpr uint32_t HI = ptx::desc_hi(G::SBO, G::SWZ), TILE = G::TILE_BYTES >> 4, STEP16 = (16 * G::RB) >> 4;
            const uint32_t LAT = (uint32_t)(M * G::RB) >> 4;
            const uint32_t lat0 = ptx::desc_lo(ptx::smem_u32(smem + SM::lat_off(bufs, stages, M, 0)), 16), td0 = ptx::desc_lo(ptx::smem_u32(tiles_s), 16);
            constexpr uint32_t MN = ptx::desc_lo(0, G::SBO) - ptx::desc_lo(0, 16);
            const uint32_t w0 = ptx::desc_lo(ptx::smem_u32(smem), 0);
            int s_stage = 0, s_wrap = 0, s_u = 0;               // of the next A and C
            int k_u = 0, k_buf = 0, k_acc = 0, k_wrap = 0;      // of the next dK
            int q_stage = 0, q_u = 0, q_tile = 0, q_buf = 0, window = 0, q_n = 0;   // of the next dQ
            auto products = [&](int n) -> bool {
                if (s_u == 0) {
                    if (!issue_wait(bar(T_FULL + s_stage), (uint32_t)s_wrap, abort_flag, kErrBwdTok | 3)) return false;
                    ptx::tc_fence_after();
                }
                const uint32_t idescS = ptx::instr_desc_bf16(128, 0, 0, 0) | (uint32_t)((s_u == nu - 1 ? wlast : UNIT) >> 3) << 17;
                uint32_t td = td0 + (uint32_t)s_stage * 3 * TILE, ld = lat0 + (uint32_t)s_u * (UNIT / 16) * STEP16;
                auto product = [&](int of, int lat, bool more) {
                    const uint32_t ad = td + (of == 0 ? 2 * TILE : TILE), bd = ld + lat * LAT;
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) ptx::mma_ss_by(lead, tm + a_col + of * ucols, ptx::desc(ad + 2 * k, HI), ptx::desc(bd + 2 * k, HI), idescS, k > 0 || more);
                };
                product(0, SM::ZL, false);
                product(0, SM::ZH, true);
                product(1, SM::DL, false);
                product(1, SM::DH, true);
                ptx::mma_commit_by(lead, bar(S_FULL + (n & 1)));
                if (++s_u == nu) {
                    s_u = 0;
                    if (++s_stage == stages) { s_stage = 0; s_wrap ^= 1; }
                }
                return true;
            };
            // dK += dS Q
            auto keys = [&]() -> bool {
                constexpr uint32_t idesc = ptx::instr_desc_bf16(128, D, 0, 1);
                if (k_u == 0) {
                    if (!issue_wait(bar(ACC_EMPTY + k_acc), (uint32_t)k_wrap ^ 1u, abort_flag, kErrBwdTok | 4)) return false;
                    ptx::tc_fence_after();
                }
                const uint32_t T = tm + acc0 + k_acc * SM::kAccStride;
                uint32_t wd = w0 + kSwDescK + (uint32_t)k_buf * (kSwBuf >> 4), qd = lat0 + SM::QR * LAT + MN + (uint32_t)k_u * (UNIT / 16) * STEP16;
                auto step = [&](int k) {
                    ptx::mma_ss_by(lead, T, ptx::desc(wd + 2 * k, kSwDescHi), ptx::desc(qd + k * STEP16, HI), idesc, (k_u > 0 || k > 0) ? 1u : 0u);
                    ptx::mma_ss_by(lead, T, ptx::desc(wd + (kSwHalf >> 4) + 2 * k, kSwDescHi), ptx::desc(qd + k * STEP16, HI), idesc, 1u);
                };
                const int steps = (k_u == nu - 1 ? wlast : UNIT) / 16;
                if (steps == UNIT / 16) {
#pragma unroll
                    for (int k = 0; k < UNIT / 16; ++k) step(k);
                } else {
                    for (int k = 0; k < steps; ++k) step(k);
                }
                if (++k_buf == bufs) k_buf = 0;
                if (++k_u == nu) {
                    k_u = 0;
                    ptx::mma_commit_by(lead, bar(ACC_FULL + k_acc));
                    if (++k_acc == 1 << log_accs) { k_acc = 0; k_wrap ^= 1; }
                }
                return true;
            };
            // dQ += dS^T K: 16 tokens per step
            auto queries = [&]() -> bool {
                constexpr uint32_t idesc = ptx::instr_desc_bf16(128, D, 1, 1);
                if (q_u == 0 && q_tile == 0 && window > 0) {
                    if (!issue_wait(bar(FL_DONE), (window - 1) & 1, abort_flag, kErrBwdTok | 5)) return false;
                    ptx::tc_fence_after();
                }
                uint32_t wd = w0 + kSwDescMn + (uint32_t)q_buf * (kSwBuf >> 4), kd = td0 + MN + (uint32_t)q_stage * 3 * TILE;
                const uint32_t to = tm + dq0 + ((q_tile & (sums_in_turn - 1)) * nu + q_u) * D;
#pragma unroll
                for (int k = 0; k < kTile / 16; ++k)
                    ptx::mma_ss_by(lead, to, ptx::desc(wd + k * (2048 >> 4), kSwDescHi), ptx::desc(kd + k * STEP16, HI), idesc, (q_tile >= sums_in_turn || k > 0) ? 1u : 0u);
                if (++q_buf == bufs) q_buf = 0;
                ++q_n;
                if (++q_u == nu) {
                    q_u = 0;
                    ptx::mma_commit_by(lead, bar(T_DONE + q_stage));
                    if (++q_stage == stages) q_stage = 0;
                    if (++q_tile == flush || q_n == units) {
                        ptx::mma_commit_by(lead, bar(FL_FULL));
                        q_tile = 0;
                        ++window;
                    }
                }
                return true;
            };
            // What says that the products of unit n + 1 are there says as well that a buffer of dS has been read: with two buffers that of unit n - 1,
            // whose sums come before those products; with three that of n - 2, and dQ of unit n - 1 may come behind them.
            // us per step, in order : late, 131072 tokens, 8 heads: D = 32, M = 32 237 : 267, 64 305 : 313, 32 x 4096, M = 128 239 : 244; D = 16, M = 32 226 : 218, 64 260 : 258; in
            // ranges, D = 8, M = 1024 2220 : 2270, D = 16 2312 : 2352.
            const bool late = bufs == 3 && D == 16 && !kRanges;
            bool ok = products(0);
            for (int n = 0; ok && n < units; ++n) {
                if (n + 1 < units) {
                    if (!issue_wait(bar(S_READ + (n & 1)), (n >> 1) & 1, abort_flag, kErrBwdTok | 6)) break;
                    ptx::tc_fence_after();
                    if (!products(n + 1)) break;
                }
                if (late && n > 0 && !queries()) break;
                if (!issue_wait(bar(P_FULL + (n & 1)), (n >> 1) & 1, abort_flag, kErrBwdTok | 7)) break;
                ptx::tc_fence_after();
                if (!keys()) break;
                if ((!late || n + 1 == units) && !queries()) break;
            }
        }
    } else if (warp == 3) {
        // Forms S and adds up dV, whose weights lie over S.
        {
            const uint32_t lead = ptx::elect_one() ? 1u : 0u;
            constexpr uint32_t HI = ptx::desc_hi(G::SBO, G::SWZ), TILE = G::TILE_BYTES >> 4, STEP16 = (16 * G::RB) >> 4;
            const uint32_t LAT = (uint32_t)(M * G::RB) >> 4;
            const uint32_t lat0 = ptx::desc_lo(ptx::smem_u32(smem + SM::lat_off(bufs, stages, M, 0)), 16), td0 = ptx::desc_lo(ptx::smem_u32(tiles_s), 16);
            constexpr uint32_t MN = ptx::desc_lo(0, G::SBO) - ptx::desc_lo(0, 16);
            int s_stage = 0, s_wrap = 0, s_u = 0, o_u = 0, o_acc = 0, o_wrap = 0;
            auto scores = [&](int n) -> bool {
                if (s_u == 0) {
                    if (!issue_wait(bar(T_FULL + s_stage), (uint32_t)s_wrap, abort_flag, kErrBwdTok | 8)) return false;
                    ptx::tc_fence_after();
                }
                const uint32_t idescS = ptx::instr_desc_bf16(128, 0, 0, 0) | (uint32_t)((s_u == nu - 1 ? wlast : UNIT) >> 3) << 17;
                uint32_t td = td0 + (uint32_t)s_stage * 3 * TILE, ld = lat0 + SM::QR * LAT + (uint32_t)s_u * (UNIT / 16) * STEP16;
#pragma unroll
                for (int k = 0; k < D / 16; ++k) ptx::mma_ss_by(lead, tm + (n & 1) * ucols, ptx::desc(td + 2 * k, HI), ptx::desc(ld + 2 * k, HI), idescS, k > 0);
                ptx::mma_commit_by(lead, bar(S_FULL + (n & 1)));
                if (++s_u == nu) {
                    s_u = 0;
                    if (++s_stage == stages) { s_stage = 0; s_wrap ^= 1; }
                }
                return true;
            };
            bool ok = true;
            for (int n = 0; ok && n < 2 && n < units; ++n) ok = scores(n);
            for (int n = 0; ok && n < units; ++n) {
                constexpr uint32_t idesc = ptx::instr_desc_bf16(128, D, 0, 1), idesc2 = ptx::instr_desc_bf16(128, 2 * D, 0, 1);
                if (!issue_wait(bar(P_FULL + (n & 1)), (n >> 1) & 1, abort_flag, kErrBwdTok | 9)) break;
                if (o_u == 0 && !issue_wait(bar(ACC_EMPTY + o_acc), (uint32_t)o_wrap ^ 1u, abort_flag, kErrBwdTok | 10)) break;
                ptx::tc_fence_after();
                const uint32_t V = tm + acc0 + o_acc * SM::kAccStride + D, w = tm + (n & 1) * ucols;
                // (MN-major; the block of c dZ lo along N is one operand further on: LBO, bits 16-29)
                const uint32_t dh = lat0 + SM::DH * LAT - ptx::desc_lo(0, 16) + (LAT << 16) + (uint32_t)o_u * (UNIT / 16) * STEP16;
                auto step = [&](int k) {                        // (hi of 16 latents, lo 8 columns on)
                    ptx::mma_ts_by(lead, V, w + 16 * k, ptx::desc(dh + k * STEP16, HI), idesc2, (o_u > 0 || k > 0) ? 1u : 0u);
                    ptx::mma_ts_by(lead, V, w + 16 * k + 8, ptx::desc(dh + k * STEP16, HI), idesc, 1u);
                };
                const int steps = (o_u == nu - 1 ? wlast : UNIT) / 16;
                if (steps == UNIT / 16) {
#pragma unroll
                    for (int k = 0; k < UNIT / 16; ++k) step(k);
                } else {
                    for (int k = 0; k < steps; ++k) step(k);
                }
                if (++o_u == nu) {
                    ptx::mma_commit_by(lead, bar(ACC_FULL + o_acc));
                    o_u = 0;
                    if (++o_acc == 1 << log_accs) { o_acc = 0; o_wrap ^= 1; }
                }
                if (n + 2 < units) ok = scores(n + 2);
            }
        }
    } else if (warp >= kSwFirstMathWarp) {
        const int cg = (warp - kSwFirstMathWarp) >> 2, set = sets == 2 ? cg >> 1 : 0, mine = sets == 2 ? cg & 1 : cg;   // columns: 16 from 16 mine on
        const int row = ((warp & 3) << 5) + lane;               // TMEM lane = token within the tile
        const uint32_t gcol = tm + ((uint32_t)((warp & 3) << 5) << 16);
        const float2 sl2p = make_float2(a.sl2, a.sl2);
        const uint32_t lead = lane == 0;
        uint32_t cst0 = ptx::smem_u32(cst + 16 * mine);         // the exponent's addends of this warp's latents, M further on -c de
        ptx::opaque(cst0);
        // this thread's first 16 bytes (8 latents) of the hi halves in its next buffer of weights; the next 8 latents are at `w ^ 16`
        const uint32_t w_first = ptx::smem_u32(smem) + (uint32_t)row * 128 + ((uint32_t)((2 * mine) ^ (row & 7)) << 4);
        uint32_t w = w_first + (uint32_t)(set % bufs) * kSwBuf, w_end = w_first + (uint32_t)bufs * kSwBuf;
        ptx::opaque(w);
        ptx::opaque(w_end);
        auto next_buffer = [&] {
            w += (uint32_t)sets * kSwBuf;
            if (w >= w_end) w -= (uint32_t)bufs * kSwBuf;
        };
        // Rows of dK and dV of the set's k-th tile: pieces of eight columns, in turn to the warps that share the tokens, to where K and V of the tile were.
        int out_stage = set % stages;                           // (where the set's next rows go)
        uint32_t out_wrap = 0;
        auto write_rows = [&](int k, float r) -> bool {
            constexpr int COLS = DR >= 16 ? DR : 8, PIECES = COLS / 4, PW = DR == 4 ? 4 : 8;
            const int i = set + k * sets, acc = i & ((1 << log_accs) - 1), s = out_stage, t = tile_at(i);
            if (!warp_wait(bar(ACC_FULL + acc), (i >> log_accs) & 1, abort_flag, kErrBwdTok | 11)) return false;
            if (!warp_wait(bar(T_DONE + s), out_wrap, abort_flag, kErrBwdTok | 17)) return false;
            ptx::tc_fence_after();
            uint32_t out = ptx::smem_u32(tiles_s) + (uint32_t)s * (3 * G::TILE_BYTES) + (uint32_t)row * (DR >= 16 ? G::RB : 16);
            ptx::opaque(out);
#pragma unroll
            for (int p0 = 0; p0 < PIECES; p0 += kSwGroups) {
                const int p = p0 + (PIECES <= 2 ? (mine + 2 * k) & (cps - 1) : mine);
                if (p >= PIECES) continue;
                for (int pp = p; pp < min(PIECES, p0 + kSwGroups); pp += cps) {
                    const int which = (pp ^ (pp >> 2)) & 1, c0 = (pp >> 1) * 8;   // dK or dV, and the first column
                    uint32_t x[8], y[8] = {};
                    const uint32_t col = gcol + acc0 + acc * SM::kAccStride + which * D + c0;
                    ptx::tmem_ld8(col, x);
                    if (which) ptx::tmem_ld8(col + D, y);
                    float4 *sums = nullptr;
                    float4 before[PW / 4];
                    if (kRanges) {
                        sums = reinterpret_cast<float4 *>(a.kvacc) + ((((size_t)(2 * which_range + which) * a.B * a.H + bh) * a.tiles + (t - a.t0)) * (DR / 4) + c0 / 4) * kTile + row;
                        if (!a.first) {
#pragma unroll
                            for (int c = 0; c < PW / 4; ++c) before[c] = sums[c * kTile];
                        }
                    }
                    ptx::tmem_wait_ld();
                    const float f = which ? r : kRanges ? 1.f : a.scale;
                    float v[PW];
#pragma unroll
                    for (int c = 0; c < PW; ++c)                // (narrow heads: the head's own columns)
                        v[c] = (__uint_as_float(DR == 4 && off != 0 ? x[(4 + c) & 7] : x[c]) + __uint_as_float(DR == 4 && off != 0 ? y[(4 + c) & 7] : y[c])) * f;
                    if (kRanges && !a.first) {                  // the earlier ranges' shares
#pragma unroll
                        for (int c = 0; c < PW / 4; ++c) {
                            v[4 * c] += before[c].x; v[4 * c + 1] += before[c].y; v[4 * c + 2] += before[c].z; v[4 * c + 3] += before[c].w;
                        }
                    }
                    if (kRanges && !a.last) {
#pragma unroll
                        for (int c = 0; c < PW / 4; ++c) sums[c * kTile] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
                    } else {
                        const float sc = kRanges && which == 0 ? a.scale : 1.f;
                        uint32_t w2[PW / 2];
#pragma unroll
                        for (int c = 0; c < PW / 2; ++c) w2[c] = ptx::pack_bf16(v[2 * c] * sc, v[2 * c + 1] * sc);
                        if constexpr (PW == 4) {                // (rows of 8 bytes are too short for a tile's copy)
                            const int n = t * kTile + row;
                            if (n < a.N) *reinterpret_cast<uint2 *>((which ? a.dV : a.dK) + (((size_t)b * a.N + n) * a.H + h) * DR) = make_uint2(w2[0], w2[1]);
                        } else {
                            ptx::sts128(out + which * G::TILE_BYTES + (DR >= 16 ? (uint32_t)(((c0 >> 3) ^ G::swz(row)) << 4) : 0u), w2);
                        }
                    }
                    __syncwarp();
                }
            }
            ptx::fence_proxy_async_smem();
            ptx::tc_fence_before();
            __syncwarp();
            ptx::mbar_arrive_if(bar(ACC_EMPTY + acc), lead);
            ptx::mbar_arrive_if(bar(T_OUT + s), lead);
            if ((out_stage += sets) >= stages) {
                out_stage -= stages;
                out_wrap ^= 1;
            }
            return true;
        };
        // Sixteen columns of a unit: W_dec (kTwo: W_enc) over S, hi and lo of 16 latents side by side, dS to shared memory.
        auto unit = [&](auto two, uint32_t col, uint32_t read, uint32_t at, float2 nldp, float2 rp, float2 nddp, float2 ndd2p) {
            constexpr bool kTwo = decltype(two)::value;
            uint32_t s[16], av[16], cv[16];
            ptx::tmem_ld16(col, s);
            ptx::tmem_ld16(gcol + a_col + 16 * mine, av);
            ptx::tmem_ld16(gcol + a_col + ucols + 16 * mine, cv);
            ptx::tmem_wait_ld();
            ptx::tc_fence_before();
            __syncwarp();
            ptx::mbar_arrive_if(read, lead);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                uint32_t hi[4], lo[4], wh[4], wl[4];
#pragma unroll
                for (int q = 0; q < 4; q += 2) {
                    const float4 ne = ptx::lds128(at + (uint32_t)(M * 4) + (8 * p + 2 * q) * 4);
                    float4 le = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (kTwo) le = ptx::lds128(at + (8 * p + 2 * q) * 4);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int o = q + e, j = 8 * p + 2 * o;
                        const float2 sv = make_float2(__uint_as_float(s[j]), __uint_as_float(s[j + 1]));
                        const float2 A = __fadd2_rn(__fadd2_rn(make_float2(__uint_as_float(av[j]), __uint_as_float(av[j + 1])), nddp), ndd2p);
                        const float2 v = __fadd2_rn(make_float2(__uint_as_float(cv[j]), __uint_as_float(cv[j + 1])), e ? make_float2(ne.z, ne.w) : make_float2(ne.x, ne.y));
                        const float2 x = __ffma2_rn(sv, sl2p, nldp);
                        float2 pw = make_float2(ptx::ex2(x.x), ptx::ex2(x.y)), ds;
                        if (kTwo) {
                            const float2 y = __ffma2_rn(sv, sl2p, __fadd2_rn(e ? make_float2(le.z, le.w) : make_float2(le.x, le.y), rp));
                            const float2 pe = make_float2(ptx::ex2(y.x), ptx::ex2(y.y));
                            ds = __ffma2_rn(pw, A, __fmul2_rn(pe, v));
                            pw = pe;
                        } else {
                            ds = __fmul2_rn(pw, __ffma2_rn(rp, v, A));
                        }
                        hi[o] = ptx::pack_bf16(ds);
                        lo[o] = ptx::pack_bf16(ptx::rest_of(ds, hi[o]));
                        wh[o] = ptx::pack_bf16(pw);
                        wl[o] = ptx::pack_bf16(ptx::rest_of(pw, wh[o]));
                    }
                }
                ptx::tmem_st4(col + 4 * p, wh);
                ptx::tmem_st4(col + 8 + 4 * p, wl);
                ptx::sts128((w ^ (p ? 16u : 0u)), hi);
                ptx::sts128((w ^ (p ? 16u : 0u)) + kSwHalf, lo);
            }
            ptx::tmem_wait_st();
        };
        // (what follows a first unsuccessful try: inline at D = 16, where it is up to 4 % quicker; a call at D = 32, where the two differ by less than 1 %)
        auto unit_wait = [&](uint32_t at, uint32_t parity, uint32_t code) { return D == 16 ? issue_wait(at, parity, abort_flag, code) : warp_wait(at, parity, abort_flag, code); };
        // The loop over the units has nothing else in it: with the rows in a branch of it, it carried some forty instructions of theirs (131072 tokens, M = 256, D =
        // 16 649 -> 622 us per step when that was changed, 32 x 4096, M = 128 259 -> 239 with what follows dd in a warp of its own).
        // Rows of a tile leave after the first unit of the set's next, when they have long been formed; at D = 32 with two sets of warps at once: the other
        // set is at work, and four tile stages are all there is room for (us per step at once : after the next unit, 131072 tokens, 8 heads: D = 32, M = 32 237 : 260, D =
        // 16, M = 16 232 : 214, D = 8, M = 32 231 : 209).
        const bool at_once = D == 32 && sets == 2;
        int n = set;                                            // unit of all
        float r_before = 0.f;
        bool ok = true;
        for (int i = set, k = 0; ok; i += sets, ++k) {          // one more turn writes the last tile's rows
            const bool more = i < nt;
            bool pending = at_once ? more : k > 0;
            if (!more && !pending) break;
            float2 nldp = make_float2(0.f, 0.f), rp = nldp, nddp = nldp, ndd2p = nldp;
            bool far = false;
            if (more) {
                const int c = i % RING;
                if (!warp_wait(bar(C_FULL + c), (i / RING) & 1, abort_flag, kErrBwdTok | 12)) break;
                const float *at = ring + c * 4 * kTile + row;
                nldp = make_float2(at[0], at[0]);
                nddp = make_float2(at[kTile], at[kTile]);
                ndd2p = make_float2(at[2 * kTile], at[2 * kTile]);
                rp = make_float2(at[3 * kTile], at[3 * kTile]);
                far = __any_sync(0xffffffffu, two_exp[c] != 0); // (the same for all: a vote says so to the compiler)
                __syncwarp();
                ptx::mbar_arrive_if(bar(C_EMPTY + c), lead);
            }
            const float r = far ? 1.f : rp.x;
            int u = 0;
            do {
                if (more) {
                    uint32_t at = cst0 + (uint32_t)u * (UNIT * 4);
                    do {
                        const uint32_t col = gcol + (n & 1) * ucols + 16 * mine, read = bar(S_READ + (n & 1));
                        if (!(ok = unit_wait(read - 8 * (S_READ - S_FULL), (n >> 1) & 1, kErrBwdTok | 13))) break;
                        ptx::tc_fence_after();
                        if (u * UNIT + 16 * mine < M) {
                            if (far) unit(std::true_type{}, col, read, at, nldp, rp, nddp, ndd2p);
                            else unit(std::false_type{}, col, read, at, nldp, rp, nddp, ndd2p);
                        } else {
                            ptx::mbar_arrive_if(read, lead);
                        }
                        ptx::fence_proxy_async_smem();
                        ptx::tc_fence_before();
                        __syncwarp();
                        ptx::mbar_arrive_if(read + 8 * (P_FULL - S_READ), lead);
                        next_buffer();
                        n += sets;
                        at += UNIT * 4;
                    } while (++u < nu && !pending);
                    if (!ok) break;
                }
                if (pending) {
                    int done = at_once ? k : k - 1;
                    asm volatile("" : "+r"(done));              // (nothing of what follows is worked out ahead)
                    const int before = set + done * sets;
                    if (!(ok = write_rows(done, at_once ? r : r_before))) break;
                    if (((before + 1) & (flush - 1)) == 0 || before + 1 == nt) {
                        const int window = before / flush;   // (after the window before, which the other set of warps may be about)
                        if (window > 0 && !(ok = warp_wait(bar(FL_DONE), (window - 1) & 1, abort_flag, kErrBwdTok | 15))) break;
                        if (!(ok = warp_wait(bar(FL_FULL), window & 1, abort_flag, kErrBwdTok | 14))) break;
                        ptx::tc_fence_after();
                        sweep_flush<D, DR>(gcol + dq0, a.part, (size_t)a.B * a.H * a.mtot, cta, r0, M, nu, min(sums_in_turn, before + 1 - window * flush), mine, cps, row, off, window > 0 || (kRanges && a.t0 > 0));
                        ptx::tc_fence_before();
                        __syncwarp();
                        ptx::mbar_arrive_if(bar(FL_DONE), lead);
                    }
                    pending = false;
                }
            } while (more && u < nu);
            if (!more) break;
            r_before = r;
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tm, 512);
    }
    if (threadIdx.x == 0 && *abort_flag != 0 && a.status != nullptr) atomicCAS(a.status, 0u, *abort_flag);
}

// ---------------------------------------------------------------------------------------------------------- ranges side by side
// dd of every token from the ranges' RowSums, in the order of the latents.
template <int kThreads>
__global__ void __launch_bounds__(kThreads)
bwd_join_dd_kernel(const float4 *sums, float *dd, int side, int BH, int N, int tiles) {
    ptx::grid_launch();
    ptx::grid_wait();
    const size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x, plane = (size_t)BH * tiles * kTile;
    const size_t bh = i / ((size_t)tiles * kTile), n = i % ((size_t)tiles * kTile);
    if (i >= plane || n >= (size_t)N) return;
    RowSums all;
    all.set(sums[i]);
#pragma unroll 4
    for (int r = 1; r < side; ++r) all.join(sums[r * plane + i]);
    const float2 d = all.mean();
    dd[bh * N + n] = d.x;
    dd[((size_t)BH + bh) * N + n] = d.y;
}

// Rows of dK and dV from the ranges' shares, in the order of the latents: a thread has four columns of a row.
template <int D, int kThreads>
__global__ void __launch_bounds__(kThreads)
bwd_join_rows_kernel(const float4 *shares, __nv_bfloat16 *dK, __nv_bfloat16 *dV, int side, int B, int H, int N, int tiles, float scale) {
    ptx::grid_launch();
    ptx::grid_wait();
    const size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x, plane = (size_t)2 * B * H * tiles * (D / 4) * kTile;
    if (i >= plane) return;
    const size_t row = i % kTile, c = i / kTile % (D / 4), t = i / kTile / (D / 4) % tiles, whh = i / kTile / (D / 4) / tiles, bh = whh % ((size_t)B * H), n = t * kTile + row;
    if (n >= (size_t)N) return;
    float4 v = shares[i];
#pragma unroll 4
    for (int r = 1; r < side; ++r) {
        const float4 x = shares[r * plane + i];
        v = make_float4(v.x + x.x, v.y + x.y, v.z + x.z, v.w + x.w);
    }
    const bool value = whh >= (size_t)B * H;
    const float sc = value ? 1.f : scale;
    const uint2 out = make_uint2(ptx::pack_bf16(v.x * sc, v.y * sc), ptx::pack_bf16(v.z * sc, v.w * sc));
    *reinterpret_cast<uint2 *>((value ? dV : dK) + ((bh / H * N + n) * H + bh % H) * D + 4 * c) = out;
}

}  // namespace flare
