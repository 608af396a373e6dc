// Tensor-core encode without a running maximum, and dZ of the backward, for bfloat16 inputs on sm_100a.
//
//   fast forms   Z'_m = sum_n 2^(S[m,n] sl2) v_n,  l_m = sum_n 2^(S[m,n] sl2)      (see kFastMaxLog2), weights rounded to bfloat16 or as two halves
//   dZ form      dZ_m = sum_n exp(S[m,n] - lse_dec[n]) dY_n                         (dY in place of V; weights as two halves)
//
// No row maximum means that the order in which a row meets its columns does not matter and that partial results simply add up.  A CTA takes
// one block of 128 latents (latents on the 128 lanes; up to 64: two adjacent heads, see kPair) and a contiguous range of token tiles; its
// four or five groups of four warps take the half tiles (units of 64 tokens) in turn, each with scores and accumulator of its own in tensor
// memory: S_unit = Q K_unit^T, weights over the scores just read, acc += W V_unit.  While a group waits for the tensor core the others
// work: five groups where tensor memory has room (64 scores and at most 32 accumulator columns each), four of 128 columns otherwise.
// The groups' accumulators are added in shared memory at the end: one partial result per CTA.
// What bounds it: 4.5 to 5.5 instructions per weight (an exponential on the special-function unit takes 2, on the FMA pipe 4.5; the two
// share the work of the fast form), issued at 2.4 per cycle and SM; the unit is 60-75 % busy.
// Measured, us, against units of 32 tokens on two buffers in a kernel with a running-maximum skeleton, four groups bound to halves of the
// tile: dZ 261 -> 190 (131072, M = 512, D = 32); weights as two halves 3692 -> 2627, 217 ->
// 185; fast 522 -> 492 (million points, M = 256); masked, 262144 tokens, M = 96: 110 -> 82; D = 8 with 64 latents in head pairs: 85 -> 40.
// Also measured: four groups 4 to 9 % slower than five; the warps of a group issuing in turn instead of a warp of its own 6 %; one guard
// warp 20 %, three no better than two.
#pragma once

#include "flare_tc.cuh"

namespace flare {

enum LeanKind { kLeanFast = 0, kLeanHiLo = 1, kLeanDz = 2 };

template <int DG, int kKind>
struct LeanGeom {
    using G = TileGeom<DG>;
    static constexpr int UNIT = 64;
    // The fast form's value operand gets a second block along N whose column 0 is all ones: accumulator column DG is the sum of the rounded
    // weights (see exp_chunk_fast); at DG = 64 there is no room and the threads add the rounded weights themselves.
    static constexpr bool kOnes = kKind == kLeanFast && DG <= 32;
    static constexpr int kAccCols = kOnes ? DG + 16 : DG;
    static constexpr int NG = UNIT + kAccCols <= 96 ? 5 : 4, COLS = NG == 5 ? 96 : 128;
    static_assert(UNIT + kAccCols <= COLS && NG * COLS <= 512, "tensor memory");
    static constexpr int kGuards = kKind == kLeanFast ? (NG == 4 ? 3 : 2) : 0;                  // warps that check the norms of the key rows
    // (warp 0: TMA; 1 to NG: MMA issue; then the guards, or in the dZ form one warp that looks Z over for the kernels behind)
    static constexpr int kFirstGuardWarp = 1 + NG, kFirstMathWarp = kFirstGuardWarp + kGuards + (kKind == kLeanDz ? 1 : 0);
    static constexpr int kThreads = (kFirstMathWarp + 4 * NG) * 32;
    static constexpr size_t kOnesBytes = kOnes ? (size_t)UNIT * G::RB : 0, kColBytes = (size_t)4 * NG * UNIT * sizeof(float);
    static constexpr size_t tail = (size_t)kTile * G::RB + ((kOnesBytes + 1023) & ~(size_t)1023) + kColBytes + 512 + 1024;
    static constexpr int stages_for() {
        int n = 8;
        while (n * 2 * (size_t)G::TILE_BYTES + tail > 227 * 1024) --n;
        return n;
    }
    static constexpr int kStages = stages_for();                                // K+V tile pairs in flight
    static constexpr size_t q_off = (size_t)kStages * 2 * G::TILE_BYTES, ones_off = q_off + (size_t)kTile * G::RB;
    static constexpr size_t col_off = ones_off + ((kOnesBytes + 1023) & ~(size_t)1023), bar_off = col_off + kColBytes;
    static constexpr size_t total = (bar_off + 512 + 1024) < kTcMinSmem ? kTcMinSmem : bar_off + 512 + 1024;
};

struct EncodeLeanArgs {
    const __nv_bfloat16 *Q;   // [H,M,D]
    const float *lse_dec;     // [B,N,H]: dZ form
    const float *Z;           // [B,H,M,D], and
    float *around;            // [B * H][1 + blocks][D], dZ form: see z_around
    const uint8_t *key_mask;  // [B,N] or null
    float *part_m, *part_l, *part_acc;
    uint32_t *status;
    uint32_t *redo;           // fast forms: set to 1 if a score may lie outside the range they are valid for
    int B, H, N, M;
    float sl2;                // scale * log2(e)
    int tiles, splits, blocks;   // ceil(N / 128); CTAs along N; blocks of 128 latents per head
};

// Sixteen columns: weights as packed bf16 (hi, and lo where there are two halves), sums into sum2.  col: per column the addend of the exponent
// (dZ: -lse_dec; masked hi/lo: 0 or -inf) or the factor (masked fast: 1 or 0); read where kCol.  odd: second chunk of a pair (see kPolyPairs).
template <int kKind, bool kCol, bool kOnes>
__device__ __forceinline__ void lean_chunk(const uint32_t *r, uint32_t *pk, uint32_t *pl, float2 sl2p, float2 &sum2, const float *col, bool odd) {
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        float4 cv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (kCol) cv = *reinterpret_cast<const float4 *>(col + 2 * k);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int j = k + e;
            const float2 s = make_float2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
            const float2 c = e ? make_float2(cv.z, cv.w) : make_float2(cv.x, cv.y);
            float2 p;
            if (kKind == kLeanFast) {
                if ((kPolyPairs >> (j + (odd ? 8 : 0))) & 1) {
                    p = exp2_fma_pipe(s, sl2p);
                } else {
                    const float2 x = __fmul2_rn(s, sl2p);
                    p = make_float2(ptx::ex2(x.x), ptx::ex2(x.y));
                }
                if (kCol) p = __fmul2_rn(p, c);
            } else {
                const float2 x = kCol ? __ffma2_rn(s, sl2p, c) : __fmul2_rn(s, sl2p);
                p = make_float2(ptx::ex2(x.x), ptx::ex2(x.y));
            }
            pk[j] = ptx::pack_bf16(p.x, p.y);
            if (kKind == kLeanHiLo) sum2 = __fadd2_rn(sum2, p);
            if (kKind == kLeanFast && !kOnes) sum2 = __fadd2_rn(sum2, make_float2(__uint_as_float(pk[j] << 16), __uint_as_float(pk[j] & 0xffff0000u)));
            if (kKind != kLeanFast) pl[j] = ptx::pack_bf16(ptx::rest_of(p, pk[j]));
        }
    }
}

// Largest squared norm among the rows [lane, lane + 32, ...) < rows of a [rows, DR] bf16 matrix (infinity if one is not finite).
template <int DR>
__device__ __forceinline__ float rows_max_norm2(const __nv_bfloat16 *src, int rows, int lane) {
    float best = 0.f;
    for (int r = lane; r < rows; r += 32) {
        float n2 = 0.f;
#pragma unroll
        for (int c = 0; c < DR; c += 4) {
            const uint2 v = *reinterpret_cast<const uint2 *>(src + (size_t)r * DR + c);
            const float x[4] = {__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u)};
            n2 = fmaf(x[0], x[0], fmaf(x[1], x[1], fmaf(x[2], x[2], fmaf(x[3], x[3], n2))));
        }
        best = fmaxf(best, n2 <= 3.0e38f ? n2 : INFINITY);
    }
    return best;
}

// grid = (heads or head pairs * blocks, splits, B): the heads side by side in a token row are worked on at the same time, so that what one
// leaves of the memory's 64-byte pieces is still in L2 for the next (heads one after the other: encode and the decode after it 3 % slower).
// kPair: at most 64 latents, H even: lanes 0-63 hold the latents of one head, 64-127 those of the next; the A operand is block-diagonal over the
// 2 D columns the two heads occupy side by side in a token row.  DRT = 8 or 4 (with D = 16): the narrow form (see narrow_offset).
// kMask: every unit reads its columns' validity: calls with a key mask and, in the form with two halves (where it costs 1 %, an addend in
// place of a product with 1, and a second body of the loop would spill), with a last partial tile; the fast form handles that in a body
// of its own (validity in every unit costs it 15 %).
template <int D, bool kPair, int kKind, int DRT, bool kMask>
__global__ void __launch_bounds__(LeanGeom<kPair ? 2 * D : D, kKind>::kThreads, 1)
encode_lean_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, EncodeLeanArgs a) {
    constexpr int DG = kPair ? 2 * D : D, DR = DRT ? DRT : D;
    using LG = LeanGeom<DG, kKind>;
    using G = TileGeom<DG>;
    static_assert(!(kPair && DRT), "head pairs are full width");
    static_assert(!(kMask && kKind == kLeanDz), "dZ knows no mask");
    static_assert(kKind != kLeanDz || (!kPair && DRT == 0), "dZ of head pairs and narrow heads is the sweeps'");
    constexpr bool kDz = kKind == kLeanDz, kTwo = kKind != kLeanFast;
    constexpr int UNIT = LG::UNIT, NG = LG::NG, nstages = LG::kStages, kThreads = LG::kThreads;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = ptx::align_1024(smem_raw);
    uint8_t *sQ = smem + LG::q_off;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + LG::bar_off);
    enum { KV_FULL = 0, KV_EMPTY = KV_FULL + nstages, S_FULL = KV_EMPTY + nstages, P_FULL = S_FULL + NG, NBARS = P_FULL + NG };
    static_assert(NBARS * 8 + 12 <= 512, "barrier area too small");
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + NBARS);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    uint32_t *any_valid = tmem_slot + 2;                        // masked two-halves form: a token of this CTA takes part

    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const int M = a.M;
    const int split = blockIdx.y, h = (kPair ? 2 : 1) * (blockIdx.x / a.blocks), lb = blockIdx.x % a.blocks, b = blockIdx.z;
    const int t_begin = (int)((long)a.tiles * split / a.splits), t_end = (int)((long)a.tiles * (split + 1) / a.splits);
    const int nt = t_end - t_begin, nu = 2 * nt;                // tiles, units of this CTA
    const int rows_here = kPair ? M : min(M - lb * kTile, kTile);
    const int off = DRT ? narrow_offset(h, DR) : 0;             // the head's first column within a tile row
    const bool guarded = LG::kGuards > 0 && lb == 0;            // the first block's CTAs check the keys against all of the head's latents
    auto bar = [&](int i) { return ptx::smem_u32(bars + i); };

    if (threadIdx.x == 0) {
        for (int i = 0; i < NBARS; ++i)                         // a tile is released by its two units and its guard
            ptx::mbar_init(bar(i), i >= P_FULL ? 4u : i >= S_FULL ? 1u : i >= KV_EMPTY ? (guarded ? 3u : 2u) : 1u);
        *abort_flag = 0;
        *any_valid = kMask ? 0u : 1u;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmK);
        ptx::prefetch_tensormap(&tmV);
    }
    if (warp == 1) ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
    if (LG::kOnes) {
        uint8_t *ones = smem + LG::ones_off;                    // a one in column 0 of every row
        for (int i = threadIdx.x; i < UNIT * (G::RB / 16); i += kThreads) {
            const int r = i / (G::RB / 16), ch = i % (G::RB / 16);
            *reinterpret_cast<uint4 *>(ones + (size_t)r * G::RB + ((ch ^ G::swz(r)) << 4)) = make_uint4(ch == 0 ? 0x00003F80u : 0u, 0, 0, 0);
        }
    }
    ptx::grid_launch();
    ptx::grid_wait();
    // rows of Q: zeros where there is no latent (or, pair and narrow forms, no feature), then the rows
    if (kPair || DRT != 0 || rows_here < kTile) {
        for (int i = threadIdx.x; i < kTile * (G::RB / 16); i += kThreads) reinterpret_cast<uint4 *>(sQ)[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
    }
#pragma unroll
    for (int w = 0; w < (kPair ? 2 : 1); ++w) {
        const size_t q0 = (size_t)(h + w) * M + lb * kTile;
        if constexpr (DR == 4) stage_rows4<DG>(sQ, a.Q + q0 * DR, rows_here, off);
        else stage_bf16<DG, DR>(sQ, a.Q + q0 * DR, rows_here, 64 * w, w * (D / 8), threadIdx.x, kThreads);
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = *tmem_slot;

    const int g = warp >= LG::kFirstMathWarp ? (warp - LG::kFirstMathWarp) >> 2 : warp - 1;   // of a math or issuing warp: its group
    const int row = ((warp & 3) << 5) + lane;                   // TMEM lane = latent within the block (or within the pair)
    const int second = kPair ? row >> 6 : 0;                    // the head of this lane's latent
    float2 l2 = make_float2(0.f, 0.f);                          // sum of this lane's weights
    const uint32_t base = tm + g * LG::COLS, gcol = base + ((uint32_t)((warp & 3) << 5) << 16);   // the group's columns: scores | accumulator
    bool ok = true;

    if (warp == 0) {
        if (ptx::elect_one()) {
            for (int i = 0; i < nt; ++i) {
                const int s = i % nstages, t = t_begin + i;
                if (!ptx::mbar_wait(bar(KV_EMPTY + s), ((i / nstages) & 1) ^ 1, abort_flag, kErrEncode | 1)) break;
                ptx::mbar_arrive_expect_tx(bar(KV_FULL + s), 2 * G::TILE_BYTES);
                uint8_t *dst = smem + (size_t)s * 2 * G::TILE_BYTES;
                ptx::tma_load_3d(ptx::smem_u32(dst), &tmK, bar(KV_FULL + s), h * DR - off, t * kTile, b);
                ptx::tma_load_3d(ptx::smem_u32(dst + G::TILE_BYTES), &tmV, bar(KV_FULL + s), h * DR - off, t * kTile, b);
            }
        }
    } else if (warp < LG::kFirstGuardWarp) {
        // One issuing thread per group: the values of a unit, the scores of the group's next and one commit, which tells the threads both that
        // those scores are there and that the value contraction (which read the weights that the scores replaced) is done.
        if (g < nu && ptx::elect_one()) {
            const uint32_t pfull = bar(P_FULL + g), sfull = bar(S_FULL + g);
            // (descriptors as 32-bit low words beside a constant high word: see ptx::desc)
            constexpr uint32_t HI = ptx::desc_hi(G::SBO, G::SWZ), STAGE = (2 * G::TILE_BYTES) >> 4, HALF = (UNIT * G::RB) >> 4;
            // the scores of unit u
            auto issue_scores = [&](int u) -> bool {
                constexpr uint32_t idescS = ptx::instr_desc_bf16(128, UNIT, 0, 0);
                const int t = u >> 1, s = t % nstages;
                if (!ptx::mbar_wait(bar(KV_FULL + s), (t / nstages) & 1, abort_flag, kErrEncode | 3)) return false;
                ptx::tc_fence_after();
                uint32_t qd = ptx::desc_lo(ptx::smem_u32(sQ), 16), kd = ptx::desc_lo(ptx::smem_u32(smem), 16) + STAGE * s + HALF * (u & 1);
                ptx::opaque(qd);
                ptx::opaque(kd);
#pragma unroll
                for (int k = 0; k < DG / 16; ++k) ptx::mma_ss(base, ptx::desc(qd + 2 * k, HI), ptx::desc(kd + 2 * k, HI), idescS, k > 0);
                return true;
            };
            // acc += W_unit V_unit: 16 token rows of the V tile per k-step as the MN-major B operand
            auto issue_values = [&](int u) {
                constexpr uint32_t idescV = ptx::instr_desc_bf16(128, LG::kAccCols, 0, 1);
                const uint32_t v0 = ptx::smem_u32(smem + G::TILE_BYTES), at = STAGE * ((u >> 1) % nstages) + HALF * (u & 1);
                // (kOnes: the second block along N starts at the tile of ones, the nearer the further the unit's rows are: LBO, bits 16-29)
                uint32_t vd = ptx::desc_lo(v0, LG::kOnes ? ptx::smem_u32(smem + LG::ones_off) - v0 : (uint32_t)G::SBO) + at - (LG::kOnes ? at << 16 : 0u);
                ptx::opaque(vd);
#pragma unroll
                for (int k = 0; k < UNIT / 16; ++k) {
                    ptx::mma_ts(base + UNIT, base + 16 * k, ptx::desc(vd + k * G::RB, HI), idescV, (u >= NG || k > 0) ? 1u : 0u);
                    if (kTwo) ptx::mma_ts(base + UNIT, base + 16 * k + 8, ptx::desc(vd + k * G::RB, HI), idescV, 1u);
                }
                ptx::mma_commit(bar(KV_EMPTY + (u >> 1) % nstages));
            };
            if (issue_scores(g)) ptx::mma_commit(sfull);
            uint32_t n = 0;
            for (int u = g; u < nu; u += NG, ++n) {
                if (!ptx::mbar_wait(pfull, n & 1, abort_flag, kErrEncode | 4)) break;
                ptx::tc_fence_after();
                issue_values(u);
                if (u + NG < nu && !issue_scores(u + NG)) break;
                ptx::mma_commit(sfull);
            }
        }
    } else if (LG::kGuards > 0 && warp >= LG::kFirstGuardWarp && warp < LG::kFirstMathWarp) {
        if (guarded) {
            // Guard warps, one tile in three each: |q| |k| sl2 <= kFastMaxLog2 for all latents of the CTA's heads and every key row of the
            // tile, checked while the tile sits in its stage.  (Whole rows in the narrow forms: they hold the neighbouring heads'
            // features too, which only makes the check stricter.)
            const float q2 = warp_max_nan(rows_max_norm2<DR>(a.Q + (size_t)h * M * DR, kPair ? 2 * M : M, lane));
            const float lim = kFastMaxLog2 / a.sl2;
            const float k2_limit = lim * lim / fmaxf(q2, 1e-30f);
            bool tame = q2 <= 3.0e38f;                          // (NaN or infinity in Q)
            for (int j = warp - LG::kFirstGuardWarp; j < nt; j += LG::kGuards) {
                const int sj = j % nstages;
                if (!warp_wait(bar(KV_FULL + sj), (j / nstages) & 1, abort_flag, kErrEncode | 9)) break;
                const float k2 = warp_max_nan(tile_max_norm2<G::RB, kPair ? 2 : 1>(smem + (size_t)sj * 2 * G::TILE_BYTES, kTile, lane));
                if (!(k2 <= k2_limit)) tame = false;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(KV_EMPTY + sj));
            }
            if (!tame && lane == 0) *a.redo = 1u;
        }
    } else if (kDz && warp < LG::kFirstMathWarp) {
        if (split == 0) {
            for (int w = 0; w < (kPair ? 2 : 1); ++w) {
                const size_t bh = (size_t)b * a.H + h + w;
                z_around<DR>(a.around + bh * (1 + a.blocks) * DR, a.Z + bh * M * DR, M, lb);
            }
        }
    } else if (warp >= LG::kFirstMathWarp) {
        const float2 sl2p = make_float2(a.sl2, a.sl2);
        const uint32_t pfull = bar(P_FULL + g), sfull = bar(S_FULL + g);
        float *col = reinterpret_cast<float *>(smem + LG::col_off) + (warp - LG::kFirstMathWarp) * UNIT;   // this warp's column constants
        // constants of this lane's columns (lane, 32 + lane) of unit u, fetched one unit ahead
        float next[2];
        bool some = false;                                      // masked: a token of this lane takes part
        auto fetch = [&](int u) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int n = t_begin * kTile + u * UNIT + e * 32 + lane;
                if (kDz) {
                    next[e] = n < a.N ? a.lse_dec[((size_t)b * a.N + n) * a.H + h + second] : INFINITY;
                } else {
                    const bool valid = n < a.N && (!kMask || a.key_mask == nullptr || a.key_mask[(size_t)b * a.N + n] != 0);
                    some = some || valid;
                    next[e] = kKind == kLeanHiLo ? (valid ? 0.f : -INFINITY) : (valid ? 1.f : 0.f);
                }
            }
        };
        uint32_t n = 0;                                         // units waited for
        auto unit = [&](auto with_col, int u) -> bool {
            constexpr bool kCol = decltype(with_col)::value;
            if (kCol) {
                if (!kDz && !kMask) fetch(u);
                __syncwarp();                                   // the previous unit's reads are done
                col[lane] = kDz ? next[0] * -1.4426950408889634f : next[0];
                col[32 + lane] = kDz ? next[1] * -1.4426950408889634f : next[1];
                __syncwarp();
                if ((kDz || kMask) && u + NG < nu) fetch(u + NG);
            }
            if (!warp_wait(sfull, n & 1, abort_flag, kErrEncode | 5)) return false;
            ptx::tc_fence_after();
            uint32_t r[2][16];
            ptx::tmem_ld16(gcol, r[0]);
#pragma unroll
            for (int q = 0; q < UNIT / 16; ++q) {               // 16 columns at a time, the next 16 on their way meanwhile
                ptx::tmem_wait_ld();
                if (q + 1 < UNIT / 16) ptx::tmem_ld16(gcol + 16 * (q + 1), r[(q + 1) & 1]);
                uint32_t pk[8], pl[8];
                lean_chunk<kKind, kCol, LG::kOnes>(r[q & 1], pk, pl, sl2p, l2, col + 16 * q, q & 1);
                ptx::tmem_st8(gcol + 16 * q, pk);               // over columns this thread has read
                if (kTwo) ptx::tmem_st8(gcol + 16 * q + 8, pl);
            }
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(pfull);
            ++n;
            return true;
        };
        if ((kDz || kMask) && g < nu) fetch(g);
        const int tail = a.N % kTile != 0 ? 2 * (a.tiles - 1 - t_begin) : nu;   // first unit of a last partial tile
        for (int u = g; ok && u < nu; u += NG) {
            if (kDz || kMask) ok = unit(std::true_type{}, u);
            else if (kKind == kLeanHiLo) ok = unit(std::false_type{}, u);
            else ok = u >= tail ? unit(std::true_type{}, u) : unit(std::false_type{}, u);
        }
        if (ok && n > 0) ok = warp_wait(sfull, n & 1, abort_flag, kErrEncode | 6);
        ptx::tc_fence_after();
        if (kMask && __any_sync(0xffffffffu, some) && lane == 0) *any_valid = 1u;
    }
    // The groups' sums, over the ring: every copy has landed and been used.  Rows of D + 1 floats: D sums, the sum of the weights.
    __syncthreads();
    constexpr int RW = D + 1;
    static_assert((size_t)NG * kTile * RW * sizeof(float) <= LG::bar_off, "the groups' sums fit over the ring");
    float *red = reinterpret_cast<float *>(smem);
    if (warp >= LG::kFirstMathWarp) {
        float *mine = red + ((size_t)g * kTile + row) * RW;
        if (g < nu) {
#pragma unroll
            for (int c0 = 0; c0 < D; c0 += 8) {
                uint32_t x[8];
                ptx::tmem_ld8(gcol + UNIT + second * D + c0, x);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < 8; ++k) mine[c0 + k] = __uint_as_float(x[k]);
            }
            if (LG::kOnes) {
                uint32_t x[8];
                ptx::tmem_ld8(gcol + UNIT + DG, x);
                ptx::tmem_wait_ld();
                l2 = make_float2(__uint_as_float(x[0]), 0.f);
            }
            mine[D] = l2.x + l2.y;
        } else {
#pragma unroll
            for (int k = 0; k <= D; ++k) mine[k] = 0.f;
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    {
        const long rows = (long)a.B * a.H * M;
        constexpr int PIECES = DR / 4 + 1;                      // of a row: 16-byte pieces, and the sum of the weights
        for (int i = threadIdx.x; i < kTile * PIECES; i += kThreads) {
            const int r = i / PIECES, c = i % PIECES, w = kPair ? r >> 6 : 0, m = kPair ? (r & 63) : lb * kTile + r;
            if (m >= M || (kDz && c == PIECES - 1)) continue;
            const size_t prow = (size_t)split * rows + ((size_t)b * a.H + h + w) * M + m;
            const float *src = red + (size_t)r * RW + (c == PIECES - 1 ? D : off + 4 * c);
            float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int gg = 0; gg < NG; ++gg)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k == 0 || c < PIECES - 1) v[k] += src[(size_t)gg * kTile * RW + k];
            if (c < PIECES - 1) {
                *reinterpret_cast<float4 *>(a.part_acc + prow * DR + 4 * c) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
                // Weights are relative to 2^0.  A sum of exactly 0 is that of no valid token: certain where the norms were checked; the form
                // with two halves takes its exponentials from the special-function unit alone, which saturates at either end, so
                // the sums show all there is to check and it has no guard, but a 0 may then be a row of weights below 2^-126.
                const bool empty = v[0] == 0.f && (kKind == kLeanFast || *any_valid == 0u);
                a.part_m[prow] = v[0] > 0.f ? 0.f : -INFINITY;
                a.part_l[prow] = v[0];
                if (!(empty || (v[0] >= kFastSumMin && v[0] <= kFastSumMax))) *a.redo = 1u;
            }
        }
    }
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tm, 512);
    }
    if (threadIdx.x == 0 && *abort_flag != 0 && a.status != nullptr) atomicCAS(a.status, 0u, *abort_flag);
}

}  // namespace flare
