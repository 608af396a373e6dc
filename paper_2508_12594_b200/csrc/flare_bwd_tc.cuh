// Tensor-core kernels of the backward for bfloat16 inputs on sm_100a (pass B: the gradients of the latent queries, keys and
// values).
//
// dQ_m = scale * sum_n dS[m,n] k_n,   dK_n = scale * sum_m dS[m,n] q_m,   dV_n = sum_m W_enc[m,n] dZ_m   with
//   dS[m,n] = W_dec[n,m] (dY_n . Z_m - dd[n]) + W_enc[m,n] (dZ_m . V_n - de[m]),
//   W_dec[n,m] = exp(S[m,n] - lse_dec[n]),  W_enc[m,n] = valid(n) exp(S[m,n] - lse_enc[m]),  S = scale * q_m . k_n.
//
// Both kernels turn three tiles that the tensor core puts side by side in tensor memory, S = q.k, A = dY.Z and C = dZ.V, into
// dS (and W_enc) over the columns just read, which feed the output contractions as their A operand.  One kind of row sits
// on the 128 lanes (latents in the dQ kernel, tokens in the token kernel), the other on the columns, in units of 64 or 32.
// Z and dZ, and dS and W_enc, enter as two bf16 halves each, because the sums cancel; for dQ at D = 64 Z, dZ and dS as three.
//
// What shapes them.  A tcgen05.mma with both operands in shared memory takes the tensor core 40 cycles at N = 16 or 32, 48 at 64 and 64
// at 128 (most of it the fetch of its A operand), one with A in tensor memory N / 2; a hand-over between threads and tensor core
// costs a warp some 100 instructions and a round trip of about 1000 cycles.  Units of 16 columns (dQ kernel at D = 32: ten MMAs of N = 16 for
// 16 tokens) ran at exactly the tensor limit.  Wider units are shared by all warps, which served better than
// groups of four warps with units of their own in both kernels.  They run for heads 64 wide, and 32 wide where the two sweeps do not (use_sweeps).
#pragma once

#include "flare_tc.cuh"

namespace flare {

// dS of a pair of columns as packed bf16 halves hi, lo, for the dQ kernel.  xd = s * sl2 + nd is the decode exponent
// (log2 units), u = A + na, v = C + nc.  Both weights come from one exponential: with K the smallest lse_enc of the CTA's latents
// (log2 units),
//     W_enc = W_dec 2^(lse_dec[n] - K) 2^(K - lse_enc[m]),    fr, fc the two factors (fc 0 for a token that takes no part),
// exact to float32 rounding wherever it matters as long as lse_dec[n] - K <= kOneExpLog2: the second factor is at most 1, so what
// underflows on the way (W_dec below 2^-126, a factor below 2^-126) is a weight below 2^(kOneExpLog2 - 126).  Tokens beyond that
// bound (or with an infinite lse_dec, how the two-query variant switches a stage off) take the form with an exponential of its own for
// W_enc, kTwo: xe = s * sl2 + ne.  (An exponential costs the special-function unit as much as the rest of a pair costs the
// issue slots: with two per pair the unit bound both kernels.)
constexpr float kOneExpLog2 = 40.f;
// kThird: dS in three parts (24 bits: all of the float32 value).
struct DsPair { uint32_t hi, lo, lo2; };
template <bool kTwo, bool kThird>
__device__ __forceinline__ DsPair ds_pair(float2 s, float2 av, float2 cv, float2 sl2p, float2 nd, float2 na, float2 nc, float2 fr_ne, float2 fc) {
    const float2 xd = __ffma2_rn(s, sl2p, nd);
    const float2 pd = make_float2(ptx::ex2(xd.x), ptx::ex2(xd.y));
    const float2 u = __fadd2_rn(av, na), v = __fadd2_rn(cv, nc);
    float2 ds;
    if (kTwo) {                                                  // fr_ne: -lse_enc[m]; fc: 0, or -inf for a token that takes no part
        const float2 xe = __ffma2_rn(s, sl2p, __fadd2_rn(fr_ne, fc));
        ds = __ffma2_rn(pd, u, __fmul2_rn(make_float2(ptx::ex2(xe.x), ptx::ex2(xe.y)), v));
    } else {
        ds = __fmul2_rn(pd, __ffma2_rn(__fmul2_rn(fr_ne, fc), v, u));
    }
    DsPair o;
    o.hi = ptx::pack_bf16(ds);
    const float2 rest = ptx::rest_of(ds, o.hi);
    o.lo = ptx::pack_bf16(rest);
    if (kThird) o.lo2 = ptx::pack_bf16(ptx::rest_of(rest, o.lo));
    return o;
}
constexpr float kBwdLog2e = 1.4426950408889634f;
// Smallest lse_enc (log2 units) of `rows` latents, leaving out those that saw no valid token (-inf); 0 if there is none.  By a full warp.
__device__ __forceinline__ float warp_lse_min(const float *lse_enc, int rows) {
    float k = INFINITY;
    for (int m = threadIdx.x & 31; m < rows; m += 32) {
        const float le = lse_enc[m];
        if (le != -INFINITY) k = fminf(k, le * kBwdLog2e);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k = fminf(k, __shfl_xor_sync(0xffffffffu, k, o));
    return k <= 3.0e38f ? k : 0.f;
}

// rows of a [rows, DR] float matrix -> bf16 halves (kThird: three parts, the third in lo2) in swizzled rows (DR >= 8), starting at
// logical chunk `chunk0` of row r0 + m; each less `centre` (null: nothing), row m times factor(m)
template <int DG, int DR, bool kThird = false, class Factor = UnitFactor>
__device__ __forceinline__ void stage_hilo(uint8_t *hi, uint8_t *lo, const float *src, int rows, int r0, int chunk0, int tid, int threads,
                                           const float *centre = nullptr, Factor factor = Factor(), uint8_t *lo2 = nullptr) {
    using G = TileGeom<DG>;
    constexpr int ZC = DR >= 8 ? DR / 8 : 1;
    for (int i = tid; i < rows * ZC; i += threads) {
        const int m = i / ZC, c = i % ZC, r = r0 + m;
        const float4 a = *reinterpret_cast<const float4 *>(src + (size_t)m * DR + c * 8);
        const float4 b = *reinterpret_cast<const float4 *>(src + (size_t)m * DR + c * 8 + 4);
        float4 ca = make_float4(0.f, 0.f, 0.f, 0.f), cb = ca;
        if (centre != nullptr) {
            ca = *reinterpret_cast<const float4 *>(centre + c * 8);
            cb = *reinterpret_cast<const float4 *>(centre + c * 8 + 4);
        }
        const float f = factor(m);
        const float z[8] = {(a.x - ca.x) * f, (a.y - ca.y) * f, (a.z - ca.z) * f, (a.w - ca.w) * f,
                            (b.x - cb.x) * f, (b.y - cb.y) * f, (b.z - cb.z) * f, (b.w - cb.w) * f};
        uint32_t vh[4], vl[4], vl2[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            vh[k] = ptx::pack_bf16(z[2 * k], z[2 * k + 1]);
            const float x = z[2 * k] - __uint_as_float(vh[k] << 16), y = z[2 * k + 1] - __uint_as_float(vh[k] & 0xffff0000u);
            vl[k] = ptx::pack_bf16(x, y);
            if (kThird) vl2[k] = ptx::pack_bf16(x - __uint_as_float(vl[k] << 16), y - __uint_as_float(vl[k] & 0xffff0000u));
        }
        const size_t o = (size_t)r * G::RB + (((chunk0 + c) ^ G::swz(r)) << 4);
        *reinterpret_cast<uint4 *>(hi + o) = make_uint4(vh[0], vh[1], vh[2], vh[3]);
        *reinterpret_cast<uint4 *>(lo + o) = make_uint4(vl[0], vl[1], vl[2], vl[3]);
        if (kThird) *reinterpret_cast<uint4 *>(lo2 + o) = make_uint4(vl2[0], vl2[1], vl2[2], vl2[3]);
    }
}
// ------------------------------------------------------------------------------- pass B, latent side (dQ)

// Units of 64 tokens, shared by sixteen warps, 16 columns each, on two alternating buffers of tensor memory (S | A | C; then the
// accumulators): while the threads work on one unit the tensor core runs the output contractions of the other and the tiles of the one after.
// Warps: 0 TMA producer, 1 MMA issue, 3 column constants, 4-19 arithmetic (warp & 3 = the quarter of the lanes it can reach).
// Measured, us, against units of 16 columns with two exponentials per pair: 131072 tokens, M = 512, D = 32, 8 heads 437 -> 392; D = 64 (2 x 20011, M = 128, 4
// heads), on the CUDA cores before, 498 -> 27 (in three parts, see kThird, 31).  Groups of four warps with units and buffers of their own: 522; 44.  Issue
// slots and the latency of tensor-memory loads share the bound (some 14 instructions per pair, two issued per cycle and SM).
constexpr int kDqUnit = 64, kDqBuf = 3 * kDqUnit, kDqAcc = 2 * kDqBuf;
constexpr int kDqThreads = 640, kDqFirstMathWarp = 4;

struct BwdDqTcArgs {
    const __nv_bfloat16 *Q;    // [H,M,D]
    const float *Z, *dZ;       // [B,H,M,D]
    const float *lse_enc, *de; // [B,H,M]
    const float *lse_dec;      // [B,N,H]
    const float *dd;           // [B,H,N] (workspace)
    const float *around;       // (workspace) a centre of the rows of Z at the head of each head's rows, see z_around
    int around_rows;
    const uint8_t *key_mask;   // [B,N] or null
    float *part;               // [P][B*H*M][D] partial dQ rows (un-scaled)
    uint32_t *status;
    int B, H, N, M;
    float sl2;                 // scale * log2(e)
    int tiles, splits, blocks; // blocks: of 128 latents per head
};

template <int D>
struct BwdDqSmem {
    using G = TileGeom<D>;
    static constexpr int kParts = D == 64 ? 3 : 2, kLat = 1 + 2 * kParts;   // parts of Z and dZ (see the kernel); with Q, latent operands
    static constexpr int kCst = 8, kAhead = 4;                                   // tiles of column constants in the ring, of them on their way
    static constexpr size_t kCstBytes = (size_t)3 * kTile * sizeof(float);     // -lse_dec, -dd, mask
    static constexpr size_t total_for(int n) {
        return (size_t)n * 3 * G::TILE_BYTES + (size_t)kLat * kTile * G::RB + kCst * kCstBytes + 768 + 1024;
    }
    static constexpr int stages_for() {
        int n = 6;
        while (n > 1 && total_for(n) > 227 * 1024) --n;
        return n;
    }
    static constexpr int kStages = stages_for();                                 // (K, V, dY) tile triples in flight
    __host__ __device__ static constexpr size_t lat_off(int which) { return (size_t)kStages * 3 * G::TILE_BYTES + (size_t)which * kTile * G::RB; }
    static constexpr size_t cst_off = lat_off(kLat);
    static constexpr size_t bar_off = cst_off + kCst * kCstBytes;
    static constexpr size_t total = total_for(kStages) < kTcMinSmem ? kTcMinSmem : total_for(kStages);
};

// grid = (heads * blocks, splits, B): heads that share token rows run at the same time; a CTA takes one block of 128 latents and a contiguous range of token tiles.
// kPadded: the launch has padded tokens (a key mask, or N not a multiple of the tile): a third constant per column, 0 or -inf.
template <int D, bool kPadded>
__global__ void __launch_bounds__(kDqThreads, 1)
bwd_dq_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                 const __grid_constant__ CUtensorMap tmG, BwdDqTcArgs a) {
    using G = TileGeom<D>;
    using SM = BwdDqSmem<D>;
    // The units take turns on as many accumulators as there is room for: the tensor core truncates each of the thousands of sums that a
    // split adds up in float32, an error that grows with their number.
    constexpr int kAccs = (512 - kDqAcc) / D;
    // D = 64: the three products carry all 24 bits of Z, dZ and dS, in three parts each, and a unit's sums go to float32 sums in registers
    // two units later, when their accumulator is free again: 16 of the 64 columns to each of the four warps that share a quarter of the lanes.
    // (This width used to run in float32 arithmetic on the CUDA cores, twenty times slower.  In halves, summed in tensor memory, as the
    // other widths are, dQ was 1.5 to 2.3 times as far from float64 as there; now 0.5 to 1.04 times, what is left being the weights in halves
    // that Z and dZ were formed with.  2 x 20011 tokens, M = 128, 4 heads, relative to the norm, float32 / halves / parts: 2.6e-6 / 4.9e-6 /
    // 2.6e-6, on features of point clouds 5.1e-6 / 7.2e-6 / 2.9e-6.  That training step: 182 us in halves, 186 with this, 192 with
    // the token kernel's third part.)
    constexpr bool kThird = SM::kParts == 3;
    static_assert(!kThird || (kAccs == 2 && D == 64), "a warp's columns, and the buffer's accumulator");
    static_assert(kAccs >= 1 && (kAccs & (kAccs - 1)) == 0, "tensor memory");
    constexpr int UNIT = kDqUnit, UPT = kTile / UNIT, nstages = SM::kStages;
    static_assert(nstages >= 2, "one tile is finished while the next begins");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = ptx::align_1024(smem_raw);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + SM::bar_off);
    enum { T_FULL = 0, T_EMPTY = T_FULL + nstages, C_FULL = T_EMPTY + nstages, C_EMPTY = C_FULL + SM::kCst, S_FULL = C_EMPTY + SM::kCst,
           P_FULL = S_FULL + 2, ACC_DONE = P_FULL + 2, NBARS = ACC_DONE + 1 };
    static_assert(NBARS * 8 + 16 + 8 * SM::kCst <= 768, "barrier area too small");
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + NBARS);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const int M = a.M;
    const int split = blockIdx.y, h = blockIdx.x / a.blocks, lb = blockIdx.x % a.blocks, b = blockIdx.z;
    const int t_begin = (int)((long)a.tiles * split / a.splits), t_end = (int)((long)a.tiles * (split + 1) / a.splits);
    const int nt = t_end - t_begin;
    const int rows_here = min(M - lb * kTile, kTile);
    auto bar = [&](int i) { return ptx::smem_u32(bars + i); };

    if (threadIdx.x == 0) {
        for (int i = 0; i < NBARS; ++i)
            ptx::mbar_init(bar(i), (i >= P_FULL && i < P_FULL + 2) || (i >= C_EMPTY && i < C_EMPTY + SM::kCst) ? 16u : 1u);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmK);
        ptx::prefetch_tensormap(&tmV);
        ptx::prefetch_tensormap(&tmG);
    }
    float *kmin = reinterpret_cast<float *>(tmem_slot + 2);     // smallest lse_enc
    volatile uint32_t *two_exp = tmem_slot + 4;                 // [kCst]: the tile needs an exponential of its own for W_enc
    if (warp == 1) ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
    ptx::grid_launch();
    ptx::grid_wait();
    if (warp == 3) {
        const float k = warp_lse_min(a.lse_enc + ((size_t)b * a.H + h) * M + lb * kTile, rows_here);
        if (lane == 0) *kmin = k;
    }
    // latent operands Q, Z_hi, Z_lo, dZ_hi, dZ_lo (D = 64: three parts of Z and dZ): zeros where there is no row, then the rows
    const float *centre = a.around + ((size_t)b * a.H + h) * a.around_rows * D;
    if (rows_here < kTile) {
        for (int i = threadIdx.x; i < SM::kLat * kTile * (G::RB / 16); i += kDqThreads)
            reinterpret_cast<uint4 *>(smem + SM::lat_off(0))[i] = make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    {
        const size_t q0 = (size_t)h * M + lb * kTile, r0 = ((size_t)b * a.H + h) * M + lb * kTile;
        constexpr int dz0 = 1 + SM::kParts;
        stage_bf16<D, D>(smem + SM::lat_off(0), a.Q + q0 * D, rows_here, 0, 0, threadIdx.x, kDqThreads);
        stage_hilo<D, D, kThird>(smem + SM::lat_off(1), smem + SM::lat_off(2), a.Z + r0 * D, rows_here, 0, 0, threadIdx.x, kDqThreads, centre, UnitFactor(),
                                 smem + SM::lat_off(3));
        stage_hilo<D, D, kThird>(smem + SM::lat_off(dz0), smem + SM::lat_off(dz0 + 1), a.dZ + r0 * D, rows_here, 0, 0, threadIdx.x, kDqThreads, nullptr,
                                 UnitFactor(), smem + SM::lat_off(SM::kLat - 1));
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = *tmem_slot;
    const float lse_min = *kmin;

    if (warp == 0) {
        if (ptx::elect_one()) {
            for (int i = 0; i < nt; ++i) {
                const int s = i % nstages;
                if (!ptx::mbar_wait(bar(T_EMPTY + s), ((i / nstages) & 1) ^ 1, abort_flag, kErrBwdDq | 1)) break;
                ptx::mbar_arrive_expect_tx(bar(T_FULL + s), 3 * G::TILE_BYTES);
                uint8_t *dst = smem + (size_t)s * 3 * G::TILE_BYTES;
                ptx::tma_load_3d(ptx::smem_u32(dst), &tmK, bar(T_FULL + s), h * D, (t_begin + i) * kTile, b);
                ptx::tma_load_3d(ptx::smem_u32(dst + G::TILE_BYTES), &tmV, bar(T_FULL + s), h * D, (t_begin + i) * kTile, b);
                ptx::tma_load_3d(ptx::smem_u32(dst + 2 * G::TILE_BYTES), &tmG, bar(T_FULL + s), h * D, (t_begin + i) * kTile, b);
            }
        }
    } else if (warp == 3) {
        // Column constants of every tile: -lse_dec, -dd, and the factor 2^(lse_dec - K) of W_enc (0 for a token that takes no part), or,
        // in a tile with a token beyond kOneExpLog2, the addend of its own exponent.  The values come by asynchronous copies, kAhead
        // tiles on their way at a time (with one tile's loads in flight this warp held the whole kernel back), and are
        // turned into constants in place.
        constexpr int AH = SM::kAhead;
        uint32_t masks[AH];                                     // mask bytes of this lane's four tokens
        auto fetch = [&](int i) -> uint32_t {
            float *cst = reinterpret_cast<float *>(smem + SM::cst_off + (i % SM::kCst) * SM::kCstBytes);
            uint32_t mk = 0x01010101u;
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) {
                const int r = e * 32 + lane, n = min((t_begin + i) * kTile + r, a.N - 1);
                const size_t nn = (size_t)b * a.N + n;
                ptx::copy_async4(ptx::smem_u32(cst + r), a.lse_dec + nn * a.H + h);
                ptx::copy_async4(ptx::smem_u32(cst + kTile + r), a.dd + ((size_t)b * a.H + h) * a.N + n);
                if (kPadded && a.key_mask != nullptr && a.key_mask[nn] == 0) mk &= ~(0xffu << (8 * e));
            }
            return mk;
        };
        bool ok = true;
#pragma unroll
        for (int k = 0; k < AH; ++k) {
            masks[k] = k < nt ? fetch(k) : 0u;
            ptx::copy_async_commit();
        }
        for (int i0 = 0; ok && i0 < nt; i0 += AH) {
#pragma unroll
            for (int k = 0; k < AH; ++k) {
                const int i = i0 + k;
                if (i >= nt) break;
                ptx::copy_async_wait<AH - 1>();
                __syncwarp();
                const int c = i % SM::kCst;
                float *cst = reinterpret_cast<float *>(smem + SM::cst_off + c * SM::kCstBytes);
                float ld[kTile / 32];
                bool part[kTile / 32], far = false;
#pragma unroll
                for (int e = 0; e < kTile / 32; ++e) {
                    const int r = e * 32 + lane;
                    const bool in = (t_begin + i) * kTile + r < a.N;
                    ld[e] = in ? cst[r] * kBwdLog2e : INFINITY;
                    part[e] = in && ((masks[k] >> (8 * e)) & 0xffu) != 0;
                    cst[r] = -ld[e];
                    cst[kTile + r] = in ? -cst[kTile + r] : 0.f;
                    far = far || (part[e] && !(ld[e] - lse_min <= kOneExpLog2));
                }
                far = __any_sync(0xffffffffu, far);
#pragma unroll
                for (int e = 0; e < kTile / 32; ++e)
                    cst[2 * kTile + e * 32 + lane] = far ? (part[e] ? 0.f : -INFINITY) : (part[e] ? ptx::ex2(ld[e] - lse_min) : 0.f);
                if (lane == 0) two_exp[c] = far ? 1u : 0u;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar(C_FULL + c));
                const int next = i + AH;
                if (next < nt) {
                    if (!(ok = warp_wait(bar(C_EMPTY + next % SM::kCst), ((next / SM::kCst) & 1) ^ 1, abort_flag, kErrBwdDq | 7))) break;
                    masks[k] = fetch(next);
                }
                ptx::copy_async_commit();
            }
        }
        ptx::copy_async_wait<0>();
    } else if (warp == 1) {
        const int units = UPT * nt;
        if (ptx::elect_one()) {
            constexpr uint32_t idescS = ptx::instr_desc_bf16(128, UNIT, 0, 0), idescQ = ptx::instr_desc_bf16(128, D, 0, 1);
            // (descriptors as 32-bit low words beside a constant high word: see ptx::desc)
            constexpr uint32_t HI = ptx::desc_hi(G::SBO, G::SWZ), TILE = G::TILE_BYTES >> 4, STEP16 = (16 * G::RB) >> 4, LAT = (kTile * G::RB) >> 4;
            const uint32_t lat0 = ptx::desc_lo(ptx::smem_u32(smem + SM::lat_off(0)), 16), k0 = ptx::desc_lo(ptx::smem_u32(smem), 16);
            constexpr uint32_t MN = ptx::desc_lo(0, G::SBO) - ptx::desc_lo(0, 16);          // K-major to MN-major
            int s_stage = 0, s_wrap = 0, s_u = 0, o_stage = 0, o_u = 0;
            // S = Q K^T | A = (Z_hi + Z_lo) dY^T | C = (dZ_hi + dZ_lo) V^T of the next unit, into buffer n & 1 (D = 64: three parts)
            auto tiles = [&](int n) -> bool {
                if (s_u == 0) {
                    if (!ptx::mbar_wait(bar(T_FULL + s_stage), (uint32_t)s_wrap, abort_flag, kErrBwdDq | 3)) return false;
                    ptx::tc_fence_after();
                }
                uint32_t kd = k0 + (uint32_t)s_stage * 3 * TILE + (uint32_t)s_u * (UNIT / 16) * STEP16, ld = lat0;
                ptx::opaque(kd);
                ptx::opaque(ld);
                const uint32_t bcol = tm + (n & 1) * kDqBuf;
#pragma unroll
                for (int i = 0; i < SM::kLat; ++i) {            // Q with K; the parts of Z with dY; those of dZ with V
                    const int of = i == 0 ? 0 : i <= SM::kParts ? 1 : 2, at = of == 0 ? 0 : (i - 1) % SM::kParts;
                    const int w = of == 0 ? 0 : 1 + (of - 1) * SM::kParts + (kThird ? SM::kParts - 1 - at : at);   // (kThird: small parts first)
                    const uint32_t col = bcol + of * UNIT, td = kd + (of == 0 ? 0 : of == 1 ? 2 * TILE : TILE);
                    const bool more = at > 0;                   // adds to an earlier part's product
#pragma unroll
                    for (int k = 0; k < D / 16; ++k)
                        ptx::mma_ss(col, ptx::desc(ld + w * LAT + 2 * k, HI), ptx::desc(td + 2 * k, HI), idescS, k > 0 || more);
                }
                ptx::mma_commit(bar(S_FULL + (n & 1)));
                if (++s_u == UPT) {
                    s_u = 0;
                    if (++s_stage == nstages) { s_stage = 0; s_wrap ^= 1; }
                }
                return true;
            };
            bool ok = true;
            for (int n = 0; ok && n < 2 && n < units; ++n) ok = tiles(n);
            for (int n = 0; ok && n < units; ++n) {
                // dQ_part += dS_unit K_unit (the parts of dS in turn): 16 token rows of the K tile per k-step as the MN-major B operand
                const uint32_t bcol = tm + (n & 1) * kDqBuf, acc = tm + kDqAcc + (n & (kAccs - 1)) * D;
                uint32_t kd = k0 + MN + (uint32_t)o_stage * 3 * TILE + (uint32_t)o_u * (UNIT / 16) * STEP16;
                ptx::opaque(kd);
                if (!ptx::mbar_wait(bar(P_FULL + (n & 1)), (n >> 1) & 1, abort_flag, kErrBwdDq | 4)) break;
                ptx::tc_fence_after();
                if constexpr (kThird) {                         // the small parts first: fewer sums are truncated at their full size
#pragma unroll
                    for (int i = 2; i >= 0; --i)
#pragma unroll
                        for (int k = 0; k < UNIT / 16; ++k)
                            ptx::mma_ts(acc, bcol + i * UNIT + 16 * k, ptx::desc(kd + k * STEP16, HI), idescQ, (i < 2 || k > 0) ? 1u : 0u);
                } else {
#pragma unroll
                    for (int k = 0; k < UNIT / 16; ++k) {
                        ptx::mma_ts(acc, bcol + 16 * k, ptx::desc(kd + k * STEP16, HI), idescQ, (n >= kAccs || k > 0) ? 1u : 0u);
                        ptx::mma_ts(acc, bcol + UNIT + 16 * k, ptx::desc(kd + k * STEP16, HI), idescQ, 1u);
                    }
                }
                if (++o_u == UPT) {
                    ptx::mma_commit(bar(T_EMPTY + o_stage));
                    o_u = 0;
                    if (++o_stage == nstages) o_stage = 0;
                }
                if (n + 2 < units) ok = tiles(n + 2);
            }
            if (ok) ptx::mma_commit(bar(ACC_DONE));
        }
    } else if (warp >= kDqFirstMathWarp) {
        const int cg = (warp - kDqFirstMathWarp) >> 2;         // the group of 16 columns this warp works on
        const int row = ((warp & 3) << 5) + lane;               // TMEM lane = latent within the block
        const uint32_t gcol = tm + ((uint32_t)((warp & 3) << 5) << 16);
        const float2 sl2p = make_float2(a.sl2, a.sl2);
        const int m = lb * kTile + row;
        // this thread's latent: -lse_enc in log2 units (-inf for a latent that saw no valid token or lies beyond M), -de
        float nle = -INFINITY, nde = 0.f;
        if (m < M) {
            const size_t r = ((size_t)b * a.H + h) * M + m;
            const float le = a.lse_enc[r];
            nle = (le == -INFINITY) ? -INFINITY : -le * kBwdLog2e;
            nde = -a.de[r];
        }
        const float fr = ptx::ex2(nle + lse_min);       // 2^(K - lse_enc)
        const float2 nlep = make_float2(nle, nle), frp = make_float2(fr, fr), ndep = make_float2(nde, nde);
        bool ok = true;
        int n = 0;
        float sum[kThird ? 16 : 1] = {};                        // (kThird) this warp's columns of the sums so far
        // (kThird) the sums of unit i, complete when the tiles of unit i + 2 are
        auto drain = [&](int i) {
            uint32_t r[16];
            ptx::tmem_ld16(gcol + kDqAcc + (i & 1) * D + cg * 16, r);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 16; ++k) sum[kThird ? k : 0] += __uint_as_float(r[k]);
        };
        for (int tile = 0; ok && tile < nt; ++tile) {
            const int c = tile % SM::kCst;
            const float *cst = reinterpret_cast<const float *>(smem + SM::cst_off + c * SM::kCstBytes) + cg * 16;
            if (!(ok = warp_wait(bar(C_FULL + c), (tile / SM::kCst) & 1, abort_flag, kErrBwdDq | 8))) break;
            auto units = [&](auto two) {
                constexpr bool kTwo = decltype(two)::value;
#pragma unroll 1
                for (int u = 0; u < UPT; ++u, ++n, cst += UNIT) {
                    const uint32_t bcol = gcol + (n & 1) * kDqBuf + cg * 16;
                    if (!(ok = warp_wait(bar(S_FULL + (n & 1)), (n >> 1) & 1, abort_flag, kErrBwdDq | 5))) break;
                    ptx::tc_fence_after();
                    uint32_t s[2][8], av[2][8], cv[2][8];
                    auto load = [&](int q) {
                        ptx::tmem_ld8(bcol + q * 8, s[q]);
                        ptx::tmem_ld8(bcol + UNIT + q * 8, av[q]);
                        ptx::tmem_ld8(bcol + 2 * UNIT + q * 8, cv[q]);
                    };
                    load(0);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {                  // eight columns at a time, the other eight on their way meanwhile
                        ptx::tmem_wait_ld();
                        if (q == 0) load(1);
                        uint32_t hi[4], lo[4], lo2[4];
#pragma unroll
                        for (int k = 0; k < 4; k += 2) {
                            const float4 nld = *reinterpret_cast<const float4 *>(cst + q * 8 + 2 * k);
                            const float4 ndd = *reinterpret_cast<const float4 *>(cst + kTile + q * 8 + 2 * k);
                            const float4 fc = *reinterpret_cast<const float4 *>(cst + 2 * kTile + q * 8 + 2 * k);
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const int j = 2 * (k + e);
                                const DsPair r = ds_pair<kTwo, kThird>(
                                    make_float2(__uint_as_float(s[q][j]), __uint_as_float(s[q][j + 1])),
                                    make_float2(__uint_as_float(av[q][j]), __uint_as_float(av[q][j + 1])),
                                    make_float2(__uint_as_float(cv[q][j]), __uint_as_float(cv[q][j + 1])), sl2p,
                                    e ? make_float2(nld.z, nld.w) : make_float2(nld.x, nld.y), e ? make_float2(ndd.z, ndd.w) : make_float2(ndd.x, ndd.y),
                                    ndep, kTwo ? nlep : frp, e ? make_float2(fc.z, fc.w) : make_float2(fc.x, fc.y));
                                hi[k + e] = r.hi;
                                lo[k + e] = r.lo;
                                if (kThird) lo2[k + e] = r.lo2;
                            }
                        }
                        // over columns this warp has read, 8 packed columns per 16 tokens: hi over S, lo over A, a third part over C
                        ptx::tmem_st4(bcol + q * 4, hi);
                        ptx::tmem_st4(bcol + UNIT + q * 4, lo);
                        if (kThird) ptx::tmem_st4(bcol + 2 * UNIT + q * 4, lo2);
                    }
                    if (kThird && n >= 2) drain(n - 2);
                    ptx::tmem_wait_st();
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar(P_FULL + (n & 1)));
                }
            };
            if (!__any_sync(0xffffffffu, two_exp[c] != 0)) units(std::false_type{});
            else units(std::true_type{});
            if (lane == 0) ptx::mbar_arrive(bar(C_EMPTY + c));
        }
        if constexpr (kThird) {
            if (ok) ok = warp_wait(bar(ACC_DONE), 0, abort_flag, kErrBwdDq | 6);
            ptx::tc_fence_after();
            for (int i = n > 2 ? n - 2 : 0; i < n; ++i) drain(i);
            if (ok && m < M) {
                const long rows = (long)a.B * a.H * M;
                float4 *dst = reinterpret_cast<float4 *>(a.part + ((size_t)split * rows + ((size_t)b * a.H + h) * M + m) * D + cg * 16);
#pragma unroll
                for (int k = 0; k < 16; k += 4) dst[k / 4] = make_float4(sum[k], sum[k + 1], sum[k + 2], sum[k + 3]);
            }
        } else if (cg == 0) {
            if (ok) ok = warp_wait(bar(ACC_DONE), 0, abort_flag, kErrBwdDq | 6);
            ptx::tc_fence_after();
            float acc[D];
#pragma unroll
            for (int k = 0; k < D; ++k) acc[k] = 0.f;
#pragma unroll 1
            for (int i = 0; i < min(kAccs, UPT * nt); ++i) {
#pragma unroll
                for (int dc = 0; dc < D / 16; ++dc) {
                    uint32_t r[16];
                    ptx::tmem_ld16(gcol + kDqAcc + i * D + dc * 16, r);
                    ptx::tmem_wait_ld();
#pragma unroll
                    for (int k = 0; k < 16; ++k) acc[dc * 16 + k] += __uint_as_float(r[k]);
                }
            }
            if (ok && m < M) {
                const long rows = (long)a.B * a.H * M;
                float4 *dst = reinterpret_cast<float4 *>(a.part + ((size_t)split * rows + ((size_t)b * a.H + h) * M + m) * D);
#pragma unroll
                for (int dc = 0; dc < D / 4; ++dc) dst[dc] = make_float4(acc[4 * dc], acc[4 * dc + 1], acc[4 * dc + 2], acc[4 * dc + 3]);
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

// ------------------------------------------------------------------------------- pass B, token side (dK, dV)
// Tokens on the lanes, latents on the columns, one sweep over the latents of a tile.  dd[n] = sum_m W_dec[n,m] A[n,m], which every dS of the
// row needs, is known only when the row is done; but it enters linearly, so it is put in at the end:
//     dK_n = scale (T_n - (dd - e)[n] U_n),   T_n = sum_m (W_dec (A - e) + W_enc (C - de))[n,m] q_m,   U_n = sum_m W_dec[n,m] q_m.
// e[n], any number that is near dd[n], keeps the two from being large and nearly equal, each with the rounding of its halves, where the rows of Z
// that a token weighs are nearly equal or one of them has most of the weight.  It comes from the stored Y (bwd_guess), which is dd up to the rounding of
// Y; A has had a row near the middle of Z taken out as well (z_around).  Against float64, what is left of dK's error when the rounding of the stored value
// is taken off, of the norm, with dd formed in a sweep of its own first : e = 0 : e from Y.  M = 64, D = 32 (which the sweeps take now), mean largest weight 0.70 4.8e-7 : 1.1e-6 : 5.7e-7
// (99th percentile of a row's 2.5e-5 : 1.9e-4 : 2.5e-6), 0.93 9.6e-6 : 1.2e-5 : 5.1e-6, 0.97 3.6e-5 : 3.8e-5 : 1.0e-5; features with
// a mean of 1, M = 128, D = 32 2.3e-4 : 2.2e-6 : 2.2e-6.  e costs a packed addition per pair of columns and a pass over Y and dY, us per training step, e = 0 -> now: 131072 tokens, M =
// 512, D = 32 1415 -> 1477; 2 x 20011, M = 128, D = 64 173 -> 180.
// And W_enc = W_dec r[n] c[m] with r = 2^(lse_dec[n] - K), c = 2^(K - lse_enc[m]) and K in the middle of the latents' lse_enc, so that with
// c dZ in the place of dZ one weight serves everything:
//     T_n = sum_m W_dec (A - e + r (C' - c de)) q_m,   C' = V (c dZ)^T,     dV_n = r sum_m W_dec (c dZ)_m,
// one exponential and one split of a weight per pair, and [dV | U] one accumulator whose contractions share their A operand.  dd goes to the
// workspace for the dQ kernel.
//
// What the factors may lose: W_dec below 2^-126 is flushed, which is a W_enc below 2^-126 r c = 2^(lse_dec[n] - lse_enc[m] - 126) (log2 units): below 2^-86 in
// tiles whose tokens have an lse_dec within kOneExpLog2 of the least lse_enc, as in the dQ kernel.  (A bound by the range of lse_enc alone would not
// do: of a range of latents lse_dec may lie far above all, and weights it flushes may then be all there is of a row of dV.)  Tiles beyond that
// (an infinite lse_dec is how the two-query variant switches a stage off) take a form of the body with an exponential of its own for W_enc,
// whose halves are a third pair of operands (kTwo): 2^(S - K) against c dZ, c at most 2^(kFoldLog2 / 2); for wider ranges of lse_enc all tiles
// do, and c is 1.
//
// Sixteen warps share units of 64 latents, 16 columns each, on two alternating buffers of tensor memory (S | A | C), as in the dQ kernel.  Rows leave the accumulators after the first unit of the next tile.
// D = 64: units of 32 shared by eight warps (the accumulators take 192 columns).
// Two sweeps over the latents (dd first; two exponentials and 26 instructions per pair, here one and 20), by groups of four warps with units of their
// own, took, us per training step -> now: 131072 tokens, M = 512, D = 32 (in two ranges, 448 latents at most) 1905 -> 1513;
// 2 x 20011, M = 128, D = 64 187 -> 178.
constexpr float kFoldLog2 = 80.f;
constexpr int kTokFirstMathWarp = 4;                            // warps: 0 TMA producer, 1 and 3 MMA issue, 2 token constants, 4 on arithmetic

struct BwdTokTcArgs {
    const __nv_bfloat16 *Q;    // [H,M,D]
    const float *Z, *dZ;       // [B,H,M,D]
    const float *lse_enc, *de; // [B,H,M]
    const float *lse_dec;      // [B,N,H]
    const uint8_t *key_mask;   // [B,N] or null
    const float *around, *e;   // (workspace) see BwdDqTcArgs; [B,N,H], see bwd_guess
    int around_rows;
    __nv_bfloat16 *dK, *dV;    // [B,N,H,D]
    float *dd;                 // [B,H,N] (workspace)
    uint32_t *status;
    int B, H, N, M;            // M: latents this launch works on (all of them, or a range)
    int mtot, m0;              // latents per head in memory, and the first one of this launch's range
    // More latents than one launch can keep in shared memory are worked off in ranges: T, dV, U and dd of a range add up with the earlier
    // ranges' in float32 sums, kvacc [3][B*N*H][D] and dd_sums (read) / dd (written: another array, since several threads
    // read what one of them replaces), and the last range writes the rows.
    int first, last;           // (without ranges both)
    float *kvacc;
    const float *dd_sums;
    float scale, sl2;
    int tiles, stages;
};

template <int D>
struct BwdTokSmem {
    using G = TileGeom<D>;
    static constexpr int UNIT = D == 64 ? 32 : 64, NCG = UNIT / 16, kThreads = (kTokFirstMathWarp + 4 * NCG) * 32;
    static constexpr int kAccStride = 4 * D;                    // columns of an accumulator: dV | U | dV's share of c dZ lo | T
    // accumulators beside two buffers of three regions of ucols columns: the largest power of two up to four (as a logarithm)
    __device__ static __forceinline__ int log2_accs(int ucols) {
        const int fit = (512 - 6 * ucols) / kAccStride;
        return fit >= 4 ? 2 : fit >= 2 ? 1 : 0;
    }
    static constexpr int kRing = 4, kPlanes = D == 64 ? 2 : 3, kRingTile = kPlanes * kTile;   // tiles of token constants on their way or in use
    static constexpr int kAlign = D == 64 ? 1024 : 512;         // (rows of 64 bytes are swizzled alike every 512: that much less to leave room for)
    // D = 64: dd[n] is subtracted from products that the dQ kernel forms of three parts of Z, so A is formed of three as well (with two,
    // dQ on features of point clouds was 4.7e-6 to 5.4e-6 of its norm from float64 instead of 2.6e-6 to 3.0e-6), as long as the third fits
    // beside two tile stages.
    static constexpr int kThirdMost = D == 64 ? 160 : 0;
    enum { ZH = 0, ZL = 1, DH = 2, QR = 3, DL = 4, Z3 = 5 };    // latent operands: Z hi, lo, c dZ hi, Q, c dZ lo (one B operand: see outputs), third part of Z
    // tiles: [stage][K | V | dY]; latent operands with M rows each (M a multiple of 16); per latent the exponent's addend and -c de;
    // per token -lse_dec, e and, but at D = 64, r; the column groups' shares of dd
    __host__ __device__ static size_t lat_off(int stages, int M, int which) {
        return (size_t)stages * 3 * G::TILE_BYTES + (size_t)which * M * G::RB;
    }
    __host__ __device__ static size_t cst_off(int stages, int M) { return lat_off(stages, M, M <= kThirdMost ? 6 : 5); }
    __host__ __device__ static size_t ring_off(int stages, int M) { return cst_off(stages, M) + 2 * sizeof(float) * M; }
    __host__ __device__ static size_t dds_off(int stages, int M) { return ring_off(stages, M) + kRing * kRingTile * sizeof(float); }
    __host__ __device__ static size_t bar_off(int stages, int M) { return dds_off(stages, M) + 4 * NCG * kTile * sizeof(float); }
    __host__ __device__ static size_t total(int stages, int M) {
        const size_t t = bar_off(stages, M) + 512 + kAlign;
        return t < kTcMinSmem ? kTcMinSmem : t;
    }
    static constexpr int kMaxStages = 6;
    // the most stages (at most kMaxStages) that fit beside the latent operands; 0 if not even one does
    __host__ static int stages(int M) {
        int s = kMaxStages;
        while (s > 0 && total(s, M) > (size_t)227 * 1024) --s;
        return s;
    }
};

// grid = (CTAs per head, H, B); a CTA takes the token tiles blockIdx.x, blockIdx.x + gridDim.x, ...  kRanges: see BwdTokTcArgs.
template <int D, bool kRanges>
__global__ void __launch_bounds__(BwdTokSmem<D>::kThreads, 1)
bwd_token_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                    const __grid_constant__ CUtensorMap tmG, BwdTokTcArgs a) {
    using G = TileGeom<D>;
    using SM = BwdTokSmem<D>;
    constexpr int UNIT = SM::UNIT, NCG = SM::NCG, kThreads = SM::kThreads, kMaxSt = SM::kMaxStages, RING = SM::kRing;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = ptx::align_smem<SM::kAlign>(smem_raw);
    const int M = a.M, stages = a.stages;
    float *cst = reinterpret_cast<float *>(smem + SM::cst_off(stages, M));      // [M] addend of W_enc's own exponent, [M] -c de
    float *ring = reinterpret_cast<float *>(smem + SM::ring_off(stages, M));    // [RING][-lse_dec (log2 units) | -e | r][token]
    float *dds = reinterpret_cast<float *>(smem + SM::dds_off(stages, M));      // [4][column group][token]
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + SM::bar_off(stages, M));
    enum { T_FULL = 0, T_EMPTY = T_FULL + kMaxSt, S_FULL = T_EMPTY + kMaxSt, P_FULL = S_FULL + 2, C_FULL = P_FULL + 2, C_EMPTY = C_FULL + RING,
           ACC_FULL = C_EMPTY + RING, ACC_EMPTY = ACC_FULL + 4, DD_FULL = ACC_EMPTY + 4, NBARS = DD_FULL + 8 };
    static_assert(NBARS * 8 + 8 + 4 * RING + 8 * kThreads / 32 <= 512 + 0, "barrier area too small");
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + NBARS);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    volatile uint32_t *two_exp = tmem_slot + 2;                 // [RING]: the tile takes the form with two exponentials
    float *extremes = reinterpret_cast<float *>(tmem_slot + 2 + RING);          // [warp][least, greatest lse_enc]

    const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
    const int h = blockIdx.y, b = blockIdx.z;
    const int nt = (a.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // tiles of this CTA
    const int nu = (M + UNIT - 1) / UNIT;                       // latent units of a tile; the last may be narrower
    const int wlast = M - (nu - 1) * UNIT;
    const int ucols = min(UNIT, (M + 31) & ~31);                // columns of a region S, A or C
    const int log_accs = SM::log2_accs(ucols);                  // accumulators in turn for the tiles
    const bool third = D == 64 && M <= SM::kThirdMost;
    auto bar = [&](int i) { return ptx::smem_u32(bars + i); };

    if (threadIdx.x == 0) {
        const uint32_t math = 4 * NCG;                          // warps that work on a unit
        for (int i = 0; i < NBARS; ++i)
            ptx::mbar_init(bar(i), i >= DD_FULL || (i >= ACC_EMPTY && i < DD_FULL) || (i >= P_FULL && i < C_FULL) ? math
                                   : i >= C_EMPTY && i < ACC_FULL ? math + 1u : i < T_EMPTY || (i >= C_FULL && i < C_EMPTY) ? 1u : 2u);   // (two issuing warps)
        *abort_flag = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmK);
        ptx::prefetch_tensormap(&tmV);
        ptx::prefetch_tensormap(&tmG);
    }
    if (warp == 1) ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
    ptx::grid_launch();
    ptx::grid_wait();
    const size_t q0 = (size_t)h * a.mtot + a.m0, r0 = ((size_t)b * a.H + h) * a.mtot + a.m0;
    const float *centre = a.around + ((size_t)b * a.H + h) * a.around_rows * D;
    float K, least, unfolded;                                   // (unfolded != 0: c is 1)
    {
        // K: the middle of the latents' lse_enc (log2 units), leaving out those that saw no valid token and those whose encode is switched off
        float lo = INFINITY, hi = -INFINITY;
        for (int m = threadIdx.x; m < M; m += kThreads) {
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
        __syncthreads();
        for (int w = 0; w < kThreads / 32; ++w) {
            lo = fminf(lo, extremes[2 * w]);
            hi = fmaxf(hi, extremes[2 * w + 1]);
        }
        K = lo <= hi ? 0.5f * (lo + hi) : 0.f;
        least = lo <= hi ? lo : 0.f;
        unfolded = lo > hi || hi - lo <= kFoldLog2 ? 0.f : 1.f;
    }
    auto factor = [&](int m) {                                  // c of latent m; 0 for those left out
        const float le = a.lse_enc[r0 + m] * kBwdLog2e;
        return le == -INFINITY || le == INFINITY ? 0.f : unfolded != 0.f ? 1.f : ptx::ex2(K - le);
    };
    {
        uint8_t *lat[5];
#pragma unroll
        for (int w = 0; w < 5; ++w) lat[w] = smem + SM::lat_off(stages, M, w);
        stage_bf16<D, D>(lat[SM::QR], a.Q + q0 * D, M, 0, 0, threadIdx.x, kThreads);
        if (third) stage_hilo<D, D, true>(lat[SM::ZH], lat[SM::ZL], a.Z + r0 * D, M, 0, 0, threadIdx.x, kThreads, centre, UnitFactor(), smem + SM::lat_off(stages, M, SM::Z3));
        else stage_hilo<D, D>(lat[SM::ZH], lat[SM::ZL], a.Z + r0 * D, M, 0, 0, threadIdx.x, kThreads, centre);
        stage_hilo<D, D>(lat[SM::DH], lat[SM::DL], a.dZ + r0 * D, M, 0, 0, threadIdx.x, kThreads, nullptr, factor);
        for (int m = threadIdx.x; m < M; m += kThreads) {
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
    const uint32_t bcols = 3 * ucols, acc0 = 2 * bcols;         // columns of a buffer; the first accumulator

    if (warp == 0) {
        if (ptx::elect_one()) {
            for (int i = 0; i < nt; ++i) {
                const int s = i % stages, t = blockIdx.x + i * gridDim.x;
                if (!ptx::mbar_wait(bar(T_EMPTY + s), ((i / stages) & 1) ^ 1, abort_flag, kErrBwdTok | 1)) break;
                ptx::mbar_arrive_expect_tx(bar(T_FULL + s), 3 * G::TILE_BYTES);
                uint8_t *dst = smem + (size_t)s * 3 * G::TILE_BYTES;
                ptx::tma_load_3d(ptx::smem_u32(dst), &tmK, bar(T_FULL + s), h * D, t * kTile, b);
                ptx::tma_load_3d(ptx::smem_u32(dst + G::TILE_BYTES), &tmV, bar(T_FULL + s), h * D, t * kTile, b);
                ptx::tma_load_3d(ptx::smem_u32(dst + 2 * G::TILE_BYTES), &tmG, bar(T_FULL + s), h * D, t * kTile, b);
            }
        }
    } else if (warp == 2) {
        // Token constants of every tile: -lse_dec, e and r (0 for a token that takes no part in the encode softmax), or, in a tile that takes
        // two exponentials, 0 or -inf in the place of r.  Fetched by asynchronous copies three tiles ahead.  (D = 64: with a plane for r as well 160
        // and 192 latents would have one tile stage instead of two.  There the last bit of e says whether a token takes part, and the arithmetic warps,
        // which have registers to spare, form r.)
        constexpr int AH = RING - 1;
        auto fetch = [&](int i) {
            float *at = ring + (i % RING) * SM::kRingTile;
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) {
                const int r = e * 32 + lane, n = min((int)(blockIdx.x + i * gridDim.x) * kTile + r, a.N - 1);
                ptx::copy_async4(ptx::smem_u32(at + r), a.lse_dec + ((size_t)b * a.N + n) * a.H + h);
                ptx::copy_async4(ptx::smem_u32(at + kTile + r), a.e + ((size_t)b * a.N + n) * a.H + h);
            }
        };
        for (int k = 0; k < AH; ++k) {
            if (k < nt) fetch(k);
            ptx::copy_async_commit();
        }
        for (int i = 0; i < nt; ++i) {
            ptx::copy_async_wait<AH - 1>();
            __syncwarp();
            float *at = ring + (i % RING) * SM::kRingTile;
            float ld[kTile / 32];
            bool part[kTile / 32], far = unfolded != 0.f;
#pragma unroll
            for (int e = 0; e < kTile / 32; ++e) {
                const int r = e * 32 + lane, n = (int)(blockIdx.x + i * gridDim.x) * kTile + r;
                const bool in = n < a.N;
                ld[e] = in ? at[r] * kBwdLog2e : INFINITY;
                part[e] = in && (a.key_mask == nullptr || a.key_mask[(size_t)b * a.N + n] != 0);
                at[r] = -ld[e];
                const float ev = at[kTile + r], ne = fabsf(ev) <= 3.0e38f ? -ev : 0.f;
                at[kTile + r] = SM::kPlanes == 3 ? ne : __uint_as_float((__float_as_uint(ne) & ~1u) | (part[e] ? 1u : 0u));
                far = far || (part[e] && !(ld[e] - least <= kOneExpLog2));
            }
            far = __any_sync(0xffffffffu, far);
#pragma unroll
            for (int e = 0; SM::kPlanes == 3 && e < kTile / 32; ++e)
                at[2 * kTile + e * 32 + lane] = far ? (part[e] ? 0.f : -INFINITY) : (part[e] ? ptx::ex2(ld[e] - K) : 0.f);
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
    } else if (warp == 1 || warp == 3) {
        // Two issuing warps: warp 1 forms S and adds up T = dS Q, whose operand dS lies over S; warp 3 forms A and C' and adds up [dV | U], whose
        // weights lie over A (kTwo: and C').  Each overwrites only what its own earlier instructions read.
        auto issue = [&](auto second) {
            constexpr bool kSecond = decltype(second)::value;
            // (descriptors as 32-bit low words beside a constant high word: see ptx::desc)
            constexpr uint32_t HI = ptx::desc_hi(G::SBO, G::SWZ), TILE = G::TILE_BYTES >> 4, STEP16 = (16 * G::RB) >> 4;
            const uint32_t LAT = (uint32_t)(M * G::RB) >> 4;    // from one latent operand to the next
            const uint32_t lat0 = ptx::desc_lo(ptx::smem_u32(smem + SM::lat_off(stages, M, 0)), 16), td0 = ptx::desc_lo(ptx::smem_u32(smem), 16);
            // K-major to MN-major; the next blocks along N of [c dZ hi | Q | c dZ lo] are one operand further on each (LBO, bits 16-29)
            constexpr uint32_t MN = ptx::desc_lo(0, G::SBO) - ptx::desc_lo(0, 16);
            const uint32_t MN3 = (LAT << 16) - ptx::desc_lo(0, 16);
            const int units = nu * nt;
            int s_stage = 0, s_wrap = 0, s_u = 0, o_u = 0, o_tile = 0, o_acc = 0, o_wrap = 0;
            bool o_two = false;
            // S^T = K Q^T, or A^T = dY Z^T | C'^T = V (c dZ)^T, of the next unit, into buffer n & 1
            auto tiles = [&](int n) -> bool {
                if (s_u == 0) {
                    if (!ptx::mbar_wait(bar(T_FULL + s_stage), (uint32_t)s_wrap, abort_flag, kErrBwdTok | 3)) return false;
                    ptx::tc_fence_after();
                }
                const uint32_t idescS = ptx::instr_desc_bf16(128, 0, 0, 0) | (uint32_t)((s_u == nu - 1 ? wlast : UNIT) >> 3) << 17;
                uint32_t td = td0 + (uint32_t)s_stage * 3 * TILE, ld = lat0 + (uint32_t)s_u * (UNIT / 16) * STEP16;
                ptx::opaque(td);
                ptx::opaque(ld);
                const uint32_t bcol = tm + (n & 1) * bcols;
                auto product = [&](int of, int lat, bool more) {   // of: S, A or C
                    const uint32_t col = bcol + of * ucols, ad = td + (of == 0 ? 0 : of == 1 ? 2 * TILE : TILE), bd = ld + lat * LAT;
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) ptx::mma_ss(col, ptx::desc(ad + 2 * k, HI), ptx::desc(bd + 2 * k, HI), idescS, k > 0 || more);
                };
                if constexpr (!kSecond) {
                    product(0, SM::QR, false);
                } else {
                    if (D == 64 && third) product(1, SM::Z3, false);   // (small parts first: fewer sums are truncated at their full size)
                    product(1, SM::ZL, D == 64 && third);
                    product(1, SM::ZH, true);
                    product(2, SM::DL, false);
                    product(2, SM::DH, true);
                }
                ptx::mma_commit(bar(S_FULL + (n & 1)));
                if (++s_u == nu) {
                    ptx::mma_commit(bar(T_EMPTY + s_stage));
                    s_u = 0;
                    if (++s_stage == stages) { s_stage = 0; s_wrap ^= 1; }
                }
                return true;
            };
            // T += dS Q, or [dV | U | dV'] += W_dec [c dZ hi | Q | c dZ lo], of unit o_u (kTwo: dV += W_enc (c dZ))
            auto outputs = [&](int n) {
                constexpr uint32_t idesc1 = ptx::instr_desc_bf16(128, D, 0, 1), idesc2 = ptx::instr_desc_bf16(128, 2 * D, 0, 1),
                                   idesc3 = ptx::instr_desc_bf16(128, 3 * D, 0, 1);
                const uint32_t bcol = tm + (n & 1) * bcols, V = tm + acc0 + o_acc * SM::kAccStride, U = V + D, V2 = U + D, T = V2 + D;
                uint32_t ld = lat0 + (uint32_t)o_u * (UNIT / 16) * STEP16;
                ptx::opaque(ld);
                const int steps = (o_u == nu - 1 ? wlast : UNIT) / 16;
                auto step = [&](auto two, int k) {
                    constexpr bool kTwo = decltype(two)::value;
                    const uint32_t acc = (o_u > 0 || k > 0) ? 1u : 0u, s = bcol + 16 * k, w = s + ucols, e = w + ucols;   // (hi, and lo 8 columns on)
                    const uint32_t qd = ld + SM::QR * LAT + MN + k * STEP16, dl = ld + SM::DL * LAT + MN + k * STEP16, dh = ld + SM::DH * LAT + k * STEP16;
                    if constexpr (!kSecond) {
                        ptx::mma_ts(T, s, ptx::desc(qd, HI), idesc1, acc);
                        ptx::mma_ts(T, s + 8, ptx::desc(qd, HI), idesc1, 1u);
                    } else if constexpr (!kTwo) {
                        ptx::mma_ts(V, w, ptx::desc(dh + MN3, HI), idesc3, acc);
                        ptx::mma_ts(V, w + 8, ptx::desc(dh + MN3, HI), idesc2, 1u);
                    } else {
                        ptx::mma_ts(V, e, ptx::desc(dh + MN, HI), idesc1, acc);
                        ptx::mma_ts(V, e + 8, ptx::desc(dh + MN, HI), idesc1, 1u);
                        ptx::mma_ts(V2, e, ptx::desc(dl, HI), idesc1, acc);
                        ptx::mma_ts(U, w, ptx::desc(qd, HI), idesc1, acc);
                        ptx::mma_ts(U, w + 8, ptx::desc(qd, HI), idesc1, 1u);
                    }
                };
                if (!kSecond || !o_two) {
                    if (steps == UNIT / 16) {
#pragma unroll
                        for (int k = 0; k < UNIT / 16; ++k) step(std::false_type{}, k);
                    } else {
                        for (int k = 0; k < steps; ++k) step(std::false_type{}, k);
                    }
                } else if constexpr (kSecond) {
                    for (int k = 0; k < steps; ++k) step(std::true_type{}, k);
                }
            };
            bool ok = true;
            for (int n = 0; ok && n < 2 && n < units; ++n) ok = tiles(n);
            for (int n = 0; ok && n < units; ++n) {
                if (!ptx::mbar_wait(bar(P_FULL + (n & 1)), (n >> 1) & 1, abort_flag, kErrBwdTok | 4)) break;
                if (o_u == 0) {
                    if (kSecond) {
                        const int c = o_tile % RING;
                        if (!ptx::mbar_wait(bar(C_FULL + c), (o_tile / RING) & 1, abort_flag, kErrBwdTok | 5)) break;
                        o_two = two_exp[c] != 0;
                        ptx::mbar_arrive(bar(C_EMPTY + c));
                    }
                    if (!ptx::mbar_wait(bar(ACC_EMPTY + o_acc), (uint32_t)o_wrap ^ 1u, abort_flag, kErrBwdTok | 6)) break;
                }
                ptx::tc_fence_after();
                outputs(n);
                if (++o_u == nu) {
                    ptx::mma_commit(bar(ACC_FULL + o_acc));
                    o_u = 0;
                    ++o_tile;
                    if (++o_acc == 1 << log_accs) { o_acc = 0; o_wrap ^= 1; }
                }
                if (n + 2 < units) ok = tiles(n + 2);
            }
        };
        if (ptx::elect_one()) {
            if (warp == 1) issue(std::false_type{});
            else issue(std::true_type{});
        }
    } else if (warp >= kTokFirstMathWarp) {
        const int mine = (warp - kTokFirstMathWarp) >> 2;       // columns: 16 from 16 mine on
        const int row = ((warp & 3) << 5) + lane;               // TMEM lane = token within the tile
        const uint32_t gcol = tm + ((uint32_t)((warp & 3) << 5) << 16);
        const float2 sl2p = make_float2(a.sl2, a.sl2);
        const float *nle = cst + 16 * mine, *nde = nle + M;
        // Rows of dK and dV of the k-th tile: pieces of eight columns, in turn to the warps that share the tokens.
        auto write_rows = [&](int k, float r, float ne) -> bool {
            constexpr int PIECES = D / 4;
            const int acc = k & ((1 << log_accs) - 1), tok_n = (int)(blockIdx.x + k * gridDim.x) * kTile + row;
            const bool in = tok_n < a.N;
            const size_t tok = ((size_t)b * a.N + (in ? tok_n : 0)) * a.H + h;
            const uint32_t V = gcol + acc0 + acc * SM::kAccStride;
            if (!warp_wait(bar(DD_FULL + (k & 3)), (k >> 2) & 1, abort_flag, kErrBwdTok | 7)) return false;
            if (!warp_wait(bar(ACC_FULL + acc), (k >> log_accs) & 1, abort_flag, kErrBwdTok | 8)) return false;
            ptx::tc_fence_after();
            const size_t plane = (size_t)a.B * a.N * a.H * D;   // of the sums over ranges
#pragma unroll 1
            for (int p = mine; p < PIECES; p += NCG) {
                const int which = (p ^ (p >> 2)) & 1, c0 = (p >> 1) * 8;   // dK or dV, and the first column
                uint32_t x[8], y[8];
                float dd = 0.f;                                 // less e
                ptx::tmem_ld8(V + (which == 0 ? 3 * D : 0) + c0, x);
                ptx::tmem_ld8(V + (which == 0 ? D : 2 * D) + c0, y);
                if (which == 0) {
                    const float *part = dds + (k & 3) * NCG * kTile + row;
                    dd = part[0] + part[kTile];
                    if (NCG == 4) dd += part[2 * kTile] + part[3 * kTile];
                    const size_t at = ((size_t)b * a.H + h) * a.N + (in ? tok_n : 0);
                    if (kRanges && !a.first) dd += a.dd_sums[at];
                    if (in && c0 == 0) a.dd[at] = !kRanges || a.last ? dd - ne : dd;
                }
                ptx::tmem_wait_ld();
                float f[8], u[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    f[c] = __uint_as_float(x[c]);
                    u[c] = __uint_as_float(y[c]);
                    if (which != 0) {
                        f[c] = (f[c] + u[c]) * r;
                        u[c] = 0.f;
                    }
                }
                if (in && kRanges) {
                    auto sums = [&](int at, float *v) {
                        float4 *sum = reinterpret_cast<float4 *>(a.kvacc + at * plane + tok * D + c0);
#pragma unroll
                        for (int c = 0; c < 8; c += 4) {        // the earlier ranges' shares
                            if (!a.first) {
                                const float4 e = sum[c / 4];
                                v[c] += e.x; v[c + 1] += e.y; v[c + 2] += e.z; v[c + 3] += e.w;
                            }
                            if (!a.last) sum[c / 4] = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
                        }
                    };
                    sums(which, f);
                    if (which == 0) sums(2, u);
                }
                if (in && (!kRanges || a.last)) {
                    const float sc = which == 0 ? a.scale : 1.f;
                    uint32_t w[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        w[c] = ptx::pack_bf16(fmaf(-dd, u[2 * c], f[2 * c]) * sc, fmaf(-dd, u[2 * c + 1], f[2 * c + 1]) * sc);
                    *reinterpret_cast<uint4 *>((which ? a.dV : a.dK) + tok * D + c0) = make_uint4(w[0], w[1], w[2], w[3]);
                }
                __syncwarp();
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar(ACC_EMPTY + acc));
            return true;
        };
        // Sixteen columns of a unit, over which its weights go: dS over S, W_dec over A, W_enc (kTwo) over C, hi and lo of 16 latents side by side.
        auto unit = [&](auto two, uint32_t col, int m, float2 nldp, float2 rp, float2 nep, float2 &d2) {
            constexpr bool kTwo = decltype(two)::value;
            uint32_t s[2][8], av[2][8], cv[2][8];
            auto load = [&](int p) {
                ptx::tmem_ld8(col + 8 * p, s[p]);
                ptx::tmem_ld8(col + ucols + 8 * p, av[p]);
                ptx::tmem_ld8(col + 2 * ucols + 8 * p, cv[p]);
            };
            load(0);
            ptx::tmem_wait_ld();
            load(1);                                            // eight columns on their way while eight are worked on
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                uint32_t hi[4], lo[4], wh[4], wl[4], eh[4], el[4];
#pragma unroll
                for (int q = 0; q < 4; q += 2) {
                    const float4 ne = *reinterpret_cast<const float4 *>(nde + m + 8 * p + 2 * q);
                    float4 le = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (kTwo) le = *reinterpret_cast<const float4 *>(nle + m + 8 * p + 2 * q);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int j = 2 * (q + e), o = q + e;
                        const float2 sv = make_float2(__uint_as_float(s[p][j]), __uint_as_float(s[p][j + 1]));
                        const float2 A = __fadd2_rn(make_float2(__uint_as_float(av[p][j]), __uint_as_float(av[p][j + 1])), nep);
                        const float2 C = make_float2(__uint_as_float(cv[p][j]), __uint_as_float(cv[p][j + 1]));
                        const float2 x = __ffma2_rn(sv, sl2p, nldp);
                        const float2 pd = make_float2(ptx::ex2(x.x), ptx::ex2(x.y));
                        const float2 v = __fadd2_rn(C, e ? make_float2(ne.z, ne.w) : make_float2(ne.x, ne.y));
                        float2 ds;
                        if (kTwo) {
                            const float2 y = __ffma2_rn(sv, sl2p, __fadd2_rn(e ? make_float2(le.z, le.w) : make_float2(le.x, le.y), rp));
                            const float2 pe = make_float2(ptx::ex2(y.x), ptx::ex2(y.y));
                            ds = __ffma2_rn(pd, A, __fmul2_rn(pe, v));
                            eh[o] = ptx::pack_bf16(pe);
                            el[o] = ptx::pack_bf16(ptx::rest_of(pe, eh[o]));
                        } else {
                            ds = __fmul2_rn(pd, __ffma2_rn(rp, v, A));
                        }
                        d2 = __ffma2_rn(pd, A, d2);
                        hi[o] = ptx::pack_bf16(ds);
                        lo[o] = ptx::pack_bf16(ptx::rest_of(ds, hi[o]));
                        wh[o] = ptx::pack_bf16(pd);
                        wl[o] = ptx::pack_bf16(ptx::rest_of(pd, wh[o]));
                    }
                }
                if (p == 0) ptx::tmem_wait_ld();                // (all sixteen have been read)
                ptx::tmem_st4(col + 4 * p, hi);
                ptx::tmem_st4(col + 8 + 4 * p, lo);
                ptx::tmem_st4(col + ucols + 4 * p, wh);
                ptx::tmem_st4(col + ucols + 8 + 4 * p, wl);
                if (kTwo) {
                    ptx::tmem_st4(col + 2 * ucols + 4 * p, eh);
                    ptx::tmem_st4(col + 2 * ucols + 8 + 4 * p, el);
                }
            }
            ptx::tmem_wait_st();
        };
        // All units of the tiles in one loop; one more turn writes the last tile's rows.
        int k = 0, u = 0;                                       // tiles done, unit of the next
        float nld = 0.f, rr = 0.f, ne = 0.f, r_before = 0.f, ne_before = 0.f;
        bool far = false;
        float2 d2 = make_float2(0.f, 0.f);
        while (true) {
            if (k < nt) {
                if (u == 0) {
                    const int c = k % RING;
                    if (!warp_wait(bar(C_FULL + c), (k / RING) & 1, abort_flag, kErrBwdTok | 9)) break;
                    const float *at = ring + c * SM::kRingTile + row;
                    nld = at[0];
                    ne = at[kTile];
                    far = __any_sync(0xffffffffu, two_exp[c] != 0);          // (the same for all: a vote says so to the compiler)
                    if constexpr (SM::kPlanes == 3) {
                        rr = at[2 * kTile];
                    } else {
                        const bool part = __float_as_uint(ne) & 1u;
                        rr = far ? (part ? 0.f : -INFINITY) : (part ? ptx::ex2(-nld - K) : 0.f);
                    }
                    d2 = make_float2(0.f, 0.f);
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(bar(C_EMPTY + c));
                }
                const int n = k * nu + u;
                const uint32_t col = gcol + (n & 1) * bcols + 16 * mine;
                if (!warp_wait(bar(S_FULL + (n & 1)), (n >> 1) & 1, abort_flag, kErrBwdTok | 10)) break;
                ptx::tc_fence_after();
                if (u * UNIT + 16 * mine < M) {
                    if (far) unit(std::true_type{}, col, u * UNIT, make_float2(nld, nld), make_float2(rr, rr), make_float2(ne, ne), d2);
                    else unit(std::false_type{}, col, u * UNIT, make_float2(nld, nld), make_float2(rr, rr), make_float2(ne, ne), d2);
                }
                if (u == nu - 1) dds[((k & 3) * NCG + mine) * kTile + row] = d2.x + d2.y;
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    ptx::mbar_arrive(bar(P_FULL + (n & 1)));
                    if (u == nu - 1) ptx::mbar_arrive(bar(DD_FULL + (k & 3)));
                }
            }
            if (u == 0 && k > 0 && !write_rows(k - 1, r_before, ne_before)) break;
            if (k >= nt) break;
            if (++u == nu) {
                u = 0;
                ++k;
                r_before = far ? 1.f : rr;
                ne_before = ne;
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

}  // namespace flare
