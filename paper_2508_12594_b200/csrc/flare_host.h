// Host-side helpers shared by the library's translation units: error text, device properties, argument checks, launch
// plans and TMA descriptors; and the launchers that each translation unit provides to the entry points.
#pragma once

#include "../../include/flare.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "flare_bwd_sweep.cuh"
#include "flare_bwd_tc.cuh"
#include "flare_common.cuh"
#include "flare_ptx.cuh"
#include "flare_tc.cuh"

namespace flare {
extern thread_local char g_cuda_error[256];   // text of the last CUDA error of this thread

inline int cuda_fail(cudaError_t e, const char *what) {
    snprintf(g_cuda_error, sizeof(g_cuda_error), "%s: %s", what, cudaGetErrorString(e));
    return FLARE_ERR_CUDA;
}

#define FLARE_CUDA(call)                                      \
    do {                                                      \
        cudaError_t e__ = (call);                             \
        if (e__ != cudaSuccess) return cuda_fail(e__, #call); \
    } while (0)

struct DeviceInfo {
    std::atomic<int> checked{0};  // 0 = not yet, 1 = ok, -1 = wrong arch, -2 = no device
    std::atomic<int> sms{148};
};
extern DeviceInfo g_dev[64];

// Properties of the current device (cached per ordinal; concurrent first calls write the same values).  Without
// a device the plan falls back to 148 SMs so that size queries still answer.
struct DeviceView {
    int checked, sms;
};
inline DeviceView device_info(int *ordinal_out = nullptr) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return DeviceView{-2, 148};
    }
    if (ordinal_out) *ordinal_out = dev;
    DeviceInfo &d = g_dev[dev];
    int checked = d.checked.load(std::memory_order_acquire);
    if (checked == 0) {
        int major = 0, sms = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return DeviceView{-2, 148};
        }
        d.sms.store(sms > 0 ? sms : 148, std::memory_order_relaxed);
        checked = (major == 10) ? 1 : -1;
        d.checked.store(checked, std::memory_order_release);
    }
    return DeviceView{checked, d.sms.load(std::memory_order_relaxed)};
}

// The opt-in to more than 48 KB of dynamic shared memory is a property of (kernel, device): one bit per device
// ordinal in a mask per kernel instantiation.  Setting it twice is harmless, so a race between host threads
// only repeats the call.
template <typename Kernel>
int ensure_big_smem(Kernel kernel, std::atomic<uint64_t> &done, int bytes = 227 * 1024) {
    int dev = 0;
    FLARE_CUDA(cudaGetDevice(&dev));
    const uint64_t bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return FLARE_OK;
    FLARE_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    done.fetch_or(bit, std::memory_order_release);
    return FLARE_OK;
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline int check_desc(const flare_desc_t *d) {
    if (d == nullptr) return FLARE_ERR_INVALID_ARG;
    if (d->B <= 0 || d->H <= 0 || d->N <= 0 || d->M <= 0 || d->D <= 0) return FLARE_ERR_INVALID_ARG;
    if (!std::isfinite(d->scale)) return FLARE_ERR_INVALID_ARG;
    if (d->dtype != FLARE_DTYPE_F32 && d->dtype != FLARE_DTYPE_BF16 && d->dtype != FLARE_DTYPE_F16) return FLARE_ERR_UNSUPPORTED;
    if (d->D != 4 && d->D != 8 && d->D != 16 && d->D != 32 && d->D != 64) return FLARE_ERR_UNSUPPORTED;
    if (d->dtype == FLARE_DTYPE_BF16 && (d->M % 16 != 0 || d->M < 16 || d->M > 2048)) return FLARE_ERR_UNSUPPORTED;
    if ((long)d->B * d->N > (1L << 31) - 1 || d->H > 65535 || d->B > 65535) return FLARE_ERR_UNSUPPORTED;
    return FLARE_OK;
}

// Launch plan of the CUDA-core kernels whose rows are latents (encode, dZ, dQ): blocks of WM groups of 8 RB latents, `splits`
// blocks along N.
struct SimtPlan {
    int RB, WM, mblocks, splits, chunk, P;
};
inline int simt_row_blocks(int D) { return D <= 16 ? 4 : D == 32 ? 2 : 1; }   // of the forward kernels: 8 RB D values of a warp's accumulators
inline SimtPlan simt_plan_for(const flare_desc_t *d, int sms, int RB) {
    SimtPlan p;
    p.RB = RB;
    const int groups = (d->M + 8 * RB - 1) / (8 * RB), tile = d->D <= 32 ? 64 : 32;
    p.WM = 1;
    while (p.WM < groups && p.WM < kSimtThreads / 32) p.WM *= 2;
    p.mblocks = (groups + p.WM - 1) / p.WM;
    const long per = (long)d->B * d->H * p.mblocks;
    long s = 2L * sms / per;                                    // two blocks per SM, in one wave
    const long most = (d->N + tile - 1) / tile;
    if (s > most) s = most;
    if (s < 1) s = 1;
    p.chunk = (int)((d->N + s - 1) / s);
    p.chunk = (p.chunk + tile - 1) / tile * tile;
    p.splits = (d->N + p.chunk - 1) / p.chunk;
    p.P = p.splits;
    return p;
}
// (up to 16 latents: single row blocks, so that fewer rows of the MMAs are empty)
inline SimtPlan simt_plan(const flare_desc_t *d, int sms) { return simt_plan_for(d, sms, d->M <= 16 ? 1 : simt_row_blocks(d->D)); }

// The tensor-core kernels take bfloat16 with D in {16, 32, 64} and a positive scale, and D = 8 or 4 as the narrow
// forms of the D = 16 kernels: a token tile of 16 feature columns then spans two or four heads, so the tensor must
// be at least 16 columns wide, and (TMA) its rows a multiple of 16 bytes.  Everything else (float32, non-positive
// scale, narrower tensors) runs on the CUDA-core kernels.  FLARE_DEBUG_PATH=simt forces the latter.
inline bool use_tc(const flare_desc_t *d) {
    static const bool forced_simt = [] {
        const char *e = std::getenv("FLARE_DEBUG_PATH");
        return e != nullptr && std::strcmp(e, "simt") == 0;
    }();
    // (a scale so small that scale * kMaskedScore no longer dwarfs every real score would let padded tokens through the
    // form that puts padding into the scores: such calls run on the CUDA cores too)
    return !forced_simt && d->dtype == FLARE_DTYPE_BF16 && d->scale > 1e-20f &&
           (d->D == 16 || d->D == 32 || d->D == 64 || (d->D == 8 && d->H >= 2) || (d->D == 4 && d->H >= 4 && d->H % 2 == 0));
}

// Small float32 and float16 forwards run as one launch (forward_small_simt_kernel): blocks per cluster, or 0 for the kernels that split the
// tokens over the whole GPU.  Sixteen blocks per head while they get an SM each, eight while two share one; a block should have one tile of 64
// tokens, or two where a tile is quick.  Measured, one launch : three, us (tokens, M, D, heads): sixteen blocks 1024, 16, 16, 2 5.3 : 7.2;
// 1024, 64, 32, 8 17.4 : 21; 2048, 16, 16, 8 8.5 : 9.7; 2048, 60, 8, 8 12.1 : 12.6; 2048, 64, 16, 4 14.1 : 11.9; 4096, 16, 16, 2 10.4 : 9.7; eight
// 512, 64, 32, 16 18 : 21; 1024, 16, 16, 32 8.8 : 12.3; 1024, 32, 16, 16 11 : 12.5; 1024, 32, 32, 16 18.5 : 16.3; 1024, 64, 32, 16 29 : 24.
inline int small_forward_wanted(const flare_desc_t *d, int sms) {
    if (use_tc(d) || d->M > 64 || d->D > 32) return 0;
    const long heads = (long)d->B * d->H;
    const int cluster = 16 * heads <= sms ? 16 : 8 * heads <= 2L * sms ? 8 : 0;
    if (cluster == 0 || d->N > cluster * (d->M * d->D <= 512 ? 128 : 64)) return 0;
    return cluster;
}

// Which form of the tensor-core forward kernels runs (flare_set_path).
extern std::atomic<int> g_path;

// With at most 64 latents a CTA encodes two adjacent heads at once (see encode_tc_kernel).
inline bool encode_head_pairs(const flare_desc_t *d) { return d->M <= 64 && d->H % 2 == 0 && d->D >= 16 && d->D <= 32; }

// The fast forms (no running maximum, see kFastMaxLog2 in flare_tc.cuh) are followed by a launch of the exact
// form that exits at once unless it is needed: two more launches per forward, which pay off from some size on.
inline bool fast_wanted(const flare_desc_t *d, bool pays) {
    const int path = g_path.load(std::memory_order_relaxed);
    return use_tc(d) && path != FLARE_PATH_EXACT && (path == FLARE_PATH_FAST || pays);
}
// Encode: the time of either form goes with the blocks of 128 lanes (of latents, or of two heads), whatever part of them is filled.
// Measured, exact against fast form with the merge behind it, us, at 65536 / 131072 / 524288 tokens x heads x blocks: D = 16, M = 96 17.8 : 16.5 /
// 21 : 18.6 / 41 : 31, masked 18.5 : 16.5 / 25 : 20.5 / 51 : 33, with log-sum-exp 18.5 : 17.7 / 22.6 : 20.7 / 43 : 37; D = 32 20.5 : 16.6 / 24 :
// 20 / 45 : 33; head pairs, at 32768 / 65536 tokens x pairs: D = 8 18.6 : 15.2 / 22 : 16.6, D = 16 14.5 : 15.8 / 16.7 : 16.5, D = 32 18.5 : 16.5 /
// 20.5 : 18.5.  D = 64: the norm check holds a tile longer than its scores (72 : 84 at a million).
inline bool lean_pairs(const flare_desc_t *d) { return d->M <= 64 && d->H % 2 == 0 && d->D >= 8 && d->D <= 32; }
inline bool use_fast_encode(const flare_desc_t *d) {
    const double work = (double)d->B * d->N * (lean_pairs(d) ? d->H / 2 : d->H) * ((d->M + 127) / 128);
    return d->D <= 32 && fast_wanted(d, work >= (lean_pairs(d) && d->D != 16 ? 3.0e4 : 6.0e4));
}
// Decode: the streaming form has no variant for head width 64.  Measured against the exact form, us, at B H N = 524288 (131072): D = 16, M = 48
// 20 : 29 (11.2 : 10.4), 64 31 : 35 (10.4 : 8.3), 96 26 : 36 (14.4 : 15.8), 144 27 : 33 (15 : 20); the exact form keeps what fills one chunk
// of its registers (M = 32: 18 : 13) and, at D = 32, 64 latents (48 : 41) and small calls up to there (M = 48: 29 : 35 from 262144 on).
// 16 latents leave half of a chunk, or of a unit, empty in either form, and the exact form, which has no form of its own for them, is slower
// than at 32: 262144 / 524288 / 2097152 rows, D = 8 18.4 : 18.4 / 22.5 : 26.7 / 43 : 68, D = 16 18.5 : 20.5 / 24.6 : 30.7 / 53 : 78, D = 32
// 24.6 : 22.5 / 32.8 : 34.8 / 90 : 96.
inline bool use_fast_decode(const flare_desc_t *d) {
    const double rows = (double)d->B * d->H * d->N;
    bool pays;
    if (d->M == 32 || (d->D == 32 && d->M == 64)) pays = false;
    else if (d->M < 64) pays = rows >= 3.0e5;
    else if (d->M == 64) pays = rows >= 5.0e5;
    else if (d->M <= 128) pays = rows >= (d->M == 128 ? 2.0e5 : d->D == 32 ? 6.0e4 : 1.2e5);
    else pays = rows >= 6.0e4;
    return d->D <= 32 && fast_wanted(d, pays);
}

// Launch plan of the tensor-core encode: `pairs` CTAs per head along the latents (two 128-latent blocks each),
// `splits` CTAs along N, about one CTA per SM in total.
struct TcEncodePlan {
    int tiles, pairs, splits, per_split, P;
};

// CTAs to split the token tiles of each of `groups` pieces of work over, one CTA per SM at a time.  A CTA costs its share of the tiles
// and about four tiles' time to start and finish (5 of 1.6 us); a launch costs as many CTAs as its fullest SM runs one after the other, so
// that one more split than fills the chip once can take twice as long and several times as many less than once (64 pieces: 2 splits leave
// 20 of 148 SMs idle, 23 in ten rounds 0.5); each split also leaves a partial result of `part_bytes` to be reduced (some 4 MB
// written and read in a tile's time).  At most 512 tiles per split keep the float32 sums on the tensor core short.
// At most `cap` splits, whatever the sums' length.
inline int balanced_splits(long groups, int tiles, int sms, size_t part_bytes, int cap) {
    const double start = 4.0, reduce = (double)part_bytes / 4.0e6;
    const int least = std::min((tiles + 511) / 512, cap), most = std::min(std::min(tiles, least + sms), cap);
    int best = least;
    double best_cost = 0.0;
    for (int s = least; s <= most; ++s) {
        const double rounds = (double)((groups * s + sms - 1) / sms);
        const double cost = rounds * ((tiles + s - 1) / s + start) + reduce * s;
        if (s == least || cost < best_cost) { best = s; best_cost = cost; }
    }
    return best;
}

// CTAs per head of the kernels of the backward that have tokens on the lanes.  As many as fill the chip once, unless that leaves enough SMs
// idle that several rounds are 2 % quicker; a CTA's start, where the head's latent operands are split and stored, counts as six units of 64
// latents against a tile, and a fifth of a tile.  us per training step, once : several rounds: 32 heads (128 of 148 CTAs : 288), 50489 tokens, M = 624, D = 16
// 2793 : 2689, 68334 tokens, M = 80, D = 8 734 : 710, 25344 tokens, M = 336, D = 32 890 : 875; 8 heads (144 : 296) of 1048576 tokens, M = 1024, D = 8
// 18813 : 18640; D = 64, where a unit has 32 latents and up to 160 of them three parts to split, 32 heads (128 : 288), 40000 tokens, M = 64 855 : 824; 40
// (120 : 280), 30000, M = 160 1611 : 1530; 64 (128 : 256), 9000, M = 96 500 : 496; the same number either way 128 heads, M = 192, and 32, 20011, M = 128.
// (A CTA per SM with a share of all heads' tiles in a row, needs a loop over heads around the kernel's body, which made every training step 5 % slower.)
// `part`: what one more CTA per head costs beyond that, in the same units (some 0.65 us): the two sweeps leave partial results of D floats per latent, two per
// CTA (the token kernel leaves none), which take about a unit per 8 MB to write and add up.  us per backward of 128 heads of 8192 tokens, M = 1024, D = 16, in seven
// rounds with 134 MB of them : once over the chip with 17 MB 1905 : 1835; M = 512, D = 8, where 34 MB do not decide, 880 : 899.
inline double token_cost(long ctas, int tiles_each, int mc, int sms) {
    const double units = (double)((mc + 63) / 64);
    return (double)((ctas + sms - 1) / sms) * (tiles_each * units + 6.0 + 0.2 * units);
}
inline int token_splits(const flare_desc_t *d, int tiles, int mc, int sms, double part = 0.0) {
    const long heads = (long)d->B * d->H;
    auto cost = [&](long s) { return token_cost(heads * s, (int)((tiles + s - 1) / s), mc, sms) + part * (double)s; };
    int best = (int)std::min<long>(std::max(1L, sms / heads), tiles);
    double best_cost = 0.98 * cost(best);
    for (int s = best + 1; s <= std::min(tiles, sms); ++s)
        if (cost(s) < best_cost) {
            best = s;
            best_cost = cost(s);
        }
    return best;
}

inline TcEncodePlan tc_encode_plan(const flare_desc_t *d, int sms) {
    TcEncodePlan p;
    p.tiles = (d->N + kTile - 1) / kTile;
    const int mb = (d->M + kTile - 1) / kTile;
    p.pairs = (mb + 1) / 2;
    long groups = (long)d->B * (encode_head_pairs(d) ? d->H / 2 : d->H) * p.pairs;
    long s = sms / groups;
    if (s < 1) s = 1;
    if (s > p.tiles) s = p.tiles;
    p.splits = (int)s;
    p.per_split = (mb == 1) ? 4 : 2;
    p.P = p.splits * p.per_split;
    return p;
}

// Launch plan of the encode without a running maximum and of dZ: one partial result per CTA.  Up to 64 latents two heads share the lanes.
struct LeanPlan { int tiles, blocks, splits; };
inline LeanPlan lean_plan(const flare_desc_t *d, int sms, int cap) {
    LeanPlan p;
    p.tiles = (d->N + kTile - 1) / kTile;
    p.blocks = lean_pairs(d) ? 1 : (d->M + kTile - 1) / kTile;
    const long groups = (long)d->B * (lean_pairs(d) ? d->H / 2 : d->H) * p.blocks;
    p.splits = balanced_splits(groups, p.tiles, sms, (size_t)d->B * d->H * d->M * (d->D + 2) * sizeof(float), cap);
    return p;
}
inline LeanPlan dz_plan(const flare_desc_t *d, int sms) { return lean_plan(d, sms, d->N); }   // (no more splits than tokens: no cap)
// alone: a call of encode by itself.  Its scratch decides whether flare_encode_static_scratch takes a problem: what the exact form brings
// into the built-in array must fit it in this form too, whose plan often splits finer (1048576 tokens, 8 heads, 2048 latents, D = 8: 4 partial
// results against 22, 2.5 MB against 14.4).  The encode of a forward, in a workspace of the caller's, keeps the finer plan.
inline LeanPlan encode_lean_plan(const flare_desc_t *d, int sms, bool alone) {
    const long rows = (long)d->B * d->H * d->M;
    const int exact = tc_encode_plan(d, sms).P;
    if (!alone || make_layout(exact, rows, d->D, false).total > FLARE_STATIC_SCRATCH_BYTES) return lean_plan(d, sms, d->N);
    const size_t part = sizeof(float) * (size_t)rows * (d->D + 2);   // (beside the header; three sections are rounded up)
    return lean_plan(d, sms, std::max(exact, (int)std::min<size_t>(d->N, (FLARE_STATIC_SCRATCH_BYTES - kHeaderBytes - 3 * kAlign) / part)));
}

// (either form of encode on the tensor cores may have to leave its partial results in the same workspace; which one runs may change with
// flare_set_path while a caller keeps the workspace.  At D = 64 there is only the exact form, see use_fast_encode.)
inline int partials_for(const flare_desc_t *d, int sms, bool alone) {
    if (!use_tc(d)) return simt_plan(d, sms).P;
    const int exact = tc_encode_plan(d, sms).P;
    return d->D <= 32 ? std::max(exact, encode_lean_plan(d, sms, alone).splits) : exact;
}

// ---- TMA descriptors (the driver entry point is looked up at run time; the library does not link libcuda)
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

inline CUtensorMapSwizzle swizzle_for(int D) {
    return D == 8 ? CU_TENSOR_MAP_SWIZZLE_NONE : D == 16 ? CU_TENSOR_MAP_SWIZZLE_32B : D == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;
}

// [B, N, H*D] bf16 viewed as a 3-D tensor (innermost H*D); box = `cols` columns (one head's D, or two adjacent
// heads' 2D) x `rows` tokens.
// (8 columns: rows of 16 bytes as they are, not swizzled)
inline int make_token_map(CUtensorMap *m, const void *base, const flare_desc_t *d, int rows, int cols = 0) {
    if (cols == 0) cols = d->D;
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) {
        snprintf(g_cuda_error, sizeof(g_cuda_error), "cuTensorMapEncodeTiled not available");
        return FLARE_ERR_CUDA;
    }
    const cuuint64_t C = (cuuint64_t)d->H * d->D;
    cuuint64_t dims[3] = {C, (cuuint64_t)d->N, (cuuint64_t)d->B};
    cuuint64_t strides[2] = {C * 2, C * 2 * (cuuint64_t)d->N};
    cuuint32_t box[3] = {(cuuint32_t)cols, (cuuint32_t)rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(cols), CU_TENSOR_MAP_L2_PROMOTION_NONE,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(g_cuda_error, sizeof(g_cuda_error), "cuTensorMapEncodeTiled(tokens) failed: %d", (int)r);
        return FLARE_ERR_CUDA;
    }
    return FLARE_OK;
}

// Q_lat [H*M, D] bf16 as a 2-D tensor; box = 16 latent rows.
inline int make_latent_map(CUtensorMap *m, const void *base, const flare_desc_t *d) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) {
        snprintf(g_cuda_error, sizeof(g_cuda_error), "cuTensorMapEncodeTiled not available");
        return FLARE_ERR_CUDA;
    }
    cuuint64_t dims[2] = {(cuuint64_t)d->D, (cuuint64_t)d->H * d->M};
    cuuint64_t strides[1] = {(cuuint64_t)d->D * 2};
    cuuint32_t box[2] = {(cuuint32_t)d->D, 16};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(d->D), CU_TENSOR_MAP_L2_PROMOTION_NONE,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        snprintf(g_cuda_error, sizeof(g_cuda_error), "cuTensorMapEncodeTiled(latents) failed: %d", (int)r);
        return FLARE_ERR_CUDA;
    }
    return FLARE_OK;
}

constexpr float kLog2e = 1.4426950408889634f;

// Header words of a workspace beyond the error flag: set by the fast form of encode / decode when its inputs are
// outside the range it is valid for; the exact form that follows runs only then.
constexpr int kRedoEncodeWord = 2, kRedoDecodeWord = 3;

// One decode launch holds all M score columns of a token tile in tensor memory: up to kDecodeMaxM latents.
constexpr int kDecodeMaxM = 512;

// Ranges of latents a decode over more than kDecodeMaxM latents is cut into, and the scratch their partial results
// take after the encode layout of the forward workspace: float32 rows [C][B*N*H][D] and log-sum-exps [C][B*N*H].
constexpr int kDecodeRange = 256;   // latents per launch when a decode is cut into ranges
inline int decode_ranges(const flare_desc_t *d) { return (d->M + kDecodeRange - 1) / kDecodeRange; }
inline bool decode_in_ranges(const flare_desc_t *d) { return use_tc(d) && d->M > kDecodeMaxM; }
inline size_t decode_range_bytes(const flare_desc_t *d) {
    if (!decode_in_ranges(d)) return 0;
    const size_t rows = (size_t)d->B * d->N * d->H;
    return align_up(sizeof(float) * decode_ranges(d) * rows * d->D) + align_up(sizeof(float) * decode_ranges(d) * rows);
}

// Plans of the backward, whose passes run on the tensor cores for the same shapes as the forward (use_tc): dz_plan for pass A, a form of
// the encode without a running maximum; tc_dq_plan for dQ.  On the CUDA cores pass A has the encode's plan, and the dQ pass, which keeps
// three operands of a latent row in registers, one with fewer rows per warp.

// Plan of the tensor-core dQ kernel: `pairs` = blocks of 128 latents per head, one partial sum per CTA.
inline TcEncodePlan tc_dq_plan(const flare_desc_t *d, int sms) {
    TcEncodePlan p;
    p.tiles = (d->N + kTile - 1) / kTile;
    p.pairs = (d->M + kTile - 1) / kTile;
    p.splits = balanced_splits((long)d->B * d->H * p.pairs, p.tiles, sms, (size_t)d->B * d->H * d->M * d->D * sizeof(float), p.tiles);
    p.per_split = 1;
    p.P = p.splits;
    return p;
}

inline SimtPlan bwd_dq_plan(const flare_desc_t *d, int sms) { return simt_plan_for(d, sms, d->D <= 16 ? 2 : 1); }

// Blocks of 128 latents of a head in dZ's kernel.
inline int latent_blocks(const flare_desc_t *d) { return (d->M + kTile - 1) / kTile; }

// How the tokens are shared out to the blocks that form e (bwd_guess): five blocks an SM, of four turns at least.
struct GuessPlan {
    int chunk, chunks, groups;
};
inline GuessPlan guess_plan(const flare_desc_t *d, int sms) {
    const int pieces = d->H * (d->D / 8), per = std::max(1, 256 / pieces);
    GuessPlan p;
    p.groups = (pieces + 255) / 256;
    const long most = std::max(1L, 5L * sms / ((long)d->B * p.groups));
    p.chunk = (int)std::max<long>((d->N + most - 1) / most, 4L * per);
    p.chunks = (d->N + p.chunk - 1) / p.chunk;
    return p;
}

struct BwdLayout {
    size_t part, dz, de, dd, e, around, dd_other, kvacc, total;
    int P;
};

// Latents one launch of the tensor-core token kernel takes: five operands of D-wide bf16 rows (six at D = 64 up to 160 latents) beside two
// tile stages; more are worked off in ranges of equal size, with three float32 planes and dd to read and write between them.  us per backward, two sweeps with
// two planes and at most 448 latents a range at D = 32 : now, 8 heads of 131072 tokens: D = 32, M = 528 1778 : 1533, 640 1922 : 1587, 1024 3126 : 2284;
// 65536, D = 64, M = 208 852 : 874, 256 939 : 904, 400 1654 : 1671; 4 heads of 131072, M = 384 1128 : 1026.
inline int token_range_most(const flare_desc_t *d) { return d->D == 64 ? 192 : 512; }
inline bool token_in_ranges(const flare_desc_t *d) { return use_tc(d) && d->M > token_range_most(d); }
inline int token_ranges(const flare_desc_t *d) { return (d->M + token_range_most(d) - 1) / token_range_most(d); }
inline int token_range(const flare_desc_t *d) { return ((d->M + token_ranges(d) - 1) / token_ranges(d) + 15) / 16 * 16; }

// Two sweeps over the tokens (flare_bwd_sweep.cuh, where both sides are measured): heads up to 16 wide, and 32 wide as long as one launch takes all latents.  Not
// where that leaves a CTA per tile and few of them, each with many units of latents: the kernels with latents on the lanes share these out.  us per backward, sweeps :
// the others, D = 32, tiles of all heads: 8, M = 208 29.3 : 29.2, M = 256 31.1 : 29.8, M = 320 35.2 : 31.9; 16, M = 256 31.1 : 30.3, M = 320 35.1 : 32.9; 32, M = 256 31.4 : 31.8, M =
// 320 35.2 : 34.6; 64, M = 256 33.8 : 35.9, M = 320 37.9 : 36.6; 96, M = 320 40.8 : 40.0; 120, M = 320 42.0 : 46.5.
inline bool use_sweeps(const flare_desc_t *d) {
    if (!use_tc(d) || d->D > 32) return false;
    const long tiles = (long)d->B * d->H * ((d->N + kTile - 1) / kTile);
    return d->D <= 16 || (d->M <= 320 && tiles > (d->M > 256 ? 100 : d->M > 224 ? 16 : 0));
}
// Latents one launch of a sweep takes: what its operands leave of shared memory (beside two tile stages) and the sums over tokens of tensor memory; more are
// worked off in ranges of about equal size, whole units of 64.
// Ranges leave float32 rows of dK and dV to one another (in the first sweep RowSums): a launch takes a chunk of each item's tokens, so that the rows stay within
// kRangeBytes (or, if that is more, within a tile to a CTA), and all ranges go over one chunk before the next.  Without a bound they are 1074 MB at 1048576 tokens of
// 8 heads, D = 16.  us per training step, no bound : 128 : 64 : 32 MB, 8 heads, M = 1024: 1048576 tokens, D = 8 17000 : 17480 : 17620 : 17870; 524288, D = 16 8830 : 9170 : 9370 : 9720;
// 131072, D = 16 2357 : 2352 : 2456 : 2534 (a chunk starts and ends as any launch does, and chunks give 144 CTAs to the 148 SMs where one launch over 1048576 tokens
// gives two rounds of 148).
constexpr size_t kRangeBytes = (size_t)128 << 20;
// Ranges side by side, each with CTAs of its own and rows that a launch of its own adds up, where one after the other (or all latents in one) leaves a few CTAs
// with many units each.  In the units of token_cost: what a sweep takes to start beyond that, and the launch that joins.  us per backward of 8 heads, one after
// the other : side by side : the three kernels before, D = 16: 128 tokens, M = 512 34.8 : 27.0 : 31.6, 1024 66.9 : 32.3 : 42.1, 2048 118 : 34 : 73; 1024 tokens, M = 768 48.8 : 39.8 :
// 47.7, 1024 72.5 : 44.3 : 55.0, 2048 127 : 61 : 94; 16384 tokens, M = 1024 279 : 247 : 293.  Beyond sixteen tiles to an SM it depends on the units alone: 65536 tokens, M = 1024, D = 8 835 : 818,
// M = 1040 854 : 909.
constexpr double kSweepStart = 5.0, kSideCost = 5.0;
struct SweepPlan { int range, ranges, side, chunk, splits, stages, bufs; };
inline size_t range_tile_bytes(const flare_desc_t *d) {         // of one tile of every item
    return sizeof(float) * kTile * (size_t)d->B * d->H * 2 * d->D;
}
inline SweepPlan sweep_ranges(const flare_desc_t *d, int sms) {
    const int most = d->D == 32 ? 320 : 768;
    SweepPlan p{};
    p.ranges = (d->M + most - 1) / most;
    p.range = p.ranges == 1 ? d->M : ((d->M + p.ranges - 1) / p.ranges + 63) / 64 * 64;
    p.ranges = (d->M + p.range - 1) / p.range;
    p.side = 1;
    const int tiles = (d->N + kTile - 1) / kTile;
    p.chunk = p.ranges == 1 ? tiles : (int)std::min<size_t>(tiles, std::max<size_t>(1, kRangeBytes / range_tile_bytes(d)));
    p.splits = token_splits(d, p.chunk, p.range, sms, (double)d->B * d->H * d->M * d->D * 2 * sizeof(float) / 8.0e6);
    if (p.chunk < tiles) {                                      // chunks of about equal size, each a whole number of tiles to a CTA
        const int chunks = (tiles + p.chunk / p.splits * p.splits - 1) / (p.chunk / p.splits * p.splits);
        p.chunk = ((tiles + chunks - 1) / chunks + p.splits - 1) / p.splits * p.splits;
        return p;
    }
    // Side by side?  Once or twice over the chip, or a tile to a CTA.
    const long heads = (long)d->B * d->H;
    if (d->D == 32 || heads * tiles > 16L * sms) return p;
    auto cost = [&](long ctas, int each, int range) { return token_cost(ctas, each, range, sms) + (double)((ctas + sms - 1) / sms) * kSweepStart; };
    double best = p.ranges * cost(heads * p.splits, (tiles + p.splits - 1) / p.splits, p.range);
    for (int range = 64; range < d->M && range <= most; range += 64) {
        const int side = (d->M + range - 1) / range;
        if (side * range_tile_bytes(d) * tiles > kRangeBytes) continue;
        for (int rounds = 1; rounds <= 2; ++rounds) {
            const int splits = (int)std::min<long>(tiles, std::max(1L, (long)rounds * sms / (heads * side)));
            const double c = cost(heads * splits * side, (tiles + splits - 1) / splits, range) + kSideCost + (double)side * range_tile_bytes(d) * tiles / 8.0e6;
            if (c < best) {
                best = c;
                p.range = range; p.ranges = p.side = side; p.splits = splits;
            }
        }
    }
    return p;
}
inline int sweep_launches(const flare_desc_t *d, const SweepPlan &p) {
    const int tiles = (d->N + kTile - 1) / kTile;
    return p.side > 1 ? 2 : p.ranges * ((tiles + p.chunk - 1) / p.chunk);
}
inline SweepPlan dz_sweep_plan(const flare_desc_t *d, int sms) {
    SweepPlan p = sweep_ranges(d, sms);
    p.bufs = 3;
    p.stages = d->D == 32 ? BwdDzSmem<32>::stages(p.range) : BwdDzSmem<16>::stages(p.range);
    return p;
}
inline SweepPlan grad_sweep_plan(const flare_desc_t *d, int sms) {
    SweepPlan p = sweep_ranges(d, sms);
    auto stages = [&](int bufs) { return d->D == 32 ? BwdGradSmem<32>::stages(bufs, p.range) : BwdGradSmem<16>::stages(bufs, p.range); };
    // Three buffers of weights want three tile stages: the issuing warp then waits for a tile before it has issued the sums that release the last but one.
    p.bufs = stages(3) >= 3 ? 3 : 2;
    p.stages = stages(p.bufs);
    return p;
}

inline BwdLayout bwd_layout(const flare_desc_t *d, int sms) {
    BwdLayout w;
    const long rows = (long)d->B * d->H * d->M;
    const int pa = simt_plan(d, sms).P, pb = bwd_dq_plan(d, sms).P;
    w.P = pa > pb ? pa : pb;
    if (use_sweeps(d)) w.P = 2 * std::max(dz_sweep_plan(d, sms).splits, grad_sweep_plan(d, sms).splits);
    else if (use_tc(d)) w.P = std::max(w.P, std::max(dz_plan(d, sms).splits, tc_dq_plan(d, sms).P));
    size_t off = kHeaderBytes;
    w.part = off; off += align_up(sizeof(float) * (size_t)w.P * rows * d->D);
    w.dz = off;   off += align_up(sizeof(float) * (size_t)rows * d->D);
    w.de = off;   off += align_up(sizeof(float) * (size_t)rows);
    w.dd = off;   off += align_up(sizeof(float) * (use_sweeps(d) ? 2 : 1) * (size_t)d->B * d->N * d->H);
    w.e = w.around = off;                                      // D = 64, and D = 32 beyond the sweeps: see bwd_guess, z_around
    if (use_tc(d) && !use_sweeps(d)) {
        w.around = off += align_up(sizeof(float) * (size_t)d->B * d->N * d->H);
        off += align_up(sizeof(float) * (size_t)(1 + latent_blocks(d)) * d->B * d->H * d->D);
    }
    w.dd_other = w.kvacc = off;                                // over latent ranges: dd so far, and float32 sums of the rows
    if (use_sweeps(d)) {                                       // (the two sweeps one after the other, in the same place: a row of either is at least a RowSums)
        const SweepPlan p = grad_sweep_plan(d, sms);
        if (p.ranges > 1) off += align_up(range_tile_bytes(d) * p.side * p.chunk);
    } else if (token_in_ranges(d)) {
        w.kvacc = off += align_up(sizeof(float) * (size_t)d->B * d->N * d->H);
        off += align_up(sizeof(float) * 3 * (size_t)d->B * d->N * d->H * d->D);
    }
    w.total = off;
    return w;
}

// ---- what the translation units provide
int encode_simt(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *V, const uint8_t *mask,
                float *pm, float *pl, float *pacc, cudaStream_t st);
// dZ form: lse_dec given, dY in place of V, partial sums of dZ to pacc
int encode_dz_simt(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *dY, const float *lse_dec,
                   float *pacc, cudaStream_t st);
// Clears the workspace header from word `first` on (one kernel for all callers: whichever call comes first loads it).
int clear_header(void *workspace, int first, cudaStream_t st);
// Blocks per cluster of a forward in one launch on the current device, or 0.  forward_small_simt: FLARE_ERR_UNSUPPORTED, and nothing launched, where the
// stream has no room for the cluster.
int small_forward_cluster(const flare_desc_t *d);
int forward_small_simt(const flare_desc_t *d, int cluster, const void *Q, const void *K, const void *V, const uint8_t *mask, float *Z, float *lse_enc,
                       void *Y, float *lse_dec, uint32_t *header, cudaStream_t st);
int decode_simt(const flare_desc_t *d, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec, cudaStream_t st);
int bwd_token_simt(const flare_desc_t *d, const void *Q, const void *K, const void *V, const uint8_t *mask, const void *dY,
                   const float *Z, const float *dZ, const float *de, const float *lse_enc, const float *lse_dec, void *dK, void *dV,
                   float *dd, cudaStream_t st);
int bwd_dq_simt(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *V, const uint8_t *mask,
                const void *dY, const float *Z, const float *dZ, const float *de, const float *dd, const float *lse_enc,
                const float *lse_dec, float *part, cudaStream_t st);
// alone: not as part of a forward (see encode_lean_plan).  keep_status: leave the error word of the workspace header as it is (a later
// part of a call in several parts)
int encode_impl(const flare_desc_t *d, const void *Q, const void *K, const void *V, const uint8_t *mask, float *Z,
                float *lse_enc, void *ws, cudaStream_t st, bool alone, bool keep_status = false);
int encode_dz_tc(const flare_desc_t *d, const LeanPlan &p, const void *Q, const void *K, const void *dY, float *part,
                 uint32_t *status, cudaStream_t st, const float *lse_dec, const float *Z, float *around);
// range_scratch: decode_range_bytes(d) bytes, or null (then more than kDecodeMaxM latents take the CUDA-core kernel)
int decode_impl(const flare_desc_t *d, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec,
                uint32_t *status, cudaStream_t st, char *range_scratch = nullptr);
// skip_pass_a: dZ and de are already in the workspace (the second of the two runs of the separate-queries variant)
int backward_impl(const flare_desc_t *d, int sms, const void *Q, const void *K, const void *V, const uint8_t *mask, const void *Y,
                  const void *dY, const float *Z, const float *lse_enc, const float *lse_dec, float *dQ, void *dK, void *dV,
                  char *ws, cudaStream_t st, bool skip_pass_a);
size_t spectral_bytes(const flare_desc_t *d, int sms);
int spectral_gram(const flare_desc_t *d, int sms, const void *Q, const void *K, const float *lse_enc, const float *lse_dec, float *G,
                  void *workspace, cudaStream_t st);
int spectral_eig(int32_t matrices, int32_t M, float *G, float *eigenvalues, float *U, int32_t sweeps, cudaStream_t st);

}  // namespace flare
