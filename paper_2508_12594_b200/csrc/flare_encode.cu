// Encode on the tensor cores: launches of the kernel's forms, the merge of the partial results.
#include "flare_host.h"
#include "flare_enc_lean.cuh"
#include "flare_reduce.cuh"

namespace flare {
namespace {

// kAlt: one latent block (M <= 128), the CTA's two slots take alternate tiles: a form of its own with a deeper K/V ring
template <int D, bool kPair, int DRT, bool kHiLo, bool kMaskBody, bool kAlt>
int launch_encode_tc_a(const flare_desc_t *d, const TcEncodePlan &p, const void *Q, const void *K, const void *V,
                       const uint8_t *mask, float *pm, float *pl, float *pacc, uint32_t *status, cudaStream_t st, bool fallback) {
    constexpr int DG = kPair ? 2 * D : D;
    CUtensorMap tmK, tmV, tmQ;
    int rc;
    if ((rc = make_token_map(&tmK, K, d, kTile, DG)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmV, V, d, kTile, DG)) != FLARE_OK) return rc;
    if (DRT != 0) tmQ = tmK;   // unused: the narrow forms stage Q with their threads
    else if ((rc = make_latent_map(&tmQ, Q, d)) != FLARE_OK) return rc;
    const size_t smem = EncodeSmem<DG, kAlt>::total();
    static std::atomic<uint64_t> smem_opt_in{0};
    if (int rc_attr = ensure_big_smem(encode_tc_kernel<D, kPair, DRT, kHiLo, kMaskBody, kAlt>, smem_opt_in, 227 * 1024)) return rc_attr;
    EncodeTcArgs a;
    a.Q = static_cast<const __nv_bfloat16 *>(Q);
    a.key_mask = mask; a.part_m = pm; a.part_l = pl; a.part_acc = pacc; a.status = status;
    a.run_if = fallback ? status + kRedoEncodeWord : nullptr;
    a.B = d->B; a.H = d->H; a.N = d->N; a.M = d->M;
    a.scale = d->scale; a.sl2 = d->scale * kLog2e;
    a.tiles = p.tiles; a.splits = p.splits; a.pairs = p.pairs; a.partials_per_split = p.per_split;
    dim3 grid(p.splits, (kPair ? d->H / 2 : d->H) * p.pairs, d->B);
    FLARE_CUDA(launch_after(encode_tc_kernel<D, kPair, DRT, kHiLo, kMaskBody, kAlt>, grid, kTcThreads, smem, st, tmK, tmV, tmQ, a));
    return FLARE_OK;
}

template <int D, bool kPair, int DRT, bool kHiLo, bool kMaskBody>
int launch_encode_tc(const flare_desc_t *d, const TcEncodePlan &p, const void *Q, const void *K, const void *V,
                     const uint8_t *mask, float *pm, float *pl, float *pacc, uint32_t *status, cudaStream_t st, bool fallback) {
    if constexpr (kPair) {
        return launch_encode_tc_a<D, kPair, DRT, kHiLo, kMaskBody, true>(d, p, Q, K, V, mask, pm, pl, pacc, status, st, fallback);
    } else {
        // (one latent block is only reached with the element tests, see encode_impl)
        if constexpr (kMaskBody)
            if (d->M <= kTile)
                return launch_encode_tc_a<D, kPair, DRT, kHiLo, kMaskBody, true>(d, p, Q, K, V, mask, pm, pl, pacc, status, st, fallback);
        return launch_encode_tc_a<D, kPair, DRT, kHiLo, kMaskBody, false>(d, p, Q, K, V, mask, pm, pl, pacc, status, st, fallback);
    }
}

template <int D, bool kPair, int kKind, int DRT, bool kMask>
int launch_lean_m(const flare_desc_t *d, const LeanPlan &p, const void *Q, const void *K, const void *V, EncodeLeanArgs a, cudaStream_t st) {
    constexpr int DG = kPair ? 2 * D : D;
    using LG = LeanGeom<DG, kKind>;
    CUtensorMap tmK, tmV;
    int rc;
    if ((rc = make_token_map(&tmK, K, d, kTile, DG)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmV, V, d, kTile, DG)) != FLARE_OK) return rc;
    static std::atomic<uint64_t> smem_opt_in{0};
    if ((rc = ensure_big_smem(encode_lean_kernel<D, kPair, kKind, DRT, kMask>, smem_opt_in, 227 * 1024)) != FLARE_OK) return rc;
    a.Q = static_cast<const __nv_bfloat16 *>(Q);
    a.B = d->B; a.H = d->H; a.N = d->N; a.M = d->M;
    a.sl2 = d->scale * kLog2e;
    a.tiles = p.tiles; a.splits = p.splits; a.blocks = p.blocks;
    FLARE_CUDA(launch_after(encode_lean_kernel<D, kPair, kKind, DRT, kMask>, dim3((kPair ? d->H / 2 : d->H) * p.blocks, p.splits, d->B), LG::kThreads, LG::total, st, tmK, tmV, a));
    return FLARE_OK;
}
template <int D, bool kPair, int kKind, int DRT>
int launch_lean_k(const flare_desc_t *d, const LeanPlan &p, const void *Q, const void *K, const void *V, const EncodeLeanArgs &a, cudaStream_t st) {
    if constexpr (kKind != kLeanDz)
        if (a.key_mask != nullptr || (kKind == kLeanHiLo && d->N % kTile != 0)) return launch_lean_m<D, kPair, kKind, DRT, true>(d, p, Q, K, V, a, st);
    return launch_lean_m<D, kPair, kKind, DRT, false>(d, p, Q, K, V, a, st);
}
template <int kKind>
int launch_lean(const flare_desc_t *d, const LeanPlan &p, const void *Q, const void *K, const void *V, const EncodeLeanArgs &a, cudaStream_t st) {
    // (dZ: what the two sweeps of the backward do not take, no narrow heads and more than 64 latents or heads 64 wide)
    if constexpr (kKind == kLeanDz)
        return d->D == 32 ? launch_lean_k<32, false, kKind, 0>(d, p, Q, K, V, a, st) : launch_lean_k<64, false, kKind, 0>(d, p, Q, K, V, a, st);
    const bool pair = lean_pairs(d);
    if constexpr (kKind != kLeanDz) switch (d->D) {
        case 4: return launch_lean_k<16, false, kKind, 4>(d, p, Q, K, V, a, st);
        case 8: return pair ? launch_lean_k<8, true, kKind, 0>(d, p, Q, K, V, a, st) : launch_lean_k<16, false, kKind, 8>(d, p, Q, K, V, a, st);
        case 16: return pair ? launch_lean_k<16, true, kKind, 0>(d, p, Q, K, V, a, st) : launch_lean_k<16, false, kKind, 0>(d, p, Q, K, V, a, st);
        case 32: return pair ? launch_lean_k<32, true, kKind, 0>(d, p, Q, K, V, a, st) : launch_lean_k<32, false, kKind, 0>(d, p, Q, K, V, a, st);
        default: return FLARE_ERR_UNSUPPORTED;                  // (use_fast_encode knows none)
    }
}

}  // namespace

int encode_impl(const flare_desc_t *d, const void *Q, const void *K, const void *V, const uint8_t *mask, float *Z,
                float *lse_enc, void *ws, cudaStream_t st, bool alone, bool keep_status) {
    const DeviceView di = device_info();
    const long rows = (long)d->B * d->H * d->M;
    const int P = partials_for(d, di.sms, alone);
    WorkspaceLayout w = make_layout(P, rows, d->D, false);
    char *base = static_cast<char *>(ws);
    float *pm = reinterpret_cast<float *>(base + w.part_m);
    float *pl = reinterpret_cast<float *>(base + w.part_l);
    float *pacc = reinterpret_cast<float *>(base + w.part_acc);
    int rc, parts = P, parts_redo = 0;                         // partial results, and those of the exact form if it replaced them
    const uint32_t *redo = nullptr;
    if (use_tc(d)) {
        if ((rc = clear_header(base, keep_status ? 1 : 0, st)) != FLARE_OK) return rc;
        TcEncodePlan p = tc_encode_plan(d, di.sms);
        uint32_t *status = reinterpret_cast<uint32_t *>(base);
        // a caller that asks for lse_enc is saving Z for the backward: weights as two bf16 halves (see exp_chunk_hilo)
        const bool fast = use_fast_encode(d);
        if (fast) {                                             // the exact form, behind it, exits at once unless the fast one raised its flag
            const LeanPlan lp = encode_lean_plan(d, di.sms, alone);
            EncodeLeanArgs a{};
            a.key_mask = mask; a.part_m = pm; a.part_l = pl; a.part_acc = pacc; a.status = status; a.redo = status + kRedoEncodeWord;
            rc = lse_enc != nullptr ? launch_lean<kLeanHiLo>(d, lp, Q, K, V, a, st) : launch_lean<kLeanFast>(d, lp, Q, K, V, a, st);
            if (rc != FLARE_OK) return rc;
            parts = lp.splits; parts_redo = p.P; redo = a.redo;
        } else {
            parts = p.P;
        }
#define FLARE_ENC3(DD, PAIR, DRT, MB, HL) launch_encode_tc<DD, PAIR, DRT, HL, MB>(d, p, Q, K, V, mask, pm, pl, pacc, status, st, fast)
#define FLARE_ENC2(DD, PAIR, DRT, MB) (lse_enc != nullptr ? FLARE_ENC3(DD, PAIR, DRT, MB, true) : FLARE_ENC3(DD, PAIR, DRT, MB, false))
        // A call with a key mask has padding in every tile and takes the form that tests every element (see
        // encode_tc_kernel).  Without a mask only a last partial tile has padding and either form serves; which one
        // is faster was measured (B200): the form without the element tests where a CTA holds two latent blocks
        // (M > 128: 0.80 -> 0.68 ms on the million-point shape, 223 -> 201 us at N = 131072, M = 512), the other
        // where two slots share one block (M <= 128: 4-5 % apart).
        const bool mask_body = mask != nullptr || d->M <= kTile;
#define FLARE_ENC(DD, PAIR, DRT) (mask_body ? FLARE_ENC2(DD, PAIR, DRT, true) : FLARE_ENC2(DD, PAIR, DRT, false))
        if (encode_head_pairs(d))
            rc = d->D == 16 ? FLARE_ENC(16, true, 0) : FLARE_ENC(32, true, 0);
        else
            rc = d->D == 4    ? FLARE_ENC(16, false, 4)
                 : d->D == 8  ? FLARE_ENC(16, false, 8)
                 : d->D == 16 ? FLARE_ENC(16, false, 0)
                 : d->D == 32 ? FLARE_ENC(32, false, 0)
                              : FLARE_ENC(64, false, 0);
#undef FLARE_ENC
#undef FLARE_ENC2
#undef FLARE_ENC3
    } else {
        SimtPlan p = simt_plan(d, di.sms);
        rc = encode_simt(d, p, Q, K, V, mask, pm, pl, pacc, st);
    }
    if (rc != FLARE_OK) return rc;
    // (the CUDA-core kernels leave nothing in the header: the merge clears it)
    FLARE_REDUCE(merge_kernel, rows, parts, d->D, st, pm, pl, pacc, Z, lse_enc, parts, redo, parts_redo, rows, use_tc(d) || keep_status ? nullptr : static_cast<uint32_t *>(ws));
    return FLARE_OK;
}

// Pass A of the backward: dY for V, lse_dec the decode log-sum-exp rows; partial sums to `part`.
int encode_dz_tc(const flare_desc_t *d, const LeanPlan &p, const void *Q, const void *K, const void *dY, float *part,
                 uint32_t *status, cudaStream_t st, const float *lse_dec, const float *Z, float *around) {
    EncodeLeanArgs a{};
    a.Z = Z; a.around = around;
    a.lse_dec = lse_dec; a.part_acc = part; a.status = status;
    return launch_lean<kLeanDz>(d, p, Q, K, dY, a, st);
}

}  // namespace flare
