// Backward: plans, workspace layout, launches of the tensor-core and CUDA-core kernels.
#include "flare_host.h"
#include "flare_bwd_sweep.cuh"
#include "flare_bwd_tc.cuh"
#include "flare_reduce.cuh"

namespace flare {
namespace {

// padded tokens: a key mask, or a last partial tile
bool has_padding(const flare_desc_t *d, const uint8_t *mask) { return mask != nullptr || d->N % kTile != 0; }

template <int D, bool kPadded>
int launch_bwd_dq_tc_n(const flare_desc_t *d, const TcEncodePlan &p, const void *K, const void *V, const void *dY, const BwdDqTcArgs &args,
                       cudaStream_t st) {
    CUtensorMap tmK, tmV, tmG;
    int rc;
    if ((rc = make_token_map(&tmK, K, d, kTile, D)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmV, V, d, kTile, D)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmG, dY, d, kTile, D)) != FLARE_OK) return rc;
    static std::atomic<uint64_t> smem_opt_in{0};
    if ((rc = ensure_big_smem(bwd_dq_tc_kernel<D, kPadded>, smem_opt_in)) != FLARE_OK) return rc;
    FLARE_CUDA(launch_after(bwd_dq_tc_kernel<D, kPadded>, dim3(d->H * p.pairs, p.splits, d->B), kDqThreads, BwdDqSmem<D>::total, st, tmK, tmV, tmG, args));
    return FLARE_OK;
}

template <int D>
int launch_bwd_dq_tc(const flare_desc_t *d, const TcEncodePlan &p, const void *Q, const void *K, const void *V, const void *dY,
                     const uint8_t *mask, const float *Z, const float *dZ, const float *lse_enc, const float *de,
                     const float *lse_dec, const float *dd, const float *around, float *part, uint32_t *status, cudaStream_t st) {
    BwdDqTcArgs a;
    a.around = around; a.around_rows = 1 + latent_blocks(d);
    a.Q = static_cast<const __nv_bfloat16 *>(Q);
    a.Z = Z; a.dZ = dZ; a.lse_enc = lse_enc; a.de = de; a.lse_dec = lse_dec; a.dd = dd;
    a.key_mask = mask; a.part = part; a.status = status;
    a.B = d->B; a.H = d->H; a.N = d->N; a.M = d->M;
    a.sl2 = d->scale * kLog2e;
    a.tiles = p.tiles; a.splits = p.splits; a.blocks = p.pairs;
    return has_padding(d, mask) ? launch_bwd_dq_tc_n<D, true>(d, p, K, V, dY, a, st) : launch_bwd_dq_tc_n<D, false>(d, p, K, V, dY, a, st);
}

template <int D, bool kRanges>
int launch_bwd_token_tc_n(const flare_desc_t *d, int sms, const void *K, const void *V, const void *dY, BwdTokTcArgs a, cudaStream_t st) {
    CUtensorMap tmK, tmV, tmG;
    int rc;
    if ((rc = make_token_map(&tmK, K, d, kTile, D)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmV, V, d, kTile, D)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmG, dY, d, kTile, D)) != FLARE_OK) return rc;
    using SM = BwdTokSmem<D>;
    a.stages = SM::stages(a.M);
    if (a.stages < 1) return FLARE_ERR_UNSUPPORTED;
    static std::atomic<uint64_t> smem_opt_in{0};
    if ((rc = ensure_big_smem(bwd_token_tc_kernel<D, kRanges>, smem_opt_in)) != FLARE_OK) return rc;
    a.tiles = (d->N + kTile - 1) / kTile;
    FLARE_CUDA(launch_after(bwd_token_tc_kernel<D, kRanges>, dim3((unsigned)token_splits(d, a.tiles, a.M, sms), d->H, d->B), SM::kThreads, SM::total(a.stages, a.M), st, tmK, tmV, tmG, a));
    return FLARE_OK;
}

// The launch's range of latents is [m0, m0 + mc); dd_sums, kvacc: see BwdTokTcArgs.
template <int D>
int launch_bwd_token_tc(const flare_desc_t *d, int sms, const void *Q, const void *K, const void *V, const void *dY,
                        const uint8_t *mask, const float *Z, const float *dZ, const float *lse_enc, const float *de,
                        const float *lse_dec, const float *around, const float *e, void *dK, void *dV, float *dd, uint32_t *status, cudaStream_t st, int m0, int mc,
                        const float *dd_sums, float *kvacc) {
    BwdTokTcArgs a;
    a.Q = static_cast<const __nv_bfloat16 *>(Q);
    a.Z = Z; a.dZ = dZ; a.lse_enc = lse_enc; a.de = de; a.lse_dec = lse_dec; a.key_mask = mask;
    a.around = around; a.around_rows = 1 + latent_blocks(d); a.e = e;
    a.dK = (__nv_bfloat16 *)dK; a.dV = (__nv_bfloat16 *)dV; a.dd = dd; a.status = status;
    a.B = d->B; a.H = d->H; a.N = d->N; a.M = mc;
    a.mtot = d->M; a.m0 = m0; a.first = m0 == 0; a.last = m0 + mc >= d->M; a.kvacc = kvacc; a.dd_sums = dd_sums;
    a.scale = d->scale; a.sl2 = d->scale * kLog2e;
    return token_in_ranges(d) ? launch_bwd_token_tc_n<D, true>(d, sms, K, V, dY, a, st) : launch_bwd_token_tc_n<D, false>(d, sms, K, V, dY, a, st);
}

template <int D, int DRT, bool kRanges>
int launch_dz_sweep(const flare_desc_t *d, const SweepPlan &p, const void *K, const void *dY, const BwdDzArgs &a, cudaStream_t st) {
    CUtensorMap tmK, tmG;
    int rc;
    if ((rc = make_token_map(&tmK, K, d, kTile, D)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmG, dY, d, kTile, D)) != FLARE_OK) return rc;
    static std::atomic<uint64_t> smem_opt_in{0};
    if ((rc = ensure_big_smem(bwd_dz_sweep_kernel<D, DRT, kRanges>, smem_opt_in)) != FLARE_OK) return rc;
    FLARE_CUDA(launch_after(bwd_dz_sweep_kernel<D, DRT, kRanges>, dim3((unsigned)(std::min(p.splits, a.tiles) * p.side), d->H, d->B), kSwThreads, BwdDzSmem<D>::total(p.stages, p.range), st,
                            tmK, tmG, a));
    return FLARE_OK;
}

template <int D, int DRT, bool kRanges>
int launch_grad_sweep(const flare_desc_t *d, const SweepPlan &p, const void *K, const void *V, const void *dY, const BwdGradArgs &a, cudaStream_t st) {
    CUtensorMap tmK, tmV, tmG, tmDK, tmDV;
    int rc;
    if ((rc = make_token_map(&tmK, K, d, kTile, D)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmV, V, d, kTile, D)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmG, dY, d, kTile, D)) != FLARE_OK) return rc;
    constexpr int out = DRT == 4 ? D : DRT ? DRT : D;           // (rows of 8 bytes do not leave by such copies)
    if ((rc = make_token_map(&tmDK, a.dK, d, kTile, out)) != FLARE_OK) return rc;
    if ((rc = make_token_map(&tmDV, a.dV, d, kTile, out)) != FLARE_OK) return rc;
    static std::atomic<uint64_t> smem_opt_in{0};
    if ((rc = ensure_big_smem(bwd_grad_sweep_kernel<D, DRT, kRanges>, smem_opt_in)) != FLARE_OK) return rc;
    FLARE_CUDA(launch_after(bwd_grad_sweep_kernel<D, DRT, kRanges>, dim3((unsigned)(std::min(p.splits, a.tiles) * p.side), d->H, d->B), kSwThreads, BwdGradSmem<D>::total(p.bufs, p.stages, p.range), st,
                            tmK, tmV, tmG, tmDK, tmDV, a));
    return FLARE_OK;
}

// bfloat16 backward of heads up to 32 wide.  skip_pass_a: as below
template <int D, int DRT>
int backward_sweeps(const flare_desc_t *d, int sms, const void *Q, const void *K, const void *V, const uint8_t *mask, const void *dY, const float *Z,
                    const float *lse_enc, const float *lse_dec, float *dQ, void *dK, void *dV, char *ws, cudaStream_t st, bool skip_pass_a) {
    const BwdLayout w = bwd_layout(d, sms);
    auto at = [&](size_t off) { return reinterpret_cast<float *>(ws + off); };
    const long rows = (long)d->B * d->H * d->M;
    const int tiles = (d->N + kTile - 1) / kTile;
    uint32_t *status = reinterpret_cast<uint32_t *>(ws);
    if (const int rc = clear_header(ws, 0, st)) return rc;
    // One launch per range of latents and chunk of tokens: all ranges over one chunk before the next.  Side by side all of them in one.
    auto sweep = [&](const SweepPlan &p, auto &&launch) -> int {
        if (p.side > 1) return launch(0, tiles, 0, p.range);
        for (int t0 = 0; t0 < tiles; t0 += p.chunk)
            for (int m0 = 0; m0 < d->M; m0 += p.range)
                if (const int rc = launch(t0, std::min(p.chunk, tiles - t0), m0, std::min(p.range, d->M - m0))) return rc;
        return FLARE_OK;
    };
    if (!skip_pass_a) {
        const SweepPlan p = dz_sweep_plan(d, sms);
        if (p.stages < p.bufs) return FLARE_ERR_UNSUPPORTED;
        if (const int rc = sweep(p, [&](int t0, int nt, int m0, int mc) -> int {
                const BwdDzArgs a{static_cast<const __nv_bfloat16 *>(Q), Z, lse_dec, at(w.part), at(w.dd), status, d->B, d->H, d->N, mc, d->M, m0, m0 == 0,
                                  p.side == 1 && m0 + mc >= d->M, reinterpret_cast<float4 *>(ws + w.dd_other), d->scale * kLog2e, nt, p.stages, t0, p.side};
                if (p.ranges == 1) return launch_dz_sweep<D, DRT, false>(d, p, K, dY, a, st);
                if constexpr (D == 16) return launch_dz_sweep<D, DRT, true>(d, p, K, dY, a, st);
                return FLARE_ERR_UNSUPPORTED;                   // (ranges at D = 32: see use_sweeps)
            }))
            return rc;
        if (p.side > 1)
            FLARE_CUDA(launch_after(bwd_join_dd_kernel<kReduceThreads>, dim3((unsigned)(((size_t)d->B * d->H * tiles * kTile + kReduceThreads - 1) / kReduceThreads)), kReduceThreads, 0, st, reinterpret_cast<const float4 *>(ws + w.dd_other), at(w.dd),
                                    p.side, d->B * d->H, d->N, tiles));
        const int slices = reduce_slices(2 * p.splits, d->D);
        const unsigned row_blocks = reduce_blocks(rows, d->D, slices);
        FLARE_CUDA(launch_after(bwd_dz_reduce_kernel<(DRT ? DRT : D) / 4>, row_blocks, kReduceThreads, 0, st, at(w.part), Z, at(w.dz), at(w.de), 2 * p.splits, rows, slices,
                                (int)row_blocks, GuessArgs{}));
    }
    const SweepPlan p = grad_sweep_plan(d, sms);
    if (p.stages < p.bufs || BwdGradSmem<D>::log2_accs(p.range) < 0) return FLARE_ERR_UNSUPPORTED;
    if (const int rc = sweep(p, [&](int t0, int nt, int m0, int mc) -> int {
            const BwdGradArgs a{static_cast<const __nv_bfloat16 *>(Q), Z, at(w.dz), lse_enc, at(w.de), lse_dec, at(w.dd), mask, static_cast<__nv_bfloat16 *>(dK),
                                static_cast<__nv_bfloat16 *>(dV), at(w.part), status, d->B, d->H, d->N, mc, d->M, m0, m0 == 0, p.side == 1 && m0 + mc >= d->M,
                                at(w.kvacc), d->scale, d->scale * kLog2e, nt, p.stages, p.bufs, t0, p.side};
            if (p.ranges == 1) return launch_grad_sweep<D, DRT, false>(d, p, K, V, dY, a, st);
            if constexpr (D == 16) return launch_grad_sweep<D, DRT, true>(d, p, K, V, dY, a, st);
            return FLARE_ERR_UNSUPPORTED;
        }))
        return rc;
    if (p.side > 1)
        FLARE_CUDA(launch_after(bwd_join_rows_kernel<DRT ? DRT : D, kReduceThreads>, dim3((unsigned)(((size_t)2 * d->B * d->H * tiles * (d->D / 4) * kTile + kReduceThreads - 1) / kReduceThreads)), kReduceThreads, 0, st,
                                reinterpret_cast<const float4 *>(ws + w.kvacc), static_cast<__nv_bfloat16 *>(dK), static_cast<__nv_bfloat16 *>(dV), p.side, d->B, d->H, d->N, tiles, d->scale));
    FLARE_REDUCE(bwd_dq_reduce_kernel, (long)d->H * d->M, d->B * 2 * p.splits, d->D, st, at(w.part), dQ, 2 * p.splits, d->B, (long)d->H * d->M, d->scale);
    return FLARE_OK;
}

template <typename T, int D>
int launch_backward_simt(const flare_desc_t *d, int sms, const void *Q, const void *K, const void *V,
                         const uint8_t *mask, const void *Y, const void *dY, const float *Z, const float *lse_enc,
                         const float *lse_dec, float *dQ, void *dK, void *dV, char *ws, cudaStream_t st,
                         bool skip_pass_a = false) {
    // skip_pass_a: dZ and de are already in the workspace (the second of the two runs of the separate-queries variant)
    if constexpr (std::is_same<T, __nv_bfloat16>::value && D <= 32) {
        if (use_sweeps(d))
            return backward_sweeps<D < 16 ? 16 : D, D < 16 ? D : 0>(d, sms, Q, K, V, mask, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a);
    }
    const BwdLayout w = bwd_layout(d, sms);
    float *part = reinterpret_cast<float *>(ws + w.part);
    float *dZ = reinterpret_cast<float *>(ws + w.dz);
    float *de = reinterpret_cast<float *>(ws + w.de);
    float *dd = reinterpret_cast<float *>(ws + w.dd);
    const long rows = (long)d->B * d->H * d->M;
    const SimtPlan pa = simt_plan(d, sms), pb = bwd_dq_plan(d, sms);
    float *around = reinterpret_cast<float *>(ws + w.around), *e = reinterpret_cast<float *>(ws + w.e);
    if (const int rc = clear_header(ws, 0, st)) return rc;
    int dz_parts = pa.P;
    bool dz_on_tc = skip_pass_a;
    if constexpr (std::is_same<T, __nv_bfloat16>::value && D >= 32) {
        if (!skip_pass_a && use_tc(d)) {
            const LeanPlan tp = dz_plan(d, sms);
            uint32_t *status = reinterpret_cast<uint32_t *>(ws);
            const int rc = encode_dz_tc(d, tp, Q, K, dY, part, status, st, lse_dec, Z, around);
            if (rc != FLARE_OK) return rc;
            dz_parts = tp.splits;
            dz_on_tc = true;
        }
    }
    if (!dz_on_tc) {
        if (const int rc = encode_dz_simt(d, pa, Q, K, dY, lse_dec, part, st)) return rc;
    }
    if (!skip_pass_a) {
        GuessArgs guess{static_cast<const __nv_bfloat16 *>(Y), static_cast<const __nv_bfloat16 *>(dY), around, e, d->H, d->N, latent_blocks(d), 0, 0, 0};
        unsigned guess_blocks = 0;                              // (the CUDA-core kernels have no use for e)
        if (dz_on_tc) {
            const GuessPlan g = guess_plan(d, sms);
            guess.chunk = g.chunk; guess.chunks = g.chunks; guess.groups = g.groups;
            guess_blocks = (unsigned)((long)d->B * g.chunks * g.groups);
        }
        const int slices = reduce_slices(dz_parts, D);
        const unsigned row_blocks = reduce_blocks(rows, D, slices);
        FLARE_CUDA(launch_after(bwd_dz_reduce_kernel<D / 4>, row_blocks + guess_blocks, kReduceThreads, 0, st, part, Z, dZ, de, dz_parts, rows, slices,
                                (int)row_blocks, guess));
    }
    bool on_tc = false;
    int dq_parts = pb.P;
    if constexpr (std::is_same<T, __nv_bfloat16>::value && D >= 32) {
        uint32_t *status = reinterpret_cast<uint32_t *>(ws);
        on_tc = use_tc(d);
        if (on_tc) {
            // more latents than one launch holds are worked off in ranges; dd alternates between two arrays, the last range's is w.dd
            float *kvacc = reinterpret_cast<float *>(ws + w.kvacc), *dd_other = reinterpret_cast<float *>(ws + w.dd_other);
            const int R = token_range(d), ranges = (d->M + R - 1) / R;
            for (int k = 0; k < ranges; ++k) {
                const int m0 = k * R;
                const bool to_dd = (ranges - 1 - k) % 2 == 0;
                if (const int rc = launch_bwd_token_tc<D>(d, sms, Q, K, V, dY, mask, Z, dZ, lse_enc, de, lse_dec, around, e, dK, dV, to_dd ? dd : dd_other, status,
                                                                st, m0, d->M - m0 < R ? d->M - m0 : R, to_dd ? dd_other : dd, kvacc))
                    return rc;
            }
            const TcEncodePlan p = tc_dq_plan(d, sms);
            if (const int rc = launch_bwd_dq_tc<D>(d, p, Q, K, V, dY, mask, Z, dZ, lse_enc, de, lse_dec, dd, around, part, status, st)) return rc;
            dq_parts = p.P;
        }
    }
    if (!on_tc) {
        if (const int rc = bwd_token_simt(d, Q, K, V, mask, dY, Z, dZ, de, lse_enc, lse_dec, dK, dV, dd, st)) return rc;
        if (const int rc = bwd_dq_simt(d, pb, Q, K, V, mask, dY, Z, dZ, de, dd, lse_enc, lse_dec, part, st)) return rc;
    }
    FLARE_REDUCE(bwd_dq_reduce_kernel, (long)d->H * d->M, d->B * dq_parts, D, st, part, dQ, dq_parts, d->B, (long)d->H * d->M, d->scale);
    return FLARE_OK;
}

template <typename T>
int backward_simt(const flare_desc_t *d, int sms, const void *Q, const void *K, const void *V, const uint8_t *mask,
                  const void *Y, const void *dY, const float *Z, const float *lse_enc, const float *lse_dec, float *dQ,
                  void *dK, void *dV, char *ws, cudaStream_t st, bool skip_pass_a) {
    switch (d->D) {
        case 4: return launch_backward_simt<T, 4>(d, sms, Q, K, V, mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a);
        case 8: return launch_backward_simt<T, 8>(d, sms, Q, K, V, mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a);
        case 16: return launch_backward_simt<T, 16>(d, sms, Q, K, V, mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a);
        case 32: return launch_backward_simt<T, 32>(d, sms, Q, K, V, mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a);
        case 64: return launch_backward_simt<T, 64>(d, sms, Q, K, V, mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a);
        default: return FLARE_ERR_UNSUPPORTED;
    }
}

}  // namespace

int backward_impl(const flare_desc_t *d, int sms, const void *Q, const void *K, const void *V, const uint8_t *mask, const void *Y,
                  const void *dY, const float *Z, const float *lse_enc, const float *lse_dec, float *dQ, void *dK, void *dV,
                  char *ws, cudaStream_t st, bool skip_pass_a) {
    return d->dtype == FLARE_DTYPE_F32
               ? backward_simt<float>(d, sms, Q, K, V, mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a)
           : d->dtype == FLARE_DTYPE_F16
               ? backward_simt<__half>(d, sms, Q, K, V, mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a)
               : backward_simt<__nv_bfloat16>(d, sms, Q, K, V, mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, ws, st, skip_pass_a);
}

}  // namespace flare
