// Decode on the tensor cores: launches of the kernel's forms, in ranges of latents where one launch cannot hold them.
#include "flare_host.h"

namespace flare {
namespace {

template <int D, int DRT, bool kPart, int kM>
int launch_decode_tc_m(const flare_desc_t *d, int sms, const void *Q, const void *K, const float *Z, void *Y,
                     float *lse_dec, uint32_t *status, cudaStream_t st, int m0, int mc, float *Ypart, bool fallback = false) {
    CUtensorMap tmK, tmQ;
    int rc;
    if ((rc = make_token_map(&tmK, K, d, kTile, D)) != FLARE_OK) return rc;
    if (DRT != 0) tmQ = tmK;   // unused: the narrow forms stage Q with their threads
    else if ((rc = make_latent_map(&tmQ, Q, d)) != FLARE_OK) return rc;
    const size_t smem = DecodeSmem<D>::total(mc);
    static std::atomic<uint64_t> smem_opt_in{0};
    if (int rc_attr = ensure_big_smem(decode_tc_kernel<D, DRT, kPart, kM>, smem_opt_in, 227 * 1024)) return rc_attr;
    DecodeTcArgs a;
    a.Q = static_cast<const __nv_bfloat16 *>(Q);
    a.Z = Z; a.Y = (__nv_bfloat16 *)Y; a.lse_dec = lse_dec; a.status = status;
    a.run_if = (fallback && status != nullptr) ? status + kRedoDecodeWord : nullptr;
    a.redo = status != nullptr ? status + kRedoDecodeWord : nullptr;
    a.B = d->B; a.H = d->H; a.N = d->N; a.M = mc;
    a.mtot = d->M; a.m0 = m0; a.Ypart = Ypart;
    a.sl2 = d->scale * kLog2e;
    a.tiles = (d->N + kTile - 1) / kTile;
    a.plan = make_decode_plan(mc, D);
    if (a.plan.cs == 0) return FLARE_ERR_UNSUPPORTED;
    long per_head = sms / ((long)d->B * d->H);
    if (per_head < 1) per_head = 1;
    if (per_head > a.tiles) per_head = a.tiles;
    dim3 grid((unsigned)per_head, d->H, d->B);
    FLARE_CUDA(launch_after(decode_tc_kernel<D, DRT, kPart, kM>, grid, kTcThreads, smem, st, tmK, tmQ, a));
    return FLARE_OK;
}

// The streaming (fast) form of decode: head widths 16 (and narrower) and 32, as many latents as fit shared memory.
template <int D>
bool decode_stream_fits(int mc) { return (D == 16 || D == 32) && DecodeStreamSmem<(D == 16 || D == 32) ? D : 16>::fits((mc + 31) & ~31); }

template <int D, int DRT, bool kPart, int kM, bool kLse>
int launch_decode_stream_l(const flare_desc_t *d, int sms, const void *Q, const void *K, const float *Z, void *Y,
                           float *lse_dec, uint32_t *status, cudaStream_t st, int m0, int mc, float *Ypart) {
    if constexpr (D == 16 || D == 32) {
        CUtensorMap tmK, tmQ;
        int rc;
        if ((rc = make_token_map(&tmK, K, d, kTile, D)) != FLARE_OK) return rc;
        if (DRT != 0) tmQ = tmK;   // unused: the narrow forms stage Q with their threads
        else if ((rc = make_latent_map(&tmQ, Q, d)) != FLARE_OK) return rc;
        const size_t smem = DecodeStreamSmem<D>::total(DecodeStreamSmem<D>::padded(mc));
        static std::atomic<uint64_t> smem_opt_in{0};
        if (int rc_attr = ensure_big_smem(decode_stream_kernel<D, DRT, kPart, kM, kLse>, smem_opt_in, 227 * 1024)) return rc_attr;
        DecodeTcArgs a;
        a.Q = static_cast<const __nv_bfloat16 *>(Q);
        a.Z = Z; a.Y = (__nv_bfloat16 *)Y; a.lse_dec = lse_dec; a.status = status;
        a.run_if = nullptr;
        a.redo = status + kRedoDecodeWord;
        a.B = d->B; a.H = d->H; a.N = d->N; a.M = mc;
        a.mtot = d->M; a.m0 = m0; a.Ypart = Ypart;
        a.sl2 = d->scale * kLog2e;
        a.tiles = (d->N + kTile - 1) / kTile;
        a.plan = DecodePlan{};
        long per_head = sms / ((long)d->B * d->H);
        const long four = (a.tiles + 3) / 4;                    // a CTA works on four tiles at a time
        if (per_head > four) per_head = four;
        if (per_head < 1) per_head = 1;
        FLARE_CUDA(launch_after(decode_stream_kernel<D, DRT, kPart, kM, kLse>, dim3((unsigned)per_head, d->H, d->B), kTcThreadsGuarded, smem, st, tmK, tmQ, a));
        return FLARE_OK;
    } else {
        return FLARE_ERR_UNSUPPORTED;
    }
}

template <int D, int DRT, bool kPart, int kM>
int launch_decode_stream_m(const flare_desc_t *d, int sms, const void *Q, const void *K, const float *Z, void *Y,
                           float *lse_dec, uint32_t *status, cudaStream_t st, int m0, int mc, float *Ypart) {
    if (lse_dec != nullptr) return launch_decode_stream_l<D, DRT, kPart, kM, true>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart);
    if constexpr (kPart) return FLARE_ERR_INVALID_ARG;          // a range of the latents always leaves its log-sum-exp
    else return launch_decode_stream_l<D, DRT, kPart, kM, false>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart);
}

// (the common latent counts as compile-time constants of the kernel)
template <int D, int DRT, bool kPart>
int launch_decode_stream(const flare_desc_t *d, int sms, const void *Q, const void *K, const float *Z, void *Y,
                         float *lse_dec, uint32_t *status, cudaStream_t st, int m0, int mc, float *Ypart) {
    if (mc == 256) return launch_decode_stream_m<D, DRT, kPart, 256>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart);
    if (mc == 128) return launch_decode_stream_m<D, DRT, kPart, 128>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart);
    if (mc == 64) return launch_decode_stream_m<D, DRT, kPart, 64>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart);
    if (mc == 512) return launch_decode_stream_m<D, DRT, kPart, 512>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart);
    return launch_decode_stream_m<D, DRT, kPart, 0>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart);
}

// The launch's range of latents is [m0, m0 + mc) (mc = 0: all of them).  The sizes that the workloads use most have
// forms of the kernel with the number of latents as a compile-time constant.  fast: the form without a row maximum
// first, then the exact form, which exits at once unless the first one found its inputs out of range (this needs
// the flag word in a workspace header: status != null).
template <int D, int DRT, bool kPart>
int launch_decode_tc_f(const flare_desc_t *d, int sms, const void *Q, const void *K, const float *Z, void *Y,
                       float *lse_dec, uint32_t *status, cudaStream_t st, int m0, int mc, float *Ypart, bool fallback) {
    if (mc == 256) return launch_decode_tc_m<D, DRT, kPart, 256>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart, fallback);
    if (mc == 128) return launch_decode_tc_m<D, DRT, kPart, 128>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart, fallback);
    if (mc == 64) return launch_decode_tc_m<D, DRT, kPart, 64>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart, fallback);
    if (mc == 32) return launch_decode_tc_m<D, DRT, kPart, 32>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart, fallback);
    if (mc == 512) return launch_decode_tc_m<D, DRT, kPart, 512>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart, fallback);
    return launch_decode_tc_m<D, DRT, kPart, 0>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart, fallback);
}

template <int D, int DRT = 0, bool kPart = false>
int launch_decode_tc(const flare_desc_t *d, int sms, const void *Q, const void *K, const float *Z, void *Y,
                     float *lse_dec, uint32_t *status, cudaStream_t st, int m0 = 0, int mc = 0, float *Ypart = nullptr,
                     bool fast = false) {
    if (mc == 0) mc = d->M;
    fast = fast && status != nullptr && decode_stream_fits<D>(mc);
    if (fast) {
        const int rc = launch_decode_stream<D, DRT, kPart>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart);
        if (rc != FLARE_OK) return rc;
    }
    return launch_decode_tc_f<D, DRT, kPart>(d, sms, Q, K, Z, Y, lse_dec, status, st, m0, mc, Ypart, fast);
}
template <int D, int DRT>
int decode_tc_any(const flare_desc_t *d, int sms, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec,
                  uint32_t *status, char *range_scratch, cudaStream_t st) {
    const bool fast = use_fast_decode(d) && status != nullptr;
    if (d->M <= kDecodeMaxM) return launch_decode_tc<D, DRT>(d, sms, Q, K, Z, Y, lse_dec, status, st, 0, 0, nullptr, fast);
    constexpr int DR = DRT ? DRT : D;
    const int C = decode_ranges(d);
    const size_t rows = (size_t)d->B * d->N * d->H;
    float *Ypart = reinterpret_cast<float *>(range_scratch);
    float *lpart = reinterpret_cast<float *>(range_scratch + align_up(sizeof(float) * C * rows * d->D));
    for (int c = 0; c < C; ++c) {
        const int m0 = c * kDecodeRange, mc = d->M - m0 < kDecodeRange ? d->M - m0 : kDecodeRange;
        const int rc = launch_decode_tc<D, DRT, true>(d, sms, Q, K, Z, nullptr, lpart + (size_t)c * rows, status, st, m0, mc,
                                                Ypart + (size_t)c * rows * DR, fast);
        if (rc != FLARE_OK) return rc;
    }
    FLARE_CUDA(launch_after(decode_combine_kernel<DR>, (unsigned)((rows + 255) / 256), 256, 0, st, Ypart, lpart, C, (long)rows, (__nv_bfloat16 *)Y, lse_dec));
    return FLARE_OK;
}

}  // namespace

// range_scratch: decode_range_bytes(d) bytes, or null (then more than kDecodeMaxM latents take the CUDA-core kernel)
int decode_impl(const flare_desc_t *d, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec,
                uint32_t *status, cudaStream_t st, char *range_scratch) {
    if (use_tc(d) && (d->M <= kDecodeMaxM || range_scratch != nullptr)) {
        const int sms = device_info().sms;
        switch (d->D) {
            case 4: return decode_tc_any<16, 4>(d, sms, Q, K, Z, Y, lse_dec, status, range_scratch, st);
            case 8: return decode_tc_any<16, 8>(d, sms, Q, K, Z, Y, lse_dec, status, range_scratch, st);
            case 16: return decode_tc_any<16, 0>(d, sms, Q, K, Z, Y, lse_dec, status, range_scratch, st);
            case 32: return decode_tc_any<32, 0>(d, sms, Q, K, Z, Y, lse_dec, status, range_scratch, st);
            default: return decode_tc_any<64, 0>(d, sms, Q, K, Z, Y, lse_dec, status, range_scratch, st);
        }
    }
    return decode_simt(d, Q, K, Z, Y, lse_dec, st);
}

}  // namespace flare
