// The CUDA-core forward kernels: float32 and float16 inputs, and the bfloat16 shapes the tensor-core kernels do not take.
#include "flare_host.h"
#include "flare_simt.cuh"

namespace flare {
namespace {

template <typename T>
int launch_encode_simt(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *V,
                       const uint8_t *mask, float *pm, float *pl, float *pacc, cudaStream_t st) {
    dim3 grid(p.splits, d->H, d->B), block(kSimtThreads);
#define FLARE_CASE(DD)                                                                                          \
    case DD:                                                                                                    \
        encode_simt_kernel<T, DD><<<grid, block, 0, st>>>((const T *)Q, (const T *)K, (const T *)V, mask, pm, pl, \
                                                          pacc, d->B, d->H, d->N, d->M, p.LM, p.chunk, d->scale); \
        break;
    switch (d->D) {
        FLARE_CASE(4) FLARE_CASE(8) FLARE_CASE(16) FLARE_CASE(32) FLARE_CASE(64)
        default: return FLARE_ERR_UNSUPPORTED;
    }
#undef FLARE_CASE
    FLARE_CUDA(cudaGetLastError());
    return FLARE_OK;
}

template <typename T>
int launch_decode_simt(const flare_desc_t *d, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec,
                       cudaStream_t st) {
    dim3 grid((d->N + kDecodeSimtThreads - 1) / kDecodeSimtThreads, d->H, d->B), block(kDecodeSimtThreads);
#define FLARE_CASE(DD)                                                                                            \
    case DD:                                                                                                      \
        decode_simt_kernel<T, DD><<<grid, block, 0, st>>>((const T *)Q, (const T *)K, Z, (T *)Y, lse_dec, d->B, d->H, \
                                                          d->N, d->M, d->scale);                                  \
        break;
    switch (d->D) {
        FLARE_CASE(4) FLARE_CASE(8) FLARE_CASE(16) FLARE_CASE(32) FLARE_CASE(64)
        default: return FLARE_ERR_UNSUPPORTED;
    }
#undef FLARE_CASE
    FLARE_CUDA(cudaGetLastError());
    return FLARE_OK;
}

}  // namespace

int encode_simt(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *V, const uint8_t *mask,
                float *pm, float *pl, float *pacc, cudaStream_t st) {
    return (d->dtype == FLARE_DTYPE_F32)   ? launch_encode_simt<float>(d, p, Q, K, V, mask, pm, pl, pacc, st)
           : (d->dtype == FLARE_DTYPE_F16) ? launch_encode_simt<__half>(d, p, Q, K, V, mask, pm, pl, pacc, st)
                                           : launch_encode_simt<__nv_bfloat16>(d, p, Q, K, V, mask, pm, pl, pacc, st);
}

int decode_simt(const flare_desc_t *d, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec, cudaStream_t st) {
    return (d->dtype == FLARE_DTYPE_F32)   ? launch_decode_simt<float>(d, Q, K, Z, Y, lse_dec, st)
           : (d->dtype == FLARE_DTYPE_F16) ? launch_decode_simt<__half>(d, Q, K, Z, Y, lse_dec, st)
                                           : launch_decode_simt<__nv_bfloat16>(d, Q, K, Z, Y, lse_dec, st);
}

}  // namespace flare
