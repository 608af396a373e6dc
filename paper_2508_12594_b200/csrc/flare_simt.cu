// Launches of the CUDA-core kernels: float32 and float16 inputs, and the bfloat16 shapes the tensor-core kernels do not take.
#include "flare_host.h"
#include "flare_simt.cuh"
#include "flare_bwd.cuh"

namespace flare {
namespace {

template <typename T, int D, int RB, bool kDz>
int launch_encode(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *V, const uint8_t *mask,
                  const float *lse_dec, float *pm, float *pl, float *pacc, cudaStream_t st) {
    const size_t smem = encode_simt_smem<T, D>(RB);
    static std::atomic<uint64_t> opt_in{0};
    if (smem > 48 * 1024)
        if (int rc = ensure_big_smem(encode_simt_kernel<T, D, RB, kDz>, opt_in, (int)smem)) return rc;
    FLARE_CUDA(launch_after(encode_simt_kernel<T, D, RB, kDz>, dim3(p.splits, d->H * p.mblocks, d->B), kSimtThreads, smem, st,
                            (const T *)Q, (const T *)K, (const T *)V, mask, lse_dec, pm, pl, pacc, d->B, d->H, d->N, d->M, p.WM, p.mblocks, p.chunk, d->scale));
    return FLARE_OK;
}
template <typename T, int D>
struct Encode {
    template <typename... A>
    static int run(bool dz, const flare_desc_t *d, const SimtPlan &p, A... a) {
        constexpr int RB = D <= 16 ? 4 : D == 32 ? 2 : 1;       // (simt_row_blocks)
        if (p.RB == 1) return dz ? launch_encode<T, D, 1, true>(d, p, a...) : launch_encode<T, D, 1, false>(d, p, a...);
        return dz ? launch_encode<T, D, RB, true>(d, p, a...) : launch_encode<T, D, RB, false>(d, p, a...);
    }
};

template <typename T, int D>
struct Decode {
    template <int RB>
    static int launch(const flare_desc_t *d, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec, cudaStream_t st) {
        const size_t smem = decode_simt_smem<T, D>();
        static std::atomic<uint64_t> opt_in{0};
        if (smem > 48 * 1024)
            if (int rc = ensure_big_smem(decode_simt_kernel<T, D, RB>, opt_in, (int)smem)) return rc;
        FLARE_CUDA(launch_after(decode_simt_kernel<T, D, RB>, dim3((d->N + 64 * RB - 1) / (64 * RB), d->H, d->B), kSimtThreads, smem, st,
                                (const T *)Q, (const T *)K, Z, (T *)Y, lse_dec, d->B, d->H, d->N, d->M, d->scale));
        return FLARE_OK;
    }
    static int run(const flare_desc_t *d, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec, cudaStream_t st) {
        constexpr int RB = D <= 16 ? 4 : D == 32 ? 2 : 1;
        // few tokens: smaller blocks of them, so that more SMs take part
        if ((long)d->B * d->H * ((d->N + 64 * RB - 1) / (64 * RB)) < 2L * device_info().sms) return launch<1>(d, Q, K, Z, Y, lse_dec, st);
        return launch<RB>(d, Q, K, Z, Y, lse_dec, st);
    }
};

// Whether the device can place a cluster of forward_small_simt_kernel, asked once per device: sixteen blocks are not a portable size, and where a
// partition of the GPU has no group of SMs with room for them a launch is refused.
template <typename T, int D, int CS>
bool small_cluster_fits() {
    static std::atomic<uint64_t> asked{0}, fits{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaGetLastError(), false;
    const uint64_t bit = 1ull << dev;
    if (!(asked.load(std::memory_order_acquire) & bit)) {
        auto kernel = forward_small_simt_kernel<T, D, CS>;
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = CS; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(CS); cfg.blockDim = dim3(kSimtThreads); cfg.dynamicSmemBytes = forward_small_smem<T, D>();
        cfg.attrs = &attr; cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes) != cudaSuccess ||
            (CS > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
            cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            clusters = 0;
        }
        if (clusters > 0) fits.fetch_or(bit, std::memory_order_relaxed);
        asked.fetch_or(bit, std::memory_order_release);
    }
    return fits.load(std::memory_order_relaxed) & bit;
}

template <typename T, int D>
struct SmallFits {
    static int run(int cluster) {
        if constexpr (D > 32) return 0;
        else return cluster == 16 ? small_cluster_fits<T, D, 16>() : small_cluster_fits<T, D, 8>();
    }
};

template <typename T, int D>
struct SmallForward {
    static int run(const flare_desc_t *d, int cluster, const void *Q, const void *K, const void *V, const uint8_t *mask, float *Z, float *lse_enc,
                   void *Y, float *lse_dec, uint32_t *header, cudaStream_t st) {
        if constexpr (D > 32) {
            return FLARE_ERR_UNSUPPORTED;
        } else {
            const size_t partials_at = encode_simt_smem<T, D>(1);
            int WM = 1;
            while (WM * 8 < d->M) WM *= 2;
            auto launch = [&](auto size) -> int {
                constexpr int CS = decltype(size)::value;
                const int chunk = ((d->N + CS - 1) / CS + 7) / 8 * 8;
                const cudaError_t e = launch_after(forward_small_simt_kernel<T, D, CS>, dim3(CS, d->H, d->B), kSimtThreads, forward_small_smem<T, D>(), st,
                                                   (const T *)Q, (const T *)K, (const T *)V, mask, Z, lse_enc, (T *)Y, lse_dec, header, d->H, d->N, d->M,
                                                   WM, chunk, d->scale, (int)partials_at);
                if (e == cudaErrorInvalidClusterSize || e == cudaErrorLaunchOutOfResources) {   // (the stream's part of the GPU is smaller than the device's)
                    cudaGetLastError();
                    return FLARE_ERR_UNSUPPORTED;
                }
                FLARE_CUDA(e);
                return FLARE_OK;
            };
            return cluster == 16 ? launch(std::integral_constant<int, 16>{}) : launch(std::integral_constant<int, 8>{});
        }
    }
};

template <typename T, int D>
struct Token {
    static int run(const flare_desc_t *d, const void *Q, const void *K, const void *V, const uint8_t *mask, const void *dY, const float *Z,
                   const float *dZ, const float *de, const float *lse_enc, const float *lse_dec, void *dK, void *dV, float *dd, cudaStream_t st) {
        constexpr int rows = BwdSimtGeom<D>::kTokRows;
        static std::atomic<uint64_t> opt_in{0};
        const size_t smem = bwd_token_simt_smem<T, D>();
        if (smem > 48 * 1024)
            if (int rc = ensure_big_smem(bwd_token_simt_kernel<T, D>, opt_in, (int)smem)) return rc;
        FLARE_CUDA(launch_after(bwd_token_simt_kernel<T, D>, dim3((d->N + rows - 1) / rows, d->H, d->B), BwdSimtGeom<D>::kTokThreads, smem, st,
                                (const T *)Q, (const T *)K, (const T *)V, mask, (const T *)dY, Z, dZ, de, lse_enc, lse_dec, (T *)dK, (T *)dV, dd, d->B, d->H, d->N, d->M, d->scale));
        return FLARE_OK;
    }
};

template <typename T, int D>
struct DQuery {
    static int run(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *V, const uint8_t *mask, const void *dY,
                   const float *Z, const float *dZ, const float *de, const float *dd, const float *lse_enc, const float *lse_dec, float *part,
                   cudaStream_t st) {
        static std::atomic<uint64_t> opt_in{0};
        const size_t smem = bwd_dq_simt_smem<T, D>();
        if (smem > 48 * 1024)
            if (int rc = ensure_big_smem(bwd_dq_simt_kernel<T, D>, opt_in, (int)smem)) return rc;
        FLARE_CUDA(launch_after(bwd_dq_simt_kernel<T, D>, dim3(p.splits, d->H * p.mblocks, d->B), kBwdThreads, smem, st,
                                (const T *)Q, (const T *)K, (const T *)V, mask, (const T *)dY, Z, dZ, de, dd, lse_enc, lse_dec, part, d->B, d->H, d->N, d->M, p.WM, p.mblocks, p.chunk, d->scale));
        return FLARE_OK;
    }
};

// Op<T, D>::run(args...) for the call's element type and head width.
template <template <typename, int> class Op, typename T, typename... A>
int by_width(int D, A... a) {
    switch (D) {
        case 4: return Op<T, 4>::run(a...);
        case 8: return Op<T, 8>::run(a...);
        case 16: return Op<T, 16>::run(a...);
        case 32: return Op<T, 32>::run(a...);
        case 64: return Op<T, 64>::run(a...);
        default: return FLARE_ERR_UNSUPPORTED;
    }
}
template <template <typename, int> class Op, typename... A>
int by_type(const flare_desc_t *d, A... a) {
    return d->dtype == FLARE_DTYPE_F32   ? by_width<Op, float>(d->D, a...)
           : d->dtype == FLARE_DTYPE_F16 ? by_width<Op, __half>(d->D, a...)
                                         : by_width<Op, __nv_bfloat16>(d->D, a...);
}

}  // namespace

int encode_simt(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *V, const uint8_t *mask,
                float *pm, float *pl, float *pacc, cudaStream_t st) {
    return by_type<Encode>(d, false, d, p, Q, K, V, mask, (const float *)nullptr, pm, pl, pacc, st);
}
int encode_dz_simt(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *dY, const float *lse_dec,
                   float *pacc, cudaStream_t st) {
    return by_type<Encode>(d, true, d, p, Q, K, dY, (const uint8_t *)nullptr, lse_dec, (float *)nullptr, (float *)nullptr, pacc, st);
}
int small_forward_cluster(const flare_desc_t *d) {
    const DeviceView di = device_info();
    const int cluster = small_forward_wanted(d, di.sms);
    return cluster != 0 && (di.checked != 1 || by_type<SmallFits>(d, cluster)) ? cluster : 0;   // (no device: what a whole one runs)
}
int forward_small_simt(const flare_desc_t *d, int cluster, const void *Q, const void *K, const void *V, const uint8_t *mask, float *Z, float *lse_enc,
                       void *Y, float *lse_dec, uint32_t *header, cudaStream_t st) {
    return by_type<SmallForward>(d, d, cluster, Q, K, V, mask, Z, lse_enc, Y, lse_dec, header, st);
}
int decode_simt(const flare_desc_t *d, const void *Q, const void *K, const float *Z, void *Y, float *lse_dec, cudaStream_t st) {
    return by_type<Decode>(d, d, Q, K, Z, Y, lse_dec, st);
}
int bwd_token_simt(const flare_desc_t *d, const void *Q, const void *K, const void *V, const uint8_t *mask, const void *dY,
                   const float *Z, const float *dZ, const float *de, const float *lse_enc, const float *lse_dec, void *dK, void *dV,
                   float *dd, cudaStream_t st) {
    return by_type<Token>(d, d, Q, K, V, mask, dY, Z, dZ, de, lse_enc, lse_dec, dK, dV, dd, st);
}
int bwd_dq_simt(const flare_desc_t *d, const SimtPlan &p, const void *Q, const void *K, const void *V, const uint8_t *mask,
                const void *dY, const float *Z, const float *dZ, const float *de, const float *dd, const float *lse_enc,
                const float *lse_dec, float *part, cudaStream_t st) {
    return by_type<DQuery>(d, d, p, Q, K, V, mask, dY, Z, dZ, de, dd, lse_enc, lse_dec, part, st);
}

}  // namespace flare
