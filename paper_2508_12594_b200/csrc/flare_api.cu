// Entry points of libflare: argument checks, workspaces, the order of the launches.  See include/flare.h for the contract.
#include <mutex>
#include "flare_host.h"
#include "flare_micro.cuh"

namespace flare {
thread_local char g_cuda_error[256] = "";
DeviceInfo g_dev[64];
std::atomic<int> g_path{FLARE_PATH_AUTO};

// Clears the workspace header from word `first` on.  (A memset waits for the launch before it and holds up the one behind: 2 us more than this, which
// overlaps with both.)
__global__ void __launch_bounds__(kHeaderBytes / 4) clear_header_kernel(uint32_t *header, int first) {
    ptx::grid_launch();
    ptx::grid_wait();
    if ((int)threadIdx.x >= first) header[threadIdx.x] = 0u;
}
int clear_header(void *workspace, int first, cudaStream_t st) {
    FLARE_CUDA(launch_after(clear_header_kernel, 1, kHeaderBytes / 4, 0, st, static_cast<uint32_t *>(workspace), first));
    return FLARE_OK;
}
}  // namespace flare

using namespace flare;

namespace {

int require_device() {
    const DeviceView di = device_info();
    if (di.checked == -2) {
        snprintf(g_cuda_error, sizeof(g_cuda_error), "no CUDA device");
        return FLARE_ERR_CUDA;
    }
    if (di.checked != 1) return FLARE_ERR_ARCH;
    return FLARE_OK;
}

// Scratch of flare_encode_static_scratch: part of the device image, shared by every call on the device.
// In host code this name is only a handle for cudaGetSymbolAddress; kernels must be given the looked-up address.
static __device__ __align__(256) unsigned char g_static_scratch[FLARE_STATIC_SCRATCH_BYTES];
std::atomic<void *> g_static_scratch_addr[64];

// Device address of g_static_scratch on the current device (looked up once per device, then cached).
int static_scratch_address(void **out) {
    int dev = -1;
    FLARE_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return FLARE_ERR_UNSUPPORTED;
    void *p = g_static_scratch_addr[dev].load(std::memory_order_acquire);
    if (p == nullptr) {
        FLARE_CUDA(cudaGetSymbolAddress(&p, g_static_scratch));
        if (p == nullptr) {
            snprintf(g_cuda_error, sizeof(g_cuda_error), "cudaGetSymbolAddress returned a null address");
            return FLARE_ERR_CUDA;
        }
        g_static_scratch_addr[dev].store(p, std::memory_order_release);
    }
    *out = p;
    return FLARE_OK;
}

// Kernels one call of `op` launches (among them the one that clears the workspace header, where it is not left to the merge).
int launches_for(const flare_desc_t *d, int op) {
    // a fast form is followed by the exact form (which may exit at once)
    const int fe = use_fast_encode(d) ? 2 : 1, f = use_fast_decode(d) ? 2 : 1;
    const int enc = fe + 1 + (use_tc(d) ? 1 : 0);               // header, encode, merge
    const int dec = decode_in_ranges(d) ? f * decode_ranges(d) + 1 : f;   // ranges of latents and their combination
    switch (op) {
        case FLARE_OP_ENCODE: return enc;
        case FLARE_OP_DECODE: return 1 + dec;                   // header (given a workspace), decode
        case FLARE_OP_FORWARD: return small_forward_cluster(d) ? 1 : enc + dec;
        case FLARE_OP_BACKWARD: {
            if (use_sweeps(d)) {                                // header; the two sweeps, each over ranges of latents and chunks of tokens, and their reductions
                const int sms = device_info().sms;
                return 1 + sweep_launches(d, dz_sweep_plan(d, sms)) + 1 + sweep_launches(d, grad_sweep_plan(d, sms)) + 1;
            }
            const int tok = token_in_ranges(d) ? (d->M + token_range(d) - 1) / token_range(d) : 1;   // (the CUDA-core kernel knows no ranges)
            return 1 + 2 + tok + 2;                             // header; dZ, its reduction; token kernel(s); dQ, its reduction
        }
        default: return 0;
    }
}

// Scratch of one flare_forward.
size_t forward_bytes(const flare_desc_t *d) {
    return make_layout(partials_for(d, device_info().sms, false), (long)d->B * d->H * d->M, d->D, true).total + decode_range_bytes(d);
}

int forward_impl(const flare_desc_t *d, const void *Q, const void *K, const void *V, const uint8_t *mask, void *Y, float *Z, float *lse_enc,
                 float *lse_dec, void *workspace, cudaStream_t st, bool keep_status) {
    const WorkspaceLayout w = make_layout(partials_for(d, device_info().sms, false), (long)d->B * d->H * d->M, d->D, true);
    if (const int cluster = small_forward_cluster(d)) {
        const int rc = forward_small_simt(d, cluster, Q, K, V, mask, Z, lse_enc, Y, lse_dec, keep_status ? nullptr : static_cast<uint32_t *>(workspace), st);
        if (rc != FLARE_ERR_UNSUPPORTED) return rc;
    }
    if (Z == nullptr) Z = reinterpret_cast<float *>(static_cast<char *>(workspace) + w.z);
    const int rc = encode_impl(d, Q, K, V, mask, Z, lse_enc, workspace, st, false, keep_status);
    if (rc != FLARE_OK) return rc;
    char *range_scratch = decode_in_ranges(d) ? static_cast<char *>(workspace) + w.total : nullptr;
    return decode_impl(d, Q, K, Z, Y, lse_dec, reinterpret_cast<uint32_t *>(workspace), st, range_scratch);
}

// Host tensors.  The copies bound such a call (67 + 67 MB in and 67 MB out take 3.7 ms, the mixer 0.1 ms), and the two directions of the link
// are independent: a batch is worked off in parts of whole items, the inputs of the next parts coming in on the caller's stream while
// a second one computes a part and takes its rows back.  3.75 -> 3.07 ms for 4 items of 65536 tokens of 128 features.  A part has at least
// 4 MB to bring in (75 us): less would no longer hide what its eight or so calls cost the host.  Items must keep the tensors' alignment.
int host_part_items(const flare_desc_t *d, size_t item_bytes, size_t workspace_bytes) {
    const size_t least = (size_t)4 << 20;
    long items = (long)((least + 2 * item_bytes - 1) / (2 * item_bytes));
    if (items >= d->B || item_bytes % 16 != 0) return d->B;
    flare_desc_t part = *d;
    part.B = (int)items;
    if (forward_bytes(&part) > workspace_bytes) return d->B;
    part.B = d->B % (int)items;                                 // the last part
    if (part.B != 0 && forward_bytes(&part) > workspace_bytes) return d->B;
    return (int)items;
}

// Second streams.  One takes 110 us to create and destroy, so a few are kept: a call takes one for itself while it queues its work and gives it
// back when it returns (a later call's work on it then simply queues behind).  At most kKept are kept in all, the rest and, with the
// library, the kept ones are destroyed.
class SideStreams {
  public:
    cudaError_t take(int device, cudaStream_t *out) {
        {
            std::lock_guard<std::mutex> lock(mutex_);
            for (int i = 0; i < kept_; ++i)
                if (device_[i] == device) {
                    *out = stream_[i];
                    --kept_;
                    device_[i] = device_[kept_];
                    stream_[i] = stream_[kept_];
                    return cudaSuccess;
                }
        }
        return cudaStreamCreateWithFlags(out, cudaStreamNonBlocking);
    }
    void give(int device, cudaStream_t stream) {
        {
            std::lock_guard<std::mutex> lock(mutex_);
            if (kept_ < kKept) {
                device_[kept_] = device;
                stream_[kept_++] = stream;
                return;
            }
        }
        cudaStreamDestroy(stream);
    }
    ~SideStreams() {
        for (int i = 0; i < kept_; ++i) cudaStreamDestroy(stream_[i]);
    }

  private:
    static constexpr int kKept = 8;
    std::mutex mutex_;
    int kept_ = 0, device_[kKept];
    cudaStream_t stream_[kKept];
};
SideStreams &side_streams() {
    static SideStreams s;
    return s;
}

int forward_host_parts(const flare_desc_t *d, int items, const void *hQ, const void *hK, const void *hV, const uint8_t *hmask, void *hY, void *dQ,
                       void *dK, void *dV, uint8_t *dmask, void *dY, void *workspace, size_t qb, size_t item_bytes, cudaStream_t st) {
    struct Side {
        int device = 0;
        cudaStream_t stream = nullptr;
        cudaEvent_t event = nullptr;
        ~Side() {
            if (event) cudaEventDestroy(event);                 // (released once what is recorded has happened)
            if (stream) side_streams().give(device, stream);
        }
    } side;
    FLARE_CUDA(cudaGetDevice(&side.device));
    FLARE_CUDA(side_streams().take(side.device, &side.stream));
    FLARE_CUDA(cudaEventCreateWithFlags(&side.event, cudaEventDisableTiming));
    auto parts = [&]() -> int {
        FLARE_CUDA(cudaMemcpyAsync(dQ, hQ, qb, cudaMemcpyHostToDevice, st));
        for (int b0 = 0; b0 < d->B; b0 += items) {
            flare_desc_t part = *d;
            part.B = std::min(items, d->B - b0);
            const size_t at = (size_t)b0 * item_bytes, n = (size_t)part.B * item_bytes, mat = (size_t)b0 * d->N;
            char *k = static_cast<char *>(dK) + at, *v = static_cast<char *>(dV) + at, *y = static_cast<char *>(dY) + at;
            FLARE_CUDA(cudaMemcpyAsync(k, static_cast<const char *>(hK) + at, n, cudaMemcpyHostToDevice, st));
            FLARE_CUDA(cudaMemcpyAsync(v, static_cast<const char *>(hV) + at, n, cudaMemcpyHostToDevice, st));
            if (hmask) FLARE_CUDA(cudaMemcpyAsync(dmask + mat, hmask + mat, (size_t)part.B * d->N, cudaMemcpyHostToDevice, st));
            FLARE_CUDA(cudaEventRecord(side.event, st));
            FLARE_CUDA(cudaStreamWaitEvent(side.stream, side.event, 0));
            const int rc = forward_impl(&part, dQ, k, v, hmask ? dmask + mat : nullptr, y, nullptr, nullptr, nullptr, workspace, side.stream, b0 > 0);
            if (rc != FLARE_OK) return rc;
            FLARE_CUDA(cudaMemcpyAsync(static_cast<char *>(hY) + at, y, n, cudaMemcpyDeviceToHost, side.stream));
        }
        return FLARE_OK;
    };
    const int rc = parts();
    // whatever was queued on the second stream comes before the caller's next work, also after an error
    FLARE_CUDA(cudaEventRecord(side.event, side.stream));
    FLARE_CUDA(cudaStreamWaitEvent(st, side.event, 0));
    return rc;
}

// ---- variants of the mixer: one latent sequence shared by all heads; separate latent queries for decode

template <typename T>
__global__ void expand_heads_kernel(const T *__restrict__ src, T *__restrict__ dst, long per_head, int H) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= per_head * H) return;
    dst[i] = src[i % per_head];
}
__global__ void sum_heads_kernel(const float *__restrict__ src, float *__restrict__ dst, long per_head, int H) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= per_head) return;
    float s = 0.f;
    for (int h = 0; h < H; ++h) s += src[(size_t)h * per_head + i];
    dst[i] = s;
}
__global__ void fill_kernel(float *__restrict__ dst, long n, float v) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = v;
}
template <typename T>
__global__ void add_into_kernel(T *__restrict__ dst, const T *__restrict__ other, long n) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T out;
    from_f32(out, to_f32(dst[i]) + to_f32(other[i]));
    dst[i] = out;
}

struct VariantLayout {
    size_t qe, qd, dq_full, dq2_full, inf_enc, inf_dec, dk2, total;   // offsets behind the operation's own workspace
};
// Scratch of the variant entry points, behind the workspace of the plain operation (base bytes).
VariantLayout variant_layout(const flare_desc_t *d, int op, int shared, int separate, size_t base) {
    VariantLayout v{};
    const size_t e = d->dtype == FLARE_DTYPE_F32 ? 4 : 2;
    const size_t q = align_up((size_t)d->H * d->M * d->D * e), qf = align_up((size_t)d->H * d->M * d->D * 4);
    size_t off = align_up(base);
    v.qe = off; if (shared) off += q;
    v.qd = off; if (shared && separate) off += q;
    if (op == FLARE_OP_BACKWARD) {
        v.dq_full = off; if (shared) off += qf;
        v.dq2_full = off; if (shared && separate) off += qf;
        v.inf_enc = off; if (separate) off += align_up(sizeof(float) * (size_t)d->B * d->H * d->M);
        v.inf_dec = off; if (separate) off += align_up(sizeof(float) * (size_t)d->B * d->N * d->H);
        v.dk2 = off; if (separate) off += align_up((size_t)d->B * d->N * d->H * d->D * e);
    }
    v.total = off;
    return v;
}

int expand_heads(const flare_desc_t *d, const void *src, void *dst, cudaStream_t st) {
    const long per = (long)d->M * d->D, n = per * d->H;
    if (d->dtype == FLARE_DTYPE_F32)
        expand_heads_kernel<float><<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const float *)src, (float *)dst, per, d->H);
    else if (d->dtype == FLARE_DTYPE_F16)
        expand_heads_kernel<__half><<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const __half *)src, (__half *)dst, per, d->H);
    else
        expand_heads_kernel<__nv_bfloat16><<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const __nv_bfloat16 *)src, (__nv_bfloat16 *)dst, per, d->H);
    FLARE_CUDA(cudaGetLastError());
    return FLARE_OK;
}

}  // namespace

extern "C" {

int flare_version(void) { return 100; }

const char *flare_status_string(int status) {
    switch (status) {
        case FLARE_OK: return "ok";
        case FLARE_ERR_INVALID_ARG: return "invalid argument";
        case FLARE_ERR_UNSUPPORTED: return "unsupported shape or dtype";
        case FLARE_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case FLARE_ERR_ARCH: return "device is not compute capability 10.x";
        case FLARE_ERR_CUDA: return "CUDA error";
        case FLARE_ERR_TIMEOUT: return "a bounded device-side wait gave up";
        default: return "unknown status";
    }
}

const char *flare_last_cuda_error(void) { return g_cuda_error; }

int flare_encode_partials(const flare_desc_t *desc) {
    if (check_desc(desc) != FLARE_OK) return 0;
    return partials_for(desc, device_info().sms, true);
}

int flare_launch_count(const flare_desc_t *desc, int op) {
    if (check_desc(desc) != FLARE_OK) return 0;
    return launches_for(desc, op);
}

size_t flare_workspace_bytes(const flare_desc_t *desc, int op) {
    if (check_desc(desc) != FLARE_OK) return 0;
    const long rows = (long)desc->B * desc->H * desc->M;
    switch (op) {
        case FLARE_OP_ENCODE: return make_layout(partials_for(desc, device_info().sms, true), rows, desc->D, false).total;
        case FLARE_OP_DECODE: return kHeaderBytes + decode_range_bytes(desc);
        case FLARE_OP_FORWARD: {
            // (room for the parts that flare_forward_host works a batch off in: fewer rows, but more CTAs along N for each)
            size_t most = forward_bytes(desc);
            flare_desc_t part = *desc;
            for (part.B = desc->B / 2; part.B >= 1; part.B /= 2) most = std::max(most, forward_bytes(&part));
            return most;
        }
        case FLARE_OP_BACKWARD: return bwd_layout(desc, device_info().sms).total;
        case FLARE_OP_SPECTRAL: return spectral_bytes(desc, device_info().sms);
        default: return 0;
    }
}

int flare_encode(const flare_desc_t *desc, const void *Q_lat, const void *K, const void *V, const uint8_t *key_mask,
                 float *Z, float *lse_enc, void *workspace, size_t workspace_bytes, flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    if (!Q_lat || !K || !V || !Z || !workspace) return FLARE_ERR_INVALID_ARG;
    if (!aligned16(Q_lat) || !aligned16(K) || !aligned16(V) || !aligned16(Z) || !aligned16(workspace) ||
        (lse_enc && !aligned16(lse_enc)))
        return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    if (workspace_bytes < flare_workspace_bytes(desc, FLARE_OP_ENCODE)) return FLARE_ERR_WORKSPACE_TOO_SMALL;
    return encode_impl(desc, Q_lat, K, V, key_mask, Z, lse_enc, workspace, (cudaStream_t)stream, true);
}

int flare_encode_static_scratch(const flare_desc_t *desc, const void *Q_lat, const void *K, const void *V,
                                const uint8_t *key_mask, float *Z, float *lse_enc, flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    if (!Q_lat || !K || !V || !Z) return FLARE_ERR_INVALID_ARG;
    if (!aligned16(Q_lat) || !aligned16(K) || !aligned16(V) || !aligned16(Z) || (lse_enc && !aligned16(lse_enc)))
        return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    const size_t need = flare_workspace_bytes(desc, FLARE_OP_ENCODE);
    if (need > (size_t)FLARE_STATIC_SCRATCH_BYTES) {
        snprintf(g_cuda_error, sizeof(g_cuda_error), "problem needs %zu bytes of scratch, the built-in array has %zu",
                 need, (size_t)FLARE_STATIC_SCRATCH_BYTES);
        return FLARE_ERR_WORKSPACE_TOO_SMALL;
    }
    void *scratch = nullptr;
    if ((rc = static_scratch_address(&scratch)) != FLARE_OK) return rc;
    // encode_impl zeroes the header words that must start at zero; every partial it later reads it first writes
    return encode_impl(desc, Q_lat, K, V, key_mask, Z, lse_enc, scratch, (cudaStream_t)stream, true);
}

int flare_decode(const flare_desc_t *desc, const void *Q_lat, const void *K, const float *Z, void *Y, float *lse_dec,
                 void *workspace, size_t workspace_bytes, flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    if (!Q_lat || !K || !Z || !Y) return FLARE_ERR_INVALID_ARG;
    if (!aligned16(Q_lat) || !aligned16(K) || !aligned16(Z) || !aligned16(Y) || (lse_dec && !aligned16(lse_dec)) ||
        (workspace && !aligned16(workspace)))
        return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    if (workspace == nullptr) return decode_impl(desc, Q_lat, K, Z, Y, lse_dec, nullptr, (cudaStream_t)stream);
    if (workspace_bytes < flare_workspace_bytes(desc, FLARE_OP_DECODE)) return FLARE_ERR_WORKSPACE_TOO_SMALL;
    if ((rc = clear_header(workspace, 0, (cudaStream_t)stream)) != FLARE_OK) return rc;
    char *range_scratch = decode_in_ranges(desc) ? static_cast<char *>(workspace) + kHeaderBytes : nullptr;
    return decode_impl(desc, Q_lat, K, Z, Y, lse_dec, static_cast<uint32_t *>(workspace), (cudaStream_t)stream,
                       range_scratch);
}

int flare_set_path(int path) {
    if (path != FLARE_PATH_AUTO && path != FLARE_PATH_EXACT && path != FLARE_PATH_FAST) return FLARE_ERR_INVALID_ARG;
    g_path.store(path, std::memory_order_relaxed);
    return FLARE_OK;
}

int flare_forward(const flare_desc_t *desc, const void *Q_lat, const void *K, const void *V, const uint8_t *key_mask,
                  void *Y, float *Z, float *lse_enc, float *lse_dec, void *workspace, size_t workspace_bytes,
                  flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    if (!Q_lat || !K || !V || !Y || !workspace) return FLARE_ERR_INVALID_ARG;
    if (!aligned16(Q_lat) || !aligned16(K) || !aligned16(V) || !aligned16(Y) || !aligned16(workspace) ||
        (Z && !aligned16(Z)) || (lse_enc && !aligned16(lse_enc)) || (lse_dec && !aligned16(lse_dec)))
        return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    if (workspace_bytes < flare_workspace_bytes(desc, FLARE_OP_FORWARD)) return FLARE_ERR_WORKSPACE_TOO_SMALL;
    return forward_impl(desc, Q_lat, K, V, key_mask, Y, Z, lse_enc, lse_dec, workspace, (cudaStream_t)stream, false);
}

int flare_backward(const flare_desc_t *desc, const void *Q_lat, const void *K, const void *V, const uint8_t *key_mask,
                   const void *Y, const void *dY, const float *Z, const float *lse_enc, const float *lse_dec,
                   float *dQ_lat, void *dK, void *dV, void *workspace, size_t workspace_bytes,
                   flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    const void *ptrs[] = {Q_lat, K, V, Y, dY, Z, lse_enc, lse_dec, dQ_lat, dK, dV, workspace};
    for (const void *p : ptrs)
        if (p == nullptr || !aligned16(p)) return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    if (workspace_bytes < flare_workspace_bytes(desc, FLARE_OP_BACKWARD)) return FLARE_ERR_WORKSPACE_TOO_SMALL;
    const int sms = device_info().sms;
    char *ws = static_cast<char *>(workspace);
    cudaStream_t st = (cudaStream_t)stream;
    return backward_impl(desc, sms, Q_lat, K, V, key_mask, Y, dY, Z, lse_enc, lse_dec, dQ_lat, dK, dV, ws, st, false);
}

int flare_forward_host(const flare_desc_t *desc, const void *hQ_lat, const void *hK, const void *hV,
                       const uint8_t *hmask, void *hY, void *dQ_lat, void *dK, void *dV, uint8_t *dmask, void *dY,
                       void *workspace, size_t workspace_bytes, flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    if (!hQ_lat || !hK || !hV || !hY || !dQ_lat || !dK || !dV || !dY || (hmask && !dmask)) return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t e = desc->dtype == FLARE_DTYPE_F32 ? 4 : 2;
    const size_t qb = (size_t)desc->H * desc->M * desc->D * e;
    const size_t tb = (size_t)desc->B * desc->N * desc->H * desc->D * e;
    if (workspace != nullptr && workspace_bytes >= flare_workspace_bytes(desc, FLARE_OP_FORWARD) && aligned16(dQ_lat) && aligned16(dK) &&
        aligned16(dV) && aligned16(dY) && aligned16(workspace)) {
        const int items = host_part_items(desc, tb / desc->B, workspace_bytes);
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (items < desc->B && cudaStreamIsCapturing(st, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone)
            return forward_host_parts(desc, items, hQ_lat, hK, hV, hmask, hY, dQ_lat, dK, dV, dmask, dY, workspace, qb, tb / desc->B, st);
        (void)cudaGetLastError();                               // (a capture elsewhere may forbid the question: one part then)
    }
    FLARE_CUDA(cudaMemcpyAsync(dQ_lat, hQ_lat, qb, cudaMemcpyHostToDevice, st));
    FLARE_CUDA(cudaMemcpyAsync(dK, hK, tb, cudaMemcpyHostToDevice, st));
    FLARE_CUDA(cudaMemcpyAsync(dV, hV, tb, cudaMemcpyHostToDevice, st));
    if (hmask) FLARE_CUDA(cudaMemcpyAsync(dmask, hmask, (size_t)desc->B * desc->N, cudaMemcpyHostToDevice, st));
    rc = flare_forward(desc, dQ_lat, dK, dV, hmask ? dmask : nullptr, dY, nullptr, nullptr, nullptr, workspace,
                       workspace_bytes, stream);
    if (rc != FLARE_OK) return rc;
    FLARE_CUDA(cudaMemcpyAsync(hY, dY, tb, cudaMemcpyDeviceToHost, st));
    return FLARE_OK;
}

size_t flare_variant_workspace_bytes(const flare_desc_t *desc, int op, int shared_latents, int separate_decode_queries) {
    if (op != FLARE_OP_FORWARD && op != FLARE_OP_BACKWARD) return 0;
    const size_t base = flare_workspace_bytes(desc, op);
    if (base == 0) return 0;
    return variant_layout(desc, op, shared_latents, separate_decode_queries, base).total;
}

int flare_forward_variant(const flare_desc_t *desc, int shared_latents, const void *Q_enc, const void *Q_dec, const void *K,
                          const void *V, const uint8_t *key_mask, void *Y, float *Z, float *lse_enc, float *lse_dec,
                          void *workspace, size_t workspace_bytes, flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    if (!Q_enc || !K || !V || !Y || !workspace) return FLARE_ERR_INVALID_ARG;
    const void *ptrs[] = {Q_enc, Q_dec, K, V, Y, Z, lse_enc, lse_dec, workspace};
    for (const void *p : ptrs)
        if (p != nullptr && !aligned16(p)) return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    const size_t base = flare_workspace_bytes(desc, FLARE_OP_FORWARD);
    const VariantLayout v = variant_layout(desc, FLARE_OP_FORWARD, shared_latents, Q_dec != nullptr, base);
    if (workspace_bytes < v.total) return FLARE_ERR_WORKSPACE_TOO_SMALL;
    cudaStream_t st = (cudaStream_t)stream;
    char *ws = static_cast<char *>(workspace);
    const void *qe = Q_enc, *qd = Q_dec ? Q_dec : Q_enc;
    if (shared_latents) {
        if ((rc = expand_heads(desc, Q_enc, ws + v.qe, st)) != FLARE_OK) return rc;
        qe = ws + v.qe;
        qd = qe;
        if (Q_dec) {
            if ((rc = expand_heads(desc, Q_dec, ws + v.qd, st)) != FLARE_OK) return rc;
            qd = ws + v.qd;
        }
    }
    const WorkspaceLayout w = make_layout(partials_for(desc, device_info().sms, false), (long)desc->B * desc->H * desc->M, desc->D, true);
    if (Z == nullptr) Z = reinterpret_cast<float *>(ws + w.z);
    if ((rc = encode_impl(desc, qe, K, V, key_mask, Z, lse_enc, workspace, st, false)) != FLARE_OK) return rc;
    char *range_scratch = decode_in_ranges(desc) ? ws + w.total : nullptr;
    return decode_impl(desc, qd, K, Z, Y, lse_dec, reinterpret_cast<uint32_t *>(workspace), st, range_scratch);
}

int flare_backward_variant(const flare_desc_t *desc, int shared_latents, const void *Q_enc, const void *Q_dec, const void *K,
                           const void *V, const uint8_t *key_mask, const void *Y, const void *dY, const float *Z,
                           const float *lse_enc, const float *lse_dec, float *dQ_enc, float *dQ_dec, void *dK, void *dV,
                           void *workspace, size_t workspace_bytes, flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    const void *need[] = {Q_enc, K, V, Y, dY, Z, lse_enc, lse_dec, dQ_enc, dK, dV, workspace};
    for (const void *p : need)
        if (p == nullptr || !aligned16(p)) return FLARE_ERR_INVALID_ARG;
    if ((Q_dec == nullptr) != (dQ_dec == nullptr)) return FLARE_ERR_INVALID_ARG;
    if ((Q_dec && !aligned16(Q_dec)) || (dQ_dec && !aligned16(dQ_dec))) return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    const size_t base = flare_workspace_bytes(desc, FLARE_OP_BACKWARD);
    const bool separate = Q_dec != nullptr;
    const VariantLayout v = variant_layout(desc, FLARE_OP_BACKWARD, shared_latents, separate, base);
    if (workspace_bytes < v.total) return FLARE_ERR_WORKSPACE_TOO_SMALL;
    cudaStream_t st = (cudaStream_t)stream;
    char *ws = static_cast<char *>(workspace);
    const int sms = device_info().sms;
    const void *qe = Q_enc, *qd = Q_dec;
    float *dqe = dQ_enc, *dqd = dQ_dec;
    const long per = (long)desc->M * desc->D;
    if (shared_latents) {
        if ((rc = expand_heads(desc, Q_enc, ws + v.qe, st)) != FLARE_OK) return rc;
        qe = ws + v.qe;
        dqe = reinterpret_cast<float *>(ws + v.dq_full);
        if (separate) {
            if ((rc = expand_heads(desc, Q_dec, ws + v.qd, st)) != FLARE_OK) return rc;
            qd = ws + v.qd;
            dqd = reinterpret_cast<float *>(ws + v.dq2_full);
        }
    }
    auto run = [&](const void *q, const float *le, const float *ld, float *dq, void *dk, bool skip_a) {
        return backward_impl(desc, sms, q, K, V, key_mask, Y, dY, Z, le, ld, dq, dk, dV, ws, st, skip_a);
    };
    if (!separate) {
        if ((rc = run(qe, lse_enc, lse_dec, dqe, dK, false)) != FLARE_OK) return rc;
    } else {
        // Two runs of the backward over the same workspace.  With lse_enc = +inf every encode weight exp(S - lse_enc) is 0,
        // so the first run (decode queries) leaves dZ, the decode term of dK and dQ_dec; with lse_dec = +inf the second
        // (encode queries; dZ kept from the first) leaves the encode term of dK, dV and dQ_enc.
        float *inf_enc = reinterpret_cast<float *>(ws + v.inf_enc), *inf_dec = reinterpret_cast<float *>(ws + v.inf_dec);
        const long ne = (long)desc->B * desc->H * desc->M, nd = (long)desc->B * desc->N * desc->H;
        fill_kernel<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(inf_enc, ne, INFINITY);
        fill_kernel<<<(unsigned)((nd + 255) / 256), 256, 0, st>>>(inf_dec, nd, INFINITY);
        FLARE_CUDA(cudaGetLastError());
        void *dk2 = ws + v.dk2;
        if ((rc = run(qd, inf_enc, lse_dec, dqd, dk2, false)) != FLARE_OK) return rc;
        if ((rc = run(qe, lse_enc, inf_dec, dqe, dK, true)) != FLARE_OK) return rc;
        const long nk = (long)desc->B * desc->N * desc->H * desc->D;
        if (desc->dtype == FLARE_DTYPE_F32)
            add_into_kernel<float><<<(unsigned)((nk + 255) / 256), 256, 0, st>>>((float *)dK, (const float *)dk2, nk);
        else if (desc->dtype == FLARE_DTYPE_F16)
            add_into_kernel<__half><<<(unsigned)((nk + 255) / 256), 256, 0, st>>>((__half *)dK, (const __half *)dk2, nk);
        else
            add_into_kernel<__nv_bfloat16><<<(unsigned)((nk + 255) / 256), 256, 0, st>>>((__nv_bfloat16 *)dK, (const __nv_bfloat16 *)dk2, nk);
        FLARE_CUDA(cudaGetLastError());
    }
    if (shared_latents) {
        sum_heads_kernel<<<(unsigned)((per + 255) / 256), 256, 0, st>>>(dqe, dQ_enc, per, desc->H);
        if (separate) sum_heads_kernel<<<(unsigned)((per + 255) / 256), 256, 0, st>>>(dqd, dQ_dec, per, desc->H);
        FLARE_CUDA(cudaGetLastError());
    }
    return FLARE_OK;
}

int flare_spectral_gram(const flare_desc_t *desc, const void *Q_lat, const void *K, const float *lse_enc,
                        const float *lse_dec, float *G, void *workspace, size_t workspace_bytes, flare_stream_t stream) {
    int rc = check_desc(desc);
    if (rc != FLARE_OK) return rc;
    const void *ptrs[] = {Q_lat, K, lse_enc, lse_dec, G, workspace};
    for (const void *p : ptrs)
        if (p == nullptr || !aligned16(p)) return FLARE_ERR_INVALID_ARG;
    if ((rc = require_device()) != FLARE_OK) return rc;
    const int sms = device_info().sms;
    if (workspace_bytes < spectral_bytes(desc, sms)) return FLARE_ERR_WORKSPACE_TOO_SMALL;
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = clear_header(workspace, 0, st)) != FLARE_OK) return rc;
    return spectral_gram(desc, sms, Q_lat, K, lse_enc, lse_dec, G, workspace, st);
}

int flare_spectral_eig(int32_t matrices, int32_t M, float *G, float *eigenvalues, float *U, int32_t sweeps, flare_stream_t stream) {
    if (matrices <= 0 || M <= 0 || M > 1024 || !G || !eigenvalues) return FLARE_ERR_INVALID_ARG;
    if (!aligned16(G) || !aligned16(eigenvalues) || (U && !aligned16(U))) return FLARE_ERR_INVALID_ARG;
    int rc = require_device();
    if (rc != FLARE_OK) return rc;
    return spectral_eig(matrices, M, G, eigenvalues, U, sweeps, (cudaStream_t)stream);
}

int flare_microbench(int which, int iters, void *scratch, size_t scratch_bytes, double *result, flare_stream_t stream) {
    if (!scratch || !result || !aligned16(scratch) || scratch_bytes < 4096 || which < 0 || which > 4) return FLARE_ERR_INVALID_ARG;
    int rc = require_device();
    if (rc != FLARE_OK) return rc;
    if (iters < 1) iters = 1;
    if (iters > 1000000) iters = 1000000;
    cudaStream_t st = (cudaStream_t)stream;
    const int sms = device_info().sms > 512 ? 512 : device_info().sms;
    unsigned long long *out = static_cast<unsigned long long *>(scratch);
    FLARE_CUDA(cudaMemsetAsync(scratch, 0, 4096, st));
    unsigned long long host[512];
    if (which <= 2) {
        if (which == 0) micro_softmax_kernel<0><<<sms, kTcThreads, 0, st>>>(iters, kLog2e, out);
        if (which == 1) micro_softmax_kernel<1><<<sms, kTcThreads, 0, st>>>(iters, kLog2e, out);
        if (which == 2) micro_softmax_kernel<2><<<sms, kTcThreads, 0, st>>>(iters, kLog2e, out);
        FLARE_CUDA(cudaGetLastError());
        FLARE_CUDA(cudaMemcpyAsync(host, out, sizeof(unsigned long long) * sms, cudaMemcpyDeviceToHost, st));
        FLARE_CUDA(cudaStreamSynchronize(st));
        double cycles = 0.0;
        for (int i = 0; i < sms; ++i) cycles += (double)host[i];
        cycles /= sms;
        *result = cycles > 0.0 ? 512.0 * 32.0 * iters / cycles : 0.0;     // 512 threads x 32 columns per round
    } else {
        static std::atomic<uint64_t> smem_opt_in{0};
        if (int rc_attr = ensure_big_smem(micro_mma_kernel, smem_opt_in, 64 * 1024)) return rc_attr;
        micro_mma_kernel<<<1, 64, 24576 + 1024, st>>>(iters, out);
        FLARE_CUDA(cudaGetLastError());
        FLARE_CUDA(cudaMemcpyAsync(host, out, sizeof(unsigned long long) * 2, cudaMemcpyDeviceToHost, st));
        FLARE_CUDA(cudaStreamSynchronize(st));
        *result = (double)host[which - 3];
    }
    return FLARE_OK;
}

int flare_check(const void *workspace, flare_stream_t stream) {
    void *builtin = nullptr;
    if (!workspace) {                                           // the built-in scratch of flare_encode_static_scratch
        const int rc = static_scratch_address(&builtin);
        if (rc != FLARE_OK) return rc;
        workspace = builtin;
    }
    uint32_t words[2] = {0, 0};
    FLARE_CUDA(cudaMemcpyAsync(words, workspace, sizeof(words), cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    FLARE_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    return words[0] == 0 ? FLARE_OK : FLARE_ERR_TIMEOUT;
}

int flare_selftest_wait(void *workspace, uint64_t budget_ns, flare_stream_t stream) {
    if (!workspace || !aligned16(workspace)) return FLARE_ERR_INVALID_ARG;
    int rc = require_device();
    if (rc != FLARE_OK) return rc;
    if (budget_ns < 1000) budget_ns = 1000;
    if (budget_ns > 100000000ull) budget_ns = 100000000ull;     // never more than a tenth of a second
    cudaStream_t st = (cudaStream_t)stream;
    FLARE_CUDA(cudaMemsetAsync(workspace, 0, kHeaderBytes, st));
    selftest_wait_kernel<<<1, 32, 0, st>>>(static_cast<uint32_t *>(workspace), (unsigned long long)budget_ns);
    FLARE_CUDA(cudaGetLastError());
    return FLARE_OK;
}

}  // extern "C"
