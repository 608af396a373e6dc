// Shared device/host helpers of libflare (CUDA path only; the CPU oracle shares none of this).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace flare {

// Launch of a kernel that calls ptx::grid_wait() before it touches global memory: its CTAs may be placed, set up their barriers and
// tensor memory and wait while the launch before it runs out, instead of starting when that has ended altogether.
// Measured, whole calls, us: training step of 16384 tokens 94.6 -> 88.2, padded batch 333 -> 317, D = 64 194 -> 182, 2-D mesh forward 113 -> 107.
// (Such kernels take no __restrict__ inputs: a read-only load might be moved ahead of the wait.)
template <typename... P, typename... A>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}


// Workspace header: 256 bytes at the start of every workspace.
//   word 0: error flag (0 = fine; otherwise a code naming the wait that gave up)
//   word 1: detail (which barrier / iteration)
constexpr size_t kHeaderBytes = 256;

// Section sizes are rounded up to this, so every section starts 256-byte aligned.
constexpr size_t kAlign = 256;
__host__ __device__ inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }

// Where the pieces of an encode/forward workspace live.  P = number of partial results per latent row.
struct WorkspaceLayout {
    size_t part_m;    // float [P][B*H*M]      running maxima (natural-log units of the scaled score)
    size_t part_l;    // float [P][B*H*M]      sums of exp(score - max)
    size_t part_acc;  // float [P][B*H*M][D]   un-normalised latent rows
    size_t z;         // float [B*H*M][D]      latent sequence when the caller passes Z = NULL
    size_t total;
};

inline WorkspaceLayout make_layout(int P, long rows, int D, bool with_z) {
    WorkspaceLayout w;
    size_t off = kHeaderBytes;
    w.part_m = off;   off += align_up(sizeof(float) * (size_t)P * rows);
    w.part_l = off;   off += align_up(sizeof(float) * (size_t)P * rows);
    w.part_acc = off; off += align_up(sizeof(float) * (size_t)P * rows * D);
    w.z = off;
    if (with_z) off += align_up(sizeof(float) * (size_t)rows * D);
    w.total = off;
    return w;
}

// Shape of the CUDA-core kernels' blocks (their launch plans need it too).
constexpr int kSimtThreads = 256;
constexpr int kBwdThreads = 256;

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void from_f32(float &dst, float x) { dst = x; }
__device__ __forceinline__ void from_f32(__nv_bfloat16 &dst, float x) { dst = __float2bfloat16_rn(x); }
__device__ __forceinline__ float to_f32(__half x) { return __half2float(x); }
__device__ __forceinline__ void from_f32(__half &dst, float x) { dst = __float2half_rn(x); }

// A row near the middle of Z [rows, D] (one head's): the mean of 32 of them.  dS holds A - dd with A[n,m] = dY_n . Z_m and
// dd[n] = sum_m W_dec[n,m] A[n,m], the weights of a token adding up to 1: unchanged when one vector is subtracted from all rows of Z, and
// where the rows are nearly equal (features with a mean) that leaves no large numbers to cancel.  The kernel that forms dd and the one that
// subtracts it take the same.  (The mean of few rows carries some of their scatter into every row: with eight, dQ was up to 1.09 times as
// far from float64 on features without a mean.)  By all warps of the block, a column each in turn.
template <int D>
__device__ __forceinline__ void z_centre(float *centre, const float *Z, int rows) {
    const int lane = threadIdx.x & 31;
    const float *row = Z + (size_t)((long)lane * rows / 32) * D;
    for (int d = threadIdx.x >> 5; d < D; d += blockDim.x >> 5) {
        float c = row[d] * (1.f / 32.f);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (lane == 0) centre[d] = c;
    }
}

// The same row of a head's Z, and how far the 128 rows from r0 on reach from it, by feature, by one warp: around [1 + blocks of 128 latents][D].
template <int D>
__device__ __forceinline__ void z_around(float *around, const float *Z, int rows, int block) {
    constexpr int L = D / 4, STEP = 32 / L;                     // lanes of a row, rows at a time
    const int lane = threadIdx.x & 31, r0 = lane / L, r1 = min(rows, block * 128 + 128);
    const float4 *z4 = reinterpret_cast<const float4 *>(Z) + lane % L;
    float c[4] = {0.f, 0.f, 0.f, 0.f}, reach[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < L; ++k) {
        const float4 z = z4[(size_t)((long)(r0 + k * STEP) * rows / 32) * L];
        c[0] += z.x; c[1] += z.y; c[2] += z.z; c[3] += z.w;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = L; o < 32; o <<= 1) c[k] += __shfl_xor_sync(0xffffffffu, c[k], o);
        c[k] *= 1.f / 32.f;
    }
#pragma unroll 8
    for (int r = block * 128 + r0; r < r1; r += STEP) {
        const float4 z = z4[(size_t)r * L];
        reach[0] = fmaxf(reach[0], fabsf(z.x - c[0])); reach[1] = fmaxf(reach[1], fabsf(z.y - c[1]));
        reach[2] = fmaxf(reach[2], fabsf(z.z - c[2])); reach[3] = fmaxf(reach[3], fabsf(z.w - c[3]));
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int o = L; o < 32; o <<= 1) reach[k] = fmaxf(reach[k], __shfl_xor_sync(0xffffffffu, reach[k], o));
    if (lane < L) {
        if (block == 0) reinterpret_cast<float4 *>(around)[lane] = make_float4(c[0], c[1], c[2], c[3]);
        reinterpret_cast<float4 *>(around + (1 + block) * D)[lane] = make_float4(reach[0], reach[1], reach[2], reach[3]);
    }
}

}  // namespace flare
