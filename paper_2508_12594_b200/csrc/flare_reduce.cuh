// Sums over the partial results that the split-N kernels leave: the log-sum-exp merge of encode, dZ and de of the backward,
// dQ.  They read a few megabytes of L2-resident partials, so what bounds them is the latency of dependent loads: a row of D
// elements is served by L = D / 4 lanes (16-byte loads) times `slices` groups of lanes, each taking every slices-th partial,
// with `slices` so large that a thread has about four independent loads (reduce_slices), and the slices meet in shuffles and,
// beyond a warp, in shared memory.  The order of every sum is fixed by the shape.
// Measured, P = 148 partials of 256 rows of 32 (a thread per element or a block of serial slices per row before): merge
// 10.8 -> 5.1, dZ with de 21.4 -> 3.5 us; P = 4, 16384 rows of 32: merge 8.3 -> 4.2, dZ with de 14.5 -> 4.1 us.
#pragma once

#include "flare_common.cuh"
#include "flare_ptx.cuh"

namespace flare {

constexpr int kReduceThreads = 256;

// Slices per row: a power of two, P / slices about four, all of a row's lanes in one block.
inline int reduce_slices(int P, int D) {
    const int L = D / 4;
    int s = 1;
    while (s * 4 < P && s * 2 * L <= kReduceThreads) s *= 2;
    return s;
}
inline unsigned reduce_blocks(long rows, int D, int slices) {
    const long per = kReduceThreads / (D / 4 * slices);
    return (unsigned)((rows + per - 1) / per);
}

struct RowMap {
    long row;          // the row this thread works on (may lie beyond the last)
    int lane, slice;   // its 16-byte piece of the row, its slice of the partials
};
template <int L>
__device__ __forceinline__ RowMap row_map(int slices) {
    const int T = L * slices, t = threadIdx.x % T;
    return RowMap{(long)blockIdx.x * (kReduceThreads / T) + threadIdx.x / T, t % L, t / L};
}

__device__ __forceinline__ float4 f4_fma(float w, float4 v, float4 a) {
    return make_float4(fmaf(w, v.x, a.x), fmaf(w, v.y, a.y), fmaf(w, v.z, a.z), fmaf(w, v.w, a.w));
}
__device__ __forceinline__ float4 f4_add(float4 v, float4 a) { return make_float4(v.x + a.x, v.y + a.y, v.z + a.z, v.w + a.w); }
__device__ __forceinline__ float4 f4_shfl_xor(float4 v, int o) {
    return make_float4(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o),
                       __shfl_xor_sync(0xffffffffu, v.z, o), __shfl_xor_sync(0xffffffffu, v.w, o));
}

// Sum of `v` over the slices of a row, valid in the threads of slice 0.  All threads of the block call it.
template <int L>
__device__ __forceinline__ float4 sum_slices(float4 v, int slices) {
    const int T = L * slices;
    for (int o = L; o < 32 && o < T; o <<= 1) v = f4_add(f4_shfl_xor(v, o), v);
    if (T > 32) {                                               // uniform over the grid
        __shared__ float4 sh[kReduceThreads / 32][L];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (lane < L) sh[warp][lane] = v;
        __syncthreads();
        const int first = threadIdx.x / T * (T / 32);           // the row's first warp
        if (threadIdx.x % T < L) {
            v = sh[first][lane];
            for (int w = 1; w < T / 32; ++w) v = f4_add(v, sh[first + w][lane]);
        }
    }
    return v;
}

// Log-sum-exp merge of the P partial results of every latent row (b, h, m):
//   m* = max_p m_p;  l = sum_p l_p exp(m_p - m*);  Z = sum_p acc_p exp(m_p - m*) / l;  lse = m* + log l.
// One pass: a thread joins its own partials relative to their maximum, four loads in flight, then the slices are joined
// relative to the row's.  `redo`: null, or a word that says, if not 0, that the exact form replaced the partial results
// by P_redo of its own.  `header`: null, or the workspace header, which is cleared here (for encode kernels that leave no
// flags in it).
template <int L>
__global__ void __launch_bounds__(kReduceThreads)
merge_kernel(const float *part_m, const float *part_l, const float *part_acc,
             float *Z, float *lse_enc, int P, const uint32_t *redo, int P_redo, long rows, uint32_t *header, int slices) {
    ptx::grid_launch();
    ptx::grid_wait();
    if (redo != nullptr && *redo != 0) P = P_redo;
    const RowMap rm = row_map<L>(slices);
    const int T = L * slices;
    if (header != nullptr && blockIdx.x == 0 && threadIdx.x < kHeaderBytes / 4) header[threadIdx.x] = 0u;
    const bool live = rm.row < rows;
    const long row = live ? rm.row : rows - 1;
    const float4 *acc4 = reinterpret_cast<const float4 *>(part_acc) + row * L + rm.lane;
    float mx = -INFINITY, l = 0.f;
    float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int p0 = rm.slice; p0 < P; p0 += 4 * slices) {
        float m[4], pl[4];
        float4 a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int p = p0 + q * slices;
            const bool in = p < P;
            const size_t i = (size_t)(in ? p : p0) * rows + row;
            m[q] = in ? part_m[i] : -INFINITY;
            pl[q] = part_l[i];
            a[q] = acc4[(size_t)(in ? p : p0) * rows * L];
        }
        const float mnew = fmaxf(fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])), mx);
        if (mnew == -INFINITY) continue;                        // no valid token in any of them
        const float f = expf(mx - mnew);
        l *= f;
        z = make_float4(z.x * f, z.y * f, z.z * f, z.w * f);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float w = expf(m[q] - mnew);
            l = w > 0.f ? fmaf(pl[q], w, l) : l;                // (a partial without valid tokens may hold anything)
            if (w > 0.f) z = f4_fma(w, a[q], z);
        }
        mx = mnew;
    }
    // the row's maximum over the slices
    __shared__ float smx[kReduceThreads / 32];
    float top = mx;
    for (int o = L; o < 32 && o < T; o <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    if (T > 32) {
        if ((threadIdx.x & 31) == 0) smx[threadIdx.x >> 5] = top;
        __syncthreads();
        const int first = threadIdx.x / T * (T / 32);
        for (int w = 0; w < T / 32; ++w) top = fmaxf(top, smx[first + w]);
    }
    const float f = mx == -INFINITY ? 0.f : expf(mx - top);
    z = sum_slices<L>(make_float4(z.x * f, z.y * f, z.z * f, z.w * f), slices);
    if (T > 32) __syncthreads();                                // (the shared array of sum_slices is used twice)
    const float4 ls = sum_slices<L>(make_float4(l * f, 0.f, 0.f, 0.f), slices);
    if (!live || rm.slice != 0) return;
    const bool none = top == -INFINITY;                         // no valid token anywhere
    const float inv = none ? 0.f : 1.f / ls.x;
    reinterpret_cast<float4 *>(Z)[rm.row * L + rm.lane] = none ? make_float4(0.f, 0.f, 0.f, 0.f)
                                                               : make_float4(z.x * inv, z.y * inv, z.z * inv, z.w * inv);
    if (lse_enc != nullptr && rm.lane == 0) lse_enc[rm.row] = none ? -INFINITY : top + logf(ls.x);
}

// A first guess e[n] of dd[n] = dY_n . Y_n for the token kernel of the backward, from the stored Y: of dY_n . (Y_n - centre), with Y_n no further from
// the centre of the rows of Z than these are (features with a mean: what rounding Y left must not be taken for a difference).  A block takes `chunk`
// tokens of a batch item, in 16-byte pieces as they lie in memory, so that a thread has the same piece of every token it reads.
struct GuessArgs {
    const __nv_bfloat16 *Y, *dY;   // [B,N,H,D]
    const float *around;           // see z_around
    float *e;                      // [B,N,H]
    int H, N, blocks;              // blocks: of latents per head
    int chunk, chunks, groups;     // groups: of at most kReduceThreads pieces of a token
};
template <int D> struct GuessGeom {
    static constexpr int F = 8, LPR = D / F;                    // features of a piece, pieces of a row
};
template <int D>
__device__ __forceinline__ void bwd_guess(int block, const GuessArgs &a) {
    using G = GuessGeom<D>;
    const int pieces = a.H * G::LPR, here = min(pieces, kReduceThreads), per = kReduceThreads / here;   // of a token, of a token in a block; tokens at a time
    const int group = block % a.groups, chunk = block / a.groups % a.chunks, b = block / a.groups / a.chunks;
    const int piece = group * kReduceThreads + threadIdx.x % here, tok = threadIdx.x / here;
    const bool live = tok < per && piece < pieces;
    const int q = live ? piece : (int)threadIdx.x % G::LPR, h = q / G::LPR, f0 = q % G::LPR * G::F;
    const float *around = a.around + ((size_t)b * a.H + h) * (1 + a.blocks) * D + f0;
    float cen[G::F], most[G::F];
#pragma unroll
    for (int k = 0; k < G::F; ++k) {
        cen[k] = around[k];
        most[k] = around[D + k];
    }
    for (int m = 2; m <= a.blocks; ++m)
#pragma unroll
        for (int k = 0; k < G::F; ++k) most[k] = fmaxf(most[k], around[m * D + k]);
    struct alignas(2 * G::F) Piece { __nv_bfloat162 w[G::F / 2]; };
    const Piece *Y = reinterpret_cast<const Piece *>(a.Y) + (size_t)b * a.N * pieces + q, *dY = reinterpret_cast<const Piece *>(a.dY) + (size_t)b * a.N * pieces + q;
    const int n1 = min(a.N, (chunk + 1) * a.chunk);
#pragma unroll 4
    for (int n = chunk * a.chunk + tok; n - tok < n1; n += per) {
        const size_t at = (size_t)min(n, n1 - 1) * pieces;
        const Piece y = Y[at], g = dY[at];
        float sum = 0.f;
#pragma unroll
        for (int k = 0; k < G::F; ++k) {
            const float yk = k & 1 ? __high2float(y.w[k / 2]) : __low2float(y.w[k / 2]), gk = k & 1 ? __high2float(g.w[k / 2]) : __low2float(g.w[k / 2]);
            sum = fmaf(gk, fminf(fmaxf(yk - cen[k], -most[k]), most[k]), sum);
        }
#pragma unroll
        for (int o = 1; o < G::LPR; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (live && f0 == 0 && n < n1) a.e[((size_t)b * a.N + n) * a.H + h] = sum;
    }
}

// dZ[row] = sum_p part[p][row] and de[row] = dZ_row . Z_row; blocks from row_blocks on: e, see bwd_guess.
template <int L>
__global__ void __launch_bounds__(kReduceThreads)
bwd_dz_reduce_kernel(const float *part, const float *Z, float *dZ, float *de, int P, long rows, int slices, int row_blocks, GuessArgs guess) {
    ptx::grid_launch();
    ptx::grid_wait();
    if ((int)blockIdx.x >= row_blocks) {
        if constexpr (L >= 8) bwd_guess<4 * L>((int)blockIdx.x - row_blocks, guess);   // (narrower heads have no use for it)
        return;
    }
    const RowMap rm = row_map<L>(slices);
    const bool live = rm.row < rows;
    const long at = (live ? rm.row : rows - 1) * L + rm.lane;
    const float4 *p4 = reinterpret_cast<const float4 *>(part) + at;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int p = rm.slice; p < P; p += slices) s = f4_add(s, p4[(size_t)p * rows * L]);
    s = sum_slices<L>(s, slices);
    const float4 z = reinterpret_cast<const float4 *>(Z)[at];
    // de is summed in double, as the CUDA-core kernels sum dZ_m . V_n: where a latent follows a single token the two cancel
    double dot = fma((double)s.w, (double)z.w, fma((double)s.z, (double)z.z, fma((double)s.y, (double)z.y, (double)s.x * (double)z.x)));
#pragma unroll
    for (int o = 1; o < L; o <<= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if (!live || rm.slice != 0) return;
    reinterpret_cast<float4 *>(dZ)[at] = s;
    if (rm.lane == 0) de[rm.row] = (float)dot;
}

// dQ[h][m] = scale * sum_b sum_p part[p][(b, h, m)]: the B * P terms of a row in index order per slice.
template <int L>
__global__ void __launch_bounds__(kReduceThreads)
bwd_dq_reduce_kernel(const float *part, float *dQ, int P, int B, long per_batch, float scale, int slices) {
    ptx::grid_launch();
    ptx::grid_wait();
    const RowMap rm = row_map<L>(slices);
    const bool live = rm.row < per_batch;
    const long at = (live ? rm.row : per_batch - 1) * L + rm.lane;
    const float4 *p4 = reinterpret_cast<const float4 *>(part) + at;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int q = rm.slice; q < B * P; q += slices) s = f4_add(s, p4[(size_t)q * per_batch * L]);   // part is [P][B][H*M] rows: q = p * B + b
    s = sum_slices<L>(s, slices);
    if (live && rm.slice == 0)
        reinterpret_cast<float4 *>(dQ)[at] = make_float4(s.x * scale, s.y * scale, s.z * scale, s.w * scale);
}

// Launch of one of the kernels above with L = D / 4 as a template parameter.
#define FLARE_REDUCE(kernel, rows_, P_, D_, st_, ...)                                            \
    do {                                                                                         \
        const int slices__ = reduce_slices(P_, D_);                                              \
        const unsigned blocks__ = reduce_blocks(rows_, D_, slices__);                            \
        switch (D_) {                                                                            \
            case 4: FLARE_CUDA(launch_after(kernel<1>, blocks__, kReduceThreads, 0, st_, __VA_ARGS__, slices__)); break;\
            case 8: FLARE_CUDA(launch_after(kernel<2>, blocks__, kReduceThreads, 0, st_, __VA_ARGS__, slices__)); break;\
            case 16: FLARE_CUDA(launch_after(kernel<4>, blocks__, kReduceThreads, 0, st_, __VA_ARGS__, slices__)); break;                 \
            case 32: FLARE_CUDA(launch_after(kernel<8>, blocks__, kReduceThreads, 0, st_, __VA_ARGS__, slices__)); break;                 \
            default: FLARE_CUDA(launch_after(kernel<16>, blocks__, kReduceThreads, 0, st_, __VA_ARGS__, slices__)); break;                \
        }                                                                                        \
        FLARE_CUDA(cudaGetLastError());                                                          \
    } while (0)

}  // namespace flare
