// Kernels of the FLARE mixer for float32 and float16 inputs (and the bfloat16 shapes the tensor-core kernels do not take).
//
// float32 inputs must meet a 1e-5 relative tolerance, which the tensor cores' reduced-mantissa float32 mode cannot.  Here
// every score q.k is summed in double precision, by the double-precision MMA (m8n8k4), and rounded once; exponentials
// are expf, the value contractions float32 FMAs.  What bounds them is the double-precision pipe: 64 multiply-adds per clock
// per SM, D of them per (row, column) pair and product, so 0.25 clocks per pair and SM at D = 16 (a thread per row with
// scalar double FMAs took 2.1 to 2.4: converting both operands of every product in the inner loop, 16 conversions per clock, was
// most of it; 0.9 now, encode and decode at D = 16).
//
// All of them share one shape.  "Rows" (latents in encode, dZ and dQ; tokens in decode and the token pass) stay in
// registers as A fragments, RB blocks of 8 rows per warp; "columns" (the other kind) stream through shared memory in tiles
// of CT, as doubles for the B fragments and as floats for the value contraction.  In a C fragment a thread holds row
// lane / 4 and columns 2 (lane % 4), + 1, so it weights two rows of the value tile per MMA and keeps a partial
// accumulator of its row over its own columns; the four lanes of a row meet once, at the end.  Row strides are padded by four
// elements: B fragments and value rows are then read without bank conflicts.
#pragma once

#include "flare_ptx.cuh"
#include "flare_common.cuh"

namespace flare {

template <int D> struct SimtGeom {
    static constexpr int CT = D <= 32 ? 64 : 32;                     // columns per tile
    static constexpr int DK = D + (D == 4 ? 0 : 4), DV = D + 4;      // padded row lengths of double and float tiles
};

// D (8x8, f64) += A (8x4, row lane / 4, k lane % 4) * B (4x8, k lane % 4, column lane / 4)
__device__ __forceinline__ void dmma(double2 &c, double a, double b) {
    asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c.x), "+d"(c.y) : "d"(a), "d"(b));
}

// Packed-pair helpers: value rows are read four floats at a time and accumulated two at a time.
template <int D>
__device__ __forceinline__ void axpy2(float2 *acc, float w, const float *row) {
    const float2 wp = make_float2(w, w);
#pragma unroll
    for (int d = 0; d < D; d += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(row + d);
        acc[d / 2] = __ffma2_rn(wp, make_float2(v.x, v.y), acc[d / 2]);
        acc[d / 2 + 1] = __ffma2_rn(wp, make_float2(v.z, v.w), acc[d / 2 + 1]);
    }
}
__device__ __forceinline__ float quad_sum(float x) {
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x + __shfl_xor_sync(0xffffffffu, x, 2);
}
__device__ __forceinline__ float quad_max(float x) {
    x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
    return fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2));
}

// A tile of CT rows of D elements on its way from global to shared memory: fetched a tile ahead by asynchronous copies into
// a raw buffer (a thread converts what it has copied itself, so the buffer needs no barrier of its own and the fetch no
// registers), 16 bytes (or a row, if that is shorter) per copy.
template <typename T, int D, int TH>
struct TileFetch {
    static constexpr int CT = SimtGeom<D>::CT;
    static constexpr int VE = (16 / (int)sizeof(T)) < D ? 16 / (int)sizeof(T) : D;   // elements per copy
    static constexpr int VB = VE * (int)sizeof(T), PR = D / VE, NV = (CT * PR + TH - 1) / TH;
    static constexpr size_t kBytes = (size_t)CT * D * sizeof(T);
    struct alignas(VB) Vec { T e[VE]; };
    Vec *raw;
    __device__ __forceinline__ explicit TileFetch(unsigned char *buffer) : raw(reinterpret_cast<Vec *>(buffer)) {}
    // row r of the tile is at src + r * stride; rows from `rows` on are zeros
    __device__ __forceinline__ void load(const T *src, size_t stride, int rows) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const int i = threadIdx.x + q * TH, r = i / PR, c = i % PR;
            if (r < CT) {
                const bool in = r < rows;
                asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(raw + i)),
                             "l"(src + (in ? (size_t)r * stride + c * VE : 0)), "n"(VB), "r"(in ? VB : 0)
                             : "memory");
            }
        }
    }
    static __device__ __forceinline__ void wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
    template <typename F>
    __device__ __forceinline__ void each(F f) const {             // f(row, first column, Vec)
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const int i = threadIdx.x + q * TH, r = i / PR, c = i % PR;
            if (r < CT) f(r, c * VE, raw[i]);
        }
    }
    // (pairs of doubles, neighbouring rows in opposite order: a quarter warp then covers all banks)
    __device__ __forceinline__ void put_double(double *dst) const {
        each([&](int r, int c, const Vec &x) {
            double2 *p = reinterpret_cast<double2 *>(dst + r * SimtGeom<D>::DK + c);
            if constexpr (VE == 4) {
                const bool odd = r & 1;
                const double2 lo = make_double2((double)to_f32(x.e[0]), (double)to_f32(x.e[1]));
                const double2 hi = make_double2((double)to_f32(x.e[2]), (double)to_f32(x.e[3]));
                p[odd] = odd ? hi : lo;
                p[!odd] = odd ? lo : hi;
            } else {
#pragma unroll
                for (int k = 0; k < VE / 2; ++k) p[k] = make_double2((double)to_f32(x.e[2 * k]), (double)to_f32(x.e[2 * k + 1]));
            }
        });
    }
    __device__ __forceinline__ void put_float(float *dst) const {
        each([&](int r, int c, const Vec &x) {
            float4 *p = reinterpret_cast<float4 *>(dst + r * SimtGeom<D>::DV + c);
#pragma unroll
            for (int k = 0; k < VE / 4; ++k)
                p[k] = make_float4(to_f32(x.e[4 * k]), to_f32(x.e[4 * k + 1]), to_f32(x.e[4 * k + 2]), to_f32(x.e[4 * k + 3]));
        });
    }
};

// A fragments of RB row blocks: row r0 + 8 rb + lane / 4, element 4 kk + lane % 4, times f; rows from `rows` on are zeros.
template <typename T, int D, int RB>
__device__ __forceinline__ void load_rows(double (&a)[RB][D / 4], const T *src, size_t stride, int r0, int rows, double f) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        const int r = r0 + 8 * rb + (lane >> 2);
#pragma unroll
        for (int kk = 0; kk < D / 4; ++kk) a[rb][kk] = r < rows ? (double)to_f32(src[(size_t)r * stride + 4 * kk + (lane & 3)]) * f : 0.0;
    }
}
// c[rb] = the 8 x 8 products of the row blocks with columns nb * 8 ... of a double tile
template <int D, int RB>
__device__ __forceinline__ void mma_block(double2 (&c)[RB], const double (&a)[RB][D / 4], const double *tile, int nb) {
    const int lane = threadIdx.x & 31;
    const double *b = tile + (nb * 8 + (lane >> 2)) * SimtGeom<D>::DK + (lane & 3);
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) c[rb] = make_double2(0.0, 0.0);
#pragma unroll
    for (int kk = 0; kk < D / 4; ++kk) {
        const double bk = b[4 * kk];
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) dmma(c[rb], a[rb][kk], bk);
    }
}

// Running softmax state of the rows of a thread, over its own columns.  The reference m is not the running maximum but a
// score within kSlack of it: exp(score - m) stays below e^20, and rescaling (a divergent branch) is rare.
constexpr float kNoScore = -1.0e30f, kSlack = 20.f;
template <int D, int RB>
struct RowState {
    float m[RB], l[RB];
    float2 acc[RB][D / 2];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) {
            m[rb] = kNoScore;
            l[rb] = 0.f;
#pragma unroll
            for (int d = 0; d < D / 2; ++d) acc[rb][d] = make_float2(0.f, 0.f);
        }
    }
    __device__ __forceinline__ void rescale(int rb, float f) {
        l[rb] *= f;
#pragma unroll
        for (int d = 0; d < D / 2; ++d) acc[rb][d] = make_float2(acc[rb][d].x * f, acc[rb][d].y * f);
    }
    // the weights of two columns of row block rb (scores of -inf weigh nothing)
    __device__ __forceinline__ float2 weights(int rb, float s0, float s1) {
        const float mx = fmaxf(s0, s1);
        if (mx > m[rb] + kSlack) {
            rescale(rb, expf(m[rb] - mx));
            m[rb] = mx;
        }
        const float2 p = make_float2(expf(s0 - m[rb]), expf(s1 - m[rb]));
        l[rb] += p.x + p.y;
        return p;
    }
    // the four lanes of every row joined; all four hold the result
    __device__ __forceinline__ void join_quad() {
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) {
            const float top = quad_max(m[rb]);
            rescale(rb, expf(m[rb] - top));
            m[rb] = top;
            l[rb] = quad_sum(l[rb]);
#pragma unroll
            for (int d = 0; d < D / 2; ++d) acc[rb][d] = make_float2(quad_sum(acc[rb][d].x), quad_sum(acc[rb][d].y));
        }
    }
};
// Element d of a row as float (d a constant after unrolling).
template <int D> __device__ __forceinline__ float pick(const float2 (&acc)[D / 2], int d) { return d & 1 ? acc[d / 2].y : acc[d / 2].x; }
// Lane q of a quad writes its quarter of a row of D elements.
template <typename T, int D>
__device__ __forceinline__ void write_quarter(T *dst, const float2 (&acc)[D / 2], float f) {
    constexpr int QD = D / 4;
    const int q = threadIdx.x & 3;
    struct alignas(sizeof(T) * QD < 16 ? sizeof(T) * QD : 16) Out { T e[QD]; } out;
#pragma unroll
    for (int k = 0; k < QD; ++k) {
        const float x01 = q & 1 ? pick<D>(acc, QD + k) : pick<D>(acc, k), x23 = q & 1 ? pick<D>(acc, 3 * QD + k) : pick<D>(acc, 2 * QD + k);
        from_f32(out.e[k], (q & 2 ? x23 : x01) * f);
    }
    *reinterpret_cast<Out *>(dst + q * QD) = out;
}

// Encode, split over N.  grid = (splits, H * mblocks, B); the block's eight warps are WM groups of 8 RB latents x WT = 8 / WM
// shares of a tile's columns.  The shares are joined in shared memory: one partial (m, l, row) per latent and split.
// kDz: the backward's dZ form: dY in place of V, weights exp(score - lse_dec[n]), no maximum and no sum.
template <typename T, int D, int RB, bool kDz>
__global__ void __launch_bounds__(kSimtThreads, 2)
encode_simt_kernel(const T *Q, const T *K, const T *V, const uint8_t *key_mask,
                   const float *lse_dec, float *part_m, float *part_l,
                   float *part_acc, int B, int H, int N, int M, int WM, int mblocks, int chunk, float scale) {
    ptx::grid_launch();
    ptx::grid_wait();
    using SG = SimtGeom<D>;
    constexpr int CT = SG::CT, RW = 8 * RB;
    extern __shared__ __align__(16) unsigned char simt_smem[];
    double *sK = reinterpret_cast<double *>(simt_smem);             // [CT][DK]
    float *sV = reinterpret_cast<float *>(sK + CT * SG::DK);        // [CT][DV]
    float *sBias = sV + CT * SG::DV;                                // [CT]: added to a column's scores
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = blockIdx.x, h = blockIdx.y / mblocks, mb = blockIdx.y % mblocks, b = blockIdx.z;
    const int WT = kSimtThreads / 32 / WM, wm = warp % WM, wt = warp / WM;
    const int rbase = mb * WM * RW, r0 = rbase + wm * RW;
    const int n0 = split * chunk, n1 = min(N, n0 + chunk);
    const size_t stride = (size_t)H * D;
    const T *Kb = K + ((size_t)b * N * H + h) * D, *Vb = V + ((size_t)b * N * H + h) * D;
    double aq[RB][D / 4];
    load_rows<T, D, RB>(aq, Q + (size_t)h * M * D, D, r0, M, (double)scale);
    RowState<D, RB> st;
    st.clear();
    using Fetch = TileFetch<T, D, kSimtThreads>;
    unsigned char *raw = reinterpret_cast<unsigned char *>(sBias + CT);
    Fetch fk(raw), fv(raw + Fetch::kBytes);
    fk.load(Kb + n0 * stride, stride, n1 - n0);
    fv.load(Vb + n0 * stride, stride, n1 - n0);
    for (int t0 = n0; t0 < n1; t0 += CT) {
        Fetch::wait();
        __syncthreads();
        fk.put_double(sK);
        fv.put_float(sV);
        if (threadIdx.x < CT) {
            const int n = t0 + threadIdx.x;
            float bias = -INFINITY;
            if (n < n1) {
                if (kDz) bias = -lse_dec[((size_t)b * N + n) * H + h];
                else if (key_mask == nullptr || key_mask[(size_t)b * N + n] != 0) bias = 0.f;
            }
            sBias[threadIdx.x] = bias;
        }
        __syncthreads();
        if (t0 + CT < n1) {
            fk.load(Kb + (size_t)(t0 + CT) * stride, stride, n1 - t0 - CT);
            fv.load(Vb + (size_t)(t0 + CT) * stride, stride, n1 - t0 - CT);
        }
        const int blocks = (min(CT, n1 - t0) + 7) / 8;
        if (r0 < M)
            for (int nb = wt; nb < blocks; nb += WT) {
                double2 c[RB];
                mma_block<D, RB>(c, aq, sK, nb);
                const int col = nb * 8 + 2 * (lane & 3);
                const float2 bias = *reinterpret_cast<const float2 *>(sBias + col);
                float2 p[RB];
#pragma unroll
                for (int rb = 0; rb < RB; ++rb) {
                    const float s0 = (float)c[rb].x + bias.x, s1 = (float)c[rb].y + bias.y;
                    p[rb] = kDz ? make_float2(expf(s0), expf(s1)) : st.weights(rb, s0, s1);
                }
#pragma unroll
                for (int d = 0; d < D; d += 4) {
                    const float4 v0 = *reinterpret_cast<const float4 *>(sV + col * SG::DV + d);
                    const float4 v1 = *reinterpret_cast<const float4 *>(sV + (col + 1) * SG::DV + d);
#pragma unroll
                    for (int rb = 0; rb < RB; ++rb) {
                        const float2 p0 = make_float2(p[rb].x, p[rb].x), p1 = make_float2(p[rb].y, p[rb].y);
                        float2 &x = st.acc[rb][d / 2], &y = st.acc[rb][d / 2 + 1];
                        x = __ffma2_rn(p1, make_float2(v1.x, v1.y), __ffma2_rn(p0, make_float2(v0.x, v0.y), x));
                        y = __ffma2_rn(p1, make_float2(v1.z, v1.w), __ffma2_rn(p0, make_float2(v0.z, v0.w), y));
                    }
                }
            }
    }
    if (kDz) {
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) st.m[rb] = 0.f;
    }
    st.join_quad();
    // the shares of the columns meet: [WT][WM * RW rows] rows of (acc, m, l)
    __syncthreads();
    constexpr int ROW = D + 4;
    float *sR = reinterpret_cast<float *>(simt_smem);
    const int rows_here = WM * RW;
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        float *dst = sR + ((size_t)wt * rows_here + wm * RW + 8 * rb + (lane >> 2)) * ROW;
        if ((lane & 3) == 0) {
            dst[D] = st.m[rb];
            dst[D + 1] = st.l[rb];
        }
        write_quarter<float, D>(dst, st.acc[rb], 1.f);
    }
    __syncthreads();
    const long rows = (long)B * H * M;
    for (int i = threadIdx.x; i < rows_here * D; i += kSimtThreads) {
        const int r = i / D, d = i % D, m = rbase + r;
        if (m >= M) continue;
        float top = kNoScore, l = 0.f, z = 0.f;
        for (int w = 0; w < WT; ++w) top = fmaxf(top, sR[((size_t)w * rows_here + r) * ROW + D]);
        for (int w = 0; w < WT; ++w) {
            const float *src = sR + ((size_t)w * rows_here + r) * ROW;
            const float f = kDz ? 1.f : expf(src[D] - top);
            l = fmaf(src[D + 1], f, l);
            z = fmaf(src[d], f, z);
        }
        const size_t prow = (size_t)split * rows + ((size_t)b * H + h) * M + m;
        part_acc[prow * D + d] = z;
        if (!kDz && d == 0) {
            part_m[prow] = top == kNoScore ? -INFINITY : top;
            part_l[prow] = l;
        }
    }
}
template <typename T, int D> inline size_t encode_simt_smem(int RB) {
    using SG = SimtGeom<D>;
    const size_t tiles = sizeof(double) * SG::CT * SG::DK + sizeof(float) * (SG::CT * SG::DV + SG::CT) + 2 * sizeof(T) * SG::CT * D;
    const size_t join = sizeof(float) * (kSimtThreads / 32) * 8 * RB * (D + 4);
    return tiles > join ? tiles : join;
}

// Decode: rows are tokens (8 RB per warp, the eight warps side by side), columns the latents.  grid = (ceil(N / (64 RB)), H, B).
template <typename T, int D, int RB>
__global__ void __launch_bounds__(kSimtThreads, 2)
decode_simt_kernel(const T *Q, const T *K, const float *Z, T *Y,
                   float *lse_dec, int B, int H, int N, int M, float scale) {
    ptx::grid_launch();
    ptx::grid_wait();
    using SG = SimtGeom<D>;
    constexpr int CT = SG::CT;
    extern __shared__ __align__(16) unsigned char simt_smem[];
    double *sQ = reinterpret_cast<double *>(simt_smem);
    float *sZ = reinterpret_cast<float *>(sQ + CT * SG::DK);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, h = blockIdx.y, b = blockIdx.z;
    const int r0 = (blockIdx.x * (kSimtThreads / 32) + warp) * 8 * RB;
    const T *Qh = Q + (size_t)h * M * D;
    const float *Zh = Z + ((size_t)b * H + h) * M * D;
    double ak[RB][D / 4];
    load_rows<T, D, RB>(ak, K + ((size_t)b * N * H + h) * D, (size_t)H * D, r0, N, (double)scale);
    RowState<D, RB> st;
    st.clear();
    unsigned char *raw = reinterpret_cast<unsigned char *>(sZ + CT * SG::DV);
    TileFetch<T, D, kSimtThreads> fq(raw);
    TileFetch<float, D, kSimtThreads> fz(raw + fq.kBytes);
    fq.load(Qh, D, M);
    fz.load(Zh, D, M);
    for (int m0 = 0; m0 < M; m0 += CT) {
        fq.wait();
        __syncthreads();
        fq.put_double(sQ);
        fz.put_float(sZ);
        __syncthreads();
        if (m0 + CT < M) {
            fq.load(Qh + (size_t)(m0 + CT) * D, D, M - m0 - CT);
            fz.load(Zh + (size_t)(m0 + CT) * D, D, M - m0 - CT);
        }
        const int mc = min(CT, M - m0);
        if (r0 < N)
            for (int nb = 0; nb < (mc + 7) / 8; ++nb) {
                double2 c[RB];
                mma_block<D, RB>(c, ak, sQ, nb);
                const int col = nb * 8 + 2 * (lane & 3);
                float2 p[RB];
#pragma unroll
                for (int rb = 0; rb < RB; ++rb)
                    p[rb] = st.weights(rb, col < mc ? (float)c[rb].x : -INFINITY, col + 1 < mc ? (float)c[rb].y : -INFINITY);
#pragma unroll
                for (int d = 0; d < D; d += 4) {
                    const float4 v0 = *reinterpret_cast<const float4 *>(sZ + col * SG::DV + d);
                    const float4 v1 = *reinterpret_cast<const float4 *>(sZ + (col + 1) * SG::DV + d);
#pragma unroll
                    for (int rb = 0; rb < RB; ++rb) {
                        const float2 p0 = make_float2(p[rb].x, p[rb].x), p1 = make_float2(p[rb].y, p[rb].y);
                        float2 &x = st.acc[rb][d / 2], &y = st.acc[rb][d / 2 + 1];
                        x = __ffma2_rn(p1, make_float2(v1.x, v1.y), __ffma2_rn(p0, make_float2(v0.x, v0.y), x));
                        y = __ffma2_rn(p1, make_float2(v1.z, v1.w), __ffma2_rn(p0, make_float2(v0.z, v0.w), y));
                    }
                }
            }
    }
    st.join_quad();
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        const int n = r0 + 8 * rb + (lane >> 2);
        if (n >= N) continue;
        const size_t tok = ((size_t)b * N + n) * H + h;
        write_quarter<T, D>(Y + tok * D, st.acc[rb], 1.f / st.l[rb]);
        if (lse_dec != nullptr && (lane & 3) == 0) lse_dec[tok] = st.m[rb] + logf(st.l[rb]);
    }
}
template <typename T, int D> inline size_t decode_simt_smem() {
    return sizeof(double) * SimtGeom<D>::CT * SimtGeom<D>::DK + sizeof(float) * SimtGeom<D>::CT * SimtGeom<D>::DV +
           (sizeof(T) + sizeof(float)) * SimtGeom<D>::CT * D;
}

}  // namespace flare
