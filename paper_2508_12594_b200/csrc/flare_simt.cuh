// Kernels of the FLARE mixer for float32 and float16 inputs (and the bfloat16 shapes the tensor-core kernels do not take).
//
// float32 inputs must meet a 1e-5 relative tolerance, which the tensor cores' reduced-mantissa float32 mode cannot.  Here
// every score q.k is summed in double precision, by the double-precision MMA (m8n8k4), and rounded once; exponentials
// are one ex2 each, put right to first order (exp_diff); the value contractions run on the double-precision MMA too, their sums in double.  What bounds them is that pipe:
// 64 multiply-adds per clock per SM, D of them per (row, column) pair and product, 0.25 clocks per pair, product and SM at D = 16.
//
// All of them share one shape.  "Rows" (latents in encode, dZ and dQ; tokens in decode and the token pass) stay in
// registers as A fragments, RB blocks of 8 rows per warp; "columns" (the other kind) stream through shared memory in tiles
// of CT, as doubles.  In a C fragment a thread holds row g = lane / 4 and two columns, what an A fragment asks of it with those two as the
// K index of two steps: the weights go from one MMA into the next in the same registers, only rounded to float and back on the way.
// (As float32 FMAs, every thread adding up whole rows over its own columns, the contractions and their shared-memory reads took
// as long again as the scores.)  Which two columns is chosen (column_slot) so that neither the fragments of the scores nor those of the values
// meet bank conflicts, with rows of D + 4 doubles.
#pragma once

#include <cooperative_groups.h>

#include "flare_ptx.cuh"
#include "flare_common.cuh"

namespace flare {

template <int D> struct SimtGeom {
    static constexpr int CT = D <= 32 ? 64 : 32;                     // columns per tile
    static constexpr int DK = D + (D == 4 ? 0 : 4);                  // padded row length of a tile of doubles
    static constexpr int NB = D < 8 ? 1 : D / 8;                     // blocks of 8 features of a row
};
// The column of a block of eight that is index j of the scores' MMA, and the other way round.  Thread q of a quad then has columns 0,1 | 2,3 | 5,4 |
// 7,6: as rows of a tile, of 8 (mod 32) banks each, the first of the four (second likewise) lie in different banks, and so do those of
// indices 0-3 and 4-7.
__host__ __device__ constexpr int column_slot(int j) { return j ^ ((j >> 2) & 1); }

// D (8x8, f64) += A (8x4, row lane / 4, k lane % 4) * B (4x8, k lane % 4, column lane / 4)
__device__ __forceinline__ void dmma(double2 &c, double a, double b) {
    asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c.x), "+d"(c.y) : "d"(a), "d"(b));
}

template <class F>
__device__ __forceinline__ F quad_sum(F x) {
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
    // kCentred: less `centre`
    template <bool kCentred = false>
    __device__ __forceinline__ void put_double(double *dst, const float *centre = nullptr) const {
        each([&](int r, int c, const Vec &x) {
            double2 *p = reinterpret_cast<double2 *>(dst + r * SimtGeom<D>::DK + c);
            auto at = [&](int k) { return (double)to_f32(x.e[k]) - (kCentred ? (double)centre[c + k] : 0.0); };
            if constexpr (VE == 4) {
                const bool odd = r & 1;
                const double2 lo = make_double2(at(0), at(1)), hi = make_double2(at(2), at(3));
                p[odd] = odd ? hi : lo;
                p[!odd] = odd ? lo : hi;
            } else {
#pragma unroll
                for (int k = 0; k < VE / 2; ++k) p[k] = make_double2(at(2 * k), at(2 * k + 1));
            }
        });
    }
};

// A fragments of RB row blocks: row r0 + 8 rb + lane / 4, element 4 kk + lane % 4, less `centre` (null: nothing), times f; rows from `rows` on
// are zeros.
template <typename T, int D, int RB>
__device__ __forceinline__ void load_rows(double (&a)[RB][D / 4], const T *src, size_t stride, int r0, int rows, double f,
                                          const float *centre = nullptr) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        const int r = r0 + 8 * rb + (lane >> 2);
#pragma unroll
        for (int kk = 0; kk < D / 4; ++kk) {
            const double c = centre != nullptr ? (double)centre[4 * kk + (lane & 3)] : 0.0;
            a[rb][kk] = r < rows ? ((double)to_f32(src[(size_t)r * stride + 4 * kk + (lane & 3)]) - c) * f : 0.0;
        }
    }
}
// c[rb] = the 8 x 8 products of the row blocks with columns nb * 8 ... of a double tile
template <int D, int RB>
__device__ __forceinline__ void mma_block(double2 (&c)[RB], const double (&a)[RB][D / 4], const double *tile, int nb) {
    const int lane = threadIdx.x & 31;
    const double *b = tile + (nb * 8 + column_slot(lane >> 2)) * SimtGeom<D>::DK + (lane & 3);
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) c[rb] = make_double2(0.0, 0.0);
#pragma unroll
    for (int kk = 0; kk < D / 4; ++kk) {
        const double bk = b[4 * kk];
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) dmma(c[rb], a[rb][kk], bk);
    }
}
// B fragments of a block of eight columns for the value contractions: v[e][j] = element 8 j + lane / 4 of the row that is the thread's
// (quad lane's) column e.
template <int D>
__device__ __forceinline__ void load_values(double (&v)[2][SimtGeom<D>::NB], const double *tile, int nb) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const double *b = tile + (nb * 8 + column_slot(2 * (lane & 3) + e)) * SimtGeom<D>::DK + (lane >> 2);
#pragma unroll
        for (int j = 0; j < SimtGeom<D>::NB; ++j) v[e][j] = D >= 8 || lane < 4 * D ? b[8 * j] : 0.0;
    }
}
// acc += weights of the thread's two columns * values: row lane / 4 of a block, elements 8 j + 2 (lane % 4), + 1
template <int D, int RB, class W>                               // W: float2 or double2
__device__ __forceinline__ void add_values(double2 (&acc)[RB][SimtGeom<D>::NB], const W (&w)[RB], const double (&v)[2][SimtGeom<D>::NB]) {
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) {
            const double we = (double)(e ? w[rb].y : w[rb].x);
#pragma unroll
            for (int j = 0; j < SimtGeom<D>::NB; ++j) dmma(acc[rb][j], we, v[e][j]);
        }
}
template <int D, int RB>
__device__ __forceinline__ void clear_rows(double2 (&acc)[RB][SimtGeom<D>::NB]) {
#pragma unroll
    for (int rb = 0; rb < RB; ++rb)
#pragma unroll
        for (int j = 0; j < SimtGeom<D>::NB; ++j) acc[rb][j] = make_double2(0.0, 0.0);
}
// The row a quad holds, times f, written by its four threads.
template <typename T, int D>
__device__ __forceinline__ void write_row(T *dst, const double2 (&acc)[SimtGeom<D>::NB], double f) {
    const int q = threadIdx.x & 3;
    if (D < 8 && 2 * q >= D) return;
    struct alignas(2 * sizeof(T)) Pair { T x, y; };
#pragma unroll
    for (int j = 0; j < SimtGeom<D>::NB; ++j) {
        Pair p;
        from_f32(p.x, (float)(acc[j].x * f));
        from_f32(p.y, (float)(acc[j].y * f));
        *reinterpret_cast<Pair *>(dst + 8 * j + 2 * q) = p;
    }
}

// exp of a score, once rounded to float, less a reference or a log-sum-exp (which was formed from scores rounded the same way: the rounding of the
// largest ones cancels; with the difference taken in double and rounded after it a weight near 1 was off by the log-sum-exp's last place,
// the largest entries of dV three times as much).  e^x = 2^y e^(x - y ln 2) with y = x log2(e) as it was rounded: what is left of x, some x / 2^24, to
// first order.  (Without, the weights of the backward over N flat scores, where x is -log N, were off by 4.7e-7 instead of 2.8e-7 at 131072 tokens, root
// mean square; what is left is the rounding of x.  expf gives the same and takes 3 % of a float16 training step more.)
__device__ __forceinline__ float exp_diff(float x) {
    const float y = x * 1.4426950408889634f, w = ptx::ex2(y);
    const float rest = fmaf(-y, -1.9046542e-9f, fmaf(-y, 0.69314718f, x));   // (ln 2 in two parts)
    return fmaf(w, fmaxf(rest, -1.f), w);                       // (x = -inf: rest is NaN, w is 0)
}

// Running softmax state of the rows of a warp.  The reference m of a row (the same in the four threads of its quad) is not the running maximum
// but a score within kSlack of it: what weighs most has a small exponent (see exp_diff; with 20, lse_enc was off by up to 1.6 of its last place), and
// rescaling, a branch of the whole warp, is rare.
constexpr float kNoScore = -1.0e30f, kSlack = 6.f;
template <int D, int RB>
struct RowState {
    float m[RB], l[RB];                                              // (l: over the thread's own columns)
    double2 acc[RB][SimtGeom<D>::NB];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) {
            m[rb] = kNoScore;
            l[rb] = 0.f;
        }
        clear_rows<D, RB>(acc);
    }
    // s: scores of the thread's two columns; their weights (0 for a score of -inf)
    __device__ __forceinline__ void weights(const float2 (&s)[RB], float2 (&p)[RB]) {
        bool far = false;
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) far = far || fmaxf(s[rb].x, s[rb].y) > m[rb] + kSlack;
        if (__any_sync(0xffffffffu, far)) {
#pragma unroll
            for (int rb = 0; rb < RB; ++rb) {
                const float mx = quad_max(fmaxf(s[rb].x, s[rb].y));
                if (mx > m[rb] + kSlack) {
                    const float f = exp_diff(m[rb] - mx);
                    m[rb] = mx;
                    l[rb] *= f;
#pragma unroll
                    for (int j = 0; j < SimtGeom<D>::NB; ++j) acc[rb][j] = make_double2(acc[rb][j].x * f, acc[rb][j].y * f);
                }
            }
        }
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) {
            p[rb] = make_float2(exp_diff(s[rb].x - m[rb]), exp_diff(s[rb].y - m[rb]));
            l[rb] += p[rb].x + p[rb].y;
        }
    }
};

// What a block of the kernels below does with the tokens n0 ... n1 - 1 (there may be none): its eight warps are WM groups of 8 RB latents, from
// rbase on, x WT = 8 / WM shares of a tile's columns.  Leaves the shares of every latent in shared memory, [WT][WM * RW rows] rows of (acc, m, l)
// of D + 4 floats.  kDz: the backward's dZ form: dY in place of V, weights exp(score - lse_dec[n]), no maximum and no sum.
template <typename T, int D, int RB, bool kDz>
__device__ __forceinline__ void encode_tokens(unsigned char *simt_smem, const T *Q, const T *K, const T *V, const uint8_t *key_mask, const float *lse_dec,
                                              int b, int h, int H, int N, int M, int WM, int rbase, int n0, int n1, float scale) {
    using SG = SimtGeom<D>;
    constexpr int CT = SG::CT, RW = 8 * RB;
    double *sK = reinterpret_cast<double *>(simt_smem);             // [CT][DK]
    double *sV = sK + CT * SG::DK;                                  // [CT][DK]
    float *sBias = reinterpret_cast<float *>(sV + CT * SG::DK);     // [CT]: added to a column's scores (in the order of the MMA's indices)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int WT = kSimtThreads / 32 / WM, wm = warp % WM, wt = warp / WM;
    const int r0 = rbase + wm * RW;
    const size_t stride = (size_t)H * D;
    const T *Kb = K + ((size_t)b * N * H + h) * D, *Vb = V + ((size_t)b * N * H + h) * D;
    using Fetch = TileFetch<T, D, kSimtThreads>;
    unsigned char *raw = reinterpret_cast<unsigned char *>(sBias + CT);
    Fetch fk(raw), fv(raw + Fetch::kBytes);
    fk.load(Kb + n0 * stride, stride, n1 - n0);
    fv.load(Vb + n0 * stride, stride, n1 - n0);
    double aq[RB][D / 4];
    load_rows<T, D, RB>(aq, Q + (size_t)h * M * D, D, r0, M, (double)scale);
    RowState<D, RB> st;
    st.clear();
    for (int t0 = n0; t0 < n1; t0 += CT) {
        Fetch::wait();
        __syncthreads();
        fk.put_double(sK);
        fv.put_double(sV);
        if (threadIdx.x < CT) {
            const int n = t0 + threadIdx.x;
            float bias = -INFINITY;
            if (n < n1) {
                if (kDz) bias = -lse_dec[((size_t)b * N + n) * H + h];
                else if (key_mask == nullptr || key_mask[(size_t)b * N + n] != 0) bias = 0.f;
            }
            sBias[column_slot(threadIdx.x)] = bias;
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
                const float2 bias = *reinterpret_cast<const float2 *>(sBias + nb * 8 + 2 * (lane & 3));
                float2 sc[RB], p[RB];
                double v[2][SG::NB];
                load_values<D>(v, sV, nb);
#pragma unroll
                for (int rb = 0; rb < RB; ++rb) {
                    sc[rb] = make_float2((float)c[rb].x + bias.x, (float)c[rb].y + bias.y);
                    if (kDz) p[rb] = make_float2(exp_diff(sc[rb].x), exp_diff(sc[rb].y));
                }
                if (!kDz) st.weights(sc, p);
                add_values<D, RB>(st.acc, p, v);
            }
    }
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        if (kDz) st.m[rb] = 0.f;
        st.l[rb] = quad_sum(st.l[rb]);
    }
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
        write_row<float, D>(dst, st.acc[rb], 1.0);
    }
    __syncthreads();
}
// Encode, split over N.  grid = (splits, H * mblocks, B).  One partial (m, l, row) per latent and split.
template <typename T, int D, int RB, bool kDz>
__global__ void __launch_bounds__(kSimtThreads, 2)
encode_simt_kernel(const T *Q, const T *K, const T *V, const uint8_t *key_mask,
                   const float *lse_dec, float *part_m, float *part_l,
                   float *part_acc, int B, int H, int N, int M, int WM, int mblocks, int chunk, float scale) {
    ptx::grid_launch();
    ptx::grid_wait();
    extern __shared__ __align__(16) unsigned char simt_smem[];
    const int split = blockIdx.x, h = blockIdx.y / mblocks, b = blockIdx.z, rbase = blockIdx.y % mblocks * WM * 8 * RB;
    const int n0 = split * chunk, n1 = min(N, n0 + chunk);
    encode_tokens<T, D, RB, kDz>(simt_smem, Q, K, V, key_mask, lse_dec, b, h, H, N, M, WM, rbase, n0, n1, scale);
    const float *sR = reinterpret_cast<const float *>(simt_smem);
    constexpr int ROW = D + 4;
    const int rows_here = WM * 8 * RB, WT = kSimtThreads / 32 / WM;
    const long rows = (long)B * H * M;
    for (int i = threadIdx.x; i < rows_here * D; i += kSimtThreads) {
        const int r = i / D, d = i % D, m = rbase + r;
        if (m >= M) continue;
        float top = kNoScore, l = 0.f, z = 0.f;
        for (int w = 0; w < WT; ++w) top = fmaxf(top, sR[((size_t)w * rows_here + r) * ROW + D]);
        for (int w = 0; w < WT; ++w) {
            const float *src = sR + ((size_t)w * rows_here + r) * ROW;
            const float f = kDz ? 1.f : exp_diff(src[D] - top);
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
    const size_t tiles = sizeof(double) * 2 * SG::CT * SG::DK + sizeof(float) * SG::CT + 2 * sizeof(T) * SG::CT * D;
    const size_t join = sizeof(float) * (kSimtThreads / 32) * 8 * RB * (D + 4);
    return tiles > join ? tiles : join;
}

// mc latents, in tiles of doubles, against the token rows of a warp
template <int D, int RB>
__device__ __forceinline__ void decode_tile(RowState<D, RB> &st, const double (&ak)[RB][D / 4], const double *sQ, const double *sZ, int mc) {
    const int lane = threadIdx.x & 31;
    for (int nb = 0; nb < (mc + 7) / 8; ++nb) {
        double2 c[RB];
        mma_block<D, RB>(c, ak, sQ, nb);
        const bool in0 = nb * 8 + column_slot(2 * (lane & 3)) < mc, in1 = nb * 8 + column_slot(2 * (lane & 3) + 1) < mc;
        float2 sc[RB], p[RB];
        double v[2][SimtGeom<D>::NB];
        load_values<D>(v, sZ, nb);
#pragma unroll
        for (int rb = 0; rb < RB; ++rb) sc[rb] = make_float2(in0 ? (float)c[rb].x : -INFINITY, in1 ? (float)c[rb].y : -INFINITY);
        st.weights(sc, p);
        add_values<D, RB>(st.acc, p, v);
    }
}
// rows r0 ... of Y and lse_dec, up to row `end`
template <typename T, int D, int RB>
__device__ __forceinline__ void decode_rows_out(const RowState<D, RB> &st, T *Y, float *lse_dec, int r0, int end, int b, int h, int N, int H) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int rb = 0; rb < RB; ++rb) {
        const int n = r0 + 8 * rb + (lane >> 2);
        const float l = quad_sum(st.l[rb]);
        if (n >= end) continue;
        const size_t tok = ((size_t)b * N + n) * H + h;
        write_row<T, D>(Y + tok * D, st.acc[rb], 1.0 / (double)l);
        if (lse_dec != nullptr && (lane & 3) == 0) lse_dec[tok] = st.m[rb] + logf(l);
    }
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
    double *sZ = sQ + CT * SG::DK;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, h = blockIdx.y, b = blockIdx.z;
    const int r0 = (blockIdx.x * (kSimtThreads / 32) + warp) * 8 * RB;
    const T *Qh = Q + (size_t)h * M * D;
    const float *Zh = Z + ((size_t)b * H + h) * M * D;
    unsigned char *raw = reinterpret_cast<unsigned char *>(sZ + CT * SG::DK);
    TileFetch<T, D, kSimtThreads> fq(raw);
    TileFetch<float, D, kSimtThreads> fz(raw + fq.kBytes);
    fq.load(Qh, D, M);
    fz.load(Zh, D, M);
    double ak[RB][D / 4];
    load_rows<T, D, RB>(ak, K + ((size_t)b * N * H + h) * D, (size_t)H * D, r0, N, (double)scale);
    RowState<D, RB> st;
    st.clear();
    for (int m0 = 0; m0 < M; m0 += CT) {
        fq.wait();
        __syncthreads();
        fq.put_double(sQ);
        fz.put_double(sZ);
        __syncthreads();
        if (m0 + CT < M) {
            fq.load(Qh + (size_t)(m0 + CT) * D, D, M - m0 - CT);
            fz.load(Zh + (size_t)(m0 + CT) * D, D, M - m0 - CT);
        }
        const int mc = min(CT, M - m0);
        if (r0 < N)
            decode_tile<D, RB>(st, ak, sQ, sZ, mc);
    }
    decode_rows_out<T, D, RB>(st, Y, lse_dec, r0, N, b, h, N, H);
}
template <typename T, int D> inline size_t decode_simt_smem() {
    return sizeof(double) * 2 * SimtGeom<D>::CT * SimtGeom<D>::DK + (sizeof(T) + sizeof(float)) * SimtGeom<D>::CT * D;
}

// The whole forward of a small problem in one launch: a cluster of CS blocks per (batch item, head), each with its share of the tokens.
// Encode as above; the blocks join their partial rows through each other's shared memory, every block its share of the latents, whose Z it
// hands to all; decode of the block's tokens against that Z.  Three launches take 2 to 3 us each whatever there is to do, and the host as long to
// queue them.  (Which problems: see small_forward_wanted.)
constexpr int kSmallMaxM = 64;
template <int D> struct SmallGeom {
    using SG = SimtGeom<D>;
    static constexpr int PS = D + 2;                                 // a partial row in shared memory: acc, m, l
    static_assert(SG::CT >= kSmallMaxM || D > 32, "all latents are one tile");
};
template <typename T, int D> inline size_t forward_small_smem() { return encode_simt_smem<T, D>(1) + sizeof(float) * kSmallMaxM * SmallGeom<D>::PS; }
template <typename T, int D, int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(kSimtThreads, 2)
forward_small_simt_kernel(const T *Q, const T *K, const T *V, const uint8_t *key_mask, float *Z, float *lse_enc, T *Y, float *lse_dec,
                          uint32_t *header, int H, int N, int M, int WM, int chunk, float scale, int partials_at) {
    ptx::grid_launch();
    ptx::grid_wait();
    using SG = SimtGeom<D>;
    constexpr int ROW = D + 4, PS = SmallGeom<D>::PS;
    extern __shared__ __align__(16) unsigned char simt_smem[];
    const int rank = blockIdx.x, h = blockIdx.y, b = blockIdx.z, warp = threadIdx.x >> 5;
    const int n0 = min(N, rank * chunk), n1 = min(N, n0 + chunk);
    if (header != nullptr && rank == 0 && h == 0 && b == 0 && threadIdx.x < kHeaderBytes / 4) header[threadIdx.x] = 0u;
    encode_tokens<T, D, 1, false>(simt_smem, Q, K, V, key_mask, nullptr, b, h, H, N, M, WM, 0, n0, n1, scale);
    const float *sR = reinterpret_cast<const float *>(simt_smem);
    float *sP = reinterpret_cast<float *>(simt_smem + partials_at);
    double *sQ = reinterpret_cast<double *>(simt_smem), *sZ = sQ + SG::CT * SG::DK;
    const int rows_here = WM * 8, WT = kSimtThreads / 32 / WM;
    for (int i = threadIdx.x; i < M * D; i += kSimtThreads) {
        const int r = i / D, d = i % D;
        float top = kNoScore, l = 0.f, z = 0.f;
        for (int w = 0; w < WT; ++w) top = fmaxf(top, sR[((size_t)w * rows_here + r) * ROW + D]);
        for (int w = 0; w < WT; ++w) {
            const float *src = sR + ((size_t)w * rows_here + r) * ROW, f = exp_diff(src[D] - top);
            l = fmaf(src[D + 1], f, l);
            z = fmaf(src[d], f, z);
        }
        sP[r * PS + d] = z;
        if (d == 0) {
            sP[r * PS + D] = top;
            sP[r * PS + D + 1] = l;
        }
    }
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    TileFetch<T, D, kSimtThreads>::wait();                           // (of a block without tokens)
    TileFetch<T, D, kSimtThreads> fq(simt_smem + sizeof(double) * 2 * SG::CT * SG::DK + sizeof(float) * SG::CT);
    fq.load(Q + (size_t)h * M * D, D, M);
    cluster.sync();                                                  // partial rows are there, and tiles and shares are done with
    fq.wait();
    fq.put_double(sQ);
    for (int i = threadIdx.x; i < ((M + 7) / 8 * 8 - M) * SG::DK; i += kSimtThreads) sZ[M * SG::DK + i] = 0.0;
    const int mine = (M - rank + CS - 1) / CS;  // latents rank, rank + CS, ...
    for (int i = threadIdx.x; i < mine * D; i += kSimtThreads) {
        const int m = rank + i / D * CS, d = i % D;
        float pm[CS], pl[CS], pz[CS], top = kNoScore;
#pragma unroll
        for (int p = 0; p < CS; ++p) {
            const float *row = cluster.map_shared_rank(sP, p) + m * PS;
            pm[p] = row[D];
            pl[p] = row[D + 1];
            pz[p] = row[d];
        }
#pragma unroll
        for (int p = 0; p < CS; ++p) top = fmaxf(top, pm[p]);
        float l = 0.f, z = 0.f;
#pragma unroll
        for (int p = 0; p < CS; ++p) {
            const float f = exp_diff(pm[p] - top);
            l = f > 0.f ? fmaf(pl[p], f, l) : l;
            z = f > 0.f ? fmaf(pz[p], f, z) : z;
        }
        const bool none = top == kNoScore;                           // no valid token anywhere
        z = none ? 0.f : z * (1.f / l);
#pragma unroll
        for (int p = 0; p < CS; ++p) cluster.map_shared_rank(sZ, p)[m * SG::DK + d] = (double)z;
        const size_t row = ((size_t)b * H + h) * M + m;
        if (Z != nullptr) Z[row * D + d] = z;
        if (lse_enc != nullptr && d == 0) lse_enc[row] = none ? -INFINITY : top + logf(l);
    }
    const T *Kh = K + ((size_t)b * N * H + h) * D;
    int r0 = n0 + warp * 8;
    double ak[1][D / 4];
    load_rows<T, D, 1>(ak, Kh, (size_t)H * D, r0, n1, (double)scale);   // (on their way across the barrier)
    cluster.sync();
    for (; r0 < n1; r0 += kSimtThreads / 32 * 8) {
        if (r0 >= n0 + kSimtThreads / 32 * 8) load_rows<T, D, 1>(ak, Kh, (size_t)H * D, r0, n1, (double)scale);
        RowState<D, 1> st;
        st.clear();
        decode_tile<D, 1>(st, ak, sQ, sZ, M);
        decode_rows_out<T, D, 1>(st, Y, lse_dec, r0, n1, b, h, N, H);
    }
}

}  // namespace flare
