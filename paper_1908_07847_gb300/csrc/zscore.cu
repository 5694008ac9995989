// Z-score normalisation of the feature table (Sec. 2.2 normalises the data
// before training; the reading: per-column mean and population standard
// deviation of the training rows, applied to every row; a column with no
// spread maps to 0), fused with the conversion to the padded layout the
// training kernels read (FP32, or bf16 with zero columns up to D_out).
//
// Statistics: two passes over the fit rows (sum, then squared deviations from
// the mean), accumulated in FP64.  Each block sums a contiguous slice of rows;
// inside a block, with D <= 256, 256 / D "row lanes" take every (256/D)-th row
// and are combined in lane order; the block partials are combined by one warp a
// column.  Every sum has a fixed order, so the statistics are bitwise
// reproducible.  The FP64 pipe (2 instructions a clock and SM) bounds a sum that
// converts and adds every element: 421 and 617 us a pass on 3M x 33 rows.  So 16
// rows at a time are first added in FP32 with their rounding errors kept
// (Knuth's two-sum; Ogita, Rump and Oishi, "Accurate sum and dot product", 2005,
// and the fused multiply-add's exact product error for the squares), and only the
// group's sum and error go to FP64: 71 and about 150 us a pass.
// The errors add up to 2^-24 of the sum and are themselves kept to 24 bits, so a
// group is off by about 2^-48 of one element, below the rounding of the FP64
// accumulator it is added to.  Groups whose values leave FP32's safe range
// (overflow, infinities, NaN, squares that would underflow) are added element by
// element in FP64.
//
// The normalisation pass is FP32: (x - m_hi) - m_lo with the mean split into two
// floats, times 1/s rounded to float; it is bound by HBM, so tiles of rows go
// through shared memory (4M x 33 floats in, 48 bf16 out, 912 MB: 292 us with an
// element a thread and its two-byte stores, 169 us).
#include <cuda_bf16.h>

#include "mlp_internal.cuh"

namespace mlp {
namespace {

constexpr int ZT = 256;

constexpr int ZG = 16;   // rows added in FP32 (with their errors) before FP64

// s + e = a + b exactly (two-sum, no overflow)
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

template <int N>
__device__ __forceinline__ void load_group(float (&v)[N], const float *p, int64_t step) {
#pragma unroll
    for (int u = 0; u < N; ++u) v[u] = __ldg(p + u * step);
}

// The same rows element by element in FP64 (kept out of line: inlined, the
// compiler ran its FP64 instructions for every group).
template <int P>
__device__ __noinline__ double add_fp64(double acc, const float *p, int64_t step, int n, double c) {
#pragma unroll 1
    for (int u = 0; u < n; ++u) {
        const double d = (double)p[u * step] - c;
        acc += P == 2 ? d * d : d;
    }
    return acc;
}

// acc += sum of v[u] (P = 1) or of (v[u] - c)^2 (P = 2, c = chi + clo up to
// 2^-49): a tree of two-sums over the group, the errors added in a fixed order.
template <int P, int N>
__device__ __forceinline__ void add_group(double &acc, const float (&v)[N], const float *p, int64_t step, double c,
                                          float chi, float clo) {
    float x[N];
    float m = 0.f, lo = 0.f;   // m: the largest |value| or |deviation|
#pragma unroll
    for (int u = 0; u < N; ++u) {
        float d = v[u], e = 0.f;
        if (P == 2) {
            // v - chi - clo as d + e, |e| <= 2^-24 |d|: exact but for e's own rounding
            two_sum(v[u], -chi, d, e);
            const float t = __fsub_rn(e, clo), s = __fadd_rn(d, t);
            e = __fsub_rn(t, __fsub_rn(s, d));
            d = s;
        }
        m = fabsf(d) < (P == 1 ? 1e36f : 1e18f) ? fmaxf(m, fabsf(d)) : 1e38f;   // NaN too: fmaxf would drop it
        x[u] = d;
        if (P == 2) {
            x[u] = __fmul_rn(d, d);
            lo = __fadd_rn(lo, __fmaf_rn(e, __fmaf_rn(2.f, d, e), __fmaf_rn(d, d, -x[u])));
        }
    }
    // squares of deviations below 1e-12 have errors that underflow
    if (m < 1e37f && (P == 1 || m > 1e-12f)) {
#pragma unroll
        for (int w = N / 2; w > 0; w >>= 1)
#pragma unroll
            for (int u = 0; u < w; ++u) {
                float e;
                two_sum(x[u], x[u + w], x[u], e);
                lo = __fadd_rn(lo, e);
            }
        acc += (double)x[0];
        acc += (double)lo;
    } else if (P == 2 && m == 0.f) {   // every value is chi, clo is 0 (a constant column)
        const double d = (double)chi - c;
        acc += (double)N * (d * d);
    } else {
        acc = add_fp64<P>(acc, p, step, N, c);
    }
}

// partial[b][j] = sum over the block's rows of (X[i][j] - centre[j])^p, p = 1 or 2
// (p = 1: the centre is 0).  GROUPS = false: fewer than four rows a lane, so that
// no group would form; the same sums without the groups' code (300 x 12 rows: 12.8 -> 12.5 us a call).
template <int P, bool GROUPS>
__global__ void __launch_bounds__(ZT) k_colsum(const float *__restrict__ X, int64_t n_fit, int D,
                                               const double *__restrict__ centre, double *__restrict__ partial) {
    __shared__ double red[ZT];
    const int b = blockIdx.x, G = gridDim.x, t = threadIdx.x;
    const int64_t r0 = n_fit * b / G, r1 = n_fit * (b + 1) / G;
    const int RL = D <= ZT ? ZT / D : 1;   // row lanes
    const int rl = D <= ZT ? t / D : 0;
    for (int j0 = 0; j0 < D; j0 += ZT) {   // one turn unless D > 256
        const int j = D <= ZT ? t % D : j0 + t;
        double acc = 0.0;
        if (rl < RL && j < D) {
            const double c = P == 2 ? centre[j] : 0.0;
            const float chi = (float)c, clo = (float)(c - (double)chi);
            int64_t i = r0 + rl;
            const float *p = X + i * D + j;
            const int64_t step = (int64_t)RL * D;
            if constexpr (GROUPS) {
                // a group's loads are in flight while the one before is added up (without
                // that the second pass waits for memory and takes 211 us)
                float v[ZG];
                bool more = i + (ZG - 1) * RL < r1;
                if (more) load_group<ZG>(v, p, step);
                while (more) {
                    const float *cur = p;
                    float w[ZG];
                    i += ZG * RL;
                    p += ZG * step;
                    more = i + (ZG - 1) * RL < r1;
                    load_group<ZG>(w, more ? p : cur, step);
                    add_group<P, ZG>(acc, v, cur, step, c, chi, clo);
#pragma unroll
                    for (int u = 0; u < ZG; ++u) v[u] = w[u];
                }
                for (; i + 3 * RL < r1; i += 4 * RL, p += 4 * step) {
                    float v4[4];
                    load_group<4>(v4, p, step);
                    add_group<P, 4>(acc, v4, p, step, c, chi, clo);
                }
            }
            for (; i < r1; i += RL, p += step) {
                const double d = (double)*p - c;
                acc += P == 2 ? d * d : d;
            }
        }
        if (D <= ZT) {
            red[t] = acc;
            __syncthreads();
            if (t < D) {
                double s = 0.0;
                for (int l = 0; l < RL; ++l) s += red[l * D + t];
                partial[(size_t)b * D + t] = s;
            }
        } else if (j < D) {
            partial[(size_t)b * D + j] = acc;
        }
    }
}

// out[j] = sum_b partial[b][j] / n_fit (P = 1: the mean), or its square root
// (P = 2: the population deviation); a warp a column (one thread a column took
// 70 us over 608 partials), or, of few partials, a thread: the warp's butterfly
// costs a call of 50 x 33 rows 1.8 us, of 1000 x 33 (12 partials) 0.7, and pays
// from some 16 partials on (1500 x 33: 15.8 us with warps, 16.7 with threads).
constexpr int FEW = 12;

template <int P>
__global__ void __launch_bounds__(ZT) k_colcombine(const double *__restrict__ partial, int G, int D, int64_t n_fit,
                                                   double *__restrict__ out) {
    const int t = blockIdx.x * ZT + threadIdx.x, lane = threadIdx.x & 31;
    const bool few = G <= FEW;
    const int j = few ? t : t >> 5;
    if (j >= D) return;
    double s = 0.0;
    for (int b = few ? 0 : lane; b < G; b += few ? 1 : 32) s += partial[(size_t)b * D + j];
    if (!few) s = warp_sum(s);
    const double v = s / (double)n_fit;
    if (few || lane == 0) out[j] = P == 2 ? sqrt(v) : v;
}

template <typename TO>
__device__ __forceinline__ TO to_out(float v);
template <>
__device__ __forceinline__ float to_out<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 to_out<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// m_hi, m_lo and 1/s (0 where s = 0) of a column
__device__ __forceinline__ float3 column_stats(double m, double s) {
    const float hi = (float)m;
    return make_float3(hi, (float)(m - (double)hi), s > 0.0 ? (float)(1.0 / s) : 0.f);
}
__device__ __forceinline__ float normalised(float x, float3 c) { return ((x - c.x) - c.y) * c.z; }

constexpr int ZU = 8;              // rows in flight a thread
constexpr int ZTILE = 32 * 1024;   // most bytes of an output tile

// Rows of a tile: ZU for each of the 256 / D row lanes, so a multiple of 8 and
// every tile of a 16-byte aligned Y starts on 16 bytes; 0 if D is above 256, the
// tile would not fit, or the table is small: k_zapply takes those.  Up to 2^16
// values one wave does it and the tile's steps are all latency: a call of 600 x 33
// rows 13.6 us without tiles and 14.2 with, 1500 x 60 17.6 and 17.8, 5000 x 33 to
// bf16 x 48 17.8 and 17.0.
int tile_rows(int64_t n, int D, int D_out, int size) {
    if (D > ZT || n * D_out <= 65536) return 0;
    const int64_t r = (int64_t)(ZT / D) * ZU;
    return r * D_out * size <= ZTILE ? (int)r : 0;
}

// A thread keeps one column's statistics in registers and takes every
// (256 / D)-th row: its loads, and its writes to the output tile in shared
// memory, run along the row with its neighbours'.  The tile (padding columns
// zeroed once) leaves in 16-byte stores while the next tile's rows load.
template <typename TO>
__global__ void __launch_bounds__(ZT) k_zapply_tiled(const float *__restrict__ X, int64_t n, int D, int D_out, int R,
                                                     const double *__restrict__ mean, const double *__restrict__ sdev,
                                                     TO *__restrict__ Y) {
    extern __shared__ __align__(16) unsigned char zraw[];
    TO *tile = (TO *)zraw;
    constexpr int V = 16 / sizeof(TO);
    const int RL = ZT / D, rl = threadIdx.x / D, j = threadIdx.x % D;
    const bool on = rl < RL;
    const float3 cs = column_stats(mean[j], sdev[j]);
    for (int i = threadIdx.x; i < R * D_out; i += ZT) tile[i] = to_out<TO>(0.f);
    __syncthreads();
    float v[ZU];
    auto load = [&](int64_t r0) {
#pragma unroll
        for (int u = 0; u < ZU; ++u) {
            const int64_t row = r0 + u * RL + rl;
            v[u] = (on && row < n) ? __ldcs(X + row * D + j) : 0.f;
        }
    };
    int64_t r0 = (int64_t)blockIdx.x * R;
    load(r0);
    for (; r0 < n; r0 += (int64_t)gridDim.x * R) {
        if (on) {
#pragma unroll
            for (int u = 0; u < ZU; ++u) tile[(u * RL + rl) * D_out + j] = to_out<TO>(normalised(v[u], cs));
        }
        load(r0 + (int64_t)gridDim.x * R);
        __syncthreads();
        const int no = (int)min((int64_t)R, n - r0) * D_out;
        TO *dst = Y + r0 * D_out;
        for (int i = V * threadIdx.x; i + V <= no; i += V * ZT) __stcs((uint4 *)(dst + i), *(const uint4 *)(tile + i));
        if (threadIdx.x < no % V) dst[no - no % V + threadIdx.x] = tile[no - no % V + threadIdx.x];
        __syncthreads();
    }
}

// Any width and alignment, an element a thread.
template <typename TO>
__global__ void __launch_bounds__(ZT) k_zapply(const float *__restrict__ X, int64_t n, int D, int D_out,
                                               const double *__restrict__ mean, const double *__restrict__ sdev,
                                               TO *__restrict__ Y) {
    extern __shared__ float zs[];   // [D] m_hi, [D] m_lo, [D] 1/s
    for (int j = threadIdx.x; j < D; j += ZT) {
        const float3 c = column_stats(mean[j], sdev[j]);
        zs[j] = c.x;
        zs[D + j] = c.y;
        zs[2 * D + j] = c.z;
    }
    __syncthreads();
    const int64_t total = n * D_out;
    const bool narrow = total < ((int64_t)1 << 32);   // 32-bit index division suffices
    for (int64_t e = (int64_t)blockIdx.x * ZT + threadIdx.x; e < total; e += (int64_t)gridDim.x * ZT) {
        const int64_t i = narrow ? (int64_t)((uint32_t)e / (uint32_t)D_out) : e / D_out;
        const int j = (int)(e - i * D_out);
        float v = 0.f;
        if (j < D) v = normalised(X[i * D + j], make_float3(zs[j], zs[D + j], zs[2 * D + j]));
        Y[e] = to_out<TO>(v);
    }
}

int zscore_blocks(int64_t n_fit) {
    int64_t g = (n_fit + 63) / 64;
    const int64_t cap = 4 * (int64_t)device_sm_count();
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace
}  // namespace mlp

extern "C" mlp_status mlp_zscore_workspace_bytes(int32_t D, uint64_t *bytes) {
    if (!bytes || D < 1) return mlp::set_error(MLP_EINVAL, "mlp_zscore_workspace_bytes: bad arguments");
    *bytes = sizeof(double) * (uint64_t)D * 4 * (uint64_t)mlp::device_sm_count();
    return MLP_OK;
}

extern "C" mlp_status mlp_zscore(const float *X, int64_t n, int32_t D, int64_t n_fit, int32_t out_prec, int32_t D_out,
                                 void *Y, double *mean, double *sdev, void *workspace, uint64_t workspace_bytes,
                                 void *stream) {
    using namespace mlp;
    if (D < 1 || D_out < D || n < 0 || (out_prec != MLP_FP32 && out_prec != MLP_BF16) || !mean || !sdev)
        return set_error(MLP_EINVAL, "mlp_zscore: bad D, D_out, n, precision or statistics pointer");
    if (n == 0) return MLP_OK;
    if (!X || !Y || !workspace || n_fit < 1 || n_fit > n)
        return set_error(MLP_EINVAL, "mlp_zscore: null buffer or n_fit outside 1..n");
    const int G = zscore_blocks(n_fit);
    if (workspace_bytes < sizeof(double) * (uint64_t)G * (uint64_t)D)
        return set_error(MLP_EINVAL, "mlp_zscore: workspace smaller than mlp_zscore_workspace_bytes");
    cudaStream_t st = (cudaStream_t)stream;
    double *partial = (double *)workspace;
    const int cols = G <= FEW ? ZT : ZT / 32;   // of a block of k_colcombine
    const int cb = (D + cols - 1) / cols;
    const int64_t RL = D <= ZT ? ZT / D : 1, lane_rows = ((n_fit + G - 1) / G + RL - 1) / RL;
    const bool groups = lane_rows >= 4;
    auto sum1 = groups ? k_colsum<1, true> : k_colsum<1, false>;
    auto sum2 = groups ? k_colsum<2, true> : k_colsum<2, false>;
    sum1<<<G, ZT, 0, st>>>(X, n_fit, D, nullptr, partial);
    k_colcombine<1><<<cb, ZT, 0, st>>>(partial, G, D, n_fit, mean);
    sum2<<<G, ZT, 0, st>>>(X, n_fit, D, mean, partial);
    k_colcombine<2><<<cb, ZT, 0, st>>>(partial, G, D, n_fit, sdev);
    const int64_t total = n * (int64_t)D_out;
    int64_t blocks = (total + ZT - 1) / ZT;
    const int64_t cap = 16 * (int64_t)device_sm_count();
    if (blocks > cap) blocks = cap;
    const size_t smem = sizeof(float) * 3 * (size_t)D;
    if (smem > 48 * 1024) return set_error(MLP_EUNSUPPORTED, "mlp_zscore: D above 4096");
    const int size = out_prec == MLP_FP32 ? 4 : 2;
    const int R = tile_rows(n, D, D_out, size);
    if (R > 0 && ((uintptr_t)Y & 15) == 0) {
        int64_t tb = (n + R - 1) / R;
        const int64_t tcap = 8 * (int64_t)device_sm_count();
        if (tb > tcap) tb = tcap;
        const size_t ts = (size_t)R * D_out * size;
        if (out_prec == MLP_FP32)
            k_zapply_tiled<float><<<(unsigned)tb, ZT, ts, st>>>(X, n, D, D_out, R, mean, sdev, (float *)Y);
        else
            k_zapply_tiled<__nv_bfloat16><<<(unsigned)tb, ZT, ts, st>>>(X, n, D, D_out, R, mean, sdev,
                                                                         (__nv_bfloat16 *)Y);
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? MLP_OK : set_error(MLP_ECUDA, cudaGetErrorString(e));
    }
    if (out_prec == MLP_FP32)
        k_zapply<float><<<(unsigned)blocks, ZT, smem, st>>>(X, n, D, D_out, mean, sdev, (float *)Y);
    else
        k_zapply<__nv_bfloat16><<<(unsigned)blocks, ZT, smem, st>>>(X, n, D, D_out, mean, sdev, (__nv_bfloat16 *)Y);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? MLP_OK : set_error(MLP_ECUDA, cudaGetErrorString(e));
}
