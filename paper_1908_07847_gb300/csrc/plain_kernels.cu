// Plain path: separate forward, output, gradient, reduction and update kernels
// for any D and H, with the hidden activations materialised in device memory.
// This is the straightforward data-parallel mapping of Sec. 2.2 of
// arXiv 1908.07847 (feed-forward, output error, backpropagation, gradient
// descent) and the baseline the fused kernels are measured against.  It also
// provides the FP64 kernels used for gradient checking.
#include "mlp_internal.cuh"

namespace mlp {

namespace {

constexpr int TJ = 64;   // hidden units per tile
constexpr int KMAX = 64; // most inputs staged at a time (with 128 rows and two tiles of 64 units: 69 KB)
constexpr int RC = 16;   // rows of a gradient chunk: a multiple of this
constexpr int NTH = 256; // threads per block

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// N consecutive shared-memory values, as 16-byte words where N and T allow
// (p aligned to them).
template <int N, typename T>
__device__ __forceinline__ void lds(T (&v)[N], const T *p) {
    constexpr int W = 16 / sizeof(T);
    if constexpr (N % W == 0) {
#pragma unroll
        for (int i = 0; i < N; i += W) {
            const uint4 q = *reinterpret_cast<const uint4 *>(p + i);
            __builtin_memcpy(&v[i], &q, 16);
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = p[i];
    }
}

// dst[k][r] = src[r][k] for rows r < nr (0 for the other rows below TR) and
// k < ks; src rows are ld apart, dst rows st = 4 mod 32 apart.  A warp takes 4
// rows x 8 inputs: whole 32-byte sectors of the rows, and all 32 banks of the
// transposed side.  Eight such patches are in flight a warp (one at a time, the
// loads' latency took longer than the products); a warp keeps its rows, so that
// no index is divided.
template <int TR, typename T, typename TX>
__device__ __forceinline__ void stage_t(T *dst, int st, const TX *src, int64_t ld, int64_t nr, int ks) {
    constexpr int R = TR >= 32 ? TR / 32 : 1, KB = 8 / R;   // patches of rows and of inputs in flight
    const int lane = threadIdx.x & 31, r0 = (threadIdx.x >> 5) * 4 + (lane >> 3);
    if (TR < 32 && r0 >= TR) return;
    for (int k0 = lane & 7; k0 < ks; k0 += 8 * KB) {
        T v[KB][R];
#pragma unroll
        for (int c = 0; c < KB; ++c)
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int k = k0 + 8 * c, r = r0 + 32 * i;
                v[c][i] = (k < ks && r < nr) ? ldx<T, TX>(src, r * ld + k) : T(0);
            }
#pragma unroll
        for (int c = 0; c < KB; ++c)
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (k0 + 8 * c < ks) dst[(k0 + 8 * c) * st + r0 + 32 * i] = v[c][i];
    }
}

// The same as asynchronous copies (T on both sides), waited for later.
template <int TR, typename T>
__device__ __forceinline__ void stage_t_async(T *dst, int st, const T *src, int64_t ld, int64_t nr, int ks) {
    const int lane = threadIdx.x & 31, r0 = (threadIdx.x >> 5) * 4 + (lane >> 3);
#pragma unroll
    for (int i = 0; i < TR / 32; ++i) {
        const int r = r0 + 32 * i;
        const T *g = src + (r < nr ? r : 0) * ld;
        const int bytes = r < nr ? (int)sizeof(T) : 0;   // the rest is zero-filled
        unsigned d = (unsigned)__cvta_generic_to_shared(dst + (lane & 7) * st + r);
        for (int k = lane & 7; k < ks; k += 8, d += 8 * st * (unsigned)sizeof(T))
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(g + k), "n"(sizeof(T)), "r"(bytes)
                         : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// ---------------------------------------------------------------------------
// z1 = X W1^T + b1 on tiles of 16 RPT rows x 64 units, h = f(z1), and each
// tile's share of z2 = h w2 (summed over the tile's units) written to
// z2part[tile_j][row].  grid: x = row tiles, y = groups of `tpb` unit tiles (a
// block keeps its rows staged over its unit tiles while they fit KMAX).
//
// Bound by the FMA pipe and, per 64 units, by the activations (about 20
// instructions each against 33..64 multiply-adds).  A thread's RPT x 4 sums
// take RPT / 4 + 1 16-byte loads a step from the transposed tiles; for RPT = 8
// a warp's three loads are 4 wavefronts against 32 multiply-adds (8 clocks of
// the SM's FMA pipes), where 4 x 4 tiles with four-byte loads were held by
// shared memory.  RPT falls to 4, 2 or 1 where the grid would not fill the
// device (forward_t).  The order of every sum is that of one pass over the
// inputs and of a fixed tree over the units, whatever RPT is.  Whole forward calls,
// 4 x 4 tiles and now: 83-166, 140024 rows 233 and 146 us; 84-37, 17620 rows 15.4
// and 12.1; 31-98, 230 rows 7.1 and 5.7; FP64 17-809, 1234 rows 129 and 89.
template <typename T, typename TX, int ACT, int RPT>
__global__ void __launch_bounds__(NTH) k_fwd_hidden(int D, int H, int64_t n, int tpb, const TX *__restrict__ X,
                                                    const T *__restrict__ W1, const T *__restrict__ b1,
                                                    const T *__restrict__ w2, T *__restrict__ hid,
                                                    T *__restrict__ z2part) {
    constexpr int TS = 16 * RPT, XST = TS + 4, WST = TJ + 4;
    extern __shared__ __align__(16) unsigned char fsm[];
    const int nsl = (D + KMAX - 1) / KMAX, ksl = (D + nsl - 1) / nsl;   // slices of the inputs
    T *Xs = (T *)fsm, *Wb = Xs + ksl * XST;                             // one buffer of rows, two of weights
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t s0 = (int64_t)blockIdx.x * TS;
    const int ntj = (H + TJ - 1) / TJ;
    const int jt0 = blockIdx.y * tpb, jt1 = min(ntj, jt0 + tpb);
    const bool vec = (H & 3) == 0 && sizeof(T) == 4 && ((uintptr_t)hid & 15) == 0;
    int buf = 0;
    auto stage_w = [&](int jt, int k0) {
        stage_t_async<TJ, T>(Wb + buf * ksl * WST, WST, W1 + (int64_t)jt * TJ * D + k0, D, H - jt * TJ, min(ksl, D - k0));
    };
    stage_w(jt0, 0);
    for (int jt = jt0; jt < jt1; ++jt) {
        const int j0 = jt * TJ;
        T acc[RPT][4];
#pragma unroll
        for (int a = 0; a < RPT; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
        for (int k0 = 0; k0 < D; k0 += ksl) {
            const int ks = min(ksl, D - k0);
            if (nsl > 1 || jt == jt0) {
                if (nsl > 1) __syncthreads();   // the previous slice has been read
                stage_t<TS, T, TX>(Xs, XST, X + s0 * D + k0, D, n - s0, ks);
            }
            cp_async_wait_all();
            __syncthreads();
            const T *xp = Xs + ty * RPT, *wp = Wb + buf * ksl * WST + tx * 4;
            // the next slice of the weights loads meanwhile, into the buffer that
            // everyone has left
            buf ^= 1;
            if (k0 + ksl < D) stage_w(jt, k0 + ksl);
            else if (jt + 1 < jt1) stage_w(jt + 1, 0);
#pragma unroll 4
            for (int k = 0; k < ks; ++k) {
                T a[RPT], b[4];
                lds<RPT>(a, xp + k * XST);
                lds<4>(b, wp + k * WST);
#pragma unroll
                for (int i = 0; i < RPT; ++i)
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) acc[i][jj] = fma(a[i], b[jj], acc[i][jj]);
            }
        }
        T bj[4], wj[4];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const int j = j0 + tx * 4 + jj;
            bj[jj] = j < H ? b1[j] : T(0);
            wj[jj] = j < H ? w2[j] : T(0);
        }
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int64_t row = s0 + ty * RPT + i;
            T zp = T(0), h[4];
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                // (FP64: an activation costs as much as 50 multiply-adds, so a last tile of one
                // to three units skips what no thread needs: 16-385, 8000 rows 277 -> 253 us)
                if (sizeof(T) == 8 && j0 + jj >= H) h[jj] = T(0);
                else h[jj] = Act<ACT>::f(acc[i][jj] + bj[jj]);
                if (j0 + tx * 4 + jj < H) zp = fma(h[jj], wj[jj], zp);
            }
            if (hid && row < n) {
                T *hp = hid + row * H + j0 + tx * 4;
                if (vec) {
                    if (j0 + tx * 4 < H) {
                        uint4 q;
                        __builtin_memcpy(&q, h, 16);
                        *reinterpret_cast<uint4 *>(hp) = q;
                    }
                } else {
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj)
                        if (j0 + tx * 4 + jj < H) hp[jj] = h[jj];
                }
            }
            // Sum over the 16 threads (tx) that share these rows: lanes of one half-warp.
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) zp += __shfl_xor_sync(0xffffffffu, zp, off);
            if (tx == 0 && row < n) z2part[(int64_t)jt * n + row] = zp;
        }
    }
}

// o = sigmoid(b2 + sum_t z2part[t]) (Eq. 1); optional output delta and
// squared-error partial per block (FP64, fixed tree order).
template <typename T>
__global__ void __launch_bounds__(256) k_fwd_output(int ntj, int64_t n, const T *__restrict__ z2part,
                                                    const T *__restrict__ b2, T *__restrict__ o,
                                                    const T *__restrict__ y, const T *__restrict__ dLdo,
                                                    T c, T *__restrict__ d2, double *__restrict__ ssep) {
    __shared__ double red[8];
    int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    double se = 0.0;
    if (i < n) {
        T z = b2[0];
        for (int t = 0; t < ntj; ++t) z += z2part[(int64_t)t * n + i];
        T oi = sigmoid_out(z);
        o[i] = oi;
        if (y) {
            T e = oi - y[i];
            d2[i] = c * e * oi * (T(1) - oi);
            se = (double)e * (double)e;
        } else if (dLdo) {
            d2[i] = dLdo[i] * oi * (T(1) - oi);
        }
    }
    if (ssep) {
        se = warp_sum(se);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = se;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < 8; ++w) s += red[w];
            ssep[blockIdx.x] = s;
        }
    }
}

// d2 = dLdo * o (1 - o) from saved outputs (autograd backward).
template <typename T>
__global__ void k_d2_upstream(int64_t n, const T *__restrict__ o, const T *__restrict__ dLdo, T *__restrict__ d2) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) d2[i] = dLdo[i] * o[i] * (T(1) - o[i]);
}

// Gradient partials over one chunk of rows (Sec. 2.2 backpropagation):
//   d1 = d2 w2 f'(h);  part[c] W1-slot (j, k) = sum_rows d1 X;
//   b1-slot = sum d1;  w2-slot = sum d2 h;  b2-slot = sum d2.
// grid: x = tiles of 64 units, y = tiles of 64 inputs, z = chunks.
//
// A thread holds 8 units x 4 inputs (three 16-byte loads for 32 multiply-adds
// a row); the tile's inputs are cut into quads, so 33 inputs cost 36 and not
// 64.  The 8 x kq thread tiles leave room for RS row subsets (2 to 32), each
// summing every RS-th row; the subsets are added in a fixed tree at the end.  The
// next slice's values load while the present one is summed (a slice's loads one
// after the other took 10,000 cycles).  Whole gradient calls, 4 x 4 tiles of 64
// inputs and now: 83-458, 105224 rows 1510 and 765 us; 65-285, 163 rows 18.9 and
// 14.6; FP64 11-24, 1018 rows 72 and 35.
constexpr int GR = 32;   // rows staged at a time

template <typename T, typename TX, int ACT>
__global__ void __launch_bounds__(NTH) k_bwd_grad(int D, int H, int64_t n, int64_t CH, const TX *__restrict__ X,
                                                  const T *__restrict__ w2, const T *__restrict__ hid,
                                                  const T *__restrict__ d2, T *__restrict__ part) {
    __shared__ __align__(16) T Ds[GR][TJ];
    __shared__ __align__(16) T Xs[GR][64];
    __shared__ T red_b1[4][TJ];
    __shared__ T red_w2[4][TJ];
    const int tid = threadIdx.x;
    const int j0 = blockIdx.x * TJ, k0 = blockIdx.y * 64;
    const int64_t c = blockIdx.z;
    const int64_t r0 = c * CH, r1 = min(n, r0 + CH);
    const int64_t P = (int64_t)(D + 2) * H + 1;
    const bool do_bias = (blockIdx.y == 0);
    const int kn = min(64, D - k0), kq = (kn + 3) >> 2;   // inputs of this tile, in quads
    const int RS = NTH / (8 * kq);                        // row subsets
    const int rs = tid / (8 * kq), t = tid - rs * 8 * kq;
    // this thread's units and inputs; neighbouring lanes along the inputs: few
    // distinct words of Ds a load, consecutive ones of Xs, and nearby stores
    const int u8 = (t / kq) * 8, k4 = (t - (t / kq) * kq) * 4;
    T acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    T gb1 = T(0), gw2 = T(0);  // for unit j0 + (tid & 63), rows (tid >> 6) + 4 i
    const int jl = tid & 63;
    const T w2j = (j0 + jl < H) ? w2[j0 + jl] : T(0);

    // this thread stages unit jl and input jl of rows sr + 4 i; the next slice's
    // values load while the present one is summed
    const int sr = tid >> 6;
    const bool jon = j0 + jl < H, kon = jl < kn;
    T hv[GR / 4], dv[GR / 4], xv[GR / 4];
    auto load = [&](int64_t rb) {
#pragma unroll
        for (int i = 0; i < GR / 4; ++i) {
            const int64_t row = rb + sr + 4 * i;
            const bool on = row < r1;
            hv[i] = on && jon ? hid[row * H + j0 + jl] : T(0);
            dv[i] = on ? d2[row] : T(0);
            xv[i] = on && kon ? ldx<T, TX>(X, row * D + k0 + jl) : T(0);
        }
    };
    load(r0);
    for (int64_t rb = r0; rb < r1; rb += GR) {
        const int nr = (int)min((int64_t)GR, r1 - rb);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < GR / 4; ++i) {
            const int s = sr + 4 * i;
            const T d1 = dv[i] * w2j * Act<ACT>::df(hv[i]);   // 0 for rows and units beyond the end
            gb1 += d1;
            gw2 = fma(dv[i], hv[i], gw2);
            Ds[s][jl] = d1;
            if (jl < 4 * kq) Xs[s][jl] = xv[i];
        }
        load(rb + GR);
        __syncthreads();
        if (rs < RS) {
#pragma unroll 2
            for (int s = rs; s < nr; s += RS) {
                T a[8], b[4];
                lds<8>(a, &Ds[s][u8]);
                lds<4>(b, &Xs[s][k4]);
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) acc[i][kk] = fma(a[i], b[kk], acc[i][kk]);
            }
        }
    }
    T *pc = part + c * P;
    // the row subsets by halving, through shared memory four units at a time (one
    // after the other, 16 subsets of a narrow tile took 60 barriers)
    for (int m = RS; m > 1;) {
        const int h = (m + 1) / 2;
        T *buf = &Ds[0][0];   // 16 values of each of at most 128 threads' tiles
        const int w = 8 * kq * (m - h);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            __syncthreads();
            if (rs >= h && rs < m)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) buf[(i * 4 + kk) * w + (rs - h) * 8 * kq + t] = acc[4 * half + i][kk];
            __syncthreads();
            if (rs < m - h)
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) acc[4 * half + i][kk] += buf[(i * 4 + kk) * w + rs * 8 * kq + t];
        }
        m = h;
    }
    if (rs == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = j0 + u8 + i;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const int k = k0 + k4 + kk;
                if (j < H && k < D) pc[(int64_t)j * D + k] = acc[i][kk];
            }
        }
    }
    if (do_bias) {
        red_b1[tid >> 6][jl] = gb1;
        red_w2[tid >> 6][jl] = gw2;
        __syncthreads();
        if (tid < TJ && j0 + tid < H) {
            T sb = red_b1[0][tid], sw = red_w2[0][tid];
            for (int q = 1; q < 4; ++q) {
                sb += red_b1[q][tid];
                sw += red_w2[q][tid];
            }
            pc[(int64_t)H * D + j0 + tid] = sb;
            pc[(int64_t)H * D + H + j0 + tid] = sw;
        }
        if (blockIdx.x == 0 && tid < 32) {
            T s = T(0);
            for (int64_t row = r0 + tid; row < r1; row += 32) s += d2[row];
            s = warp_sum(s);
            if (tid == 0) pc[P - 1] = s;
        }
    }
}

// g[p] = sum over chunks c = 0..C-1 of part[c][p], scattered to the four
// gradient arrays and, with weights given, w -= lr g; the last block sums the
// squared-error partials (FP64, fixed order) into the loss.  Eight threads a
// value: every eighth chunk each, then the eight in order (256 chunks in one
// thread's order took 31 us in FP64).
template <typename T>
struct Finish {
    T *gW1, *gb1, *gw2, *gb2;
    T *W1, *b1, *w2, *b2;
    T lr;
    const double *ssep;
    int64_t nsse;
    double scale;
    double *loss;
    int loss_add;
    int *status;
};

template <typename T>
__global__ void __launch_bounds__(256) k_finish(int D, int H, int C, const T *__restrict__ part, Finish<T> f) {
    if (f.loss && blockIdx.x == gridDim.x - 1) {
        __shared__ double red[8];
        double s = 0.0;
        for (int64_t i = threadIdx.x; i < f.nsse; i += 256) s += f.ssep[i];
        s = warp_sum(s);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < 8; ++w) t += red[w];
            t *= f.scale;
            *f.loss = f.loss_add ? *f.loss + t : t;
            if (f.status && !isfinite(t)) atomicOr(f.status, ST_NONFINITE);
        }
        return;
    }
    __shared__ T sum[8][32];
    const int64_t P = (int64_t)(D + 2) * H + 1;
    const int64_t HD = (int64_t)H * D;
    const int q = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int64_t p = (int64_t)blockIdx.x * 32 + l;
    T v = T(0);
    if (p < P) {
        const T *pp = part + p;
#pragma unroll 4
        for (int c = q; c < C; c += 8) v += pp[(int64_t)c * P];
    }
    sum[q][l] = v;
    __syncthreads();
    if (q != 0 || p >= P) return;
    T g = sum[0][l];
#pragma unroll
    for (int i = 1; i < 8; ++i) g += sum[i][l];
    T *gp, *wp;
    if (p < HD) gp = f.gW1 + p, wp = f.W1 + p;
    else if (p < HD + H) gp = f.gb1 + (p - HD), wp = f.b1 + (p - HD);
    else if (p < HD + 2 * H) gp = f.gw2 + (p - HD - H), wp = f.w2 + (p - HD - H);
    else gp = f.gb2, wp = f.b2;
    *gp = g;
    if (f.W1) *wp -= f.lr * g;
}

// gX = d1 W1, d1 recomputed from hid, d2, w2.  grid: x = row tiles, y = tiles
// of 64 inputs.  A thread holds RPT rows x 4 inputs; the tile's inputs are cut
// into quads (33 inputs cost 36), the rows fill the block: 256 / quads rows
// times RPT.
template <typename T, int RPT>
__host__ __device__ inline int input_rows(int D) {
    const int kn = D < 64 ? D : 64;
    return (NTH / ((kn + 3) / 4)) * RPT;
}

template <typename T, int ACT, int RPT>
__global__ void __launch_bounds__(NTH) k_bwd_input(int D, int H, int64_t n, const T *__restrict__ W1,
                                                   const T *__restrict__ w2, const T *__restrict__ hid,
                                                   const T *__restrict__ d2, T *__restrict__ gX) {
    constexpr int JS = 16;                           // units staged at a time
    extern __shared__ __align__(16) unsigned char gsm[];
    const int TR = input_rows<T, RPT>(D), DST = TR + 1;
    T *Ws = (T *)gsm;                                // [JS][64], inputs beyond D zero
    T *Ds = Ws + JS * 64;                            // [JS][TR + 1]
    const int tid = threadIdx.x;
    const int64_t s0 = (int64_t)blockIdx.x * TR;
    const int k0 = blockIdx.y * 64;
    const int kn = min(64, D - k0), kq = (min(64, D) + 3) >> 2;
    const int kg = tid % kq, rg = tid / kq;
    const bool on = rg < NTH / kq;
    T acc[RPT][4];
#pragma unroll
    for (int a = 0; a < RPT; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    for (int j0 = 0; j0 < H; j0 += JS) {
        const int nj = min(JS, H - j0);
        __syncthreads();
        {
            const int j = tid % JS;                  // four loads in flight a thread
            const T w2j = j < nj ? w2[j0 + j] : T(0);
            for (int s = tid / JS; s < TR; s += 4 * (NTH / JS)) {
                T hv[4], dv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int su = s + u * (NTH / JS);
                    const int64_t row = s0 + su;
                    const bool in = su < TR && row < n && j < nj;
                    hv[u] = in ? hid[row * H + j0 + j] : T(0);
                    dv[u] = in ? d2[row] : T(0);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int su = s + u * (NTH / JS);
                    if (su < TR) Ds[j * DST + su] = dv[u] * w2j * Act<ACT>::df(hv[u]);
                }
            }
        }
        {
            const int k = tid & 63;
            T wv[JS / 4];
#pragma unroll
            for (int u = 0; u < JS / 4; ++u) {
                const int j = (tid >> 6) + 4 * u;
                wv[u] = (j < nj && k < kn) ? W1[(int64_t)(j0 + j) * D + k0 + k] : T(0);
            }
#pragma unroll
            for (int u = 0; u < JS / 4; ++u) Ws[((tid >> 6) + 4 * u) * 64 + k] = wv[u];
        }
        __syncthreads();
        if (on) {
#pragma unroll 4
            for (int j = 0; j < nj; ++j) {
                T b[4];
                lds<4>(b, Ws + j * 64 + 4 * kg);
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const T a = Ds[j * DST + rg * RPT + i];
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) acc[i][kk] = fma(a, b[kk], acc[i][kk]);
                }
            }
        }
    }
    if (!on) return;
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int64_t row = s0 + rg * RPT + i;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const int k = k0 + 4 * kg + kk;
            if (row < n && k < D) gX[row * D + k] = acc[i][kk];
        }
    }
}

// w -= lr g over the four arrays
template <typename T>
__global__ void k_update(int64_t HD, int64_t H, T lr, T *__restrict__ W1, T *__restrict__ b1, T *__restrict__ w2,
                         T *__restrict__ b2, const T *__restrict__ gW1, const T *__restrict__ gb1,
                         const T *__restrict__ gw2, const T *__restrict__ gb2) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < HD) W1[i] -= lr * gW1[i];
    else if (i < HD + H) b1[i - HD] -= lr * gb1[i - HD];
    else if (i < HD + 2 * H) w2[i - HD - H] -= lr * gw2[i - HD - H];
    else if (i == HD + 2 * H) b2[0] -= lr * gb2[0];
}

template <typename T>
__global__ void k_gnorm_partial(int64_t P, const T *__restrict__ g, double *part) {
    __shared__ double red[8];
    double s = 0.0;
    for (int64_t p = (int64_t)blockIdx.x * 256 + threadIdx.x; p < P; p += (int64_t)gridDim.x * 256) {
        double v = (double)g[p];
        s += v * v;
    }
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

__global__ void k_sqrt_sum(int m, const double *part, double *out) {
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < m; ++i) t += part[i];
        *out = sqrt(t);
    }
}

template <typename T>
__global__ void k_labels(int64_t n, const T *__restrict__ o, int8_t *__restrict__ lab) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) lab[i] = (o[i] >= T(0.5)) ? 1 : 0;
}

// ---------------------------------------------------------------- dispatch

template <typename T, typename TX, int ACT, int RPT>
void launch_hidden(int D, int H, int64_t n, const void *X, const void *W1, const void *b1, const void *w2, void *hid,
                   const PlainWork &w, int sms, cudaStream_t st) {
    const int nsl = (D + KMAX - 1) / KMAX, ksl = (D + nsl - 1) / nsl;
    const size_t smem = sizeof(T) * (size_t)ksl * (16 * RPT + 4 + 2 * (TJ + 4));
    if (smem > 48 * 1024)
        cudaFuncSetAttribute((void *)k_fwd_hidden<T, TX, ACT, RPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int64_t gx = cdiv(n, 16 * RPT);
    const int ntj = (int)cdiv(H, TJ);
    // unit tiles a block: few enough that the grid has eight blocks an SM, or in
    // FP64, where a block of several tiles takes long, 32 (64-512, 17394 rows: 1403 and 1356 us)
    int64_t gy = cdiv((sizeof(T) == 8 ? 32 : 8) * (int64_t)sms, gx);
    if (gy > ntj) gy = ntj;
    const int tpb = (int)cdiv(ntj, gy);
    k_fwd_hidden<T, TX, ACT, RPT><<<dim3((unsigned)gx, (unsigned)cdiv(ntj, tpb)), NTH, smem, st>>>(
        D, H, n, tpb, (const TX *)X, (const T *)W1, (const T *)b1, (const T *)w2, (T *)hid, (T *)w.z2part);
}

template <typename T, typename TX, int ACT>
void hidden_act(int D, int H, int64_t n, const void *X, const void *W1, const void *b1, const void *w2, void *hid,
                const PlainWork &w, cudaStream_t st) {
    const int sms = device_sm_count();
    if constexpr (sizeof(T) == 8) {
        // the FP64 pipe (2 multiply-adds a clock and SM) is all that counts: many
        // small blocks spread evenly
        launch_hidden<T, TX, ACT, 1>(D, H, n, X, W1, b1, w2, hid, w, sms, st);
    } else {
        // 128-row tiles where they still give two blocks an SM, 64-row tiles down
        // to one (84-37, 17620 rows: 16.9 us with 276 tiles of 64 rows, 21.0 with
        // 551 of 32; 80-149, 1043 rows: 13.4 with 51 and 10.5 with 99)
        const int64_t tj = cdiv(H, TJ);
        if (cdiv(n, 128) * tj >= 2 * (int64_t)sms) launch_hidden<T, TX, ACT, 8>(D, H, n, X, W1, b1, w2, hid, w, sms, st);
        else if (cdiv(n, 64) * tj >= sms) launch_hidden<T, TX, ACT, 4>(D, H, n, X, W1, b1, w2, hid, w, sms, st);
        else launch_hidden<T, TX, ACT, 2>(D, H, n, X, W1, b1, w2, hid, w, sms, st);
    }
}

template <typename T, typename TX>
cudaError_t forward_t(int act, int D, int H, int64_t n, const void *X, const void *W1, const void *b1,
                      const void *w2, const void *b2, void *hid, void *o, const void *y, const void *dLdo,
                      double c, const PlainWork &w, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int prec = sizeof(T) == 8 ? MLP_FP64 : (sizeof(TX) == 2 ? MLP_BF16 : MLP_FP32);
    if (split_forward_takes(prec, D, H, n, hid != nullptr)) {
        const cudaError_t e = split_forward(prec, act, D, H, n, X, W1, b1, w2, hid, w.z2part, st);
        if (e != cudaSuccess) return e;
    } else if (act == MLP_ACT_TANH) hidden_act<T, TX, MLP_ACT_TANH>(D, H, n, X, W1, b1, w2, hid, w, st);
    else hidden_act<T, TX, MLP_ACT_SIGMOID>(D, H, n, X, W1, b1, w2, hid, w, st);
    k_fwd_output<T><<<(unsigned)cdiv(n, 256), 256, 0, st>>>((int)cdiv(H, TJ), n, (const T *)w.z2part,
                                                            (const T *)b2, (T *)o, (const T *)y,
                                                            (const T *)dLdo, (T)c, (T *)w.d2,
                                                            (y != nullptr) ? w.ssep : nullptr);
    return cudaGetLastError();
}

template <typename T, int ACT, int RPT>
void launch_input(int D, int H, int64_t n, const void *W1, const void *w2, const void *hid, void *gX,
                  const PlainWork &w, cudaStream_t st) {
    const int TR = input_rows<T, RPT>(D);
    const size_t smem = sizeof(T) * 16 * (64 + (size_t)TR + 1);
    k_bwd_input<T, ACT, RPT><<<dim3((unsigned)cdiv(n, TR), (unsigned)cdiv(D, 64)), NTH, smem, st>>>(
        D, H, n, (const T *)W1, (const T *)w2, (const T *)hid, (const T *)w.d2, (T *)gX);
}

template <typename T, typename TX, int ACT>
void backward_act(int D, int H, int64_t n, const void *X, const void *W1, const void *w2, const void *hid, void *gX,
                  const PlainWork &w, cudaStream_t st) {
    dim3 g2((unsigned)cdiv(H, TJ), (unsigned)cdiv(D, 64), (unsigned)w.C);
    k_bwd_grad<T, TX, ACT><<<g2, NTH, 0, st>>>(D, H, n, w.CH, (const TX *)X, (const T *)w2, (const T *)hid,
                                               (const T *)w.d2, (T *)w.part);
    if (!gX) return;
    // rows a thread: four, or one where that would leave SMs without a block (D
    // small: 64 row groups of four are 256 rows) and in FP64
    if (sizeof(T) == 8 || cdiv(n, input_rows<T, 4>(D)) * cdiv(D, 64) < 2 * (int64_t)device_sm_count() ||
        input_rows<T, 4>(D) > 512)
        launch_input<T, ACT, 1>(D, H, n, W1, w2, hid, gX, w, st);
    else
        launch_input<T, ACT, 4>(D, H, n, W1, w2, hid, gX, w, st);
}

template <typename T, typename TX>
cudaError_t backward_t(int act, int D, int H, int64_t n, const void *X, const void *W1, const void *w2,
                       const void *hid, void *gW1, void *gb1, void *gw2, void *gb2, void *gX,
                       const PlainFinish &fin, const PlainWork &w, cudaStream_t st) {
    const int64_t P = (int64_t)(D + 2) * H + 1;
    if (n == 0) {
        cudaMemsetAsync(gW1, 0, sizeof(T) * (size_t)H * D, st);
        cudaMemsetAsync(gb1, 0, sizeof(T) * (size_t)H, st);
        cudaMemsetAsync(gw2, 0, sizeof(T) * (size_t)H, st);
        cudaMemsetAsync(gb2, 0, sizeof(T), st);
        if (fin.loss && !fin.loss_add) cudaMemsetAsync(fin.loss, 0, sizeof(double), st);
        return cudaGetLastError();   // a zero gradient leaves the weights as they are
    }
    if (act == MLP_ACT_TANH) backward_act<T, TX, MLP_ACT_TANH>(D, H, n, X, W1, w2, hid, gX, w, st);
    else backward_act<T, TX, MLP_ACT_SIGMOID>(D, H, n, X, W1, w2, hid, gX, w, st);
    Finish<T> f;
    f.gW1 = (T *)gW1;
    f.gb1 = (T *)gb1;
    f.gw2 = (T *)gw2;
    f.gb2 = (T *)gb2;
    f.W1 = (T *)fin.W1;
    f.b1 = (T *)fin.b1;
    f.w2 = (T *)fin.w2;
    f.b2 = (T *)fin.b2;
    f.lr = (T)fin.lr;
    f.ssep = w.ssep;
    f.nsse = cdiv(n, 256);
    f.scale = 0.5 * fin.c_loss;
    f.loss = fin.loss;
    f.loss_add = fin.loss_add ? 1 : 0;
    f.status = fin.status;
    k_finish<T><<<(unsigned)(cdiv(P, 32) + (fin.loss ? 1 : 0)), 256, 0, st>>>(D, H, w.C, (const T *)w.part, f);
    return cudaGetLastError();
}

}  // namespace

size_t plain_workspace_bytes(int prec, int D, int H, int64_t n, int sms) {
    PlainWork w;
    plain_workspace_carve(nullptr, prec, D, H, n, sms, &w);
    return (size_t)(uintptr_t)w.part + (size_t)w.C * ((size_t)(D + 2) * H + 1) *
                                           (prec == MLP_FP64 ? sizeof(double) : sizeof(float));
}

void plain_workspace_carve(void *base, int prec, int D, int H, int64_t n, int sms, PlainWork *w) {
    size_t es = (prec == MLP_FP64) ? sizeof(double) : sizeof(float);
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    int64_t nn = n > 0 ? n : 1;
    int tiles = (int)(cdiv(H, TJ) * cdiv(D, 64));
    // Enough row chunks for about two blocks per SM, at least 16 rows each.
    int64_t C = cdiv(2 * (int64_t)sms, tiles);
    C = C < 1 ? 1 : C;
    int64_t maxC = cdiv(nn, RC);
    if (C > maxC) C = maxC;
    int64_t CH = cdiv(cdiv(nn, C), RC) * RC;
    C = cdiv(nn, CH);
    size_t off = 0;
    char *b = (char *)base;
    w->z2part = b + off;
    off = al(off + es * (size_t)cdiv(H, TJ) * (size_t)nn);
    w->d2 = b + off;
    off = al(off + es * (size_t)nn);
    w->ssep = (double *)(b + off);
    off = al(off + sizeof(double) * (size_t)cdiv(nn, 256));
    w->part = b + off;
    w->C = (int)C;
    w->CH = CH;
}

cudaError_t plain_forward(int prec, int act, int D, int H, int64_t n, const void *X, const void *W1,
                          const void *b1, const void *w2, const void *b2, void *hid, void *o, const void *y,
                          const void *dLdo, double c, const PlainWork &w, cudaStream_t st) {
    if (prec == MLP_FP64)
        return forward_t<double, double>(act, D, H, n, X, W1, b1, w2, b2, hid, o, y, dLdo, c, w, st);
    if (prec == MLP_BF16)
        return forward_t<float, uint16_t>(act, D, H, n, X, W1, b1, w2, b2, hid, o, y, dLdo, c, w, st);
    return forward_t<float, float>(act, D, H, n, X, W1, b1, w2, b2, hid, o, y, dLdo, c, w, st);
}

cudaError_t plain_backward(int prec, int act, int D, int H, int64_t n, const void *X, const void *W1,
                           const void *w2, const void *hid, void *gW1, void *gb1, void *gw2, void *gb2,
                           void *gX, const PlainFinish &fin, const PlainWork &w, cudaStream_t st) {
    if (prec == MLP_FP64)
        return backward_t<double, double>(act, D, H, n, X, W1, w2, hid, gW1, gb1, gw2, gb2, gX, fin, w, st);
    if (prec == MLP_BF16)
        return backward_t<float, uint16_t>(act, D, H, n, X, W1, w2, hid, gW1, gb1, gw2, gb2, gX, fin, w, st);
    return backward_t<float, float>(act, D, H, n, X, W1, w2, hid, gW1, gb1, gw2, gb2, gX, fin, w, st);
}

cudaError_t plain_d2_upstream(int prec, int64_t n, const void *o, const void *dLdo, void *d2, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (prec == MLP_FP64)
        k_d2_upstream<double><<<(unsigned)cdiv(n, 256), 256, 0, st>>>(n, (const double *)o, (const double *)dLdo,
                                                                      (double *)d2);
    else
        k_d2_upstream<float><<<(unsigned)cdiv(n, 256), 256, 0, st>>>(n, (const float *)o, (const float *)dLdo,
                                                                     (float *)d2);
    return cudaGetLastError();
}

cudaError_t plain_update(int prec, int D, int H, double lr, void *W1, void *b1, void *w2, void *b2,
                         const void *gW1, const void *gb1, const void *gw2, const void *gb2, cudaStream_t st) {
    const int64_t HD = (int64_t)H * D;
    const unsigned grid = (unsigned)cdiv(HD + 2 * (int64_t)H + 1, 256);
    if (prec == MLP_FP64)
        k_update<double><<<grid, 256, 0, st>>>(HD, H, lr, (double *)W1, (double *)b1, (double *)w2, (double *)b2,
                                               (const double *)gW1, (const double *)gb1, (const double *)gw2,
                                               (const double *)gb2);
    else
        k_update<float><<<grid, 256, 0, st>>>(HD, H, (float)lr, (float *)W1, (float *)b1, (float *)w2, (float *)b2,
                                              (const float *)gW1, (const float *)gb1, (const float *)gw2,
                                              (const float *)gb2);
    return cudaGetLastError();
}

cudaError_t plain_gnorm(int prec, int64_t P, const void *g, double *scratch64, double *out, cudaStream_t st) {
    // Two fixed-order levels: 64 block partials in scratch64, then one serial sum.
    if (prec == MLP_FP64) k_gnorm_partial<double><<<64, 256, 0, st>>>(P, (const double *)g, scratch64);
    else k_gnorm_partial<float><<<64, 256, 0, st>>>(P, (const float *)g, scratch64);
    k_sqrt_sum<<<1, 32, 0, st>>>(64, scratch64, out);
    return cudaGetLastError();
}

cudaError_t plain_labels(int prec, int64_t n, const void *o, int8_t *labels, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (prec == MLP_FP64) k_labels<double><<<(unsigned)cdiv(n, 256), 256, 0, st>>>(n, (const double *)o, labels);
    else k_labels<float><<<(unsigned)cdiv(n, 256), 256, 0, st>>>(n, (const float *)o, labels);
    return cudaGetLastError();
}

}  // namespace mlp
