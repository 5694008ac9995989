// Forward pass of the general path on the tensor cores at FP32 accuracy:
// z1 = X W1^T + b1, h = f(z1) (Sec. 2.2 and Eq. 1 of arXiv 1908.07847) and the
// partial z2 = h w2 of every 64 units, for up to 64 inputs.
//
// An FP32 value is the exact sum of three bf16 ones (8 bits each, rounded to
// nearest, remainders exact), so x w is the sum of nine exact bf16 products, of
// which the three below 2^-24 x w are left out; for bf16 rows only w is cut, and
// nothing is left out.  tcgen05.mma adds them in FP32, but rounds towards zero at
// every accumulation, so the small products go first: three (D <= 48) or four
// accumulations meet a sum of full size.  For FP32 rows the steps' large products
// are shared between two accumulators, added rounded to nearest, so at most two do;
// bf16 rows keep one (two take the tensor memory of the third block an SM: the
// 200003 rows below 368 -> 412 us).  Measured against 64 bits, root mean square
// error / sum |x w| (chains of FP32 multiply-adds in brackets), D = 16, 33, 48, 64:
//   x N(0, 1), w U(-1, 1)   1.7 1.5 1.1 1.0e-8 (2.6), bf16 rows 1.7 - 1.4 1.3e-8
//   both U(0, 1)            5.1 6.0 5.0 5.7e-8 (6.2 8.4 10 11), bf16 5.1 - 6.9 8.3e-8
//   x exp(3 N(0, 1)), w U(0, 1), where mostly one term counts and the bias adds up:
//                           6.1 11 10 12e-8 (6.8 9.4 11 13), bf16 6.1 - 16 23e-8
//
// One block takes 128 units (W1's parts stay in shared memory) and walks over
// tiles of 128 rows: M = 128 rows, N = 128 units, K = 16 at a time, 64 clocks an
// instruction; 18 to 24 of them for FP32 rows, 9 to 12 for bf16.  Thread r of a
// quarter owns row r (its tensor-memory lane) and half of the units, so z2 is
// summed in the thread.  What is left bounds the kernel: about 20 instructions
// of activation an element and its two special-function operations.  Two (FP32
// rows) or three blocks an SM run at different points of their tiles, which
// overlaps loads, products and activations without a pipeline inside the block.
// 200003 bf16 rows x 48-2048: 1467 us by FP32 multiply-adds (half of them, half
// activations), 359 us here; 100003 x 33-512 with the activations stored: 179 and
// 136 us.
//
// Values that the parts cannot carry (infinities, NaN, magnitudes from 2^60, and
// for cut operands below 2^-100) send the tile through plain FP32 multiply-adds,
// after the block's other tiles (plain_tile): in a loop of its own, so that the
// units are cut once and its registers are not the products' (in the same loop
// they cost 200003 bf16 rows x 48-2048 7 %).
#include <type_traits>

#include "tc_common.cuh"

namespace mlp {

namespace {

using namespace tcd;

constexpr int SNT = 256;         // threads
constexpr int SR = 128;          // rows of a tile
constexpr int SU = 128;          // units of a block
constexpr uint32_t PART = 16384; // one part of a tile: 128 rows of 128 bytes (64 inputs), 128-byte swizzle

template <typename TX> constexpr int x_parts = std::is_same<TX, float>::value ? 3 : 1;
template <typename TX> constexpr int tm_cols = x_parts<TX> == 3 ? 2 * SU : SU;   // tensor memory: accumulators of SU columns
constexpr int WIN = 2048;        // a block's tiles between two turns of its plain ones
template <typename TX> constexpr uint32_t split_smem = (x_parts<TX> + 3) * PART + 2 * SU * 4 + 64 + WIN / 8 + 1024;

// Whether a value can go through the parts; zero always can.
__device__ __forceinline__ bool part_safe(float v, bool cut) {
    const float a = fabsf(v);
    return a < 1.152921504606846976e18f && (!cut || a > 7.8886e-31f || a == 0.f);
}

// Eight values into three bf16 parts.
__device__ __forceinline__ void split8(const float (&v)[8], uint4 (&p)[3]) {
    float r[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = v[i];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            w[i] = pack_bf16(r[2 * i], r[2 * i + 1]);
            r[2 * i] -= __uint_as_float(w[i] << 16);
            r[2 * i + 1] -= __uint_as_float(w[i] & 0xffff0000u);
        }
        p[q] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// The tile of rows from row0 and units from j0 by FP32 multiply-adds, in chains
// over the inputs as the general kernel's.  wf: the units' weights, the inputs
// padded with zeros to a multiple of four; xf: room for the rows, four inputs of a
// row at (k / 4) SR + row, later for the shares of z2.  A lane takes four rows and
// eight units at a time: 12 16-byte loads (a weight's is a broadcast, but takes as
// long) for 128 multiply-adds.  Every tile plain (a column of weights of 1e-32):
// 200003 bf16 rows x 48-2048 32.8 ms with operands loaded for each multiply-add, 2.3
// with one row a lane, 1.72 here; a training step of 64-512 whose weights are NaN,
// two epochs of 20011 rows, 4.63 and 0.46 ms.
template <typename TX, int ACT>
__device__ __forceinline__ void plain_tile(int D, int H, int64_t n, const TX *__restrict__ X, const float *wf, float *xf,
                                           const float *b1s, const float *w2s, float *__restrict__ hid,
                                           float *__restrict__ z2part, int64_t row0, int j0) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ld = (D + 3) & ~3;
    for (int i = tid; i < SR * ld; i += SNT) {
        const int s = i / ld, k = i - s * ld;
        xf[((k >> 2) * SR + s) * 4 + (k & 3)] = (row0 + s < n && k < D) ? ldx<float, TX>(X, (row0 + s) * D + k) : 0.f;
    }
    __syncthreads();
    const bool hvec = (H & 3) == 0 && ((uintptr_t)hid & 15) == 0;
    float zp[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int u0 = 16 * warp; u0 < 16 * warp + 16; u0 += 8) {
        float z[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int u = 0; u < 8; ++u) z[i][u] = 0.f;
        const float *wr = wf + u0 * ld, *xr = xf + 4 * lane;
#pragma unroll 1
        for (int k = 0; k < ld; k += 4, wr += 4, xr += 4 * SR) {
            float4 x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = *(const float4 *)(xr + 128 * i);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float4 w = *(const float4 *)(wr + u * ld);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    z[i][u] = fmaf(x[i].x, w.x, z[i][u]);
                    z[i][u] = fmaf(x[i].y, w.y, z[i][u]);
                    z[i][u] = fmaf(x[i].z, w.z, z[i][u]);
                    z[i][u] = fmaf(x[i].w, w.w, z[i][u]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t row = row0 + 32 * i + lane;
            float *hp = hid + row * H + j0 + u0;
            const bool store = hid && row < n;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                z[i][u] = Act<ACT>::f(z[i][u] + b1s[u0 + u]);
                // (a unit beyond the end may be infinity times 0)
                if (j0 + u0 + u < H) {
                    zp[i] = fmaf(z[i][u], w2s[u0 + u], zp[i]);
                    if (store && !hvec) hp[u] = z[i][u];
                }
            }
            if (store && hvec) {
#pragma unroll
                for (int u = 0; u < 8; u += 4)
                    if (j0 + u0 + u < H) *(float4 *)(hp + u) = make_float4(z[i][u], z[i][u + 1], z[i][u + 2], z[i][u + 3]);
            }
        }
    }
    __syncthreads();   // the rows have been read
#pragma unroll
    for (int i = 0; i < 4; ++i) xf[warp * SR + 32 * i + lane] = zp[i];
    __syncthreads();
    const int r = tid & (SR - 1), half = tid >> 7;
    const float *zr = xf + 4 * half * SR + r;
    if (row0 + r < n && j0 + 64 * half < H)
        z2part[(int64_t)((j0 >> 6) + half) * n + row0 + r] = (zr[0] + zr[SR]) + (zr[2 * SR] + zr[3 * SR]);
    __syncthreads();   // the shares have been read
}

template <typename TX, int ACT>
__global__ void __launch_bounds__(SNT, x_parts<TX> == 3 ? 2 : 3)
k_fwd_split(int D, int H, int64_t n, const TX *__restrict__ X, const float *__restrict__ W1,
            const float *__restrict__ b1, const float *__restrict__ w2, float *__restrict__ hid,
            float *__restrict__ z2part) {
    constexpr int NX = x_parts<TX>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *xs = sm, *ws = sm + NX * PART;
    float *b1s = (float *)(ws + 3 * PART), *w2s = b1s + SU;
    const uint32_t bar = s32(w2s + SU);
    uint32_t *tmem_slot = (uint32_t *)(w2s + SU) + 4;
    volatile int *abort = (volatile int *)(tmem_slot + 1);
    uint32_t *pmask = (uint32_t *)(w2s + SU) + 16;    // of a window of tiles, the plain ones
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int j0 = blockIdx.y * SU;
    const int nks = (D + 15) >> 4, nq = 2 * nks;      // steps of 16 inputs, groups of 8
    if (tid == 0) {
        mbar_init(bar, 1);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(tmem_slot)),
                     "n"(tm_cols<TX>));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // this block's units in parts; whether one cannot be
    auto split_units = [&]() -> bool {
        bool bad = false;
        for (int i = tid; i < SU * nq; i += SNT) {
            const int j = i / nq, k8 = (i - j * nq) * 8;
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                v[u] = (j0 + j < H && k8 + u < D) ? W1[(int64_t)(j0 + j) * D + k8 + u] : 0.f;
                bad |= !part_safe(v[u], true);
            }
            uint4 p[3];
            split8(v, p);
#pragma unroll
            for (int q = 0; q < 3; ++q) *(uint4 *)(ws + q * PART + kmajor_off(j, k8)) = p[q];
        }
        return bad;
    };
    bool wbad = split_units();
    for (int j = tid; j < SU; j += SNT) {
        b1s[j] = j0 + j < H ? b1[j0 + j] : 0.f;
        w2s[j] = j0 + j < H ? w2[j0 + j] : 0.f;
    }
    tc_fence_before();
    wbad = __syncthreads_or(wbad);
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int q = warp & 3, half = warp >> 2, r = q * 32 + lane, c0 = half * 64;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + c0;
    const int tiles = (int)((n + SR - 1) / SR);       // rows that fit the memory: far below 2^31
    const int cn = min(64, H - j0 - c0);              // this thread's units (none if <= 0)
    const bool xvec = NX == 1 && (D & 7) == 0 && ((uintptr_t)X & 15) == 0;
    const bool hvec = (H & 3) == 0 && ((uintptr_t)hid & 15) == 0;
    int use = 0;                                       // MMA batches issued
    bool dead = false;                                 // a wait gave up: no further MMAs
    for (int t0 = blockIdx.x; t0 < tiles; t0 += WIN * (int)gridDim.x) {
        const int t1 = min(tiles, t0 + WIN * (int)gridDim.x);
        if (tid < WIN / 32) pmask[tid] = wbad ? ~0u : 0u;
        bool later = wbad;                             // there are plain tiles
        int bit = 0;
        for (int t = t0; t < t1 && !wbad; t += gridDim.x, ++bit) {
            const int64_t row0 = (int64_t)t * SR, row = row0 + r;
            // ---- rows into parts
            bool bad = false;
#pragma unroll 2
            for (int i = tid; i < SR * nq; i += SNT) {
                const int s = i / nq, k8 = (i - s * nq) * 8;
                const bool in = row0 + s < n;
                const TX *src = X + (row0 + s) * D + k8;
                const uint32_t off = kmajor_off(s, k8);
                if constexpr (NX == 1) {
                    uint32_t w[4] = {0u, 0u, 0u, 0u};
                    if (in && xvec && k8 < D) {
                        const uint4 v = __ldg((const uint4 *)src);
                        w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
                    } else if (in) {
#pragma unroll
                        for (int u = 0; u < 8; ++u)
                            if (k8 + u < D) w[u >> 1] |= (uint32_t)src[u] << (16 * (u & 1));
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        bad |= !part_safe(__uint_as_float(w[u] << 16), false) | !part_safe(__uint_as_float(w[u] & 0xffff0000u), false);
                    *(uint4 *)(xs + off) = make_uint4(w[0], w[1], w[2], w[3]);
                } else {
                    float v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = (in && k8 + u < D) ? (float)src[u] : 0.f;
#pragma unroll
                    for (int u = 0; u < 8; ++u) bad |= !part_safe(v[u], true);
                    uint4 p[3];
                    split8(v, p);
#pragma unroll
                    for (int c = 0; c < 3; ++c) *(uint4 *)(xs + c * PART + off) = p[c];
                }
            }
            proxy_fence();
            const bool plain = __syncthreads_or(bad) || dead;
            if (!plain) {
                if (tid == 0) {
                    tc_fence_after();
                    const uint32_t id = idesc_bf16(SR, SU, 0, 0);
                    const uint64_t xd = sdesc(s32(xs), 16, 1024, 2), wd = sdesc(s32(ws), 16, 1024, 2);
                    // (part of x, part of w), the smallest products first
                    constexpr int XP[6] = {2, 0, 1, 1, 0, 0}, WP[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
                    for (int c = 0; c < (NX == 3 ? 6 : 3); ++c) {
                        // of the large products, the steps from k2 on go to the second accumulator
                        const int k2 = NX == 3 && c == 5 ? (nks + 1) >> 1 : 4;
                        const uint64_t xa = xd + (NX == 3 ? XP[c] : 0) * (PART >> 4);
                        const uint64_t wb = wd + (NX == 3 ? WP[c] : 2 - c) * (PART >> 4);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            if (ks < nks)
                                mma_bf16(ks < k2 ? tmem : tmem + SU, xa + 2 * ks, wb + 2 * ks, id,
                                         ks != k2 && (c > 0 || ks > 0) ? 1u : 0u);
                    }
                    mma_commit(bar);
                }
                __syncwarp();
                dead = !mbar_wait(bar, use++ & 1, abort);
                tc_fence_after();
            }
            if (__syncthreads_or(plain || dead)) {   // everyone the same way
                dead |= !plain;
                later = true;
                if (tid == 0) pmask[bit >> 5] |= 1u << (bit & 31);
                continue;
            }
            // ---- h = f(z1 + b1), this thread's row and 64 units
            float zp[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
            for (int c = 0; c < 64; c += 32) {
                float z[32];
                tmem_ld32(lane_base + c, z);
                if (NX == 3 && nks > 1) {
#pragma unroll
                    for (int v = 0; v < 32; v += 16) {
                        float z2[16];
                        tmem_ld16(lane_base + SU + c + v, z2);
#pragma unroll
                        for (int u = 0; u < 16; ++u) z[v + u] += z2[u];
                    }
                }
#pragma unroll
                for (int u = 0; u < 32; u += 4) {
                    const float4 bv = *(const float4 *)(b1s + c0 + c + u), wv = *(const float4 *)(w2s + c0 + c + u);
                    z[u] = Act<ACT>::f(z[u] + bv.x);
                    z[u + 1] = Act<ACT>::f(z[u + 1] + bv.y);
                    z[u + 2] = Act<ACT>::f(z[u + 2] + bv.z);
                    z[u + 3] = Act<ACT>::f(z[u + 3] + bv.w);
                    // units beyond the end have w2 = 0 and a finite h
                    zp[0] = fmaf(z[u], wv.x, zp[0]);
                    zp[1] = fmaf(z[u + 1], wv.y, zp[1]);
                    zp[2] = fmaf(z[u + 2], wv.z, zp[2]);
                    zp[3] = fmaf(z[u + 3], wv.w, zp[3]);
                }
                if (hid && row < n) {
                    float *hp = hid + row * H + j0 + c0 + c;
                    if (hvec) {
#pragma unroll
                        for (int u = 0; u < 32; u += 4)
                            if (c + u < cn) *(float4 *)(hp + u) = make_float4(z[u], z[u + 1], z[u + 2], z[u + 3]);
                    } else {
#pragma unroll
                        for (int u = 0; u < 32; ++u)
                            if (c + u < cn) hp[u] = z[u];
                    }
                }
            }
            if (row < n && cn > 0) z2part[(int64_t)((j0 + c0) >> 6) * n + row] = (zp[0] + zp[1]) + (zp[2] + zp[3]);
            // the next tile's parts and products overwrite what was read here
            tc_fence_before();
            __syncthreads();
        }
        if (!later) continue;
        // the plain tiles, with rows and units as they are in the parts' place
        __syncthreads();
        float *xf = (float *)sm, *wf = xf + SR * 64;
        const int ld = (D + 3) & ~3;
        for (int i = tid; i < SU * ld; i += SNT) {
            const int j = i / ld, k = i - j * ld;
            wf[i] = (j0 + j < H && k < D) ? W1[(int64_t)(j0 + j) * D + k] : 0.f;
        }
        bit = 0;
        for (int t = t0; t < t1; t += gridDim.x, ++bit)
            if (pmask[bit >> 5] >> (bit & 31) & 1u)
                plain_tile<TX, ACT>(D, H, n, X, wf, xf, b1s, w2s, hid, z2part, (int64_t)t * SR, j0);
        if (t1 < tiles && !wbad) split_units();
        __syncthreads();
    }
    // drain (a wait that gave up may have left products in flight), then free
    if (tid == 0) {
        mma_commit(bar);
        mbar_wait(bar, use & 1, abort, true);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(tm_cols<TX>));
}

template <typename TX, int ACT>
cudaError_t launch(int D, int H, int64_t n, const void *X, const void *W1, const void *b1, const void *w2, void *hid,
                   void *z2part, cudaStream_t st) {
    auto kern = k_fwd_split<TX, ACT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)split_smem<TX>);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (n + SR - 1) / SR, chunks = (H + SU - 1) / SU;
    // one wave of resident blocks
    int64_t gx = (x_parts<TX> == 3 ? 2 : 3) * (int64_t)device_sm_count() / chunks;
    gx = gx < 1 ? 1 : (gx > tiles ? tiles : gx);
    kern<<<dim3((unsigned)gx, (unsigned)chunks), SNT, split_smem<TX>, st>>>(
        D, H, n, (const TX *)X, (const float *)W1, (const float *)b1, (const float *)w2, (float *)hid,
        (float *)z2part);
    return cudaGetLastError();
}

}  // namespace

// From 12 to 64 inputs (what the parts' tiles hold), more than one tile of 64
// units, and enough tiles of 128 x 128.  Whole forward calls, FP32 multiply-adds
// against this: 12-512 4096 rows (128 tiles) 8.4 and 8.4 us, 8192 rows 12.3 and
// 9.8; 33-512 2048 rows 7.4 and 10.4, 4096 rows 11.2 and 10.5; 33-96 16384 rows
// 11.2 and 10.7; bf16 48-2048 1024 rows 13.7 and 9.9.  Storing the activations, a
// row a thread, costs more here, the more so the fewer the inputs: 16-512 65536
// rows 69.3 and 74.0; 33-512 4096 rows 11.3 and 13.2, 8192 rows 17.8 and 17.9,
// 65536 rows 95.4 and 91.7; 64-512 4096 rows 15.6 and 14.6.  Rows of hid that do
// not start on 16 bytes are stored four bytes at a time (56-433, 2060 rows: a
// gradient call 36 us, 28 with multiply-adds).
bool split_forward_takes(int prec, int D, int H, int64_t n, bool hid) {
    if (prec == MLP_FP64 || D < 12 || D > 64 || H <= 64) return false;
    const int64_t tiles = ((n + SR - 1) / SR) * ((H + SU - 1) / SU);
    if (hid && ((H & 3) != 0 || D <= 32 || D * tiles < 8192)) return false;
    return tiles >= 128;
}

cudaError_t split_forward(int prec, int act, int D, int H, int64_t n, const void *X, const void *W1, const void *b1,
                          const void *w2, void *hid, void *z2part, cudaStream_t st) {
    if (prec == MLP_BF16)
        return act == MLP_ACT_TANH ? launch<uint16_t, MLP_ACT_TANH>(D, H, n, X, W1, b1, w2, hid, z2part, st)
                                   : launch<uint16_t, MLP_ACT_SIGMOID>(D, H, n, X, W1, b1, w2, hid, z2part, st);
    return act == MLP_ACT_TANH ? launch<float, MLP_ACT_TANH>(D, H, n, X, W1, b1, w2, hid, z2part, st)
                               : launch<float, MLP_ACT_SIGMOID>(D, H, n, X, W1, b1, w2, hid, z2part, st);
}

}  // namespace mlp
