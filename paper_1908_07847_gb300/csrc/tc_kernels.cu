// BF16 tensor-core (tcgen05) training of many independent D-H-1 networks, one
// block per network for all epochs (Sec. 2.2 of arXiv 1908.07847: feed-forward,
// output error, backpropagation, full-batch gradient descent, no momentum).
//
// Tiles of 128 rows of X (bf16, loaded by TMA, 128-byte swizzle, column D set to
// 1) are worked on as two halves of 64 rows; hidden units lie along the
// tensor-memory lanes, rows along the columns.  Per half:
//   forward    Z1^T = [W1/2 | b1/2] [X | 1]^T    tcgen05.mma M = 128 units (once
//                                    per 128), N = 64 rows, K = D + 1; A = bf16
//                                    [W1/2 | b1/2], B = the rows, both K-major;
//                                    FP32 z1/2 in tensor memory;
//   epilogue   a thread owns a unit of every 128 and 32 rows: h = sigmoid(z1) =
//              1/2 + tanh(z1/2)/2 in bf16 pairs (or, for tanh hidden units, h =
//              tanh(z1) with W1 and b1 unscaled); z2 = h w2 summed over the warp's
//              units by a halving butterfly (FP32) and over the four lane
//              quarters through shared memory; a lane a row, o = sigmoid(z2 + b2)
//              and d2 = c (o - y) o (1 - o); then gw2 += h d2 (FP32, in the
//              thread) and d1 / w2 = d2 f'(h) in bf16 pairs back to tensor
//              memory, over Z1;
//   gradient   [gW1 | gb1] / w2 += d1^T [X | 1]    M = 128 units, N = 64, K = 64
//                                    rows, A = d1 in tensor memory, B = the rows
//                                    read as MN-major; column D is gb1.
// At the end of an epoch the epilogue threads read the accumulators (one hidden
// unit per lane), multiply by w2, update the FP32 master weights in global memory
// (w -= lr g) and rebuild the bf16 copy of W1 for the next epoch.
//
// What bounds a tile is the special-function unit (32,768 tanh for H = 256: 1.0
// us).  With rows along the lanes (h^T and d1^T as shared-memory operands, gw2 as
// a third product) the MMAs and the epilogue moved 4,500 of shared memory's
// 128-byte wavefronts a tile, 2.2 us, and one tile in flight left the pipes idle
// between its steps: 3.3 us a tile.  Here h never leaves the registers and d1 not
// the tensor memory: about 1,500 wavefronts.  The two halves run in two groups of
// eight warps, so one's activations overlap the other's z2, d2 and gradient, and
// a third Z1 buffer lets the forwards run ahead.  MMAs are issued from unrolled
// loops over base descriptors plus constants (an instruction costs 48 cycles from
// shared memory, N/2 from tensor memory; 121 with descriptors rebuilt in a
// runtime loop).  1024 nets 48-256-1 of 4096 to 16384 rows, 8 epochs: 13.95 ms
// before, 12.12 ms now; issue slots bind next (61 % busy, 14,200 warp
// instructions a tile).
// For H = 128 a group has one unit block, so the serial part of a half tile shows:
// with 40 to 56 inputs within 5 % of the form before either way, with 8 to 32 up
// to 14 % slower (27 nets of 500 to 2100 rows, D = 16: 273 and 297 us).  That form
// is not kept for such nets: a net's bits would follow what else is in its plan.
//
// Roles: warp 0 sets the ones column and issues the forward MMAs, warp 1 the TMA
// loads and the gradient MMAs, warps 2..17 run the epilogue.  Every wait is
// bounded; on a timeout the block records MLP_ETIMEOUT, stops issuing, drains
// what it issued (again bounded), frees its tensor memory and leaves.
#include <mutex>

#include "tc_common.cuh"

namespace mlp {

namespace {

constexpr int TR = 128;           // rows per tile
constexpr int SUB = 64;           // rows of a half tile
constexpr int HMAX = 256;
constexpr int NSTAGE = 6;         // X tiles in shared memory
constexpr int NZ1 = 3;            // Z1 / d1 buffers in tensor memory
// Barriers of the two hand-overs between MMAs and epilogue.  A parity wait sees
// one phase back, so a barrier must not complete twice before its waiter has
// looked.  One barrier a group would: the forward of half tile s only waits for
// the buffer's last reader, s - 3, a half of the other group, so s - 2 and s can
// both be done while a thread of their group still looks for s - 2.  Here the
// next phase of a barrier needs the same buffer again, hence everyone's work on
// the one before.
constexpr int NZ1F = 2 * NZ1;     // forward done: a group and buffer
constexpr int NDF = NZ1;          // d1 written: a buffer
constexpr int NEPI = 16;          // epilogue warps: two groups of 4 lane quarters x 2 row halves
constexpr int NT = (2 + NEPI) * 32;  // threads: forward warp, gradient and TMA warp, epilogue warps
constexpr uint32_t NEPI_T = NEPI * 32;
constexpr uint32_t NGRP_T = NEPI_T / 2;   // threads of an epilogue group
constexpr uint32_t TM_GW1 = 0;    // tensor-memory columns: gW1 | gb1 of unit block b at 64 b
constexpr uint32_t TM_Z1 = 128;   // three Z1 / d1 buffers of 128 columns, unit block b at 64 b

// shared-memory layout (bytes); operand tiles 1024-byte aligned
constexpr uint32_t SM_X = 0;                               // NSTAGE x 16 KB
constexpr uint32_t SM_W1 = SM_X + NSTAGE * 16384;          // H x 128 B
constexpr uint32_t SM_GS = SM_W1 + HMAX * 128;             // FP32 gradient at the end of an epoch: H x (D + 2), D <= 56
constexpr uint32_t SM_GWP = SM_GS + HMAX * 58 * 4;         // 4 shares of gw2
constexpr uint32_t SM_ZX = SM_GWP + 4 * HMAX * 4;          // z2: 2 groups x 2 parities x 4 quarters x 64 rows
constexpr uint32_t SM_D2 = SM_ZX + 2 * 2 * 4 * 64 * 4;     // d2 pairs: 16 warps x 16
constexpr uint32_t SM_B1 = SM_D2 + NEPI * 64;              // fp32 b1
constexpr uint32_t SM_W2 = SM_B1 + HMAX * 4;               // fp32 w2
constexpr uint32_t SM_BAR = SM_W2 + HMAX * 4;              // mbarriers
constexpr uint32_t SM_MISC = SM_BAR + 256;                 // tmem slot, flags, reductions
constexpr uint32_t SM_TOTAL = SM_MISC + 256;
constexpr uint32_t SM_ALLOC = SM_TOTAL + 1024;             // + alignment slack
static_assert(SM_ALLOC <= 227 * 1024, "shared memory");

// 16-byte aligned: the host packs the descriptors sizeof(TcNet) apart.
struct __align__(16) TcNet {
    const CUtensorMap *tmap;  // X: bf16 [n x D], box 64 x 128, 128-byte swizzle
    const float *y;           // n labels
    float *params;            // packed FP32 [W1 (H x D), b1, w2, b2]
    double *loss_hist;        // [epochs] or NULL
    double *gnorm_hist;       // [epochs] or NULL
    int64_t n;
    int32_t H;
    int32_t pad;
};

struct TcArgs {
    const TcNet *nets;
    const int *order;
    int n_nets;
    int D;
    int epochs;
    float lr;
    int loss_mean;
    int act;                  // hidden activation (mlp_activation)
    int *status;
    int *next;                // nets taken after the first wave (zeroed before the launch), or NULL
};

using namespace tcd;

template <int ACT>
__global__ void __launch_bounds__(NT, 1) k_tc_batched(TcArgs a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *sm = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sb = s32(sm);
    float *b1s = (float *)(sm + SM_B1);
    float *w2s = (float *)(sm + SM_W2);
    const uint32_t bar0 = sb + SM_BAR;
    // TMA -> MMA: FULL (a stage); gradient MMA -> TMA: EMPTY (a stage); forward
    // MMA -> epilogue: Z1F (a group and Z1 buffer); epilogue -> gradient MMA: DF (a
    // buffer's d1 written); gradient MMA -> forward: GD (a buffer read), ->
    // epilogue: EPOCH; epilogue -> forward: W (weights updated); among epilogue
    // threads: EPI (a group), EPIA (both).
    constexpr int I_EMPTY = NSTAGE, I_Z1F = I_EMPTY + NSTAGE, I_GD = I_Z1F + NZ1F, I_DF = I_GD + NZ1,
                  I_EPOCH = I_DF + NDF, I_W = I_EPOCH + 1, I_EPI = I_W + 1, I_EPIA = I_EPI + 2, I_DRAIN = I_EPIA + 1,
                  NBAR = I_DRAIN + 2;
    static_assert(8 * NBAR <= SM_MISC - SM_BAR, "barriers");
    const uint32_t BAR_FULL = bar0, BAR_EMPTY = bar0 + 8 * I_EMPTY, BAR_Z1F = bar0 + 8 * I_Z1F,
                   BAR_GD = bar0 + 8 * I_GD, BAR_DF = bar0 + 8 * I_DF, BAR_EPOCH = bar0 + 8 * I_EPOCH,
                   BAR_W = bar0 + 8 * I_W, BAR_EPI = bar0 + 8 * I_EPI, BAR_EPIA = bar0 + 8 * I_EPIA,
                   BAR_DRAIN = bar0 + 8 * I_DRAIN;
    uint32_t *tmem_slot = (uint32_t *)(sm + SM_MISC);
    volatile int *abort = (volatile int *)(sm + SM_MISC + 16);
    float *red = (float *)(sm + SM_MISC + 64);     // 4 warps x (sse, gb2)
    double *gnr = (double *)(sm + SM_MISC + 128);  // 16 epilogue warps' squared gradient norms
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int D = a.D;
    // Hidden activation from the forward accumulator: the sigmoid as
    // 1/2 + tanh(z/2)/2 (the operands hold W1/2 and b1/2, so the accumulator
    // is z/2), tanh (Sec. 2.2's other activation) directly from z.
    constexpr bool tanh_act = ACT == MLP_ACT_TANH;
    constexpr float wscale = tanh_act ? 1.0f : 0.5f;
    // h = act_a tanh(acc) + act_b; the tanh form keeps the sigmoid's instruction
    // pattern (one packed fma after the tanh)
    constexpr uint32_t act_a = tanh_act ? BF2_ONE : BF2_HALF, act_b = tanh_act ? 0u : BF2_HALF;
    auto bar_count = [&](int i) -> uint32_t {
        if ((i >= I_DF && i < I_DF + NDF) || i == I_EPI || i == I_EPI + 1) return NGRP_T;
        if (i == I_W || i == I_EPIA) return NEPI_T;
        return 1;
    };

    if (tid == 0) {
        for (int i = 0; i < NBAR; ++i) mbar_init(bar0 + 8 * i, bar_count(i));
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(s32(tmem_slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // Nets go to blocks in decreasing cost: block b takes net b first, then
    // each block that finishes takes the next net not yet taken (one atomic
    // increment), so the longest nets start first and no block waits on a
    // fixed share; which block trains a net does not change its result.
    int *s_idx = (int *)(sm + SM_MISC + 32);
    auto next_net = [&](int cur) -> int {
        if (!a.next) return cur + (int)gridDim.x;
        __syncthreads();
        if (tid == 0) *s_idx = (int)gridDim.x + atomicAdd(a.next, 1);
        __syncthreads();
        return *s_idx;
    };
    for (int idx = blockIdx.x; idx < a.n_nets; idx = next_net(idx)) {
        const TcNet nd = a.nets[a.order ? a.order[idx] : idx];
        const int H = nd.H, NB = H / 128;
        const int64_t n = nd.n;
        const int T = (int)((n + TR - 1) / TR);
        const float c = a.loss_mean ? 1.0f / (float)n : 1.0f;
        float *P = nd.params;
        const int HD = H * D;

        // ---- weights into shared memory: bf16 [W1/2 | b1/2] (swizzled, zero
        // padded; column D meets the ones column of X), b1 and w2 (FP32)
        for (int i = tid; i < H * 64; i += NT) {
            const int j = i >> 6, k = i & 63;
            const float v = (k < D) ? P[j * D + k] : (k == D ? P[HD + j] : 0.f);
            *(__nv_bfloat16 *)(sm + SM_W1 + kmajor_off(j, k)) = __float2bfloat16_rn(wscale * v);
        }
        for (int j = tid; j < H; j += NT) {
            b1s[j] = P[HD + j];
            w2s[j] = P[HD + H + j];
        }
        proxy_fence();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();

        if (T == 0 || a.epochs == 0) {
            if (tid == 0)
                for (int e = 0; e < a.epochs; ++e) {
                    if (nd.loss_hist) nd.loss_hist[e] = 0.0;
                    if (nd.gnorm_hist) nd.gnorm_hist[e] = 0.0;
                }
            continue;
        }

        // Barrier phase counters restart for every net: the previous net's
        // waits were all completed, so re-initialising is safe after a sync.
        if (tid == 0) {
            for (int i = 0; i < NBAR; ++i) {
                asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar0 + 8 * i));
                mbar_init(bar0 + 8 * i, bar_count(i));
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncthreads();

        const int total = a.epochs * T;   // tiles of the launch (below 2^31: the host checks)
        if (warp == 0) {
            // ================= forward MMAs =================
            // whole warp: all lanes set the ones column, lane 0 issues
            const uint32_t id_fwd = idesc_bf16(128, SUB, 0, 0);
            const int nks = D / 16 + 1;   // K = D + 1 in steps of 16
            const uint64_t xd0 = sdesc(sb + SM_X, 16, 1024, 2);
            const uint64_t wd0 = sdesc(sb + SM_W1, 16, 1024, 2);
            int t = 0, e = 0, s = 0, sph = 0, buf = 0, bph = 1;   // bph: parity of GD's phase before
            bool go = true;
            for (int it = 0; it < total && go; ++it) {
                go = __all_sync(0xffffffffu, mbar_wait(BAR_FULL + 8 * s, sph, abort));
                if (!go) break;
#pragma unroll
                for (int i = 0; i < TR / 32; ++i)
                    *(__nv_bfloat16 *)(sm + SM_X + 16384 * s + kmajor_off(lane + 32 * i, D)) = __float2bfloat16_rn(1.0f);
                proxy_fence();
                go = t > 0 || e == 0 || mbar_wait(BAR_W, (e - 1) & 1, abort);   // this epoch's weights
                go = __all_sync(0xffffffffu, go);
                for (int g = 0; g < 2 && go; ++g) {
                    // the buffer's previous d1 has been read
                    go = __all_sync(0xffffffffu, mbar_wait(BAR_GD + 8 * buf, bph, abort));
                    if (!go) break;
                    if (lane == 0) {
                        tc_fence_after();
                        const uint64_t xd = xd0 + (uint32_t)(s * (16384 >> 4) + g * (8192 >> 4));
                        for (int b = 0; b < NB; ++b) {
                            const uint64_t wd = wd0 + (uint32_t)(b * (16384 >> 4));
                            const uint32_t dt = tmem + TM_Z1 + 128 * buf + 64 * b;
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks)
                                if (ks < nks) mma_bf16(dt, wd + ks * 2, xd + ks * 2, id_fwd, ks > 0 ? 1u : 0u);
                        }
                        mma_commit(BAR_Z1F + 8 * (NZ1 * g + buf));
                    }
                    __syncwarp();
                    if (++buf == NZ1) { buf = 0; bph ^= 1; }
                }
                if (++s == NSTAGE) { s = 0; sph ^= 1; }
                if (++t == T) { t = 0; ++e; }
            }
            if (lane == 0) {
                mma_commit(BAR_DRAIN);
                mbar_wait(BAR_DRAIN, 0, abort, true);
            }
        } else if (warp == 1) {
            // ================= TMA loads and gradient MMAs =================
            if (lane == 0) {
                const uint32_t id_gw1 = idesc_bf16(128, 64, 0, 1);
                const uint64_t xd0 = sdesc(sb + SM_X, 16384, 1024, 2);
                int lt = 0, ls = 0, lph = 1, issued = 0;    // row tile, stage and EMPTY parity of the next load
                auto load = [&]() -> bool {
                    if (!mbar_wait(BAR_EMPTY + 8 * ls, lph, abort)) return false;
                    mbar_expect_tx(BAR_FULL + 8 * ls, 16384);
                    tma_load_2d(sb + SM_X + 16384 * ls, nd.tmap, 0, lt * TR, BAR_FULL + 8 * ls);
                    ++issued;
                    if (++lt == T) lt = 0;
                    if (++ls == NSTAGE) { ls = 0; lph ^= 1; }
                    return true;
                };
                bool ok = true;
                while (ok && issued < NSTAGE && issued < total) ok = load();
                int t = 0, s = 0, sph = 0, buf = 0, bph = 0;
                for (int it = 0; it < total && ok; ++it) {
                    // the stage of tile it - 1 is free once its MMAs are done
                    if (it > 0 && issued < total && !load()) { ok = false; break; }
                    if (!mbar_wait(BAR_FULL + 8 * s, sph, abort)) { ok = false; break; }
                    for (int g = 0; g < 2; ++g) {
                        // [gW1 | gb1] / w2 += d1^T [X | 1]
                        if (!mbar_wait(BAR_DF + 8 * buf, bph, abort)) { ok = false; break; }
                        tc_fence_after();
                        const uint64_t xd = xd0 + (uint32_t)(s * (16384 >> 4) + g * (8192 >> 4));
                        for (int b = 0; b < NB; ++b) {
                            const uint32_t at = tmem + TM_Z1 + 128 * buf + 64 * b, dt = tmem + TM_GW1 + 64 * b;
#pragma unroll
                            for (int kk = 0; kk < SUB / 16; ++kk)
                                mma_bf16_ta(dt, at + 8 * kk, xd + kk * (2048 >> 4), id_gw1,
                                            (t > 0 || g > 0 || kk > 0) ? 1u : 0u);
                        }
                        mma_commit(BAR_GD + 8 * buf);
                        if (++buf == NZ1) { buf = 0; bph ^= 1; }
                    }
                    if (!ok) break;
                    mma_commit(BAR_EMPTY + 8 * s);
                    if (++s == NSTAGE) { s = 0; sph ^= 1; }
                    if (++t == T) {
                        t = 0;
                        mma_commit(BAR_EPOCH);
                    }
                }
                // drain: every issued load and MMA completes before the block moves on
                for (int q = (issued > NSTAGE ? issued - NSTAGE : 0); q < issued; ++q)
                    mbar_wait(BAR_FULL + 8 * (q % NSTAGE), (q / NSTAGE) & 1, abort, true);
                mma_commit(BAR_DRAIN + 8);
                mbar_wait(BAR_DRAIN + 8, 0, abort, true);
            }
        } else {
            // ===== epilogue: lane = hidden unit, columns = rows; a group takes one half of every tile =====
            const int q = warp & 3;                 // tensor-memory lane quarter
            const int g = (warp - 2) >> 3;          // group: rows 64 g .. of a tile
            const int rh = ((warp - 2) >> 2) & 1;   // rows 32 rh .. of the group's
            const int u0 = q * 32 + lane;           // unit in a block of 128 = lane
            const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
            const int rl = 64 * g + 32 * rh + lane; // the row whose output this lane works out
            float *zx = (float *)(sm + SM_ZX) + 512 * g;                       // [2][4 quarters][64 rows]
            uint32_t *dsm = (uint32_t *)(sm + SM_D2) + 16 * (warp - 2);        // 32 rows' d2 in bf16 pairs
            float b2 = P[HD + 2 * H];
            int it = 0, buf = g, bph = 0, epi_use = 0;   // bph: parity of this group's use of a buffer
            bool ok = true;
            // Barrier of all epilogue threads with a bounded wait (an mbarrier, so
            // that a block that aborts cannot leave it hanging).
            auto epi_sync = [&]() -> bool {
                mbar_arrive(BAR_EPIA);
                return mbar_wait(BAR_EPIA, epi_use++ & 1, abort);
            };
            for (int e = 0; e < a.epochs && ok; ++e) {
                float sse = 0.f, gb2s = 0.f, gw2a[2] = {0.f, 0.f};
                uint32_t w2h[2];                    // this thread's output weights, a bf16 twice
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float w = b < NB ? w2s[128 * b + u0] : 0.f;
                    w2h[b] = pack_bf16(w, w);
                }
                float y_next = rl < n ? nd.y[rl] : 0.f;   // label of this lane's row, one tile ahead
                for (int t = 0; t < T; ++t, ++it) {
                    const int64_t row = (int64_t)t * TR + rl;
                    const bool valid = row < n;
                    const float yv = y_next;
                    if (row + TR < n) y_next = nd.y[row + TR];
                    const uint32_t zc = lane_base + TM_Z1 + 128 * buf;
                    if (!mbar_wait(BAR_Z1F + 8 * (NZ1 * g + buf), bph, abort)) { ok = false; break; }
                    tc_fence_after();
                    // pass 1: h in bf16 pairs of rows, and the warp's share of z2 = h w2
                    // (FP32), 16 rows at a time
                    uint32_t hp[2][16];
                    float *zw = zx + 256 * (it & 1) + 64 * q + 32 * rh;
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        float pr[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) pr[i] = 0.f;
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            if (b >= NB) break;
                            float z[16];
                            tmem_ld16(zc + 64 * b + 32 * rh + 16 * k, z);
#pragma unroll
                            for (int u = 0; u < 8; ++u) {
                                const uint32_t h = hfma2(tanh_bf2(pack_bf16(z[2 * u], z[2 * u + 1])), act_a, act_b);
                                hp[b][8 * k + u] = h;
                                fma_rows(h, w2h[b], pr[2 * u], pr[2 * u + 1]);
                            }
                        }
                        // sums over the warp's units: halve the rows a lane holds at each step
#pragma unroll
                        for (int off = 16; off >= 2; off >>= 1) {
                            const bool up = lane & off;
                            const int m = off / 2;   // rows left after this step
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                if (i >= m) break;
                                const float keep = up ? pr[i + m] : pr[i], send = up ? pr[i] : pr[i + m];
                                pr[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                            }
                        }
                        pr[0] += __shfl_xor_sync(0xffffffffu, pr[0], 1);
                        if ((lane & 1) == 0) zw[16 * k + (lane >> 1)] = pr[0];   // row bits = lane bits 4..1
                    }
                    tc_fence_before();
                    mbar_arrive(BAR_EPI + 8 * g);
                    if (!mbar_wait(BAR_EPI + 8 * g, it & 1, abort)) { ok = false; break; }
                    tc_fence_after();
                    const float *zr = zx + 256 * (it & 1) + 32 * rh + lane;
                    const float o = sigmoid_bf(((zr[0] + zr[64]) + (zr[128] + zr[192])) + b2);
                    const float err = o - yv;
                    const float d2 = valid ? c * err * o * (1.0f - o) : 0.f;
                    if (valid) sse = fmaf(err, err, sse);
                    gb2s += d2;
                    const float d2n = __shfl_xor_sync(0xffffffffu, d2, 1);
                    if ((lane & 1) == 0) dsm[lane >> 1] = pack_bf16(d2, d2n);
                    __syncwarp();
                    // pass 2: gw2 += h d2 (FP32), d1 / w2 = d2 f'(h) in bf16 pairs over Z1, as
                    // the A operand of the gradient
                    uint32_t dp[16];
#pragma unroll
                    for (int i = 0; i < 16; i += 4) {
                        const uint4 v = *(const uint4 *)(dsm + i);
                        dp[i] = v.x, dp[i + 1] = v.y, dp[i + 2] = v.z, dp[i + 3] = v.w;
                    }
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        if (b >= NB) break;
                        float d1[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const uint32_t h = hp[b][i];
                            gw2a[b] = dot2_bf16(h, dp[i], gw2a[b]);
                            // f'(h): h (1 - h) for the sigmoid, 1 - h^2 for tanh
                            const uint32_t f = tanh_act ? hfma2(h ^ 0x80008000u, h, BF2_ONE)
                                                        : hmul2(h, hfma2(h, BF2_NEG1, BF2_ONE));
                            d1[i] = __uint_as_float(hmul2(f, dp[i]));
                        }
                        tmem_st16(zc + 64 * b + 16 * rh, d1);
                    }
                    tc_fence_before();
                    mbar_arrive(BAR_DF + 8 * buf);
                    buf = buf == 0 ? NZ1 - 1 : buf - 1;   // two half tiles on, modulo 3
                    if (buf == g) bph ^= 1;               // the group has used all three
                }
                if (!ok) break;
                // ---- end of epoch: reductions and the update
                if (!mbar_wait(BAR_EPOCH, e & 1, abort)) { ok = false; break; }
                tc_fence_after();
                const float ws = warp_sum(sse), wg = warp_sum(gb2s);
                // fixed order over the four warps of quarter 0 (every quarter has the same rows)
                if (q == 0 && lane == 0) {
                    red[2 * (2 * g + rh)] = ws;
                    red[2 * (2 * g + rh) + 1] = wg;
                }
                float *gwp = (float *)(sm + SM_GWP);   // [group, half][H] shares of gw2
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    if (b < NB) gwp[HMAX * (2 * g + rh) + 128 * b + u0] = gw2a[b];
                // The gradient rows go to shared memory so that the FP32 master weights
                // in global memory are updated with coalesced accesses: a row per thread
                // there would touch a cache line per lane and load.  Block of units of
                // this thread: its group (H = 256) or 0 (H = 128); columns by its half.
                float *gs = (float *)(sm + SM_GS);     // H x D gradient, row-major, then gb1, gw2
                if (g < NB) {
                    const int j = g * 128 + u0;
                    const float w2j = w2s[j];
#pragma unroll
                    for (int c16 = 0; c16 < 32; c16 += 16) {
                        const int k0 = 32 * rh + c16;
                        if (k0 > D) break;
                        float gv[16];
                        tmem_ld16(lane_base + TM_GW1 + 64 * g + k0, gv);
#pragma unroll
                        for (int u = 0; u < 16; ++u) {
                            if (k0 + u < D) gs[j * D + k0 + u] = w2j * gv[u];
                            else if (k0 + u == D) gs[HD + j] = w2j * gv[u];   // the ones column: gb1
                        }
                    }
                }
                if (!epi_sync()) { ok = false; break; }
                const int et = (warp - 2) * 32 + lane;   // epilogue thread 0..511
                double sse_t = 0.0;
                float gb2 = 0.f;
                for (int w = 0; w < 4; ++w) {
                    sse_t += (double)red[2 * w];
                    gb2 += red[2 * w + 1];
                }
                if (et < H) {
                    const int j = et;
                    const float gw2 = (gwp[j] + gwp[HMAX + j]) + (gwp[2 * HMAX + j] + gwp[3 * HMAX + j]);
                    gs[HD + H + j] = gw2;       // kept for the gradient norm
                    const float nb1 = b1s[j] - a.lr * gs[HD + j];
                    const float nw2 = w2s[j] - a.lr * gw2;
                    P[HD + j] = nb1;
                    P[HD + H + j] = nw2;
                    b1s[j] = nb1;
                    w2s[j] = nw2;
                    *(__nv_bfloat16 *)(sm + SM_W1 + kmajor_off(j, D)) = __float2bfloat16_rn(wscale * nb1);
                }
                // w -= lr g over the flat H x D array, 16 loads in flight per thread
                for (int i0 = et; i0 < HD; i0 += (int)NEPI_T * 16) {
                    float w[16];
#pragma unroll
                    for (int v = 0; v < 16; ++v) {
                        const int i = i0 + v * (int)NEPI_T;
                        w[v] = i < HD ? P[i] : 0.f;
                    }
#pragma unroll
                    for (int v = 0; v < 16; ++v) {
                        const int i = i0 + v * (int)NEPI_T;
                        if (i < HD) {
                            const int j = i / D, k = i - j * D;
                            w[v] -= a.lr * gs[i];
                            P[i] = w[v];
                            *(__nv_bfloat16 *)(sm + SM_W1 + kmajor_off(j, k)) = __float2bfloat16_rn(wscale * w[v]);
                        }
                    }
                }
                b2 -= a.lr * gb2;
                if (et == 0) {
                    P[HD + 2 * H] = b2;
                    const double L = 0.5 * (a.loss_mean ? 1.0 / (double)n : 1.0) * sse_t;
                    if (nd.loss_hist) nd.loss_hist[e] = L;
                    if (!isfinite(L)) atomicOr(a.status, ST_NONFINITE);
                }
                proxy_fence();
                tc_fence_before();
                if (!epi_sync()) { ok = false; break; }
                // FP64 squared norm of the gradient this update applied (only when
                // asked for): each thread's elements of [gW1, gb1, gw2] in index order, a
                // fixed butterfly per warp, the warps in order, then gb2.  (The pointer
                // is read here, not kept in registers for the epoch.)
                double *const gnorm_hist = a.nets[a.order ? a.order[idx] : idx].gnorm_hist;
                if (gnorm_hist) {
                    double gn = 0.0;
                    for (int i = et; i < HD + 2 * H; i += (int)NEPI_T) gn = fma((double)gs[i], (double)gs[i], gn);
                    gn = warp_sum(gn);
                    if (lane == 0) gnr[warp - 2] = gn;
                    if (!epi_sync()) { ok = false; break; }
                    if (et == 0) {
                        double u = 0.0;
                        for (int w = 0; w < NEPI; ++w) u += gnr[w];
                        gnorm_hist[e] = sqrt(fma((double)gb2, (double)gb2, u));
                    }
                }
                mbar_arrive(BAR_W);
            }
        }
        if (*abort && tid == 0) atomicOr(a.status, ST_TIMEOUT);
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (*abort) break;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static std::mutex mu;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::lock_guard<std::mutex> lk(mu);
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

}  // namespace

static_assert(sizeof(TcNet) % 16 == 0, "descriptor stride");
size_t tc_desc_bytes() { return sizeof(TcNet); }
size_t tc_tmap_bytes() { return sizeof(CUtensorMap); }

bool tc_supported(int D, int H) { return D >= 8 && D <= 56 && D % 8 == 0 && (H == 128 || H == 256); }

// Encodes the tensor map of one net's X (bf16 n x D, row-major) into *map.
cudaError_t tc_encode_map(void *map, const void *X, int D, int64_t n) {
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    if (((uintptr_t)X & 15) != 0) return cudaErrorInvalidValue;
    cuuint64_t dims[2] = {(cuuint64_t)D, (cuuint64_t)(n > 0 ? n : 1)};
    cuuint64_t strides[1] = {(cuuint64_t)D * 2};
    cuuint32_t box[2] = {64, TR};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn((CUtensorMap *)map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(X), dims, strides,
                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Fills the device-side descriptor (host image) of one net.
void tc_fill_desc(void *desc, const void *tmap_dev, const float *y, float *params, double *loss_hist,
                  double *gnorm_hist, int64_t n, int H) {
    TcNet *d = (TcNet *)desc;
    d->tmap = (const CUtensorMap *)tmap_dev;
    d->y = y;
    d->params = params;
    d->loss_hist = loss_hist;
    d->gnorm_hist = gnorm_hist;
    d->n = n;
    d->H = H;
    d->pad = 0;
}

cudaError_t tc_batched_train(const void *descs_dev, const int *order_dev, int n_nets, int D, int epochs, float lr,
                             int loss_mean, int act, int *status, int *next, cudaStream_t st) {
    if (n_nets == 0 || epochs == 0) return cudaSuccess;
    auto kern = act == MLP_ACT_TANH ? k_tc_batched<MLP_ACT_TANH> : k_tc_batched<MLP_ACT_SIGMOID>;
    static bool attr_set[2] = {false, false};
    if (!attr_set[act == MLP_ACT_TANH]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM_ALLOC);
        if (e != cudaSuccess) return e;
        attr_set[act == MLP_ACT_TANH] = true;
    }
    TcArgs a;
    a.nets = (const TcNet *)descs_dev;
    a.order = order_dev;
    a.n_nets = n_nets;
    a.D = D;
    a.epochs = epochs;
    a.lr = lr;
    a.loss_mean = loss_mean;
    a.act = act;
    a.status = status;
    const int grid = n_nets < device_sm_count() ? n_nets : device_sm_count();
    a.next = nullptr;
    if (next && n_nets > grid) {
        cudaError_t e = cudaMemsetAsync(next, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
        a.next = next;
    }
    kern<<<grid, NT, SM_ALLOC, st>>>(a);
    return cudaGetLastError();
}

}  // namespace mlp
