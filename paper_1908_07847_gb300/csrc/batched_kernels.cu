// Many independent networks in one launch (Sec. 2.1 of arXiv 1908.07847 trains
// the male and female subsets as separate networks; here thousands of nets with
// their own hidden width H <= 128 and row count n).  One block trains one net
// for all epochs without leaving the chip: its rows of X (when they fit) and
// its master weights live in shared memory, the row engine (row_engine.cuh)
// runs forward and backward with one hidden neuron per lane, and the per-epoch
// gradient reduction and update (Sec. 2.2: full-batch gradient descent, no
// momentum) run in shared memory in a fixed order.  Blocks take nets in the
// order given (the host sorts them by cost, largest first).
#include "row_engine.cuh"

namespace mlp {

namespace {

constexpr int BNT = RE_NT;       // threads per block
constexpr int BCAP = 256;        // rows staged in shared memory at a time

constexpr int RING = 32;         // epochs whose losses are finished together

// RB1, RBN: rows a lane keeps in flight for H <= 32 and above, whole deals of one
// and RE_RB rows in both forms: a net's bits do not depend on the plan's size.
template <int DP, int WU, int ACT, int RB1, int RBN, bool ONE>
__device__ __forceinline__ void net_body(const BatchNet &nd, int D, int epochs, float lr, int loss_mean,
                                         int *status, float *Xs, float *ys, float *Wm, float *part,
                                         float *zx, double (*s_sse)[RE_NW], double *s_gn) {
    using Eng = RowEngine<DP, WU, ACT, RB1, RBN, 1, RE_RB>;
    Eng eng;
    eng.setup(nd.H, D);
    constexpr int NG = Eng::NG;
    const int64_t n = nd.n;
    const int P = (D + 2) * nd.H + 1;
    const int tid = threadIdx.x;

    for (int i = tid; i < P; i += BNT) Wm[i] = nd.params[i];
    const bool resident = n <= BCAP;
    auto load_rows = [&](int64_t r0, int cn) {
        const float *Xg = nd.X + r0 * D;
        for (int i = tid; i < cn * D; i += BNT) {
            int s = i / D, k = i - s * D;
            Xs[s * DP + k] = Xg[i];
        }
        for (int i = tid; i < cn; i += BNT) ys[i] = nd.y[r0 + i];
    };
    if (resident) load_rows(0, (int)n);
    __syncthreads();
    const float c = loss_mean ? 1.0f / (float)n : 1.0f;
    const double C = loss_mean ? 1.0 / (double)n : 1.0;

    // The loss of epochs first.. (warp 0): a dozen dependent FP64 operations each.
    // ONE: RING epochs' at a time, a lane each, while the next epoch runs; with
    // two blocks an SM the other block fills that gap, and the registers this
    // takes cost more (2 to 6 %).
    constexpr int HELD = ONE ? RING : 1;
    auto finish_losses = [&](int first, int cnt) {
        if (tid < cnt) {
            const double *v = s_sse[(first + tid) & (2 * HELD - 1)];
            double t = 0.0;
            for (int q = 0; q < NG; ++q) t += v[q];
            const double L = 0.5 * C * t;
            if (nd.loss_hist) nd.loss_hist[first + tid] = L;
            if (!isfinite(L)) atomicOr(status, ST_NONFINITE);
        }
    };
    for (int e = 0; e < epochs; ++e) {
        eng.load_weights(Wm);
        for (int64_t cs = 0; cs < n; cs += BCAP) {
            const int cn = (int)min((int64_t)BCAP, n - cs);
            if (!resident) {
                __syncthreads();
                load_rows(cs, cn);
                __syncthreads();
            }
            eng.rows(Xs, ys, cn, c, zx);
        }
        eng.write_group(part, s_sse[e & (2 * HELD - 1)]);
        __syncthreads();
        // Update, and the FP64 squared norm of the gradient it applies: each
        // thread's values in index order, then a fixed butterfly per warp and
        // the warps in order.
        // (FP64 arithmetic is slow on this part: only when asked for.)
        double gn = 0.0;
        const bool want_gn = nd.gnorm_hist != nullptr;
        constexpr int PF = ONE ? 4 : 1;   // parameters in flight a thread
        for (int base = tid; base < P; base += PF * BNT) {
            float g[PF];
#pragma unroll
            for (int u = 0; u < PF; ++u) {
                const int p = PF > 1 ? min(base + u * BNT, P - 1) : base;
                g[u] = part[p];
#pragma unroll
                for (int q = 1; q < NG; ++q) g[u] += part[q * P + p];
            }
#pragma unroll
            for (int u = 0; u < PF; ++u) {
                const int p = base + u * BNT;
                if (PF > 1 && p >= P) break;
                Wm[p] -= lr * g[u];
                if (want_gn) gn = fma((double)g[u], (double)g[u], gn);
            }
        }
        if (want_gn) {
            gn = warp_sum(gn);
            if ((tid & 31) == 0) s_gn[tid >> 5] = gn;
        }
        __syncthreads();
        if (want_gn && tid == 0) {
            double u = 0.0;
            for (int q = 0; q < RE_NW; ++q) u += s_gn[q];
            nd.gnorm_hist[e] = sqrt(u);
        }
        if ((e & (HELD - 1)) == HELD - 1) finish_losses(e + 1 - HELD, HELD);
    }
    finish_losses(epochs & ~(HELD - 1), epochs & (HELD - 1));
    for (int i = tid; i < P; i += BNT) nd.params[i] = Wm[i];
    __syncthreads();
}

// ONE: one block an SM, for plans of at most one net an SM: a lane then keeps
// as many rows in flight as the fused kernel's (two subsets of 46 and 44 rows, 16
// units: 2.92 -> 2.32 us an epoch with the losses finished in groups).  Otherwise two blocks an SM and,
// for H <= 32, one row in flight: the second row's registers spill there
// (measured 4.7 % slower on the 4096-net workload).
template <int DP, int ACT, bool ONE>
__global__ void __launch_bounds__(BNT, (DP <= 36 && !ONE ? 2 : 1)) k_batched_train(const BatchNet *__restrict__ nets,
                                                         const int *__restrict__ order, int n_nets, int D,
                                                         int epochs, float lr, int loss_mean, int *status,
                                                         int part_floats, int wm_floats) {
    constexpr int RB1 = ONE && DP <= 36 ? 3 : 1, RBN = ONE ? 8 : RE_RB;
    extern __shared__ __align__(16) float smem[];
    __shared__ double s_sse[2 * RING][RE_NW];
    __shared__ double s_gn[RE_NW];
    float *Xs = smem;                      // BCAP x DP
    float *ys = Xs + BCAP * DP;            // BCAP
    float *Wm = ys + BCAP;                 // wm_floats
    float *part = Wm + wm_floats;          // part_floats
    float *zx = part + part_floats;        // z2 exchange
    for (int i = threadIdx.x; i < BCAP * DP; i += BNT) Xs[i] = 0.f;
    __syncthreads();
    for (int idx = blockIdx.x; idx < n_nets; idx += gridDim.x) {
        const BatchNet nd = nets[order ? order[idx] : idx];
        if (nd.n <= 0 || nd.H <= 0) {
            if (threadIdx.x == 0)
                for (int e = 0; e < epochs; ++e) {
                    if (nd.loss_hist) nd.loss_hist[e] = 0.0;
                    if (nd.gnorm_hist) nd.gnorm_hist[e] = 0.0;
                }
            continue;
        }
        if (nd.H <= 32)
            net_body<DP, 1, ACT, RB1, RBN, ONE>(nd, D, epochs, lr, loss_mean, status, Xs, ys, Wm, part, zx, s_sse, s_gn);
        else if (nd.H <= 64)
            net_body<DP, 2, ACT, RB1, RBN, ONE>(nd, D, epochs, lr, loss_mean, status, Xs, ys, Wm, part, zx, s_sse, s_gn);
        else
            net_body<DP, 4, ACT, RB1, RBN, ONE>(nd, D, epochs, lr, loss_mean, status, Xs, ys, Wm, part, zx, s_sse, s_gn);
    }
}

template <int DP>
void *pick(int act, bool one) {
    if (act == MLP_ACT_TANH)
        return one ? (void *)k_batched_train<DP, MLP_ACT_TANH, true> : (void *)k_batched_train<DP, MLP_ACT_TANH, false>;
    return one ? (void *)k_batched_train<DP, MLP_ACT_SIGMOID, true> : (void *)k_batched_train<DP, MLP_ACT_SIGMOID, false>;
}

int dp_for(int D) {
    if (D <= 8) return 8;
    if (D <= 16) return 16;
    if (D <= 36) return 36;
    if (D <= 48) return 48;
    if (D <= 64) return 64;
    return 0;
}

}  // namespace

bool batched_shape_supported(int D, int shape) {
    if (shape == BATCH_SHAPE_U1) return dp_for(D) != 0;
    if (shape == BATCH_SHAPE_U2_RB1) return batched_u2_supported(D, 1);
    if (shape == BATCH_SHAPE_U2_RB2) return batched_u2_supported(D, 2);
    if (shape == BATCH_SHAPE_U2_3B) return batched_u2_supported(D, 3);
    if (shape == BATCH_SHAPE_TILED128 || shape == BATCH_SHAPE_TILED64 || shape == BATCH_SHAPE_TILED32)
        return batched_tiled_supported(D, 128);
    return false;
}

int batched_max_H() { return 128; }
int batched_max_D() { return 64; }

void batched_smem_layout(int D, int Hmax, int *part_floats, int *wm_floats, size_t *bytes) {
    const int DP = dp_for(D);
    const int pf = re_part_floats(D, Hmax);
    const int wm = ((D + 2) * Hmax + 1 + 3) & ~3;
    *part_floats = pf;
    *wm_floats = wm;
    *bytes = sizeof(float) * ((size_t)BCAP * DP + BCAP + wm + pf + RE_ZX);
}

cudaError_t batched_train(int act, int D, int Hmax, int64_t nmax, const BatchNet *nets_dev, const int *order_dev,
                          int n_nets, int epochs, float lr, int loss_mean, int *status, int shape, cudaStream_t st) {
    if (shape == BATCH_SHAPE_TILED128 || shape == BATCH_SHAPE_TILED64 || shape == BATCH_SHAPE_TILED32)
        return batched_train_tiled(act, D, Hmax, nmax, nets_dev, order_dev, n_nets, epochs, lr, loss_mean, status,
                                   shape == BATCH_SHAPE_TILED32 ? 32 : (shape == BATCH_SHAPE_TILED64 ? 64 : 128), st);
    if (shape != BATCH_SHAPE_U1)
        return batched_train_u2(act, D, Hmax, nets_dev, order_dev, n_nets, epochs, lr, loss_mean, status,
                                shape == BATCH_SHAPE_U2_RB2 ? 2 : (shape == BATCH_SHAPE_U2_3B ? 3 : 1), st);
    const int DP = dp_for(D);
    if (DP == 0 || Hmax > 128) return cudaErrorInvalidValue;
    if (n_nets == 0 || epochs == 0) return cudaSuccess;
    void *fn = nullptr;
    const bool one = n_nets <= device_sm_count();
    switch (DP) {
        case 8: fn = pick<8>(act, one); break;
        case 16: fn = pick<16>(act, one); break;
        case 36: fn = pick<36>(act, one); break;
        case 48: fn = pick<48>(act, one); break;
        default: fn = pick<64>(act, one); break;
    }
    int pf, wm;
    size_t smem;
    batched_smem_layout(D, Hmax, &pf, &wm, &smem);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&nets_dev, (void *)&order_dev, (void *)&n_nets, (void *)&D, (void *)&epochs,
                    (void *)&lr, (void *)&loss_mean, (void *)&status, (void *)&pf, (void *)&wm};
    return cudaLaunchKernel(fn, dim3((unsigned)n_nets), dim3(BNT), args, smem, st);
}

}  // namespace mlp
