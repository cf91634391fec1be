// Training of the per-atom preconditioner network on the GPU: mean squared
// error between z(f) and the recorded target t over a data set, plain
// backpropagation through the two layers, and Adam (Kingma & Ba 2015).
// Hand-written kernels, FP32 arithmetic; weights are handed to inference as
// FP16.  Minibatches are drawn with the SplitMix64 counter stream.
//
// Loss per sample: (z - t)^2; minibatch loss = mean.  Gradients:
//   dz = 2 (z - t) / B,  dw2_k = dz h_k,  db2 = dz,
//   dh_k = dz w2_k [a_k > 0],  dW1_ki = dh_k f_i,  db1_k = dh_k.
// Partial gradients are summed in a fixed order, so training is
// deterministic.
//
// Bound: latency (a step of 16,384 rows is 44 MFLOP, under a microsecond of
// FP32).  A warp takes 32 rows, a thread two hidden units, whose weights,
// activations and 14 gradient sums stay in registers.  All steps of a call run in one cooperative launch: a step's gradient is summed over a
// cluster of 8 blocks through distributed shared memory, over the clusters
// through global memory at one grid barrier, and every block takes the Adam
// step for itself (same sums, same order), so that the weights never leave
// the SM; the next step's rows are gathered while the barrier is pending.
// 16,384 rows: 320 + 27 us a step with all 449 sums per thread in local memory,
// 11.3 us as two kernels a step, 8.7 us now.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "ffmin.h"
#include "mlp.cuh"

namespace ffm {

namespace cg = cooperative_groups;

constexpr int MT = 128;           // threads per training block, one row each
constexpr int MLP_ROWS = 256;     // rows of MLP_NW floats that the scratch holds
#ifndef FFMIN_MLP_CLUSTER
#define FFMIN_MLP_CLUSTER 8
#endif
constexpr int MLP_CLUSTER = FFMIN_MLP_CLUSTER;  // blocks per cluster
// clusters, at most; all of a launch's blocks have to be resident at once, and
// a launch that finds too few SMs (128 blocks need 43) is repeated with fewer
#ifndef FFMIN_MLP_CLUSTERS
#define FFMIN_MLP_CLUSTERS 16
#endif
constexpr int MLP_CLUSTERS = FFMIN_MLP_CLUSTERS;
constexpr int MLP_NV = MLP_NW + 1;                    // summed values: the gradient, the loss
#ifndef FFMIN_MLP_STEPS
#define FFMIN_MLP_STEPS 4096
#endif
constexpr int MLP_STEPS = FFMIN_MLP_STEPS;  // steps per launch (their losses wait in the scratch)
// polls of the grid barrier before a block gives up (about a second)
#ifndef FFMIN_MLP_POLLS
#define FFMIN_MLP_POLLS (1 << 22)
#endif

// a run of training steps; lr == 0: one gradient, no update
struct MlpRun {
    const float *feat, *target;
    int64_t n;
    int batch, steps, step0, sample;  // step0: steps taken before; sample: minibatches from the stream
    uint64_t seed;
    float lr;
    float *w32, *adam;
    float *part;               // [2][MLP_CLUSTERS][MLP_NV]
    unsigned int *sync;        // [0] barrier count, [1] set when a block gave up
    float *losses, *grad_out;  // losses [steps]; grad_out optional
    uint16_t *w16;             // optional: FP16 copy for inference
};

__device__ __forceinline__ uint64_t mix64(uint64_t seed, uint64_t k) {
    uint64_t z = seed + (k + 1) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// Samples of minibatch t are index t batch + k of the SplitMix64 stream when
// sample != 0, else rows [0, batch) of the data in order.  CS: blocks per
// cluster; 1 where the SMs at hand cannot hold a cluster
template <int CS>
__global__ void __launch_bounds__(MT) k_mlp_train(MlpRun o) {
    constexpr int SLICE = (MLP_NV + CS - 1) / CS;  // sums per block of a cluster
    cg::cluster_group cl = cg::this_cluster();
    __shared__ float4 sw[MLP_H][2];        // per hidden unit: W1 (5), b1, w2
    __shared__ float4 sf[MT / 32][32][2];  // per row of the warp: features (5), dz
    __shared__ float acc[MT / 32][MLP_NV];
    __shared__ float sum[MLP_NV];          // the block's sums, read by the cluster
    __shared__ float wt[MLP_NW], am[MLP_NW], av[MLP_NW];
    __shared__ float unbias[2];
    __shared__ int gave_up, failed;  // this block at the last grid barrier; some block of the cluster
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int rank = (int)cl.block_rank(), cluster = blockIdx.x / CS, clusters = gridDim.x / CS;
    const float be1 = 0.9f, be2 = 0.999f, eps = 1e-8f;
    const float inv_b = 1.0f / (float)o.batch;
    for (int k = tid; k < MLP_NW; k += MT) {
        wt[k] = o.w32[k];
        if (o.lr > 0.f) {
            am[k] = o.adam[k];
            av[k] = o.adam[MLP_NW + k];
        }
    }
    if (tid == 0) failed = 0;
    float f[MLP_IN], tg = 0.f;
    // rows are counted in 64 bits: a 32-bit index of a batch near 2^31 would
    // wrap before it reached the end, and the loop would never end
    const int64_t first = (int64_t)blockIdx.x * MT, stride = (int64_t)gridDim.x * MT;
    auto gather = [&](int t, int64_t s0) {  // this thread's row of minibatch t, from s0 on
        const int64_t s = s0 + tid;
#pragma unroll
        for (int i = 0; i < MLP_IN; i++) f[i] = 0.f;
        tg = 0.f;
        if (s >= o.batch) return;
        const uint64_t q = (uint64_t)(o.step0 + t) * (uint64_t)o.batch + (uint64_t)s;
        const int64_t row = o.sample ? (int64_t)__umul64hi(mix64(o.seed, q), (uint64_t)o.n) : s;
#pragma unroll
        for (int i = 0; i < MLP_IN; i++) f[i] = o.feat[row * MLP_IN + i];
        tg = o.target[row];
    };
    gather(0, first);
    for (int t = 0; t < o.steps; t++) {
        __syncthreads();  // wt of this step
        if (tid < MLP_H) {
            const float *w1 = wt + MLP_W1 + tid * MLP_IN;
            sw[tid][0] = make_float4(w1[0], w1[1], w1[2], w1[3]);
            sw[tid][1] = make_float4(w1[4], wt[MLP_B1 + tid], wt[MLP_W2 + tid], 0.f);
        }
        __syncthreads();
        const float b2 = wt[MLP_B2];
        float g[2][MLP_IN + 2] = {};  // of units lane, lane + 32: W1, b1, w2
        float wu[2][MLP_IN + 2], gb2 = 0.f, loss = 0.f;
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const float4 p = sw[lane + 32 * u][0], q = sw[lane + 32 * u][1];
            wu[u][0] = p.x; wu[u][1] = p.y; wu[u][2] = p.z; wu[u][3] = p.w;
            wu[u][4] = q.x; wu[u][5] = q.y; wu[u][6] = q.z;
        }
        for (int64_t s0 = first; s0 < o.batch; s0 += stride) {
            if (s0 != first) gather(t, s0);
            // The warp's 32 rows, two hidden units per thread: the units'
            // activations stay in registers for the backward pass, and their
            // shares of z are summed over the lanes by halving (31 exchanges
            // for 32 rows), which leaves row `lane` in lane `lane`
            sf[w][lane][0] = make_float4(f[0], f[1], f[2], f[3]);
            sf[w][lane][1] = make_float4(f[4], 0.f, 0.f, 0.f);
            __syncwarp();
            float act[32][2], z[32];
#pragma unroll
            for (int m = 0; m < 32; m++) {
                const float4 p = sf[w][m][0];
                const float p4 = sf[w][m][1].x;
                z[m] = 0.f;
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    float a = fmaf(wu[u][0], p.x, wu[u][5]);
                    a = fmaf(wu[u][1], p.y, a);
                    a = fmaf(wu[u][2], p.z, a);
                    a = fmaf(wu[u][3], p.w, a);
                    a = fmaf(wu[u][4], p4, a);
                    act[m][u] = fmaxf(a, 0.f);
                    z[m] = fmaf(wu[u][6], act[m][u], z[m]);
                }
            }
#pragma unroll
            for (int q = 16; q > 0; q >>= 1) {
                const bool up = lane & q;
#pragma unroll
                for (int m = 0; m < q; m++) {
                    const float keep = up ? z[m + q] : z[m], send = up ? z[m] : z[m + q];
                    z[m] = keep + __shfl_xor_sync(0xffffffffu, send, q);
                }
            }
            const float r = s0 + tid < o.batch ? (z[0] + b2) - tg : 0.f;
            loss += r * r;
            const float dz = 2.f * r * inv_b;
            gb2 += dz;
            sf[w][lane][1].y = dz;
            __syncwarp();
#pragma unroll
            for (int m = 0; m < 32; m++) {
                const float4 p = sf[w][m][0];
                const float2 q = *reinterpret_cast<const float2 *>(&sf[w][m][1]);
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const float h = act[m][u];
                    const float dh = h > 0.f ? q.y * wu[u][6] : 0.f;
                    g[u][0] = fmaf(dh, p.x, g[u][0]);
                    g[u][1] = fmaf(dh, p.y, g[u][1]);
                    g[u][2] = fmaf(dh, p.z, g[u][2]);
                    g[u][3] = fmaf(dh, p.w, g[u][3]);
                    g[u][4] = fmaf(dh, q.x, g[u][4]);
                    g[u][5] += dh;
                    g[u][6] = fmaf(q.y, h, g[u][6]);
                }
            }
            __syncwarp();
        }
        // the block's sums, warps in order
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int k = lane + 32 * u;
#pragma unroll
            for (int i = 0; i < MLP_IN; i++) acc[w][MLP_W1 + k * MLP_IN + i] = g[u][i];
            acc[w][MLP_B1 + k] = g[u][5];
            acc[w][MLP_W2 + k] = g[u][6];
        }
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) {
            gb2 += __shfl_xor_sync(0xffffffffu, gb2, q);
            loss += __shfl_xor_sync(0xffffffffu, loss, q);
        }
        if (lane == 0) {
            acc[w][MLP_B2] = gb2;
            acc[w][MLP_NW] = loss;
        }
        __syncthreads();
        for (int k = tid; k < MLP_NV; k += MT) sum[k] = (acc[0][k] + acc[1][k]) + (acc[2][k] + acc[3][k]);
        cl.sync();
        if (failed) break;  // the whole cluster: no block reads the sums of one that has left
        // the cluster's sums, one slice per block, blocks in order
        float *part = o.part + (int64_t)(t & 1) * MLP_CLUSTERS * MLP_NV;
#pragma unroll
        for (int u = 0; u < SLICE; u += MT) {
            const int k = rank * SLICE + u + tid;
            if (u + tid < SLICE && k < MLP_NV) {
                float x[CS];
#pragma unroll
                for (int r = 0; r < CS; r++) x[r] = *cl.map_shared_rank(&sum[k], r);
#pragma unroll
                for (int q = 1; q < CS; q *= 2)
#pragma unroll
                    for (int r = 0; r < CS; r += 2 * q) x[r] += x[r + q];
                part[cluster * MLP_NV + k] = x[0];
            }
        }
        cl.sync();
        // grid barrier: every cluster has its sums of this step in memory
        // (the two buffers alternate, so no cluster writes over sums that
        // another still reads: it arrives here again only after reading them).
        // The cluster barrier orders every block's slice before this thread,
        // whose fence releases them with its arrival to the pollers' acquire
        if (rank == 0 && tid == 0) {
            __threadfence();
            atomicAdd(&o.sync[0], 1u);
        }
        if (t + 1 < o.steps) gather(t + 1, first);
        if (tid == MT - 1) {  // Adam's bias corrections of this step
            const float step = (float)(o.step0 + t + 1);
            unbias[0] = 1.f - powf(be1, step);
            unbias[1] = 1.f - powf(be2, step);
        }
        if (tid == 0) {
            const unsigned want = (unsigned)(t + 1) * (unsigned)clusters;
            long long polls = 0;
            unsigned got;
            do {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(&o.sync[0]) : "memory");
            } while (got < want && ++polls < FFMIN_MLP_POLLS && *(volatile unsigned int *)&o.sync[1] == 0u);
            gave_up = got < want;
            if (got < want) {
                // its cluster leaves together behind the next cluster barrier
                // (another block of it may have seen the count in time); the
                // other clusters run out of arrivals or see the word
                *(volatile unsigned int *)&o.sync[1] = 1u;
                for (int r = 0; r < CS; r++) *cl.map_shared_rank(&failed, r) = 1;
            }
        }
        __syncthreads();
        if (gave_up) continue;
        // the gradient over the clusters, then one Adam step: every load of a
        // thread's (up to four) parameters in flight together
        constexpr int KT = (MLP_NV + MT - 1) / MT;
        float x[KT][MLP_CLUSTERS];
#pragma unroll
        for (int h = 0; h < KT; h++) {
            const int k = tid + h * MT;
#pragma unroll
            for (int q = 0; q < MLP_CLUSTERS; q++)
                x[h][q] = q < clusters && k < MLP_NV ? __ldcg(part + q * MLP_NV + k) : 0.f;
        }
        const float d1 = unbias[0], d2 = unbias[1];
#pragma unroll
        for (int h = 0; h < KT; h++) {
            const int k = tid + h * MT;
#pragma unroll
            for (int q = MLP_CLUSTERS / 2; q > 0; q >>= 1)
#pragma unroll
                for (int r = 0; r < q; r++) x[h][r] += x[h][r + q];
            const float gk = x[h][0];
            if (k == MLP_NW && blockIdx.x == 0) o.losses[t] = gk / (float)o.batch;
            if (k >= MLP_NW) continue;
            if (o.grad_out && blockIdx.x == 0 && t == o.steps - 1) o.grad_out[k] = gk;
            if (o.lr > 0.f) {
                const float m = am[k] = be1 * am[k] + (1.f - be1) * gk;
                const float v = av[k] = be2 * av[k] + (1.f - be2) * gk * gk;
                wt[k] -= o.lr * (m / d1) / (sqrtf(v / d2) + eps);
            }
        }
    }
    __syncthreads();
    if (blockIdx.x == 0) {
        for (int k = tid; k < MLP_NW; k += MT) {
            if (o.lr > 0.f) {
                o.w32[k] = wt[k];
                o.adam[k] = am[k];
                o.adam[MLP_NW + k] = av[k];
            }
            if (o.w16) {
                __half hv = __float2half_rn(wt[k]);
                o.w16[k] = *reinterpret_cast<uint16_t *>(&hv);
            }
        }
    }
    cl.sync();  // no block leaves while its sums may be read
}

// all blocks resident (cooperative): the grid barrier ends
static cudaError_t launch_train(const MlpRun &o, int clusters, int cs, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * cs);
    cfg.blockDim = dim3(MT);
    cfg.stream = s;
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cs;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cs == 1 ? cudaLaunchKernelEx(&cfg, k_mlp_train<1>, o) : cudaLaunchKernelEx(&cfg, k_mlp_train<MLP_CLUSTER>, o);
}

}  // namespace ffm

using namespace ffm;

extern "C" ffmin_status ffmin_mlp_train(const float *feat_dev, const float *target_dev, int64_t n_samples,
                                        int32_t steps, int32_t batch, float lr, uint64_t seed, float *w32_dev,
                                        float *adam_dev, float *work_dev, float *loss_host, uint16_t *w16_dev,
                                        void *cuda_stream) {
    if (!feat_dev || !target_dev || n_samples < 1 || steps < 0 || batch < 1 || !w32_dev || !work_dev)
        return FFMIN_ERR_INVALID_ARG;
    if (steps > 0 && (!adam_dev || !(lr > 0.f))) return FFMIN_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    MlpRun o{};
    o.feat = feat_dev;
    o.target = target_dev;
    o.n = n_samples;
    o.batch = steps > 0 ? batch : (int)std::min<int64_t>(batch, n_samples);
    o.sample = steps > 0 ? 1 : 0;
    o.seed = seed;
    o.lr = steps > 0 ? lr : 0.f;
    o.w32 = w32_dev;
    o.adam = adam_dev;
    o.part = work_dev;                                                // [2][MLP_CLUSTERS][MLP_NV]
    o.losses = o.part + (size_t)2 * MLP_CLUSTERS * MLP_NV;            // [MLP_STEPS]
    float *tail = work_dev + (size_t)MLP_ROWS * MLP_NW;               // [MLP_ROWS + 1], then the gradient
    o.sync = reinterpret_cast<unsigned int *>(tail);
    static_assert(2 * MLP_CLUSTERS * MLP_NV + MLP_STEPS <= MLP_ROWS * MLP_NW, "the losses fit in the scratch");
    const int nsteps = steps > 0 ? steps : 1;
    const int64_t blocks = ((int64_t)o.batch + MT - 1) / MT;
    int cs = MLP_CLUSTER, clusters = (int)std::min<int64_t>(MLP_CLUSTERS, (blocks + cs - 1) / cs);
    for (int t = 0; t < nsteps; t += MLP_STEPS) {
        o.step0 = t;
        o.steps = std::min(MLP_STEPS, nsteps - t);
        const bool last = t + o.steps == nsteps;
        o.grad_out = last ? tail + MLP_ROWS + 1 : nullptr;
        o.w16 = last ? w16_dev : nullptr;
        if (cudaMemsetAsync(o.sync, 0, 2 * sizeof(unsigned int), s) != cudaSuccess) return FFMIN_ERR_CUDA;
        cudaError_t e;
        while ((e = launch_train(o, clusters, cs, s)) != cudaSuccess) {
            // refused: too few SMs at hand (a share of the GPU) for so many
            // blocks, or, at the end, for a cluster
            if ((clusters == 1 && cs == 1) ||
                (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorLaunchOutOfResources &&
                 e != cudaErrorInvalidClusterSize))
                return FFMIN_ERR_CUDA;
            (void)cudaGetLastError();
            if (clusters > 1) {
                clusters = (clusters + 1) / 2;
            } else {
                cs = 1;
                clusters = (int)std::min<int64_t>(MLP_CLUSTER, blocks);
            }
        }
        unsigned int gave_up[2] = {0u, 0u};
        if (cudaMemcpyAsync(gave_up, o.sync, sizeof(gave_up), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            (loss_host && cudaMemcpyAsync(loss_host + t, o.losses, sizeof(float) * (size_t)o.steps,
                                          cudaMemcpyDeviceToHost, s) != cudaSuccess) ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return FFMIN_ERR_CUDA;
        if (gave_up[1]) return FFMIN_ERR_TIMEOUT;
    }
    return cudaGetLastError() == cudaSuccess ? FFMIN_OK : FFMIN_ERR_CUDA;
}

extern "C" int64_t ffmin_mlp_work_floats(void) {
    return (int64_t)MLP_ROWS * MLP_NW + MLP_ROWS + 1 + MLP_NW;
}
