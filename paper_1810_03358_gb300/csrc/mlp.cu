// Training of the per-atom preconditioner network on the GPU: mean squared
// error between z(f) and the recorded target t over a data set, plain
// backpropagation through the two layers, and Adam (Kingma & Ba 2015).
// Hand-written kernels, FP32 arithmetic; weights are handed to inference as
// FP16.  Minibatches are drawn with the SplitMix64 counter stream.
//
// Loss per sample: (z - t)^2; minibatch loss = mean.  Gradients:
//   dz = 2 (z - t) / B,  dw2_k = dz h_k,  db2 = dz,
//   dh_k = dz w2_k [a_k > 0],  dW1_ki = dh_k f_i,  db1_k = dh_k.
// Per-block partial gradients are summed in a fixed order by a second kernel,
// so a step is deterministic.
//
// Bound: latency (a step of 16,384 rows is 44 MFLOP, under a microsecond of
// FP32).  Forward with one thread per row, backward with one thread per two
// hidden units, whose 14 gradient sums stay in registers; the start's form
// kept all 449 sums per thread in local memory and added them over the block
// one parameter at a time (320 us a step, 27 us for the Adam kernel).  The
// two kernels of a step are launched programmatically dependent, so that the
// next one's rows are gathered while this one ends, and the losses stay on
// the device until the last step.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "ffmin.h"
#include "mlp.cuh"

namespace ffm {

constexpr int MT = 128;          // threads per training block, one row each
constexpr int MLP_ROWS = 256;    // partial-gradient rows of the scratch
constexpr int MLP_BLOCKS = 152;  // blocks per minibatch gradient, at most
// the scratch rows that no block uses hold the losses of up to this many steps
constexpr int MLP_LOSSES = (MLP_ROWS - MLP_BLOCKS) * MLP_NW;
constexpr int AT = 1024, AP = 32;  // Adam kernel: threads, parameters per block

// programmatic dependent launch: let the next kernel of the stream start /
// wait for the previous one to have finished
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint64_t mix64(uint64_t seed, uint64_t k) {
    uint64_t z = seed + (k + 1) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// partial gradient of one block over its share of the minibatch; samples of
// the minibatch are index (base + k) of the SplitMix64 stream when sample
// != 0, else rows [0, batch) of the data in order
__global__ void __launch_bounds__(MT) k_mlp_grad(const float *feat, const float *target, int64_t n,
                                                 const float *w32, int batch, uint64_t seed, uint64_t base,
                                                 int sample, float *part, float *loss_part) {
    __shared__ float4 sw[MLP_H][2];        // per hidden unit: W1 (5), b1, w2
    __shared__ float4 sf[MT / 32][32][2];  // per row of the warp: features (5), dz
    __shared__ float acc[MT / 32][MLP_NW];
    __shared__ float lsum[MT / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    pdl_trigger();
    float f[MLP_IN], t = 0.f;
    const float inv_b = 1.0f / (float)batch;
    float g[2][MLP_IN + 2] = {};  // of units lane, lane + 32: W1, b1, w2
    float gb2 = 0.f, loss = 0.f;
    float wu[2][MLP_IN + 2];
    float b2 = 0.f;
    for (int s0 = blockIdx.x * MT; s0 < batch; s0 += gridDim.x * MT) {
        const int s = s0 + threadIdx.x;
        const bool on = s < batch;
#pragma unroll
        for (int i = 0; i < MLP_IN; i++) f[i] = 0.f;
        if (on) {
            const int64_t row = sample ? (int64_t)__umul64hi(mix64(seed, base + s), (uint64_t)n) : s;
#pragma unroll
            for (int i = 0; i < MLP_IN; i++) f[i] = feat[row * MLP_IN + i];
            t = target[row];
        }
        if (s0 == (int)blockIdx.x * MT) {  // the weights, once the previous step has written them
            pdl_wait();
            for (int k = threadIdx.x; k < MLP_H; k += MT) {
                const float *w1 = w32 + MLP_W1 + k * MLP_IN;
                sw[k][0] = make_float4(w1[0], w1[1], w1[2], w1[3]);
                sw[k][1] = make_float4(w1[4], w32[MLP_B1 + k], w32[MLP_W2 + k], 0.f);
            }
            b2 = w32[MLP_B2];
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const float4 p = sw[lane + 32 * u][0], q = sw[lane + 32 * u][1];
                wu[u][0] = p.x; wu[u][1] = p.y; wu[u][2] = p.z; wu[u][3] = p.w;
                wu[u][4] = q.x; wu[u][5] = q.y; wu[u][6] = q.z;
            }
        }
        // forward: one row per thread
        float z = b2;
#pragma unroll 8
        for (int k = 0; k < MLP_H; k++) {
            const float4 p = sw[k][0], q = sw[k][1];
            float a = fmaf(p.x, f[0], q.y);
            a = fmaf(p.y, f[1], a);
            a = fmaf(p.z, f[2], a);
            a = fmaf(p.w, f[3], a);
            a = fmaf(q.x, f[4], a);
            z = fmaf(q.z, fmaxf(a, 0.f), z);
        }
        const float r = on ? z - t : 0.f;
        loss += r * r;
        const float dz = 2.f * r * inv_b;
        gb2 += dz;
        sf[w][lane][0] = make_float4(f[0], f[1], f[2], f[3]);
        sf[w][lane][1] = make_float4(f[4], dz, 0.f, 0.f);
        __syncwarp();
        // backward: two hidden units per thread, the warp's rows in order
#pragma unroll 4
        for (int m = 0; m < 32; m++) {
            const float4 p = sf[w][m][0], q = sf[w][m][1];
#pragma unroll
            for (int u = 0; u < 2; u++) {
                float a = fmaf(wu[u][0], p.x, wu[u][5]);
                a = fmaf(wu[u][1], p.y, a);
                a = fmaf(wu[u][2], p.z, a);
                a = fmaf(wu[u][3], p.w, a);
                a = fmaf(wu[u][4], q.x, a);
                const float h = fmaxf(a, 0.f);
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
    // the warps' sums in warp order
#pragma unroll
    for (int u = 0; u < 2; u++) {
        const int k = lane + 32 * u;
#pragma unroll
        for (int i = 0; i < MLP_IN; i++) acc[w][MLP_W1 + k * MLP_IN + i] = g[u][i];
        acc[w][MLP_B1 + k] = g[u][5];
        acc[w][MLP_W2 + k] = g[u][6];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        gb2 += __shfl_xor_sync(0xffffffffu, gb2, o);
        loss += __shfl_xor_sync(0xffffffffu, loss, o);
    }
    if (lane == 0) {
        acc[w][MLP_B2] = gb2;
        lsum[w] = loss;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < MLP_NW; k += MT) {
        float v = acc[0][k];
#pragma unroll
        for (int q = 1; q < MT / 32; q++) v += acc[q][k];
        part[(int64_t)blockIdx.x * MLP_NW + k] = v;
    }
    if (threadIdx.x == 0) {
        float v = lsum[0];
#pragma unroll
        for (int q = 1; q < MT / 32; q++) v += lsum[q];
        loss_part[blockIdx.x] = v;
    }
}

// Sum of the block partials (thread (q, k) of a block takes the blocks q,
// q + 32, ... of parameter k, then the 32 sums in order); then one Adam step
// on the FP32 master weights (when lr > 0) and the FP16 copy for inference
__global__ void __launch_bounds__(AT) k_mlp_adam(const float *part, const float *loss_part, int nblocks, int batch,
                                                 float *w32, float *adam, int step, float lr, float *grad_out,
                                                 float *loss_out, uint16_t *w16) {
    __shared__ float sums[AT / AP][AP + 1];
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const int p = threadIdx.x & (AP - 1), q = threadIdx.x / AP, k = blockIdx.x * AP + p;
    pdl_trigger();
    pdl_wait();
    // the loss counts as one more parameter, behind the last
    float v = 0.f;
    if (k < MLP_NW) {
        for (int b = q; b < nblocks; b += AT / AP) v += part[(int64_t)b * MLP_NW + k];
    } else if (k == MLP_NW) {
        for (int b = q; b < nblocks; b += AT / AP) v += loss_part[b];
    }
    sums[q][p] = v;
    __syncthreads();
    if (q != 0 || k > MLP_NW) return;
    float gk = 0.f;
#pragma unroll
    for (int r = 0; r < AT / AP; r++) gk += sums[r][p];
    if (k == MLP_NW) {
        if (loss_out) *loss_out = gk / (float)batch;
        return;
    }
    if (grad_out) grad_out[k] = gk;
    if (lr > 0.f) {
        float m = adam[k] = b1 * adam[k] + (1.f - b1) * gk;
        float vv = adam[MLP_NW + k] = b2 * adam[MLP_NW + k] + (1.f - b2) * gk * gk;
        const float mh = m / (1.f - powf(b1, (float)step));
        const float vh = vv / (1.f - powf(b2, (float)step));
        w32[k] -= lr * mh / (sqrtf(vh) + eps);
    }
    if (w16) {
        __half hv = __float2half_rn(w32[k]);
        w16[k] = *reinterpret_cast<uint16_t *>(&hv);
    }
}

template <typename... A, typename... B>
static cudaError_t launch_dependent(void (*kernel)(A...), int grid, int block, cudaStream_t s, bool dependent, B... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, A(args)...);
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
    float *part = work_dev;                                    // [MLP_BLOCKS][MLP_NW]
    float *losses = part + (size_t)MLP_BLOCKS * MLP_NW;        // [MLP_LOSSES]
    float *loss_part = work_dev + (size_t)MLP_ROWS * MLP_NW;   // [MLP_ROWS]
    float *grad_dev = loss_part + MLP_ROWS + 1;                // [MLP_NW]
    const int nsteps = steps > 0 ? steps : 1;
    const int sample = steps > 0 ? 1 : 0;
    const int b = steps > 0 ? batch : (int)std::min<int64_t>(batch, n_samples);
    const int blocks = (int)std::min<int64_t>(MLP_BLOCKS, ((int64_t)b + MT - 1) / MT);
    int kept = 0;  // steps whose losses have been copied
    for (int t = 0; t < nsteps; t++) {
        // the first kernel waits for whatever the stream held before; the
        // others depend on the kernel before them alone
        if (launch_dependent(k_mlp_grad, blocks, MT, s, t > kept, feat_dev, target_dev, n_samples,
                             (const float *)w32_dev, b, seed, (uint64_t)t * (uint64_t)batch, sample, part,
                             loss_part) != cudaSuccess)
            return FFMIN_ERR_CUDA;
        const bool last = t == nsteps - 1;
        if (launch_dependent(k_mlp_adam, (MLP_NW + AP) / AP, AT, s, true, (const float *)part,
                             (const float *)loss_part, blocks, b, w32_dev, adam_dev, t + 1, steps > 0 ? lr : 0.f,
                             last ? grad_dev : (float *)nullptr, losses + (t - kept),
                             last ? w16_dev : (uint16_t *)nullptr) != cudaSuccess)
            return FFMIN_ERR_CUDA;
        if (last || t - kept + 1 == MLP_LOSSES) {
            if (loss_host && cudaMemcpyAsync(loss_host + kept, losses, sizeof(float) * (size_t)(t - kept + 1),
                                             cudaMemcpyDeviceToHost, s) != cudaSuccess)
                return FFMIN_ERR_CUDA;
            kept = t + 1;
        }
    }
    if (cudaStreamSynchronize(s) != cudaSuccess) return FFMIN_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? FFMIN_OK : FFMIN_ERR_CUDA;
}

extern "C" int64_t ffmin_mlp_work_floats(void) {
    return (int64_t)MLP_ROWS * MLP_NW + MLP_ROWS + 1 + MLP_NW;
}
