// Deterministic block and per-system reductions shared by the per-tile
// kernels: every block stores its partial sums; the last block of a system to
// finish (atomic ticket per system, no waiting) sums the system's blocks in a
// fixed order and runs its control step, so the systems of a batch do not
// wait for one another and no further launch is needed.
#pragma once

#include "ffmin_internal.cuh"

namespace ffm {

constexpr int NW = TI / 32;

template <int NR>
__device__ inline void block_reduce_store(double (&v)[NR], unsigned maxmask, double *dst) {
    __shared__ double sh[NW][NR];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NR; k++) {
        double x = v[k];
        const bool mx = (maxmask >> k) & 1u;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double y = __shfl_xor_sync(0xffffffffu, x, o);
            x = mx ? fmax(x, y) : x + y;
        }
        if (lane == 0) sh[w][k] = x;
    }
    __syncthreads();
    if (threadIdx.x < NR) {
        const int k = threadIdx.x;
        const bool mx = (maxmask >> k) & 1u;
        double x = sh[0][k];
        for (int j = 1; j < NW; j++) x = mx ? fmax(x, sh[j][k]) : x + sh[j][k];
        dst[k] = x;
    }
}

__device__ inline bool last_block(unsigned int *cnt) {
    __shared__ int am_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned t = atomicAdd(cnt, 1u);
        am_last = (t == gridDim.x - 1);
        if (am_last) __threadfence();
    }
    __syncthreads();
    return am_last != 0;
}

// Block reduction of nv <= NV values through shared memory: every thread
// stores its values; column k is summed (or, for the bits of maxmask,
// maximised) in RSTRANDS interleaved strands (strand s: threads s,
// s + RSTRANDS, ... in order), then its strand results in strand order.
// One FP64 operation per thread and value, where a shuffle tree costs five
// (the FP64 pipe is the scarce unit of the kernels that use it), and a
// dependent chain of TI / RSTRANDS + RSTRANDS operations instead of TI (a
// dependent FP64 operation takes hundreds of cycles when the pipe is shared).
constexpr int RSTRANDS = 8;
template <int NV>
__device__ inline double (*columns_buffer())[TI + 1] {
    __shared__ double sh[NV][TI + 1];
    return sh;
}
template <int NV>
__device__ inline void block_reduce_columns(const double (&v)[NV], int nv, unsigned maxmask, double *dst) {
    double (*sh)[TI + 1] = columns_buffer<NV>();
    __shared__ double part[NV][RSTRANDS];
#pragma unroll
    for (int k = 0; k < NV; k++)
        if (k < nv) sh[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int u = threadIdx.x; u < nv * RSTRANDS; u += TI) {
        const int k = u / RSTRANDS, s = u % RSTRANDS;
        const bool mx = (maxmask >> k) & 1u;
        double x = sh[k][s];
#pragma unroll 4
        for (int t = s + RSTRANDS; t < TI; t += RSTRANDS) x = mx ? fmax(x, sh[k][t]) : x + sh[k][t];
        part[k][s] = x;
    }
    __syncthreads();
    if (threadIdx.x < nv) {
        const int k = threadIdx.x;
        const bool mx = (maxmask >> k) & 1u;
        double x = part[k][0];
#pragma unroll
        for (int s = 1; s < RSTRANDS; s++) x = mx ? fmax(x, part[k][s]) : x + part[k][s];
        dst[k] = x;
    }
}

// ticket of a block among its system's: true in the last one, which then may
// read what the others stored (the thread with the ticket fences for the
// block, the barrier passes it on: a fence in all of 16 warps took 5,000
// cycles, during which the shuffles behind it waited)
__device__ inline bool sys_last_block(unsigned int *cnt, int ntile) {
    __shared__ int am_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        am_last = atomicAdd(cnt, 1u) == (unsigned)ntile - 1u;
        if (am_last) {
            *cnt = 0u;  // for the next launch
            __threadfence();
        }
    }
    __syncthreads();
    return am_last != 0;
}

// Sums of up to 8 values over a system's tiles by a warp: value k of tile t at
// r[k vs + t ts]; lane l takes tiles l, l + 32, ... in order, then the lanes
// are combined 16 apart, 8 apart, ... 1 apart, sharing the values out on the
// way (9 additions for 8 values; the FP64 unit takes 64 cycles for each,
// however many lanes are on).  Stored to out[k].
__device__ inline void warp_sums8(const double *r, int64_t vs, int64_t ts, int t0, int t1, int nv, double *out) {
    const int lane = threadIdx.x & 31;
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = 0.0;
#pragma unroll 2
    for (int t = t0 + lane; t < t1; t += 32) {
        double y[8];
#pragma unroll
        for (int k = 0; k < 8; k++) y[k] = k < nv ? __ldcg(&r[k * vs + t * ts]) : 0.0;
#pragma unroll
        for (int k = 0; k < 8; k++)
            if (k < nv) x[k] += y[k];
    }
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int k = 0; k < h; k++) {
            const double keep = up ? x[k + h] : x[k], send = up ? x[k] : x[k + h];
            x[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
        }
    }
    x[0] += __shfl_xor_sync(0xffffffffu, x[0], 2);
    x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
    if ((lane & 3) == 0 && (lane >> 2) < nv) out[lane >> 2] = x[0];
}
// the same for one value at r[t]
__device__ inline void warp_sum1(const double *r, int t0, int t1, double *out) {
    const int lane = threadIdx.x & 31;
    double x = 0.0;
    for (int t = t0 + lane; t < t1; t += 8 * 32) {
        double y[8];
#pragma unroll
        for (int k = 0; k < 8; k++) y[k] = t + 32 * k < t1 ? __ldcg(&r[t + 32 * k]) : 0.0;
#pragma unroll
        for (int k = 0; k < 8; k++)
            if (t + 32 * k < t1) x += y[k];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) *out = x;
}
// largest of non-negative values (no NaN) over a system's tiles by a warp, as integers
__device__ inline void warp_max(const double *r, int t0, int t1, double *out) {
    const int lane = threadIdx.x & 31;
    unsigned long long x = 0ULL;
    for (int t = t0 + lane; t < t1; t += 32) {
        const unsigned long long y = (unsigned long long)__double_as_longlong(__ldcg(&r[t]));
        x = y > x ? y : x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
        x = y > x ? y : x;
    }
    if (lane == 0) *out = __longlong_as_double((long long)x);
}
// the first nv reduction values of a per-tile kernel (c.red), by the block
__device__ inline void sys_sums(const Ctx &c, const SysState &S, int nv, double *out) {
    for (int k = 8 * (threadIdx.x >> 5); k < nv; k += 8 * (blockDim.x >> 5))
        warp_sums8(c.red + k, 1, NRED, S.tile0, S.tile0 + S.ntile, min(8, nv - k), out + k);
    __syncthreads();
}

// A system's control state on its way to shared memory from the start of the
// kernel (asynchronous copies by the whole block), so that the control step, a
// long chain of dependent reads and writes of the state, runs on a copy that
// is there when the last block gets to it.  async_wait, then a barrier, before
// the first use.
static_assert(sizeof(SysState) % 8 == 0, "SysState is copied in 8-byte words");
__device__ inline void async_copy8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ inline void async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ inline void prefetch_state(SysState *dst, const SysState *src) {
    for (int k = threadIdx.x; k < (int)(sizeof(SysState) / 8); k += blockDim.x)
        async_copy8(reinterpret_cast<unsigned long long *>(dst) + k, reinterpret_cast<const unsigned long long *>(src) + k);
}

// control step of system b by warp 0 on the prefetched copy sS: fn(sS) is
// called by the whole warp
template <typename Fn>
__device__ inline void sys_control(const Ctx &c, int b, SysState &sS, Fn fn) {
    if (threadIdx.x >= 32) return;
    fn(sS);
    __syncwarp();
    const unsigned long long *s = reinterpret_cast<const unsigned long long *>(&sS);
    unsigned long long *d = reinterpret_cast<unsigned long long *>(&c.st[b]);
    for (int k = threadIdx.x; k < (int)(sizeof(SysState) / 8); k += 32) d[k] = s[k];
}

}  // namespace ffm
