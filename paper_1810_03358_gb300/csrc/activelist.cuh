// Active lists of the pair kernels' work queues.
#pragma once

#include "ffmin_internal.cuh"

namespace ffm {

// For each work queue: the systems with an evaluation request in its
// precision and kind and the exclusive prefix of their item counts, in system
// order, by one warp per queue (called by a block of at least N_LISTS warps).  Also resets the queues' counters.
__device__ inline void active_lists(const Ctx &c) {
    const int lane = threadIdx.x & 31, L = threadIdx.x >> 5;
    if (L >= N_LISTS) return;
    if (lane == 0) c.counters[L == LIST_F64 ? CNT_PAIR64 : (L == LIST_F32_E ? CNT_PAIR32E : CNT_PAIR)] = 0;
    int32_t *A = c.act + L * (2 * c.n_sys + 2);
    // each queue on the symmetric list of its precision when the object has one
    const int2 *items = L == LIST_F64 ? (c.sym64 ? c.sys_items64 : c.sys_items)
                                      : (L == LIST_F32_E && c.sym32 ? c.sys_items32 : c.sys_items);
    // 256 systems at a time: the loads of their states together (two dependent
    // ones for every 32 took 36 us for 1,024 systems, behind all tiles' trial
    // points), then warp scans over 32
    constexpr int U = 8;
    __shared__ int len[N_LISTS][U][32];
    int n_items = 0, n_act = 0;
    for (int b0 = 0; b0 < c.n_sys; b0 += 32 * U) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int b = b0 + 32 * u + lane;
            if (b >= c.n_sys) break;
            const int kind = c.st[b].ev_kind, mode = c.st[b].mode, n = items[b].y;
            const int mine = kind == EV_NONE ? -1 : (mode == 1 ? LIST_F64 : (kind == EV_E ? LIST_F32_E : LIST_F32_EG));
            len[L][u][lane] = mine == L ? n : 0;
        }
#pragma unroll 1
        for (int u = 0; b0 + 32 * u < c.n_sys && u < U; u++) {
            const int b = b0 + 32 * u + lane, n = b < c.n_sys ? len[L][u][lane] : 0;
            int sum = n;  // inclusive scan
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, sum, o);
                if (lane >= o) sum += v;
            }
            const unsigned on = __ballot_sync(0xffffffffu, n > 0);
            if (n > 0) {
                const int k = n_act + __popc(on & ((1u << lane) - 1u));
                A[2 + k] = n_items + sum - n;
                A[2 + c.n_sys + k] = b;
            }
            n_items += __shfl_sync(0xffffffffu, sum, 31);
            n_act += __popc(on);
        }
    }
    if (lane == 0) {
        A[0] = n_act;
        A[1] = n_items;
    }
}

}  // namespace ffm
