// Per-tile kernels of the minimizer pipeline (one 128-thread block per
// 128-atom tile, one thread per atom; finalize: a cluster of four blocks).
//
//   prepare   trial point XT = base + h * dir * scale (FP64, fused multiply-add
//             per component) and the pair-kernel positions (float4/double4_32a)
//   finalize  per-atom sum of the pair kernel's partial rows in a fixed order,
//             bonded terms of Section 2 gathered per atom (no atomics),
//             energy / gradient reductions, then the control step
//   update    accept a point, push an L-BFGS pair, FGM vector updates
//   dir       search directions: a G + b R + sum c_j S_j + sum c_j Y_j,
//             scaled by gamma (and the learned diagonal), with their dots
//
// Reductions are deterministic: every block writes its partial sums, the
// last block of a system to finish (atomic ticket) sums the system's blocks
// in a fixed order and runs its control step.  No thread ever waits.
//
// This file is compiled without contraction of a*b+c into FMA so that the
// scalar control arithmetic and the vector updates round like their
// textbook statements; fused multiply-adds appear only where written.
#include <cooperative_groups.h>

#include <cmath>
#include <utility>

#include "activelist.cuh"
#include "bonded.cuh"
#include "control.cuh"
#include "mlp.cuh"
#include "reduce.cuh"

namespace ffm {

namespace cg = cooperative_groups;

// <a, b> of two 3-vectors with explicit FMA (this unit is compiled without
// implicit contraction; the vector kernels are FP64-pipe bound)
__device__ __forceinline__ double dot3_fma(const double *a, const double *b) {
    return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2]));
}

// ---------------------------------------------------------------- prepare
// trial point of atom a: base + h (dir sc), and the pair-kernel positions
__device__ __forceinline__ void prepare_atom(const Ctx &c, int a, const double *base, const double *dir, double h,
                                             double sc, int mode, bool delta) {
    double *xt = vslot(c, V_XT) + 3 * a;
    double b[3], p[3];
    for (int k = 0; k < 3; k++) b[k] = base[3 * a + k];
    if (dir) {
        for (int k = 0; k < 3; k++) p[k] = fma(h, dir[3 * a + k] * sc, b[k]);
    } else {
        for (int k = 0; k < 3; k++) p[k] = b[k];
    }
    for (int k = 0; k < 3; k++) xt[k] = p[k];
    const double q = c.qs[a];
    if (mode == 0 && delta) {
        // difference trial: base position and the displacement, each rounded
        // once to FP32 (the displacement keeps its full relative precision)
        c.posf[a] = make_float4((float)b[0], (float)b[1], (float)b[2], (float)q);
        c.dispf[a] = make_float4((float)(p[0] - b[0]), (float)(p[1] - b[1]), (float)(p[2] - b[2]), 0.f);
    } else if (mode == 0) {
        c.posf[a] = make_float4((float)p[0], (float)p[1], (float)p[2], (float)q);
    } else {
        c.posd[a] = make_double4_32a(p[0], p[1], p[2], q);
    }
}

__global__ void __launch_bounds__(TI) k_prepare(Ctx c) {
    if (blockIdx.x == c.n_tiles) {  // the work queues, beside the tiles' trial points
        active_lists(c);
        return;
    }
    const Tile t = c.tiles[blockIdx.x];
    const SysState &S = c.st[t.sys];
    if (S.ev_kind == EV_NONE) return;
    const int i = threadIdx.x;
    if (i >= t.na) return;
    prepare_atom(c, t.a0 + i, vslot(c, S.ev_base), S.ev_dir >= 0 ? vslot(c, S.ev_dir) : nullptr, S.ev_h, S.ev_scale,
                 S.mode, S.ev_delta);
}

// One evaluation outside a minimization in three launches (this, the pair
// kernel of the kind, the finalize): the point is read where the caller has
// it, and block 0 sets every system's request and the work queues.  Uploading the states,
// copying the point and the active lists were half of a small evaluation.
__global__ void __launch_bounds__(TI) k_prepare_eval(Ctx c, EvalReq r) {
    const Tile &t = c.tiles[blockIdx.x];
    if (threadIdx.x < t.na) prepare_atom(c, t.a0 + threadIdx.x, r.base, r.dir, r.h, 1.0, r.mode, r.delta != 0);
    if (blockIdx.x != 0) return;
    for (int b = threadIdx.x; b < c.n_sys; b += TI) {
        SysState &S = c.st[b];
        S.active = 1;
        S.phase = PH_EVAL_ONLY;
        S.upd.op = U_NONE;
        S.dir[0].on = S.dir[1].on = 0;
        S.ev_kind = r.kind;
        S.ev_delta = r.delta;
        S.ne = S.neg = 0;
        S.mode = r.mode;
        S.epair_base = S.epair_last;
    }
    if (threadIdx.x == 0) {
        *c.nactive = c.n_sys;
        c.nmode[0] = r.mode == 0 ? c.n_sys : 0;
        c.nmode[1] = r.mode == 0 ? 0 : c.n_sys;
    }
    __syncthreads();
    active_lists(c);
}

cudaError_t launch_prepare_eval(const Ctx &c, const EvalReq &r, cudaStream_t s) {
    k_prepare_eval<<<c.n_tiles, TI, 0, s>>>(c, r);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- finalize
// Bound: latency (a chain of about ten loads, barriers and short FP64 sums; an
// FP64 operation holds a quarter of an SM for 64 cycles however few of its
// lanes are on).  A tile is a cluster of four blocks, 32 atoms each (or one block,
// 32 atoms after 32): warp w < 4
// sums the atoms' partial rows w, w + 4, ... (strand w; combined as
// (0 + 1) + (2 + 3)), warps 4 and 5 gather their bonded terms, then one warp
// finishes each component; the first block receives the atoms' contributions
// in its shared memory, forms the tile's sums and, in the system's last tile,
// the control step.  One block of 512 threads a tile took 16.2 us for 500 atoms
// and 22 us for 3,334 (FP64), half of them with one SM's FP64 pipe saturated and
// a sixth in fences executed by every warp; now 12.4 and 14.6 us.  The sums keep one
// order in every version of this kernel (strands, then the columns of
// block_reduce_columns, then the tiles): a MIXED minimization amplifies any
// other rounding.
constexpr int FIN_STRANDS = 4;
constexpr int FIN_PARTS = TI / 32;
constexpr int FIN_NT = 32 * (FIN_STRANDS + 2);

// exact FP32 -> FP64 on the integer pipe (the conversion instruction runs at
// the FP64 rate); the FP32 kernels flush denormals, which read as zero
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
    unsigned hi = m >= 0x7f800000u ? (m >> 3) | 0x70000000u : (m >> 3) + 0x38000000u;  // inf, NaN : normal
    const bool zero = m < 0x00800000u;
    hi = zero ? 0u : hi;
    return __hiloint2double((int)(hi | (u & 0x80000000u)), zero ? 0 : (int)(u << 29));
}

struct Row4 {
    double x, y, z, w;
};
__device__ __forceinline__ Row4 row_at(const double4_32a *rows, int64_t slot, int i) {
    const double4_32a p = rows[slot * TI + i];
    return Row4{p.x, p.y, p.z, p.w};
}

// sum of m FP32 rows FIN_STRANDS * TI apart from p on, in order, added to a;
// eight rows in flight (an object of 30,000 atoms has 20 a strand)
__device__ __forceinline__ void rows_f32(const float4 *p, int m, Row4 &a) {
    constexpr int U = 8, ST = FIN_STRANDS * TI;
    for (int q = 0; q < m; q += U, p += U * ST) {
        float4 v[U];
        const bool full = q + U <= m;
#pragma unroll
        for (int u = 0; u < U; u++) v[u] = full || q + u < m ? __ldcs(p + u * ST) : float4{0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (!full && q + u >= m) break;
            a.x += widen(v[u].x);
            a.y += widen(v[u].y);
            a.z += widen(v[u].z);
            a.w += widen(v[u].w);
        }
    }
}
// the same for energies alone
__device__ __forceinline__ void rows_f32(const float *p, int m, double &a) {
    constexpr int U = 16, ST = FIN_STRANDS * TI;
    for (int q = 0; q < m; q += U, p += U * ST) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; u++) v[u] = q + u < m ? __ldcs(p + u * ST) : 0.f;
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (q + u >= m) break;
            a += widen(v[u]);
        }
    }
}

// this strand's share (w, w + 4, ...) of the sum over q < n of f(q), in order,
// added to a; XYZ / W: the components that count; four or eight loads in flight
template <bool XYZ, bool W, typename F>
__device__ __forceinline__ void strand_sum(int n, int w, Row4 &a, F f) {
    constexpr int U = XYZ ? 4 : 8;
    for (int q = w; q < n; q += 4 * U) {
        Row4 p[U];
#pragma unroll
        for (int u = 0; u < U; u++) p[u] = q + 4 * u < n ? f(q + 4 * u) : Row4{0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (q + 4 * u >= n) break;
            if (XYZ) { a.x += p[u].x; a.y += p[u].y; a.z += p[u].z; }
            if (W) a.w += p[u].w;
        }
    }
}

// FP64 rows of atom i of tile t on the symmetric list: the j-side rows the
// tile received from the rows of the tiles at or left of it, then its own
// row's i-side rows (every part of every item)
template <bool GRAD>
__device__ __forceinline__ void sym_rows(const Ctx &c, const Tile &t, int tile0, int ntile, int i, int w, Row4 &a) {
    const int T = t.tloc, C = t.r64.chunk, P = t.r64.split;
    if (GRAD)
        strand_sum<true, false>(T + 1, w, a, [&](int I) {
            const int q = T - I;
            return row_at(c.gpd, (int64_t)c.tiles[tile0 + I].r64.slot + (int64_t)(q / C) * (P + C) + P + q % C, i);
        });
    strand_sum<GRAD, true>((ntile - T + C - 1) / C * P, w, a, [&](int m) {
        return row_at(c.gpd, (int64_t)t.r64.slot + (int64_t)(m / P) * (P + C) + m % P, i);
    });
}

// the control step's value for each of finalize's sums
__device__ __forceinline__ int fin_value(int k) {
    return k == 0 ? RF_E : (k == 1 ? RF_EPAIR : (k == 2 ? RF_GG : (k == 3 ? RF_GTG : RF_GTR)));
}

// CS: blocks per tile, four, or one that takes the tile's 32 atoms in turn, for
// objects of so many tiles that only the work of a block counts (its chain of
// loads, the state that it fetches, its ticket).  BLOCKS: resident blocks per SM, 4
// (80 registers, the shortest chain), 6 (56) for objects of more tiles than SMs,
// which run in waves, or 8 (40).  Us with 4 and 6 blocks of four per tile: 79 tiles
// 19.7, 19.8 (with gradient) and 11.7, 14.1; 157 tiles 33.9, 29.8 and 17.3, 17.1.
// Whole L-BFGS runs of batches, MIXED, ms, with four per tile at 6, one per tile at 6
// and at 8: 660 tiles 6.08, 6.13, 6.19; 1,024 tiles (500 atoms each) 8.85, 8.89, 8.39,
// (2,000) 11.19, 11.28, 10.78, (60) 11.99, 11.02, 10.29; 4,096 tiles 30.5, 28.8, 28.2.
template <int CS, int BLOCKS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(FIN_NT, BLOCKS) k_finalize(Ctx c, double *g_out) {
    const int tile = blockIdx.x / CS, rank = blockIdx.x % CS;
    const Tile &t = c.tiles[tile];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;  // w: strand, then bonded terms
    int i = 32 * rank + lane, a = t.a0 + i;
    bool real = i < t.na;
    constexpr int NSUM = 5;  // E, Epair and, with a gradient, g.g, g.G, g.R
    __shared__ double part[FIN_STRANDS][4][32], bond[2][4][32];
    __shared__ double sg[3 * 32], sr[3 * 32], sgt[3][32];  // current gradient, direction, new gradient
    // first block of the cluster: the tile's contributions
    __shared__ double val[NSUM][TI];
    __shared__ unsigned long long gmax[3 * FIN_PARTS];
    __shared__ int badf[4 * FIN_PARTS];
    __shared__ double strands[NSUM][RSTRANDS], tot[RF_N];
    __shared__ SysState sS;
    cg::cluster_group cl = cg::this_cluster();
    // bonded terms: the even entries of an atom's incidence list in warp 4,
    // the odd ones in warp 5
    constexpr int U = 5;  // an atom in a chain has 9 or 10 entries
    int k1 = 0, kb = 0;
    if (real && w >= FIN_STRANDS) {
        k1 = c.inc_off[a + 1];
        kb = c.inc_off[a] + w - FIN_STRANDS;
    }
    const SysState &S = c.st[t.sys];
    const int kind = S.ev_kind, mode = S.mode, ntile = S.ntile, tile0 = S.tile0;
    if (kind == EV_NONE) return;  // the whole cluster
    cg::cluster_group::arrival_token started{};
    if constexpr (CS > 1) started = cl.barrier_arrive();
    const bool grad = kind == EV_EG;
    if (rank == 0) prefetch_state(&sS, &S);
    for (int part32 = rank;; part32 += CS) {  // 32 atoms of the tile
        if (grad) {
            const int64_t o = 3 * ((int64_t)t.a0 + 32 * part32);
            const int n = 3 * min(32, max(0, t.na - 32 * part32));
            for (int k = threadIdx.x; k < n; k += FIN_NT) {
                async_copy8(&sg[k], vslot(c, V_G) + o + k);
                async_copy8(&sr[k], vslot(c, V_R) + o + k);
            }
        }
        if (w < FIN_STRANDS) {
            Row4 r = Row4{0.0, 0.0, 0.0, 0.0};
            if (real) {
                if (mode == 0 && c.sym32 && !grad) {
                    // energies on the symmetric list, each pair counted once
                    const int C = t.r32.chunk, n = (ntile - t.tloc + C - 1) / C;
                    rows_f32(c.gpf_sym + ((int64_t)t.r32.slot + w) * TI + i, (n - w + 3) / FIN_STRANDS, r.w);
                } else if (mode == 0) {
                    rows_f32(c.gpf + ((int64_t)t.item0 + w) * TI + i, (t.nitem - w + 3) / FIN_STRANDS, r);
                    r.w *= 0.5;  // every pair was counted in both of its rows
                } else if (c.sym64) {
                    if (grad) sym_rows<true>(c, t, tile0, ntile, i, w, r);
                    else sym_rows<false>(c, t, tile0, ntile, i, w, r);
                } else {
                    strand_sum<true, true>(t.nitem, w, r, [&](int it) { return row_at(c.gpd, t.item0 + it, i); });
                    r.w *= 0.5;
                }
            }
            part[w][0][lane] = r.x; part[w][1][lane] = r.y; part[w][2][lane] = r.z; part[w][3][lane] = r.w;
        } else {
            // evaluated once per term by the pair kernel's bonded items; an atom
            // takes its terms' energies (as owner) and position gradients
            Row4 bo = Row4{0.0, 0.0, 0.0, 0.0};
            for (; kb < k1; kb += 2 * U) {
                int2 in[U];
                Row4 p[U];
#pragma unroll
                for (int u = 0; u < U; u++) in[u] = kb + 2 * u < k1 ? c.inc[kb + 2 * u] : make_int2(-1, 0);
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int type = in[u].x >> 2, pos = in[u].x & 3;
                    if (in[u].x < 0) continue;
                    p[u].w = pos == 0 ? c.te[bonded_index(c, type, in[u].y)] : 0.0;
                    if (grad) {
                        const double *g = c.tg + 3 * bonded_grad_slot(c, type, in[u].y, pos);
                        p[u].x = g[0]; p[u].y = g[1]; p[u].z = g[2];
                    }
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (in[u].x < 0) break;
                    if ((in[u].x & 3) == 0) bo.w += p[u].w;
                    if (grad) { bo.x += p[u].x; bo.y += p[u].y; bo.z += p[u].z; }
                }
            }
            double (*b)[32] = bond[w - FIN_STRANDS];
            b[0][lane] = bo.x; b[1][lane] = bo.y; b[2][lane] = bo.z; b[3][lane] = bo.w;
        }
        async_wait();
        __syncthreads();
        if constexpr (CS > 1) cl.barrier_wait(std::move(started));  // the first block's shared memory is there
        // the first block's shared memory
        auto first = [&](auto *p) {
            if constexpr (CS > 1) return cl.map_shared_rank(p, 0);
            else return p;
        };
        double *tv = first(&val[0][0]) + i;
        auto finite = [](double x) { return ((unsigned)__double2hiint(x) & 0x7ff00000u) != 0x7ff00000u; };
        if (w < 4 && (grad || w == 3)) {  // component w of the gradient, or the energy
            double x = 0.0, q = 0.0;
            if (real) {
                q = (part[0][w][lane] + part[1][w][lane]) + (part[2][w][lane] + part[3][w][lane]);
                x = q + (bond[0][w][lane] + bond[1][w][lane]);
            }
            const unsigned bad = __ballot_sync(0xffffffffu, !finite(x));
            if (lane == 0) first(&badf[0])[4 * part32 + w] = bad != 0u;
            if (w == 3) {
                tv[0] = x;
                tv[TI] = q;
            } else {
                sgt[w][lane] = x;
                if (real) {
                    vslot(c, V_GT)[3 * (int64_t)a + w] = x;
                    if (g_out) g_out[3 * (int64_t)a + w] = x;
                }
                // the largest |component|, as an integer (a NaN counts as 0)
                const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu, lo = (unsigned)__double2loint(x);
                const bool nan = hi > 0x7ff00000u || (hi == 0x7ff00000u && lo != 0u);
                const unsigned mh = __reduce_max_sync(0xffffffffu, nan ? 0u : hi);
                const unsigned ml = __reduce_max_sync(0xffffffffu, !nan && hi == mh ? lo : 0u);
                if (lane == 0) first(&gmax[0])[3 * part32 + w] = (unsigned long long)mh << 32 | ml;
            }
        }
        if (grad) {
            __syncthreads();
            if (w < 3) {
                double x = 0.0;
                if (real) {
                    const double g0 = sgt[0][lane], g1 = sgt[1][lane], g2 = sgt[2][lane];
                    const double *o = w == 1 ? sg : sr;
                    const double o0 = w == 0 ? g0 : o[3 * lane], o1 = w == 0 ? g1 : o[3 * lane + 1],
                                 o2 = w == 0 ? g2 : o[3 * lane + 2];
                    x = fma(g0, o0, fma(g1, o1, g2 * o2));
                }
                tv[(2 + w) * TI] = x;
            }
        }
        if (CS == FIN_PARTS || part32 + CS >= FIN_PARTS) break;
        i += 32 * CS;
        a += 32 * CS;
        real = i < t.na;
        k1 = kb = 0;
        if (real && w >= FIN_STRANDS) {
            k1 = c.inc_off[a + 1];
            kb = c.inc_off[a] + w - FIN_STRANDS;
        }
        __syncthreads();  // the buffers of the next 32 atoms
    }
    if constexpr (CS == 1) __syncthreads();
    if constexpr (CS > 1) cl.sync();
    if (rank != 0) return;
    // the tile's sums, in the order of block_reduce_columns: values 0 to 3 in
    // warp 0, value 4 in warp 1
    const int nsum = grad ? NSUM : 2;
    if (w < 2) {
        const int k = 4 * w + lane / RSTRANDS, s = lane % RSTRANDS;
        if (k < nsum) {
            double x = val[k][s];
#pragma unroll
            for (int u = s + RSTRANDS; u < TI; u += RSTRANDS) x += val[k][u];
            strands[k][s] = x;
        }
        __syncwarp();
        const int k1v = 4 * w + lane;
        if (lane < 4 && k1v < NSUM) {
            double x = 0.0;
            if (k1v < nsum) {
                x = strands[k1v][0];
#pragma unroll
                for (int q = 1; q < RSTRANDS; q++) x += strands[k1v][q];
            }
            c.redf[(int64_t)k1v * c.n_tiles + tile] = x;
            tot[fin_value(k1v)] = 0.0 + x;  // of a system of one tile
        }
    } else if (w == 2) {
        unsigned long long m = grad && lane < 3 * FIN_PARTS ? gmax[lane] : 0ULL;
        const bool bad = lane < 4 * FIN_PARTS && (grad || (lane & 3) == 3) && badf[lane];
        const unsigned any_bad = __ballot_sync(0xffffffffu, bad);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, m, o);
            m = y > m ? y : m;
        }
        if (lane == 0) {
            const double gi = __longlong_as_double((long long)m), fb = any_bad ? 1.0 : 0.0;
            c.redf[(int64_t)5 * c.n_tiles + tile] = gi;
            c.redf[(int64_t)6 * c.n_tiles + tile] = fb;
            tot[RF_GINF] = gi;
            tot[RF_BAD] = fb;
        }
    }
    if (ntile > 1) {
        if (!sys_last_block(&c.tickets[STAGE_FIN * c.n_sys + t.sys], ntile)) return;
        const double *rd = c.redf + (int64_t)w * c.n_tiles;
        if (w < NSUM) {
            warp_sum1(rd, tile0, tile0 + ntile, &tot[fin_value(w)]);
        } else {
            warp_max(rd, tile0, tile0 + ntile, &tot[RF_GINF]);
            warp_max(rd + c.n_tiles, tile0, tile0 + ntile, &tot[RF_BAD]);
        }
    }
    __syncthreads();
    sys_control(c, t.sys, sS, [&](SysState &W) {
        if (lane == 0) on_eval_done(c, W, t.sys, tot);
    });
}

// ---------------------------------------------------------------- update
__global__ void __launch_bounds__(TI) k_update(Ctx c) {
    const Tile t = c.tiles[blockIdx.x];
    const SysState &S = c.st[t.sys];
    const int op = S.upd.op;
    const int i = threadIdx.x;
    __shared__ SysState sS;
    if (op == U_NONE) return;
    prefetch_state(&sS, &c.st[t.sys]);
    if (op == U_PUSH) {
        double v[RU_N];
#pragma unroll
        for (int k = 0; k < RU_N; k++) v[k] = 0.0;
        if (i < t.na) {
            const int64_t off = 3 * (int64_t)(t.a0 + i);
            double *X = vslot(c, V_X) + off, *G = vslot(c, V_G) + off;
            const double *XT = vslot(c, V_XT) + off, *GT = vslot(c, V_GT) + off;
            double *Ss = vslot(c, V_S0 + S.upd.stage) + off, *Ys = vslot(c, V_Y0 + S.upd.stage) + off;
            double s[3], y[3];
            for (int k = 0; k < 3; k++) {
                s[k] = XT[k] - X[k];
                y[k] = GT[k] - G[k];
                Ss[k] = s[k];
                Ys[k] = y[k];
            }
            v[RU_SY] = dot3_fma(s, y);
            v[RU_YY] = dot3_fma(y, y);
            if (S.rec_ptr && S.rec_every > 0 && S.iter % S.rec_every == 0) {
                const int slot = S.iter / S.rec_every - 1;
                if (slot < S.rec_slots) {
                    double *r = S.rec_ptr + ((int64_t)slot * c.n_atoms + t.a0 + i) * 4;
                    r[0] = v[RU_SY];
                    r[1] = v[RU_YY];
                    r[2] = sqrt(G[0] * G[0] + G[1] * G[1] + G[2] * G[2]);
                    r[3] = 1.0;
                }
            }
            v[RU_SG] = dot3_fma(s, GT);
            const int nS = S.upd.nS;
#pragma unroll
            for (int j = 0; j < NRING; j++) {
                if (j < nS) {
                    const double *sj = vslot(c, V_S0 + S.upd.sS[j]) + off;
                    v[ru_sjy(j)] = dot3_fma(sj, y);
                    v[ru_sjg(j)] = dot3_fma(sj, GT);
                }
            }
            for (int k = 0; k < 3; k++) { X[k] = XT[k]; G[k] = GT[k]; }
        }
        block_reduce_columns<RU_N>(v, ru_count(S.upd.nS), 0u, &c.red[(int64_t)blockIdx.x * NRED]);
    } else if (op == U_OGM) {
        double v[1] = {0.0};
        if (i < t.na) {
            const int64_t off = 3 * (int64_t)(t.a0 + i);
            double *X = vslot(c, V_X) + off, *G = vslot(c, V_G) + off, *W = vslot(c, V_W) + off;
            double *R = vslot(c, V_R) + off, *X0 = vslot(c, V_X0) + off, *DS = vslot(c, V_DS) + off;
            const double *XT = vslot(c, V_XT) + off, *GT = vslot(c, V_GT) + off;
            const UpdOp &u = S.upd;
            double rr[3];
            for (int k = 0; k < 3; k++) {
                double x = X[k], g = G[k];
                if (u.accept) { x = XT[k]; g = GT[k]; X[k] = x; G[k] = g; }
                double x0, ds;
                if (u.restart) {
                    x0 = x;
                    ds = g;
                    X0[k] = x0;
                } else {
                    x0 = X0[k];
                    ds = u.accept ? fma(u.h, g, DS[k]) : DS[k];
                }
                DS[k] = ds;
                W[k] = fma(u.a, x, u.b * x0);
                const double r = -fma(u.a, g, u.inv * ds);
                R[k] = r;
                rr[k] = r;
            }
            v[0] = dot3_fma(rr, rr);
        }
        block_reduce_columns<1>(v, 1, 0u, &c.red[(int64_t)blockIdx.x * NRED]);
    } else if (i < t.na) {
        const int64_t off = 3 * (int64_t)(t.a0 + i);
        double *X = vslot(c, V_X) + off, *G = vslot(c, V_G) + off, *W = vslot(c, V_W) + off;
        double *P = vslot(c, V_P) + off, *XB = vslot(c, V_XB) + off;
        const double *XT = vslot(c, V_XT) + off, *GT = vslot(c, V_GT) + off;
        switch (op) {
        case U_ACCEPT:
            for (int k = 0; k < 3; k++) { X[k] = XT[k]; G[k] = GT[k]; }
            break;
        case U_FGM_W:
            for (int k = 0; k < 3; k++) { W[k] = XT[k]; G[k] = GT[k]; }
            if (S.upd.best) for (int k = 0; k < 3; k++) XB[k] = XT[k];
            if (S.upd.restart)  // a (re)start at XT: x^k = x^{k-1} = XT
                for (int k = 0; k < 3; k++) { X[k] = XT[k]; P[k] = 0.0; }
            break;
        case U_FGM_ACCEPT: {
            const double *R = vslot(c, V_R) + off;
            const double h = S.upd.h, inv = S.upd.inv;
            for (int k = 0; k < 3; k++) {
                const double xn = fma(h, R[k] * inv, W[k]);
                P[k] = S.upd.restart ? 0.0 : xn - X[k];
                X[k] = xn;
                if (S.upd.best) XB[k] = xn;
            }
            break;
        }
        case U_FGM_RESET:
            for (int k = 0; k < 3; k++) { X[k] = W[k]; P[k] = 0.0; }
            break;
        case U_FGM_BEST_W:
            for (int k = 0; k < 3; k++) XB[k] = W[k];
            break;
        case U_HB: {  // Eq. 8, formed as the oracle forms it
            // accept the evaluated point (XT, GT): x^{k+1}, or at the start
            // x^0 itself with x^{-1} = x^0; then form the next iterate
            double *XTw = vslot(c, V_XT) + off;
            const double a = S.upd.a, b = S.upd.b;
            for (int k = 0; k < 3; k++) {
                const double x = XT[k], g = GT[k];
                const double xp = S.upd.accept ? X[k] : x;
                X[k] = x;
                G[k] = g;
                P[k] = xp;
                XTw[k] = fma(b, x - xp, fma(-a, g, x));
            }
            break;
        }
        default:
            break;
        }
    }
    async_wait();
    if (!sys_last_block(&c.tickets[STAGE_UPD * c.n_sys + t.sys], S.ntile)) return;
    __shared__ double tot[RU_N];
    sys_sums(c, S, op == U_PUSH ? ru_count(S.upd.nS) : (op == U_OGM ? 1 : 0), tot);
    sys_control(c, t.sys, sS, [&](SysState &W) { warp_update_done(c, W, tot); });
}

// ---------------------------------------------------------------- direction
template <int WHICH>
__global__ void __launch_bounds__(TI) k_dir(Ctx c) {
    const Tile t = c.tiles[blockIdx.x];
    const SysState &S = c.st[t.sys];
    const DirOp &d = S.dir[WHICH];
    const int i = threadIdx.x;
    double v[NRING];
#pragma unroll
    for (int k = 0; k < NRING; k++) v[k] = 0.0;
    __shared__ SysState sS;
    if (!d.on) return;
    prefetch_state(&sS, &c.st[t.sys]);
    __shared__ float w_mlp[MLP_NW];
    if (d.use_d) {  // learned H0 diagonal: FP16 weights -> FP32 in shared memory
        for (int k = threadIdx.x; k < MLP_NW; k += blockDim.x)
            w_mlp[k] = __half2float(__ushort_as_half(c.mlp_w[k]));
        __syncthreads();
    }
    if (i < t.na) {
        const int64_t off = 3 * (int64_t)(t.a0 + i);
        const double *G = vslot(c, V_G) + off;
        double *R = vslot(c, V_R) + off;
        double acc[3];
        for (int k = 0; k < 3; k++) {
            double x = 0.0;
            if (d.a != 0.0) x = d.a * G[k];
            if (d.b != 0.0) x = fma(d.b, R[k], x);
            acc[k] = x;
        }
        for (int j = 0; j < d.nY; j++) {
            const double *y = vslot(c, V_Y0 + d.sY[j]) + off;
            const double cy = d.cY[j];
            for (int k = 0; k < 3; k++) acc[k] = fma(cy, y[k], acc[k]);
        }
        for (int j = 0; j < d.nS; j++) {
            const double *s = vslot(c, V_S0 + d.sS[j]) + off;
            const double cs = d.cS[j];
            for (int k = 0; k < 3; k++) acc[k] = fma(cs, s[k], acc[k]);
        }
        double dscale = 1.0;
        if (d.use_d) {
            const int a = t.a0 + i;
            float f[MLP_IN];
            const double gn = sqrt(G[0] * G[0] + G[1] * G[1] + G[2] * G[2]);
            mlp_features(c.feat[3 * a], c.feat[3 * a + 1], c.feat[3 * a + 2], c.ncount[a], (float)gn, f);
            dscale = (double)mlp_scale(w_mlp, f);
        }
        for (int k = 0; k < 3; k++) {
            acc[k] = d.use_d ? (d.outer * dscale) * acc[k] : d.outer * acc[k];
            R[k] = acc[k];
        }
        if (d.dots == 1) {
            v[RD_RR] = dot3_fma(acc, acc);
            v[RD_GR] = dot3_fma(G, acc);
        } else if (d.dots == 2) {
#pragma unroll
            for (int j = 0; j < NRING; j++) {
                if (j < d.nY) {
                    const double *y = vslot(c, V_Y0 + d.sY[j]) + off;
                    v[j] = dot3_fma(y, acc);
                }
            }
        }
    }
    const int nv = d.dots == 2 ? d.nY : 2;
    block_reduce_columns<NRING>(v, nv, 0u, &c.red[(int64_t)blockIdx.x * NRED]);
    async_wait();
    if (!sys_last_block(&c.tickets[(WHICH == 0 ? STAGE_DIR1 : STAGE_DIR2) * c.n_sys + t.sys], S.ntile)) return;
    __shared__ double tot[NRING + 1];
    sys_sums(c, S, nv, tot);
    sys_control(c, t.sys, sS, [&](SysState &W) { warp_dir_done(c, W, WHICH, tot); });
}

// Neighbours within 8 A of every atom inside its own system, at x.  Block
// (tile, chunk): the tile's atoms against j-atoms staged in FP32 through shared
// memory, chunk y of every NC_CHUNKS-th j-tile; counts add up in out (zero
// before).  Each thread used to convert every j-atom of its system itself
// (conversions run at the FP64 rate), on as many SMs as there are tiles:
// 1,207 us for 32 systems of 200 to 5,000 atoms, 96 us now.
constexpr int NC_CHUNKS = 8;
__global__ void __launch_bounds__(TI) k_ncount(Ctx c, const double *x, int32_t *out) {
    __shared__ float4 sj[TI];
    const Tile &t = c.tiles[blockIdx.x];
    const SysState &S = c.st[t.sys];
    const int i = threadIdx.x, a = t.a0 + (i < t.na ? i : 0), end = S.atom0 + S.natoms;
    const float xi = (float)x[3 * a], yi = (float)x[3 * a + 1], zi = (float)x[3 * a + 2];
    int n = 0;
    for (int jt = S.atom0 + blockIdx.y * TI; jt < end; jt += NC_CHUNKS * TI) {
        const int j = jt + i;
        __syncthreads();
        if (j < end) sj[i] = make_float4((float)x[3 * j], (float)x[3 * j + 1], (float)x[3 * j + 2], 0.f);
        __syncthreads();
        const int m = min(TI, end - jt);
#pragma unroll 8
        for (int k = 0; k < m; k++) {
            const float dx = sj[k].x - xi, dy = sj[k].y - yi, dz = sj[k].z - zi;
            n += (jt + k != a && dx * dx + dy * dy + dz * dz < 64.f) ? 1 : 0;
        }
    }
    if (i < t.na && n) atomicAdd(&out[a], n);
}

cudaError_t launch_ncount(const Ctx &c, const double *x, int32_t *out, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(int32_t) * (size_t)c.n_atoms, s);
    if (e != cudaSuccess) return e;
    k_ncount<<<dim3(c.n_tiles, NC_CHUNKS), TI, 0, s>>>(c, x, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- basin hopping
// one block per tile, one thread per atom; the offset is formed as the
// oracle forms it (this unit has no implicit FMA contraction)
__global__ void __launch_bounds__(TI) k_mbh_perturb(Ctx c, const double *best, double *out, double step,
                                                   uint64_t seed, int64_t hop) {
    const Tile t = c.tiles[blockIdx.x];
    const int i = threadIdx.x;
    if (i >= t.na) return;
    const SysState &S = c.st[t.sys];
    const int a = t.a0 + i;
    const uint64_t base = (uint64_t)hop * (uint64_t)(3 * S.natoms) + 3ull * (uint64_t)(a - S.atom0);
    for (int k = 0; k < 3; k++) {
        const double u = (double)(splitmix64(seed + (uint64_t)t.sys, base + k) >> 11) * 0x1.0p-53;
        out[3 * a + k] = best[3 * a + k] + step * (2.0 * u - 1.0);
    }
}

__global__ void __launch_bounds__(TI) k_mbh_accept(Ctx c, const int32_t *flags, const double *x, double *best) {
    const Tile t = c.tiles[blockIdx.x];
    const int i = threadIdx.x;
    if (i >= t.na || !flags[t.sys]) return;
    const int a = t.a0 + i;
    for (int k = 0; k < 3; k++) best[3 * a + k] = x[3 * a + k];
}

cudaError_t launch_mbh_perturb(const Ctx &c, const double *best, double *out, double step, uint64_t seed,
                               int64_t hop, cudaStream_t s) {
    k_mbh_perturb<<<c.n_tiles, TI, 0, s>>>(c, best, out, step, seed, hop);
    return cudaGetLastError();
}
cudaError_t launch_mbh_accept(const Ctx &c, const int32_t *flags, const double *x, double *best, cudaStream_t s) {
    k_mbh_accept<<<c.n_tiles, TI, 0, s>>>(c, flags, x, best);
    return cudaGetLastError();
}

cudaError_t launch_prepare(const Ctx &c, cudaStream_t s) {
    k_prepare<<<c.n_tiles + 1, TI, 0, s>>>(c);
    return cudaGetLastError();
}
cudaError_t launch_finalize(const Ctx &c, cudaStream_t s, double *g_out) {
    if (c.n_tiles <= c.sms) k_finalize<FIN_PARTS, 4><<<c.n_tiles * FIN_PARTS, FIN_NT, 0, s>>>(c, g_out);
    else if (c.n_tiles <= 5 * c.sms) k_finalize<FIN_PARTS, 6><<<c.n_tiles * FIN_PARTS, FIN_NT, 0, s>>>(c, g_out);
    else k_finalize<1, 8><<<c.n_tiles, FIN_NT, 0, s>>>(c, g_out);
    return cudaGetLastError();
}
cudaError_t launch_update(const Ctx &c, cudaStream_t s) {
    k_update<<<c.n_tiles, TI, 0, s>>>(c);
    return cudaGetLastError();
}
cudaError_t launch_dir(const Ctx &c, int which, cudaStream_t s) {
    if (which == 0) k_dir<0><<<c.n_tiles, TI, 0, s>>>(c);
    else k_dir<1><<<c.n_tiles, TI, 0, s>>>(c);
    return cudaGetLastError();
}

}  // namespace ffm
