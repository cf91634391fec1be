// Per-tile kernels of the minimizer pipeline (one 128-thread block per
// 128-atom tile, one thread per atom) and the bonded terms.
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
// last block to finish (atomic ticket) sums each system's blocks in a fixed
// order and runs that system's control step.  No thread ever waits.
//
// This file is compiled without contraction of a*b+c into FMA so that the
// scalar control arithmetic and the vector updates round like their
// textbook statements; fused multiply-adds appear only where written.
#include <cmath>

#include "bonded.cuh"
#include "control.cuh"
#include "mlp.cuh"
#include "reduce.cuh"

namespace ffm {

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
    const Tile t = c.tiles[blockIdx.x];
    const SysState &S = c.st[t.sys];
    if (S.ev_kind == EV_NONE) return;
    const int i = threadIdx.x;
    if (i >= t.na) return;
    prepare_atom(c, t.a0 + i, vslot(c, S.ev_base), S.ev_dir >= 0 ? vslot(c, S.ev_dir) : nullptr, S.ev_h, S.ev_scale,
                 S.mode, S.ev_delta);
}

// One evaluation outside a minimization in three launches (this, the pair
// kernel of the kind, the finalize; one more for 8 systems and up): the point
// is read where the caller has it, and block 0 sets every system's request
// and the one work queue that the evaluation uses.  Uploading the states,
// copying the point and the active lists were half of a small evaluation.
__global__ void __launch_bounds__(TI) k_prepare_eval(Ctx c, EvalReq r) {
    const Tile &t = c.tiles[blockIdx.x];
    if (threadIdx.x < t.na) prepare_atom(c, t.a0 + threadIdx.x, r.base, r.dir, r.h, 1.0, r.mode, r.delta != 0);
    if (blockIdx.x != 0) return;
    __shared__ int wsum[NW];
    __shared__ int base;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int2 *items = r.list == LIST_F64 ? (c.sym64 ? c.sys_items64 : c.sys_items)
                                           : (r.list == LIST_F32_E && c.sym32 ? c.sys_items32 : c.sys_items);
    int32_t *A = c.act + r.list * (2 * c.n_sys + 2);
    if (threadIdx.x == 0) {
        base = 0;
        c.counters[r.list == LIST_F64 ? CNT_PAIR64 : (r.list == LIST_F32_E ? CNT_PAIR32E : CNT_PAIR)] = 0;
        *c.nactive = c.n_sys;
        c.nmode[0] = r.mode == 0 ? c.n_sys : 0;
        c.nmode[1] = r.mode == 0 ? 0 : c.n_sys;
        A[0] = c.n_sys;
    }
    __syncthreads();
    for (int b0 = 0; b0 < c.n_sys; b0 += TI) {
        const int b = b0 + threadIdx.x;
        int n = 0;
        if (b < c.n_sys) {
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
            n = items[b].y;
        }
        int sum = n;  // inclusive scan within the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += u;
        }
        if (lane == 31) wsum[w] = sum;
        __syncthreads();
        int p = base + sum - n;
        for (int v = 0; v < w; v++) p += wsum[v];
        if (b < c.n_sys) {
            A[2 + b] = p;
            A[2 + c.n_sys + b] = b;
        }
        __syncthreads();
        if (threadIdx.x == TI - 1) base = p + n;
        __syncthreads();
    }
    if (threadIdx.x == 0) A[1] = base;
}

cudaError_t launch_prepare_eval(const Ctx &c, const EvalReq &r, cudaStream_t s) {
    k_prepare_eval<<<c.n_tiles, TI, 0, s>>>(c, r);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- finalize
// Bound: latency and the FP64 pipe (16 cycles per warp operation and SM).
// One block per tile, four threads per atom: strand s of an atom sums its
// partial rows s, s + 4, ..., the strands are combined through shared memory
// as (0 + 1) + (2 + 3).  One thread per atom took 25 us for 500 atoms and 31 us
// for 3,334 (cold caches).  The sums keep one order in every version of this
// kernel (strands, then the columns of block_reduce_columns, then the tiles):
// a MIXED minimization amplifies any other rounding.
constexpr int FIN_STRANDS = 4;
constexpr int FIN_NT = TI * FIN_STRANDS;

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
__device__ __forceinline__ Row4 row_at(const float4 *rows, int64_t slot, int i) {
    const float4 p = rows[slot * TI + i];
    return Row4{widen(p.x), widen(p.y), widen(p.z), widen(p.w)};
}
__device__ __forceinline__ Row4 row_at(const double4_32a *rows, int64_t slot, int i) {
    const double4_32a p = rows[slot * TI + i];
    return Row4{p.x, p.y, p.z, p.w};
}

// this strand's share (w, w + 4, ...) of the sum over q < n of f(q), added to
// a; XYZ / W: the components that count
template <bool XYZ, bool W, typename F>
__device__ __forceinline__ void strand_sum(int n, int w, Row4 &a, F f) {
    int q = w;
    for (; q + 12 < n; q += 16) {  // four loads in flight
        Row4 p[4];
#pragma unroll
        for (int u = 0; u < 4; u++) p[u] = f(q + 4 * u);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            if (XYZ) { a.x += p[u].x; a.y += p[u].y; a.z += p[u].z; }
            if (W) a.w += p[u].w;
        }
    }
    for (; q < n; q += 4) {
        const Row4 p = f(q);
        if (XYZ) { a.x += p.x; a.y += p.y; a.z += p.z; }
        if (W) a.w += p.w;
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

// sum (or max) of finalize value k over a system's tiles, fixed order, by a
// whole warp; the result is valid on every lane
__device__ double fin_sys_sum(const Ctx &c, const SysState &S, int k, bool mx) {
    const int lane = threadIdx.x & 31, t1 = S.tile0 + S.ntile;
    const double *r = c.redf + (int64_t)k * c.n_tiles;
    double x = 0.0;
#pragma unroll 4
    for (int t = S.tile0 + lane; t < t1; t += 32) {
        const double y = __ldcg(&r[t]);
        x = mx ? fmax(x, y) : x + y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double y = __shfl_xor_sync(0xffffffffu, x, o);
        x = mx ? fmax(x, y) : x + y;
    }
    return x;
}

__global__ void __launch_bounds__(FIN_NT) k_finalize(Ctx c, double *g_out) {
    const Tile &t = c.tiles[blockIdx.x];
    const SysState &S = c.st[t.sys];
    const int kind = S.ev_kind, mode = S.mode;
    const int i = threadIdx.x % TI, w = threadIdx.x / TI;  // atom, strand
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ Row4 part[FIN_STRANDS][TI];
    __shared__ Row4 bond[TI];
    __shared__ double val[RF_N][TI + 1];
    __shared__ double strands[RF_N][RSTRANDS];
    const unsigned maxmask = (1u << RF_GINF) | (1u << RF_BAD);
    if (kind != EV_NONE) {
        const bool real = i < t.na, grad = kind == EV_EG;
        const int a = t.a0 + i;
        Row4 r = Row4{0.0, 0.0, 0.0, 0.0}, bo = r;
        if (real) {
            if (mode == 0 && c.sym32 && !grad) {
                // energies on the symmetric list, each pair counted once
                const int C = t.r32.chunk;
                strand_sum<false, true>((S.ntile - t.tloc + C - 1) / C, w, r, [&](int q) {
                    return Row4{0.0, 0.0, 0.0, widen(c.gpf_sym[((int64_t)t.r32.slot + q) * TI + i])};
                });
            } else if (mode == 0) {
                strand_sum<true, true>(t.nitem, w, r, [&](int it) { return row_at(c.gpf, t.item0 + it, i); });
                r.w *= 0.5;  // every pair was counted in both of its rows
            } else if (c.sym64) {
                if (grad) sym_rows<true>(c, t, S.tile0, S.ntile, i, w, r);
                else sym_rows<false>(c, t, S.tile0, S.ntile, i, w, r);
            } else {
                strand_sum<true, true>(t.nitem, w, r, [&](int it) { return row_at(c.gpd, t.item0 + it, i); });
                r.w *= 0.5;
            }
            // bonded terms: evaluated once per term by the pair kernel's
            // bonded items; every atom gathers its terms' energies (as owner)
            // and position gradients through its incidence list, the even
            // entries in strand 2, the odd ones in strand 3
            if (w >= 2) {
                const int k1 = c.inc_off[a + 1];
#pragma unroll 2
                for (int k = c.inc_off[a] + w - 2; k < k1; k += 2) {
                    const int2 in = c.inc[k];
                    const int type = in.x >> 2, pos = in.x & 3;
                    if (pos == 0) bo.w += c.te[bonded_index(c, type, in.y)];
                    if (grad) {
                        const double *g = c.tg + 3 * bonded_grad_slot(c, type, in.y, pos);
                        bo.x += g[0]; bo.y += g[1]; bo.z += g[2];
                    }
                }
            }
        }
        part[w][i] = r;
        if (w == 3) bond[i] = bo;
        __syncthreads();
        if (w == 2) {  // the whole atom
            double v[RF_N];
#pragma unroll
            for (int k = 0; k < RF_N; k++) v[k] = 0.0;
            if (real) {
                const Row4 r0 = part[0][i], r1 = part[1][i], r3 = part[3][i], b1 = bond[i];
                const double ep = (r0.w + r1.w) + (r.w + r3.w);
                const double e = ep + (bo.w + b1.w);
                v[RF_EPAIR] = ep;
                v[RF_E] = e;
                bool bad = !isfinite(e);
                if (grad) {
                    const double g0 = ((r0.x + r1.x) + (r.x + r3.x)) + (bo.x + b1.x);
                    const double g1 = ((r0.y + r1.y) + (r.y + r3.y)) + (bo.y + b1.y);
                    const double g2 = ((r0.z + r1.z) + (r.z + r3.z)) + (bo.z + b1.z);
                    double *gt = vslot(c, V_GT) + 3 * a;
                    gt[0] = g0; gt[1] = g1; gt[2] = g2;
                    if (g_out) { g_out[3 * a] = g0; g_out[3 * a + 1] = g1; g_out[3 * a + 2] = g2; }
                    const double *G = vslot(c, V_G) + 3 * a;
                    const double *R = vslot(c, V_R) + 3 * a;
                    v[RF_GG] = fma(g0, g0, fma(g1, g1, g2 * g2));
                    v[RF_GINF] = fmax(fabs(g0), fmax(fabs(g1), fabs(g2)));
                    v[RF_GTG] = fma(g0, G[0], fma(g1, G[1], g2 * G[2]));
                    v[RF_GTR] = fma(g0, R[0], fma(g1, R[1], g2 * R[2]));
                    bad = bad || !isfinite(g0) || !isfinite(g1) || !isfinite(g2);
                }
                v[RF_BAD] = bad ? 1.0 : 0.0;
            }
#pragma unroll
            for (int k = 0; k < RF_N; k++) val[k][i] = v[k];
        }
        __syncthreads();
        // the tile's sums, in the order of block_reduce_columns
        if (threadIdx.x < RF_N * RSTRANDS) {
            const int k = threadIdx.x / RSTRANDS, s = threadIdx.x % RSTRANDS;
            const bool mx = (maxmask >> k) & 1u;
            double x = val[k][s];
#pragma unroll
            for (int u = s + RSTRANDS; u < TI; u += RSTRANDS) x = mx ? fmax(x, val[k][u]) : x + val[k][u];
            strands[k][s] = x;
        }
        __syncthreads();
        if (threadIdx.x < RF_N) {
            const int k = threadIdx.x;
            const bool mx = (maxmask >> k) & 1u;
            double x = strands[k][0];
#pragma unroll
            for (int s = 1; s < RSTRANDS; s++) x = mx ? fmax(x, strands[k][s]) : x + strands[k][s];
            c.redf[(int64_t)k * c.n_tiles + blockIdx.x] = x;
        }
    }
    if (c.sep_reduce || !last_block(&c.counters[CNT_FIN])) return;
    // fewer than 8 systems: the last block sums every system's tiles, one
    // (system, value) per warp at a time, then warp 0 runs the control steps
    // in system order on a shared-memory copy of the state
    __shared__ double tot[LB_MAX_SYS][RF_N];
    __shared__ SysState sS;
    const int n = c.n_sys < LB_MAX_SYS ? c.n_sys : LB_MAX_SYS;
    for (int u = warp; u < n * RF_N; u += FIN_NT / 32) {
        const SysState &Sb = c.st[u / RF_N];
        if (Sb.ev_kind == EV_NONE) continue;
        const double x = fin_sys_sum(c, Sb, u % RF_N, (maxmask >> (u % RF_N)) & 1u);
        if (lane == 0) tot[u / RF_N][u % RF_N] = x;
    }
    __syncthreads();
    if (warp == 0) {
        for (int b = 0; b < n; b++) {
            if (c.st[b].ev_kind == EV_NONE) continue;
            warp_copy_state(&sS, &c.st[b]);
            if (lane == 0) on_eval_done(c, sS, b, tot[b]);
            __syncwarp();
            warp_copy_state(&c.st[b], &sS);
        }
    }
    if (threadIdx.x == 0) c.counters[CNT_FIN] = 0;
}

// ---------------------------------------------------------------- update
__global__ void __launch_bounds__(TI) k_update(Ctx c) {
    const Tile t = c.tiles[blockIdx.x];
    const SysState &S = c.st[t.sys];
    const int op = S.upd.op;
    const int i = threadIdx.x;
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
    } else if (op != U_NONE && i < t.na) {
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
    if (c.sep_reduce || !last_block(&c.counters[CNT_UPD])) return;
    last_block_systems<RU_N>(
        c, RU_N, 0u, [](const SysState &S) { return S.upd.op != U_NONE; },
        [&](SysState &S, const double *tot) { on_update_done(c, S, tot); },
        [](const SysState &S) { return S.upd.op == U_PUSH ? ru_count(S.upd.nS) : (S.upd.op == U_OGM ? 1 : 0); });
    __syncthreads();
    if (threadIdx.x == 0) c.counters[CNT_UPD] = 0;
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
    const bool on = d.on != 0;
    __shared__ float w_mlp[MLP_NW];
    if (on && d.use_d) {  // learned H0 diagonal: FP16 weights -> FP32 in shared memory
        for (int k = threadIdx.x; k < MLP_NW; k += blockDim.x)
            w_mlp[k] = __half2float(__ushort_as_half(c.mlp_w[k]));
        __syncthreads();
    }
    if (on && i < t.na) {
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
    if (on) block_reduce_columns<NRING>(v, d.dots == 2 ? d.nY : 2, 0u, &c.red[(int64_t)blockIdx.x * NRED]);
    if (c.sep_reduce || !last_block(&c.counters[WHICH == 0 ? CNT_DIR1 : CNT_DIR2])) return;
    last_block_systems<NRING>(
        c, 2, 0u, [](const SysState &S) { return S.dir[WHICH].on != 0; },
        [&](SysState &S, const double *tot) { on_dir_done(c, S, WHICH, tot); },
        [](const SysState &S) { return S.dir[WHICH].dots == 2 ? S.dir[WHICH].nY : 2; });
    __syncthreads();
    if (threadIdx.x == 0) c.counters[WHICH == 0 ? CNT_DIR1 : CNT_DIR2] = 0;
}

// one block per system: the system's tile partials of every value are summed
// by the block's warps in tile order, then thread 0 runs the control step
template <int STAGE>
__global__ void __launch_bounds__(TI) k_sysreduce(Ctx c) {
    SysState &S = c.st[blockIdx.x];
    int nv;
    unsigned maxmask = 0u;
    if (STAGE == 0) {
        if (S.upd.op == U_NONE) return;
        nv = S.upd.op == U_PUSH ? ru_count(S.upd.nS) : (S.upd.op == U_OGM ? 1 : 0);
    } else if (STAGE == 1 || STAGE == 2) {
        const DirOp &d = S.dir[STAGE - 1];
        if (!d.on) return;
        nv = d.dots == 2 ? d.nY : 2;
    } else {
        if (S.ev_kind == EV_NONE) return;
        nv = RF_N;
        maxmask = (1u << RF_GINF) | (1u << RF_BAD);
    }
    __shared__ double tot[NRED];
    __shared__ SysState sS;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int k = w; k < nv; k += NW) {
        const double x = STAGE == 3 ? fin_sys_sum(c, S, k, (maxmask >> k) & 1u)
                                    : warp_sys_sum(c, S, k, (maxmask >> k) & 1u);
        if (lane == 0) tot[k] = x;
    }
    __syncthreads();
    if (w != 0) return;
    // the control step on a shared-memory copy of the state
    warp_copy_state(&sS, &S);
    if (lane == 0) {
        if (STAGE == 0) on_update_done(c, sS, tot);
        else if (STAGE == 1) on_dir_done(c, sS, 0, tot);
        else if (STAGE == 2) on_dir_done(c, sS, 1, tot);
        else on_eval_done(c, sS, blockIdx.x, tot);
    }
    __syncwarp();
    warp_copy_state(&S, &sS);
}

cudaError_t launch_sysreduce(const Ctx &c, int stage, cudaStream_t s) {
    switch (stage) {
    case 0: k_sysreduce<0><<<c.n_sys, TI, 0, s>>>(c); break;
    case 1: k_sysreduce<1><<<c.n_sys, TI, 0, s>>>(c); break;
    case 2: k_sysreduce<2><<<c.n_sys, TI, 0, s>>>(c); break;
    default: k_sysreduce<3><<<c.n_sys, TI, 0, s>>>(c); break;
    }
    return cudaGetLastError();
}

// neighbours within 8 A of every atom inside its own system, from X
__global__ void __launch_bounds__(TI) k_ncount(Ctx c, const double *x, int32_t *out) {
    const Tile t = c.tiles[blockIdx.x];
    const SysState &S = c.st[t.sys];
    const int i = threadIdx.x;
    if (i >= t.na) return;
    const int a = t.a0 + i;
    const float xi = (float)x[3 * a], yi = (float)x[3 * a + 1], zi = (float)x[3 * a + 2];
    int n = 0;
    for (int j = S.atom0; j < S.atom0 + S.natoms; j++) {
        const float dx = (float)x[3 * j] - xi, dy = (float)x[3 * j + 1] - yi, dz = (float)x[3 * j + 2] - zi;
        n += (j != a && dx * dx + dy * dy + dz * dz < 64.f) ? 1 : 0;
    }
    out[a] = n;
}

cudaError_t launch_ncount(const Ctx &c, const double *x, int32_t *out, cudaStream_t s) {
    k_ncount<<<c.n_tiles, TI, 0, s>>>(c, x, out);
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
    k_prepare<<<c.n_tiles, TI, 0, s>>>(c);
    return cudaGetLastError();
}
cudaError_t launch_finalize(const Ctx &c, cudaStream_t s, double *g_out) {
    k_finalize<<<c.n_tiles, FIN_NT, 0, s>>>(c, g_out);
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
