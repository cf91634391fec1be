// Gradient-free moves with FP64 terms (arXiv 1810.03358, Section 3; the move
// itself is described in parab.cu): a whole run of moves in one launch, for
// the sequential search and for the parts of a parallel epoch.
//
// Bound: latency.  A move is two dependent rounds, 7 rows and then the vertex
// row, each a sum over all atoms and the bonded terms of the moving atom, so
// the rounds stay on the chip: one thread-block cluster per part, every block
// with its own copy of the part's positions, partial sums exchanged through
// distributed shared memory at one cluster barrier a round, and the decision
// taken by every block alike (same sums, same order).  As two launches a move
// the sequential search cost 66 us a move at 500 atoms.
//
// Warps of a block: 14 pair warps (7 positions times two halves of the
// block's atoms; the vertex row over all 14) and one warp for the bonded terms
// (terms spread over the cluster's blocks, positions over the lanes), whose
// square roots and arc tangents take longer than a small system's pair sums
// and overlap them.  Pair terms are formed on the integer pipes
// (pair64.cuh), atom i's factors outside the sums.
//
// This file is compiled without implicit contraction (as parab.cu), so that
// positions and the far-field test round like their statements.
#include <cooperative_groups.h>

#include "bonded.cuh"
#include "ffmin_internal.cuh"
#include "pair64.cuh"

namespace ffm {

namespace cg = cooperative_groups;

constexpr int MV_PAIR_WARPS = 14;
constexpr int MV_THREADS = 32 * (MV_PAIR_WARPS + 1);
constexpr int MV_CLUSTER = 8;      // largest (portable) cluster
// partial sums of a block and round: one per pair warp, one bonded per position
constexpr int MV_PART = MV_PAIR_WARPS + 7;

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// SH: positions and this block's share of the parameters in shared memory;
// otherwise a private copy in global memory and the object's arrays
template <bool SH>
__global__ void __launch_bounds__(MV_THREADS, 1) k_moves64(Ctx c, MovesArgs a) {
    cg::cluster_group cl = cg::this_cluster();
    const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank(), part = blockIdx.x / CS;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n = a.n, sh = (n + CS - 1) / CS, j0 = min(n, rank * sh), nj = min(n, j0 + sh) - j0;
    extern __shared__ double dyn[];
    __shared__ double rows[MV_CLUSTER][MV_PART], vrow[MV_CLUSTER][MV_PAIR_WARPS + 1];
    __shared__ double s_f[8], s_pv[3];
    double *V = SH ? dyn : a.view + (int64_t)blockIdx.x * 3 * n;
    double *pq = dyn + 3 * n, *p6 = pq + sh, *p12 = p6 + sh;  // SH: the share's parameters
    const double *X = vslot(c, V_X);
    for (int t = tid; t < 3 * n; t += MV_THREADS) V[t] = X[t];
    if (SH) {
        for (int t = tid; t < nj; t += MV_THREADS) {
            const double2 p = c.pard[j0 + t];
            pq[t] = c.qs[j0 + t];
            p6[t] = p.x;
            p12[t] = p.y;
        }
    }
    const bool seq = a.list == nullptr;
    const int l0 = seq ? 0 : a.loff[part], cnt = seq ? n : a.loff[part + 1] - l0;
    const int moves = seq ? a.moves : a.allowed[part];
    const uint64_t base = ((uint64_t)part << 40) + a.base;
    cl.sync();  // every block has its copy (and started: its shared memory may be written)

    // this thread's share of a row: atom i at p, current position x0, atoms
    // t0, t0 + stride, ... of the block's share
    auto row = [&](int i, const double *p, const double *x0, int t0, int stride) -> double {
        double s1 = 0.0, s6 = 0.0, s12 = 0.0, ex = 0.0;
        const double qi = c.qs[i];
        const double2 ci = c.pard[i];
        // full warps: the fallback below votes
        for (int tb = t0 - lane; tb < nj; tb += stride) {
            const int t = tb + lane, tc = t < nj ? t : nj - 1, j = j0 + tc;
            const bool on = t < nj && j != i;
            const double xj = V[3 * j], yj = V[3 * j + 1], zj = V[3 * j + 2];
            const double qj = SH ? pq[tc] : c.qs[j];
            const double c6j = SH ? p6[tc] : c.pard[j].x, c12j = SH ? p12[tc] : c.pard[j].y;
            double dx = xj - p[0], dy = yj - p[1], dz = zj - p[2];
            if (!on) { dx = 1.0; dy = 0.0; dz = 0.0; }
            Inv64 v;
            bool ok = inv64(dx, dy, dz, v);
            double r1 = inv64_r1(v), r6 = inv64_r6(v), r12 = inv64_r12(v);
            bool far = false;
            if (a.taylor_r2 > 0.0) {  // linearised Coulomb term of a far atom
                double ex0 = xj - x0[0], ey0 = yj - x0[1], ez0 = zj - x0[2];
                far = on && ex0 * ex0 + ey0 * ey0 + ez0 * ez0 >= a.taylor_r2;
                if (!far) { ex0 = 1.0; ey0 = 0.0; ez0 = 0.0; }
                Inv64 v0;
                const bool ok0 = inv64(ex0, ey0, ez0, v0);
                const double dd = ex0 * (p[0] - x0[0]) + ey0 * (p[1] - x0[1]) + ez0 * (p[2] - x0[2]);
                const double i0 = inv64_r1(v0);
                if (far) {
                    r1 = fma(i0 * inv64_r2(v0), dd, i0);
                    ok = ok && ok0;
                }
            }
            if (__any_sync(0xffffffffu, !ok)) {  // out of range: the FP64 formula
                const double ri = rsqrt(dx * dx + dy * dy + dz * dz), ri2 = ri * ri, ri6 = ri2 * ri2 * ri2;
                double ec = qi * qj * ri;
                if (far) {
                    const double ex0 = xj - x0[0], ey0 = yj - x0[1], ez0 = zj - x0[2];
                    const double r02 = ex0 * ex0 + ey0 * ey0 + ez0 * ez0, e0 = qi * qj * rsqrt(r02);
                    ec = e0 + e0 / r02 * (ex0 * (p[0] - x0[0]) + ey0 * (p[1] - x0[1]) + ez0 * (p[2] - x0[2]));
                }
                const double e = ec + ri6 * (ci.y * c12j * ri6 - ci.x * c6j) * (1.0 / 6.0);
                ex += on ? e : 0.0;
            } else if (on) {
                s1 = fma(qj, r1, s1);
                s6 = fma(c6j, r6, s6);
                s12 = fma(c12j, r12, s12);
            }
        }
        return ex + (qi * s1 + (ci.y * s12 - ci.x * s6) * (1.0 / 6.0));
    };

    for (int m = 0; m < moves; m++) {
        const int pick = (int)__umul64hi(splitmix64(a.seed, base + (uint64_t)m), (uint64_t)cnt);
        const int i = seq ? pick : a.list[l0 + pick];
        const double x0[3] = {V[3 * i], V[3 * i + 1], V[3 * i + 2]};
        const int k0 = c.inc_off[i], k1 = c.inc_off[i + 1];
        // ---- the 7 rows: current position and +-delta along x, y, z
        if (w < MV_PAIR_WARPS) {
            const int q = w % 7;
            double p[3] = {x0[0], x0[1], x0[2]};
#pragma unroll
            for (int k = 0; k < 3; k++) {
                if (q == 1 + 2 * k) p[k] = p[k] + a.delta;
                if (q == 2 + 2 * k) p[k] = p[k] - a.delta;
            }
            const double e = warp_sum(row(i, p, x0, (w / 7) * 32 + lane, 64));
            if (lane < CS) cl.map_shared_rank(&rows[rank][w], lane)[0] = e;
        } else if (lane < 7) {  // bonded terms of atom i: one position per lane
            double p[3] = {x0[0], x0[1], x0[2]};
#pragma unroll
            for (int k = 0; k < 3; k++) {
                if (lane == 1 + 2 * k) p[k] = p[k] + a.delta;
                if (lane == 2 + 2 * k) p[k] = p[k] - a.delta;
            }
            double e = 0.0;
            for (int k = k0 + rank; k < k1; k += CS) {
                const int2 in = c.inc[k];
                e += bonded_term(c, V, in.x >> 2, in.y, in.x & 3, nullptr, nullptr, i, p);
            }
            for (int r = 0; r < CS; r++) cl.map_shared_rank(&rows[rank][MV_PAIR_WARPS + lane], r)[0] = e;
        }
        __syncwarp();
        cl.sync();
        if (w == 0) {  // sums over the blocks: lane = position + 8 * (block mod 4)
            const int q = lane & 7, r0 = lane >> 3;
            double f = 0.0;
            if (q < 7)
                for (int r = r0; r < CS; r += 4) f += (rows[r][q] + rows[r][q + 7]) + rows[r][MV_PAIR_WARPS + q];
            f += __shfl_xor_sync(0xffffffffu, f, 8);
            f += __shfl_xor_sync(0xffffffffu, f, 16);
            // per-axis parabola vertex
            const double f0 = __shfl_sync(0xffffffffu, f, 0);
            const int ax = lane < 3 ? lane : 0;
            const double fp = __shfl_sync(0xffffffffu, f, 1 + 2 * ax), fm = __shfl_sync(0xffffffffu, f, 2 + 2 * ax);
            const double curv = fm - 2.0 * f0 + fp;
            const double ts = curv > 0.0 ? a.delta * (fm - fp) / (2.0 * curv) : 0.0;
            if (lane < 3) s_pv[lane] = x0[lane] + ts;
            if (lane < 7) s_f[lane] = f;
        }
        __syncthreads();
        // ---- the vertex row
        const double pv[3] = {s_pv[0], s_pv[1], s_pv[2]};
        if (w < MV_PAIR_WARPS) {
            const double e = warp_sum(row(i, pv, x0, w * 32 + lane, 32 * MV_PAIR_WARPS));
            if (lane < CS) cl.map_shared_rank(&vrow[rank][w], lane)[0] = e;
        } else {
            // one term per lane: the terms of one block of the cluster
            double e = 0.0;
            for (int k = k0 + rank + CS * lane; k < k1; k += CS * 32) {
                const int2 in = c.inc[k];
                e += bonded_term(c, V, in.x >> 2, in.y, in.x & 3, nullptr, nullptr, i, pv);
            }
            e = warp_sum(e);
            if (lane < CS) cl.map_shared_rank(&vrow[rank][MV_PAIR_WARPS], lane)[0] = e;
        }
        __syncwarp();
        cl.sync();
        if (w == 0) {
            double f = 0.0;
            for (int t = lane; t < CS * (MV_PAIR_WARPS + 1); t += 32)
                f += vrow[t / (MV_PAIR_WARPS + 1)][t % (MV_PAIR_WARPS + 1)];
            f = warp_sum(f);
            if (lane == 0) {
                // the best of the 8 points, ties to the earlier one
                int best = 0;
                double fb = s_f[0];
                for (int q = 1; q < 7; q++)
                    if (s_f[q] < fb) { fb = s_f[q]; best = q; }
                double pb[3] = {x0[0], x0[1], x0[2]};
                for (int k = 0; k < 3; k++) {
                    if (best == 1 + 2 * k) pb[k] = pb[k] + a.delta;
                    if (best == 2 + 2 * k) pb[k] = pb[k] - a.delta;
                }
                const bool vert = f < fb;
                for (int k = 0; k < 3; k++) V[3 * i + k] = vert ? pv[k] : pb[k];
            }
        }
        __syncthreads();
    }
    // results: the sequential search writes X (every block its share: all
    // have read X before the first barrier); a part's atoms wait in the
    // view, since blocks of other parts may still have to read X
    if (seq) {
        double *Xw = vslot(c, V_X);
        for (int t = 3 * j0 + tid; t < 3 * (j0 + nj); t += MV_THREADS) Xw[t] = V[t];
    } else if (rank == 0) {
        for (int t = a.moff[part] + tid; t < a.moff[part + 1]; t += MV_THREADS) {
            const int j = a.members[t];
            for (int k = 0; k < 3; k++) a.merged[3 * j + k] = V[3 * j + k];
        }
    }
    cl.sync();  // no block leaves while its shared memory may be written
}

// blocks per part: the largest power of two up to MV_CLUSTER that lets every
// part run at once
int moves_cluster(int parts, int sms) {
    int cs = 1;
    while (cs < MV_CLUSTER && 2 * cs * parts <= sms) cs *= 2;
    return cs;
}
// dynamic shared memory of the SH form, or 0 when it does not fit
static size_t moves_smem(int n, int cs) {
    const size_t b = sizeof(double) * (3 * (size_t)n + 3 * (size_t)((n + cs - 1) / cs));
    return b <= 208 * 1024 ? b : 0;
}
// doubles of private copies that a launch needs in MovesArgs::view
int64_t moves_view_doubles(int n, int parts, int cs) { return moves_smem(n, cs) ? 0 : (int64_t)3 * n * parts * cs; }

cudaError_t launch_moves64(const Ctx &c, const MovesArgs &a, int parts, int cs, cudaStream_t s) {
    const size_t smem = moves_smem(a.n, cs);
    cudaError_t e = cudaSuccess;
    if (smem) e = cudaFuncSetAttribute(k_moves64<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 208 * 1024);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(parts * cs);
    cfg.blockDim = dim3(MV_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cs;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return smem ? cudaLaunchKernelEx(&cfg, k_moves64<true>, c, a) : cudaLaunchKernelEx(&cfg, k_moves64<false>, c, a);
}

}  // namespace ffm
