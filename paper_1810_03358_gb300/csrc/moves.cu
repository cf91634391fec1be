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
// The FP64 unit takes an instruction of a warp every 64 cycles of an SM
// quarter, however many lanes are on, so a move is counted in FP64
// instructions per warp.  Rows: one j-atom per thread at all 7 positions (they
// share two coordinates of three), coordinates in fixed point, terms on the
// integer pipes (pair64.cuh), 24 instructions an atom and 7 rows; the lanes
// share the 7 sums out by halving (9 additions, not 35).  Bonded terms on
// warps of their own, one per kind, lane = (term, position), in forms of their
// own: 10 instructions for a bond, about 35 for an angle, 45 for a torsion.
// 500 atoms: 66 us a move as two launches, 16 us with the terms in plain FP64
// and a warp per position, 8.7 us now; 3,334 atoms 68 and 14.3 us.
//
// This file is compiled without implicit contraction (as parab.cu), so that
// positions and the far-field test round like their statements.
#include <cooperative_groups.h>

#include <cmath>

#include "bonded.cuh"
#include "ffmin_internal.cuh"
#include "pair64.cuh"

namespace ffm {

namespace cg = cooperative_groups;

constexpr int MV_PAIR_WARPS = 12;
constexpr int MV_BOND_WARPS = 4;   // bonds, angles, torsions, exclusion corrections
constexpr int MV_WARPS = MV_PAIR_WARPS + MV_BOND_WARPS;
constexpr int MV_THREADS = 32 * MV_WARPS;
constexpr int MV_CLUSTER = 8;      // largest (portable) cluster
// fast rows: coordinates within this (differences below 2^62 units), an axis
// offset of at most 0.2 A, and pairs at least 1/2 A apart along some axis
constexpr double MV_FIX_MAX = 112.0, MV_DELTA_MAX = 0.2;
// fixed-point coordinate of one beyond: its difference from any in range is at
// least 2^62 (and below 2^63)
constexpr long long MV_FAR = 3LL << 61;
// arc tangents: sine and cosine at multiples of pi / MV_ATAN
constexpr int MV_ATAN = 128;

// Sums over the warp of 8 values per lane: lane l returns value l / 4 (three
// exchanges share the values out, two more add within the groups of 4)
__device__ __forceinline__ double sum8(double (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int k = 0; k < h; k++) {
            const double keep = up ? v[k + h] : v[k], send = up ? v[k] : v[k + h];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
        }
    }
    double x = v[0];
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x;
}
__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// x^-1/2 and 1/x of a normal positive double, on the integer pipes
__device__ __forceinline__ Inv64 inv_of(double x) {
    const u64 u = bits64(x);
    const int e = (int)(u >> 52) - 1023;
    Inv64 v;  // x = R 2^(2 E - 60), E = floor(e / 2)
    inv64_back(((u & 0xfffffffffffffULL) | 0x10000000000000ULL) << (8 + (e & 1)), e >> 1, v);
    return v;
}
__device__ __forceinline__ bool normal_positive(double x) {
    const u64 u = bits64(x);
    return u >= 0x0010000000000000ULL && u < 0x7ff0000000000000ULL;
}
__device__ __forceinline__ double dot_fma(const double *a, const double *b) {
    return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2]));
}
__device__ __forceinline__ void cross_fma(const double *a, const double *b, double *o) {
    o[0] = fma(a[1], b[2], -(a[2] * b[1]));
    o[1] = fma(a[2], b[0], -(a[0] * b[2]));
    o[2] = fma(a[0], b[1], -(a[1] * b[0]));
}

// Energy of one bonded term with atom i at p (bonded.cuh has the formulas;
// degenerate geometries go there).  Angle: theta = theta_k + atan(t) with
// theta_k the table angle nearest to the FP32 arc tangent, t = sin / cos of
// theta - theta_k by the addition theorems, |t| < 0.0123, and the arc
// tangent's series to t^9 (the next term is below 2^-66).  Torsion: the four
// terms are polynomials in cos phi.
template <int TYPE>
__device__ __forceinline__ double bonded_energy(const Ctx &c, const double2 *tab, const double *x, int term, int pos,
                                                int i, const double *p) {
    if (TYPE == 0) {
        const int2 ij = c.bidx[term];
        const double2 kp = c.bpar[term];
        double xi[3], xj[3], d[3];
        ld3(x, ij.x, xi, i, p);
        ld3(x, ij.y, xj, i, p);
        for (int k = 0; k < 3; k++) d[k] = xi[k] - xj[k];
        const double dd = dot_fma(d, d);
        const double r = normal_positive(dd) ? dd * inv64_r1(inv_of(dd)) : sqrt(dd);
        return kp.x * (r - kp.y) * (r - kp.y);
    }
    if (TYPE == 1) {
        const int4 q = c.aidx[term];
        const double2 kp = c.apar[term];
        double xi[3], xj[3], xk[3], u[3], v[3], w[3];
        ld3(x, q.x, xi, i, p);
        ld3(x, q.y, xj, i, p);
        ld3(x, q.z, xk, i, p);
        for (int k = 0; k < 3; k++) { u[k] = xi[k] - xj[k]; v[k] = xk[k] - xj[k]; }
        cross_fma(u, v, w);
        const double ww = dot_fma(w, w), uv = dot_fma(u, v);
        const double cr = normal_positive(ww) ? ww * inv64_r1(inv_of(ww)) : sqrt(ww);
        const int k = __float2int_rn(atan2f((float)cr, (float)uv) * (float)(MV_ATAN / 3.14159265358979323846));
        const double2 sc = tab[k < 0 ? 0 : (k > MV_ATAN ? MV_ATAN : k)];  // sine, cosine
        const double num = fma(cr, sc.y, -(uv * sc.x)), den = fma(uv, sc.y, cr * sc.x);
        if (!normal_positive(den)) return bonded_term(c, x, 1, term, pos, nullptr, nullptr, i, p);
        const double t = num * inv64_r2(inv_of(den));
        const double z = t * t;
        const double s = fma(z, fma(z, fma(z, 1.0 / 9.0, -1.0 / 7.0), 1.0 / 5.0), -1.0 / 3.0);
        const double th = fma((double)k, 3.14159265358979323846 / MV_ATAN, fma(t * z, s, t));
        if (!(z < 0.01)) return bonded_term(c, x, 1, term, pos, nullptr, nullptr, i, p);  // FP32 range left
        return kp.x * (th - kp.y) * (th - kp.y);
    }
    if (TYPE == 2) {
        const int4 q = c.didx[term];
        const double4_32a V = c.dpar[term];
        double xi[3], xj[3], xk[3], xl[3], b1[3], b2[3], b3[3], m[3], n[3];
        ld3(x, q.x, xi, i, p);
        ld3(x, q.y, xj, i, p);
        ld3(x, q.z, xk, i, p);
        ld3(x, q.w, xl, i, p);
        for (int k = 0; k < 3; k++) { b1[k] = xj[k] - xi[k]; b2[k] = xk[k] - xj[k]; b3[k] = xl[k] - xk[k]; }
        cross_fma(b1, b2, m);
        cross_fma(b2, b3, n);
        const double mm = dot_fma(m, m), nn = dot_fma(n, n), pr = mm * nn;
        if (mm < 1e-12 || nn < 1e-12 || !normal_positive(pr))
            return bonded_term(c, x, 2, term, pos, nullptr, nullptr, i, p);
        const double cp = dot_fma(m, n) * inv64_r1(inv_of(pr));
        const double t = cp * cp, c2 = fma(2.0, t, -1.0), c3 = cp * fma(4.0, t, -3.0), c4 = fma(2.0 * c2, c2, -1.0);
        return 0.5 * fma(V.x, 1.0 + cp, fma(V.y, 1.0 - c2, fma(V.z, 1.0 + c3, V.w * (1.0 - c4))));
    }
    return bonded_term(c, x, 3, term, pos, nullptr, nullptr, i, p);
}

// Bonded energy of atom i's terms of one kind (k0 .. k1: its incidence list,
// sorted by kind) at NP positions, by one warp: lane q < NP returns the sum at
// position q.  pos3: the positions, [NP][3]; buf: 32 doubles of the warp.
template <int TYPE, int NP>
__device__ __forceinline__ double bonded_rows(const Ctx &c, const double2 *tab, const double *x, int k0, int k1, int i,
                                              const double (*pos3)[3], double *buf) {
    const int lane = threadIdx.x & 31;
    double sum = 0.0;
    for (int kb = k0; kb < k1; kb += 32) {
        const int2 in = kb + lane < k1 ? c.inc[kb + lane] : make_int2(-1, 0);
        const unsigned mine = __ballot_sync(0xffffffffu, in.x >= 0 && (in.x >> 2) == TYPE);
        const int first = mine ? __ffs((int)mine) - 1 : 0, cnt = __popc(mine);
        constexpr int PER = 32 / NP;  // terms per pass
        for (int r0 = 0; r0 < cnt; r0 += PER) {
            const int r = r0 + lane / NP, q = lane % NP;
            const int src = first + (r < cnt ? r : 0);
            const int x4 = __shfl_sync(0xffffffffu, in.x, src), term = __shfl_sync(0xffffffffu, in.y, src);
            double e = 0.0;
            if (lane < PER * NP && r < cnt) {
                const double p[3] = {pos3[q][0], pos3[q][1], pos3[q][2]};
                e = bonded_energy<TYPE>(c, tab, x, term, x4 & 3, i, p);
            }
            buf[lane] = e;
            __syncwarp();
            if (lane < NP)
                for (int u = 0; u < PER && r0 + u < cnt; u++) sum += buf[u * NP + lane];
            __syncwarp();
        }
    }
    return sum;
}

// |x| < MV_FIX_MAX for the three coordinates (false for a NaN), on the integer pipe
__device__ __forceinline__ bool in_fix(const double *x) {
    constexpr unsigned lim = 0x405C0000u;  // the high word of 112.0
    static_assert(MV_FIX_MAX == 112.0, "lim is MV_FIX_MAX");
    unsigned m = 0u;
    for (int k = 0; k < 3; k++) m = max(m, (unsigned)__double2hiint(x[k]) & 0x7fffffffu);
    return m < lim;
}

// SH: positions and this block's share of the parameters in shared memory;
// otherwise a private copy in global memory and the object's arrays.
// GEN: rows from FP64 differences, for what the fixed-point rows leave out: a
// larger offset, the far field, systems beyond the range.  Nine FP64 instructions
// more for an atom's 7 rows (with the far field about 35), and the alignment of
// the significands: 3,334 atoms 19.4 us a move (22.6), 41 (70) in plain FP64 terms.
// A kernel of its own, since its code beside the other rows cost those 3 % (4.54
// -> 4.71 ms for 500 moves of 500 atoms).
template <bool SH, bool GEN>
__global__ void __launch_bounds__(MV_THREADS, 1) k_moves64(Ctx c, MovesArgs a) {
    cg::cluster_group cl = cg::this_cluster();
    const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank(), part = blockIdx.x / CS;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n = a.n, sh = (n + CS - 1) / CS, j0 = min(n, rank * sh), nj = min(n, j0 + sh) - j0;
    extern __shared__ double dyn[];
    __shared__ double2 tab[MV_ATAN + 1];
    __shared__ double wsum[MV_WARPS][8];                   // sums of this block's warps
    __shared__ double crow[MV_CLUSTER][8], cvert[MV_CLUSTER];  // sums of the cluster's blocks
    __shared__ double pos[8][3];                           // the 7 positions and the vertex
    __shared__ double buf[MV_BOND_WARPS][32];
    __shared__ double s_f[8];
    double *V = SH ? dyn : a.view + (int64_t)blockIdx.x * (3 * (int64_t)n + 3 * sh);
    long long *F = reinterpret_cast<long long *>(V + 3 * n);             // the share in fixed point
    double *pq = V + 3 * n + 3 * sh, *p6 = pq + sh, *p12 = p6 + sh;      // SH: the share's parameters
    const double *X = vslot(c, V_X);
    for (int t = tid; t < 3 * n; t += MV_THREADS) V[t] = X[t];
    for (int t = tid; t < 3 * nj; t += MV_THREADS) {
        const double x = X[3 * j0 + t];
        long long f;
        fix64(x, f);
        F[t] = fabs(x) < MV_FIX_MAX ? f : MV_FAR;
    }
    if (SH) {
        for (int t = tid; t < nj; t += MV_THREADS) {
            const double2 p = c.pard[j0 + t];
            pq[t] = c.qs[j0 + t];
            p6[t] = p.x;
            p12[t] = p.y;
        }
    }
    if (tid <= MV_ATAN) {
        double sn, cs;
        sincospi((double)tid / MV_ATAN, &sn, &cs);
        tab[tid] = make_double2(sn, cs);
    }
    const bool seq = a.list == nullptr;
    const int l0 = seq ? 0 : a.loff[part], cnt = seq ? n : a.loff[part + 1] - l0;
    const int moves = seq ? a.moves : a.allowed[part];
    const uint64_t base = ((uint64_t)part << 40) + a.base;
    cl.sync();  // every block has its copy (and started: its shared memory may be written)

    // FP64 form of the pair term of atoms i (at p, current position x0) and
    // j0 + t, with the far field; for the pairs that the integer forms leave out
    auto pair_plain = [&](int i, const double *p, const double *x0, int t) -> double {
        const int j = j0 + t;
        const double dx = V[3 * j] - p[0], dy = V[3 * j + 1] - p[1], dz = V[3 * j + 2] - p[2];
        const double ri = rsqrt(dx * dx + dy * dy + dz * dz), ri2 = ri * ri, ri6 = ri2 * ri2 * ri2;
        const double qq = c.qs[i] * c.qs[j];
        const double c6 = c.pard[i].x * c.pard[j].x, c12 = c.pard[i].y * c.pard[j].y;
        const double lj = ri6 * (c12 * ri6 - c6) * (1.0 / 6.0);
        if (GEN && a.taylor_r2 > 0.0) {
            const double ex = V[3 * j] - x0[0], ey = V[3 * j + 1] - x0[1], ez = V[3 * j + 2] - x0[2];
            const double r02 = ex * ex + ey * ey + ez * ez;
            if (r02 >= a.taylor_r2) {
                const double e0 = qq * rsqrt(r02), dd = ex * (p[0] - x0[0]) + ey * (p[1] - x0[1]) + ez * (p[2] - x0[2]);
                return e0 + e0 / r02 * dd + lj;
            }
        }
        return qq * ri + lj;
    };

    // the linearised far field of atom j about the moving atom's current position
    // x0: Coulomb energy e0 + fac (d . displacement), d = x_j - x0; false: near
    auto far_field = [&](const double *x0, int j, double w1, double (&d)[3], double &e0, double &fac) -> bool {
        if (!(a.taylor_r2 > 0.0)) return false;
        for (int k = 0; k < 3; k++) d[k] = V[3 * j + k] - x0[k];
        const double r02 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        if (!(r02 >= a.taylor_r2)) return false;
        Inv64 v;
        if (inv64(d[0], d[1], d[2], v)) {
            e0 = w1 * inv64_r1(v);
            fac = e0 * inv64_r2(v);
        } else {
            e0 = w1 * rsqrt(r02);
            fac = e0 / r02;
        }
        return true;
    };
    // plain terms of one pair at the positions of a mask
    auto plain_rows = [&](int i, const double *x0, int t, unsigned mask, double (&acc)[8]) {
#pragma unroll 1
        for (int q = 0; q < 7; q++) {
            if (!((mask >> q) & 1u)) continue;
            const double e = pair_plain(i, pos[q], x0, t);
#pragma unroll
            for (int k = 0; k < 7; k++)
                if (k == q) acc[k] += e;
        }
    };
    // GEN: the 7 rows of one pair, 9 FP64 differences (the positions share two
    // coordinates of three) and 21 accumulations
    auto general_rows = [&](int i, const double *x0, int t, double w1, double w6, double w12, double (&acc)[8]) {
        const int j = j0 + t;
        double e0, fac, ex[3];
        const bool far = far_field(x0, j, w1, ex, e0, fac);
        double d0[3], dp[3], dm[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const double x = V[3 * j + k];
            d0[k] = x - pos[0][k];
            dp[k] = x - pos[1 + 2 * k][k];
            dm[k] = x - pos[2 + 2 * k][k];
        }
        unsigned out = 0u;
#pragma unroll
        for (int q = 0; q < 7; q++) {
            double d[3] = {d0[0], d0[1], d0[2]};
            const int k = q > 0 ? (q - 1) / 2 : 0;
            if (q > 0) d[k] = q & 1 ? dp[k] : dm[k];
            Inv64 v;
            if (!inv64(d[0], d[1], d[2], v)) {
                out |= 1u << q;
                continue;
            }
            if (far) acc[q] += q > 0 ? e0 + fac * (ex[k] * (pos[q][k] - x0[k])) : e0;
            else acc[q] = fma(w1, inv64_r1(v), acc[q]);
            acc[q] = fma(w6, inv64_r6(v), acc[q]);
            acc[q] = fma(w12, inv64_r12(v), acc[q]);
        }
        if (out) plain_rows(i, x0, t, out, acc);
    };

    for (int m = 0; m < moves; m++) {
        const int pick = (int)__umul64hi(splitmix64(a.seed, base + (uint64_t)m), (uint64_t)cnt);
        const int i = seq ? pick : a.list[l0 + pick];
        const int k0 = c.inc_off[i], k1 = c.inc_off[i + 1];
        if (tid < 21) {  // current position and +-delta along x, y, z
            const int q = tid / 3, k = tid % 3;
            double x = V[3 * i + k];
            if (q == 1 + 2 * k) x = x + a.delta;
            if (q == 2 + 2 * k) x = x - a.delta;
            pos[q][k] = x;
        }
        const double qi = c.qs[i], c6i = c.pard[i].x * (1.0 / 6.0), c12i = c.pard[i].y * (1.0 / 6.0);
        __syncthreads();
        const double x0[3] = {pos[0][0], pos[0][1], pos[0][2]};
        const bool fix = !GEN && in_fix(x0);
        // ---- the 7 rows
        if (w < MV_PAIR_WARPS) {
            double acc[8] = {};
            if (GEN) {
                for (int t = w * 32 + lane; t < nj; t += 32 * MV_PAIR_WARPS) {
                    const int j = j0 + t;
                    if (j == i) continue;
                    general_rows(i, x0, t, qi * (SH ? pq[t] : c.qs[j]), -(c6i * (SH ? p6[t] : c.pard[j].x)),
                                 c12i * (SH ? p12[t] : c.pard[j].y), acc);
                }
            } else if (w * 32 < nj && fix) {
                long long f0[3], fp[3], fm[3];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    fix64(pos[0][k], f0[k]);
                    fix64(pos[1 + 2 * k][k], fp[k]);
                    fix64(pos[2 + 2 * k][k], fm[k]);
                }
                for (int t = w * 32 + lane; t < nj; t += 32 * MV_PAIR_WARPS) {
                    const int j = j0 + t;
                    if (j == i) continue;
                    u64 s0[3], sp[3], sm[3], any = 0;
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        const long long x = F[3 * t + k];
                        s0[k] = abs64(x - f0[k]);
                        sp[k] = abs64(x - fp[k]);
                        sm[k] = abs64(x - fm[k]);
                        any |= s0[k];
                    }
                    if ((unsigned)(any >> 53) - 1u >= 511u) {  // closer than 1/2 A along every axis, or MV_FAR
                        plain_rows(i, x0, t, 127u, acc);
                        continue;
                    }
                    const double w1 = qi * (SH ? pq[t] : c.qs[j]);
                    const double w6 = -(c6i * (SH ? p6[t] : c.pard[j].x)), w12 = c12i * (SH ? p12[t] : c.pard[j].y);
                    const int nz = clz_hi(any) - 2;  // a bit to spare for the offset
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        s0[k] = sqh(s0[k] << nz);
                        sp[k] = sqh(sp[k] << nz);
                        sm[k] = sqh(sm[k] << nz);
                    }
                    const u64 R0 = s0[0] + s0[1] + s0[2];
#pragma unroll
                    for (int q = 0; q < 7; q++) {
                        u64 R = R0;
                        if (q > 0) {
                            const int k = (q - 1) / 2;
                            R = (q & 1 ? sp[k] : sm[k]) + s0[(k + 1) % 3] + s0[(k + 2) % 3];
                        }
                        const int e2 = (clz_hi(R) - 2) & ~1;  // R into [2^60, 2^62)
                        Inv64 v;
                        inv64_back(R << e2, 8 - nz - e2 / 2, v);
                        acc[q] = fma(w1, inv64_r1(v), acc[q]);
                        acc[q] = fma(w6, inv64_r6(v), acc[q]);
                        acc[q] = fma(w12, inv64_r12(v), acc[q]);
                    }
                }
            } else if (!fix) {  // an atom beyond the range moves
                for (int t = w * 32 + lane; t < nj; t += 32 * MV_PAIR_WARPS)
                    if (j0 + t != i) plain_rows(i, x0, t, 127u, acc);
            }
            __syncwarp();
            double s = 0.0;
            if (w * 32 < nj) s = sum8(acc);
            if ((lane & 3) == 0) wsum[w][lane >> 2] = s;
        } else {
            const int type = w - MV_PAIR_WARPS;
            double e = 0.0;
            if (type % CS == rank) {
                if (type == 0) e = bonded_rows<0, 7>(c, tab, V, k0, k1, i, pos, buf[type]);
                else if (type == 1) e = bonded_rows<1, 7>(c, tab, V, k0, k1, i, pos, buf[type]);
                else if (type == 2) e = bonded_rows<2, 7>(c, tab, V, k0, k1, i, pos, buf[type]);
                else e = bonded_rows<3, 7>(c, tab, V, k0, k1, i, pos, buf[type]);
            }
            if (lane < 8) wsum[w][lane] = lane < 7 ? e : 0.0;
        }
        __syncthreads();
        if (w == 0) {  // the block's sums: lane = position + 8 * (warp mod 4), then to every block
            const int q = lane & 7, r0 = lane >> 3;
            double f = (wsum[r0][q] + wsum[r0 + 4][q]) + (wsum[r0 + 8][q] + wsum[r0 + 12][q]);
            f += __shfl_xor_sync(0xffffffffu, f, 8);
            f += __shfl_xor_sync(0xffffffffu, f, 16);
            for (int r = r0; r < CS; r += 4) cl.map_shared_rank(&crow[rank][q], r)[0] = f;
        }
        __syncwarp();
        cl.sync();
        if (w == 0) {  // over the blocks, then the per-axis parabola vertex
            const int q = lane & 7, r0 = lane >> 3;
            double f = r0 < CS ? crow[r0][q] : 0.0;
            if (CS > 4) f += crow[r0 + 4][q];
            if (CS > 1) f += __shfl_xor_sync(0xffffffffu, f, 8);
            if (CS > 2) f += __shfl_xor_sync(0xffffffffu, f, 16);
            const double f0 = __shfl_sync(0xffffffffu, f, 0);
            const int ax = lane < 3 ? lane : 0;
            const double fp = __shfl_sync(0xffffffffu, f, 1 + 2 * ax), fm = __shfl_sync(0xffffffffu, f, 2 + 2 * ax);
            const double curv = fm - 2.0 * f0 + fp;
            const double ts = curv > 0.0 ? a.delta * (fm - fp) / (2.0 * curv) : 0.0;
            if (lane < 3) pos[7][lane] = x0[lane] + ts;
            if (lane < 7) s_f[lane] = f;
        }
        __syncthreads();
        // ---- the vertex row
        const double pv[3] = {pos[7][0], pos[7][1], pos[7][2]};
        double e = 0.0;
        if (w < MV_PAIR_WARPS) {
            if (w * 32 < nj) {
                long long f[3];
                const bool fit = fix && in_fix(pv);
#pragma unroll
                for (int k = 0; k < 3; k++) fix64(pv[k], f[k]);
                for (int t = w * 32 + lane; t < nj; t += 32 * MV_PAIR_WARPS) {
                    const int j = j0 + t;
                    if (j == i) continue;
                    const double w1 = qi * (SH ? pq[t] : c.qs[j]);
                    Inv64 v;
                    u64 ax, ay, az;
                    int nz;
                    if (GEN ? !inv64(V[3 * j] - pv[0], V[3 * j + 1] - pv[1], V[3 * j + 2] - pv[2], v)
                            : (!fit ||
                               !inv64_fix(F[3 * t] - f[0], F[3 * t + 1] - f[1], F[3 * t + 2] - f[2], v, ax, ay, az, nz) ||
                               nz == 0)) {  // nz: MV_FAR
                        e += pair_plain(i, pv, x0, t);
                        continue;
                    }
                    double e0, fac, d[3];
                    if (GEN && far_field(x0, j, w1, d, e0, fac))
                        e += e0 + fac * (d[0] * (pv[0] - x0[0]) + d[1] * (pv[1] - x0[1]) + d[2] * (pv[2] - x0[2]));
                    else
                        e = fma(w1, inv64_r1(v), e);
                    e = fma(-(c6i * (SH ? p6[t] : c.pard[j].x)), inv64_r6(v), e);
                    e = fma(c12i * (SH ? p12[t] : c.pard[j].y), inv64_r12(v), e);
                }
                __syncwarp();
                e = warp_sum(e);
            }
        } else {
            const int type = w - MV_PAIR_WARPS;
            if (type % CS == rank) {
                if (type == 0) e = bonded_rows<0, 1>(c, tab, V, k0, k1, i, &pos[7], buf[type]);
                else if (type == 1) e = bonded_rows<1, 1>(c, tab, V, k0, k1, i, &pos[7], buf[type]);
                else if (type == 2) e = bonded_rows<2, 1>(c, tab, V, k0, k1, i, &pos[7], buf[type]);
                else e = bonded_rows<3, 1>(c, tab, V, k0, k1, i, &pos[7], buf[type]);
            }
        }
        if (lane == 0) wsum[w][0] = e;
        __syncthreads();
        if (w == 0) {
            double f = lane < MV_WARPS ? wsum[lane][0] : 0.0;
#pragma unroll
            for (int o = MV_WARPS / 2; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
            if (lane < CS) cl.map_shared_rank(&cvert[rank], lane)[0] = f;
        }
        __syncwarp();
        cl.sync();
        if (w == 0) {
            double f = lane < CS ? cvert[lane] : 0.0;
            for (int o = CS / 2; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
            f = __shfl_sync(0xffffffffu, f, 0);
            // the best of the 8 points, ties to the earlier one: doubles as
            // ordered integers (a NaN is above everything), the point in
            // the last comparison
            double mine = lane < 7 ? s_f[lane] : f;
            const double f0 = __shfl_sync(0xffffffffu, mine, 0);
            u64 key = bits64(mine + 0.0);
            key = (key >> 63) ? ~key : key | 0x8000000000000000ULL;
            if (mine != mine) key = ~0ULL;
            int best = lane & 7;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                const u64 k2 = __shfl_xor_sync(0xffffffffu, key, o);
                const int b2 = __shfl_xor_sync(0xffffffffu, best, o);
                if (k2 < key || (k2 == key && b2 < best)) { key = k2; best = b2; }
            }
            best = __shfl_sync(0xffffffffu, f0 != f0 ? 0 : best, 0);
            if (lane < 3) {
                const double x = pos[best][lane];
                V[3 * i + lane] = x;
                if (i >= j0 && i < j0 + nj) {
                    long long f;
                    fix64(x, f);
                    F[3 * (i - j0) + lane] = fabs(x) < MV_FIX_MAX ? f : MV_FAR;
                }
            }
        }
        __syncthreads();
    }
    // results: the sequential search writes X (every block its share: all
    // have read X before the first barrier); a part's atoms are merged from
    // a buffer of their own, since blocks of other parts may still have to
    // read X
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
constexpr size_t MV_SMEM = 208 * 1024;  // of 227 KB, beside the static arrays
// dynamic shared memory of the SH form, or 0 when it does not fit
static size_t moves_smem(int n, int cs) {
    const size_t b = sizeof(double) * (3 * (size_t)n + 6 * (size_t)((n + cs - 1) / cs));
    return b <= MV_SMEM ? b : 0;
}
// doubles of private copies that a launch needs in MovesArgs::view
int64_t moves_view_doubles(int n, int parts, int cs) {
    return moves_smem(n, cs) ? 0 : (int64_t)parts * cs * (3 * (int64_t)n + 3 * ((n + cs - 1) / cs));
}

// whether a run takes the GEN rows; x: the positions, on the host.  A pair with
// an atom beyond the range costs the fixed-point rows a plain evaluation, so a
// few such atoms (one that a move has thrown out) are no reason
bool moves_general(const double *x, int n, double delta, double taylor_r2) {
    if (!(delta <= MV_DELTA_MAX) || taylor_r2 > 0.0) return true;
    int far = 0;
    for (int i = 0; i < n; i++) {
        const double *p = x + 3 * (size_t)i;
        far += !(std::fabs(p[0]) < MV_FIX_MAX && std::fabs(p[1]) < MV_FIX_MAX && std::fabs(p[2]) < MV_FIX_MAX);
    }
    return far > n / 256;
}

// Whether a sequential search of n atoms moves by launches over all SMs
// (parab.cu) instead of on one cluster: a move there costs two launches however
// small it is, here the time of eight SMs.  Us a move there, fixed-point rows, GEN
// (offset 0.3 A), and with the far field there and GEN: 7,000 atoms 32, 17, 27, and
// 37, 33; 10,000 36, 22, 35, and 39, 45; 14,000 34, 26, 44, and 38, 56; 30,000 54, 46,
// 86, and 62, 111; 60,000 70, 82, 164, and 85, 214.
bool moves_on_grid(int n, bool gen) { return n > (gen ? 8000 : 40000); }

template <bool SH>
static cudaError_t launch_moves(const Ctx &c, const MovesArgs &a, bool gen, const cudaLaunchConfig_t &cfg) {
    return gen ? cudaLaunchKernelEx(&cfg, k_moves64<SH, true>, c, a) : cudaLaunchKernelEx(&cfg, k_moves64<SH, false>, c, a);
}

cudaError_t launch_moves64(const Ctx &c, const MovesArgs &a, bool gen, int parts, int cs, cudaStream_t s) {
    const size_t smem = moves_smem(a.n, cs);
    cudaError_t e = cudaSuccess;
    if (smem)
        e = cudaFuncSetAttribute(gen ? k_moves64<true, true> : k_moves64<true, false>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MV_SMEM);
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
    return smem ? launch_moves<true>(c, a, gen, cfg) : launch_moves<false>(c, a, gen, cfg);
}

}  // namespace ffm
