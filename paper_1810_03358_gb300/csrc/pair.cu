// Non-bonded pair energy and gradient: the O(N^2) hot loop of the method.
//
// E_cul + E_vdw over all atom pairs (arXiv 1810.03358, Section 2), evaluated
// as a row sweep parallel over the outer sum (Section 3: one inner sum per
// GPU thread).  Every thread owns one i-atom of a 128-atom tile in registers
// and walks a j-chunk staged through shared memory; the pair (i, j) is
// evaluated in row i and again in row j, so no force is ever scattered and
// no atomic touches a force (Newton's third law is not used).
//
// Work items are (i-tile, j-chunk) pairs taken from a device queue (reset with
// its active list before each launch) by a persistent grid; each item writes its
// partial row sums (gx, gy, gz, row energy) to its own slot, and the
// finalize kernel sums the slots of an atom in a fixed order, so results are
// deterministic for a given chunking.  Bonded-term items share the queue.
//
// Per pair (d = x_j - x_i, r^-1 = rsqrt(r^2), q' = q sqrt(C), and the
// per-atom Lennard-Jones factors c6 = a sigma^3, c12 = a sigma^6 with
// a = sqrt(24 eps), so that c6_i c6_j = 24 eps_ij sigma_ij^6 and
// c12_i c12_j = 24 eps_ij sigma_ij^12 under the geometric combining rule):
//   e_cul  = q'_i q'_j r^-1
//   6 e_lj = r^-6 (C12 r^-6 - C6),              C6 = c6_i c6_j, C12 = c12_i c12_j
//   F      = (e_cul + r^-6 (2 C12 r^-6 - C6)) r^-2,   grad_i += F d
// which is C q_i q_j / r + 4 sqrt(eps_i eps_j)((s/r)^12 - (s/r)^6) and its
// derivative.  The row energy sum_j (e_cul + e_lj) counts each pair twice;
// the finalize kernel halves it.  The FP32 kernel flushes denormals (none
// occur for separations above 1e-6 A) and takes r^-1 from the hardware
// reciprocal square root (rsqrt.approx.ftz.f32).
#include <cooperative_groups.h>

#include <cstdio>
#include <type_traits>

#include "activelist.cuh"
#include "bonded.cuh"
#include "ffmin_internal.cuh"
#include "pair64.cuh"

namespace ffm {

namespace cg = cooperative_groups;

__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <typename T> struct VT;
template <> struct VT<float> {
    using V4 = float4;
    using V2 = float2;
    static __device__ __forceinline__ float rsq(float x) { return rsqrt_approx(x); }
};
template <> struct VT<double> {
    using V4 = double4_32a;
    using V2 = double2;
    static __device__ __forceinline__ double rsq(double x) { return rsqrt(x); }
};

// The scaled partners of the thread's i-atoms (exclusion variant; sorted by
// index), walked along a j tile 32 atoms at a time: one bit each, and the
// scale of the partner at bit k from the number of bits below it.  A pair
// without a bit has scale 1.  (A lookup of every pair in the atom's list made
// a masked tile cost 10 plain ones; looking up only the pairs with a bit, still
// a chain of dependent loads in nearly every step near the diagonal, kept it
// at 900 cycles a step: 1,000 atoms E + grad 72 -> 45 us, 5,000 86 -> 61.)
template <int IPT>
struct XCursor {
    const Ctx *c;
    int cur[IPT], end[IPT], base[IPT];
    unsigned m[IPT];
    __device__ __forceinline__ void begin(const Ctx *cx, const int *ig, int jt) {  // ig: -1 for padding
        c = cx;
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            cur[u] = end[u] = 0;
            if (ig[u] < 0) continue;
            cur[u] = c->xs_off[ig[u]];
            end[u] = c->xs_off[ig[u] + 1];
            while (cur[u] < end[u] && c->xs_part[cur[u]] < jt) cur[u]++;
        }
    }
    __device__ __forceinline__ void window(int j0) {
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            m[u] = 0u;
            base[u] = cur[u];
            for (; cur[u] < end[u]; cur[u]++) {
                const int d = c->xs_part[cur[u]] - j0;
                if (d >= 32) break;
                m[u] |= 1u << d;
            }
        }
    }
    __device__ __forceinline__ float scale(int u, int k) const {
        return (m[u] >> k) & 1u ? c->xs_val[base[u] + __popc(m[u] & ((1u << k) - 1u))] : 1.f;
    }
};

// IPT i-atoms per thread share every j load from shared memory.  DM: 0 an
// off-diagonal tile; 1 the i-tile itself (j == i skipped); 2 the i-tile
// itself on the symmetric list (only j > i: each pair once).  MASK: the j
// tile holds scaled partners of the i tile (exclusion variant, FP32): every
// pair is multiplied by its scale s_ij inside the sums (ig: the i atoms'
// global indices, -1 for padding; jt: the j tile's first atom).
template <typename T, int IPT, bool GRAD, int DM, bool MASK = false>
__device__ __forceinline__ void sweep(const typename VT<T>::V4 *__restrict__ sp,
                                      const typename VT<T>::V2 *__restrict__ sq,
                                      const typename VT<T>::V4 (&pi)[IPT],
                                      const typename VT<T>::V2 (&ci)[IPT], const int (&dk)[IPT],
                                      T (&gx)[IPT], T (&gy)[IPT], T (&gz)[IPT], T (&ec)[IPT],
                                      T (&lj)[IPT], const Ctx *cx = nullptr, const int *ig = nullptr,
                                      int jt = 0) {
    // the masked form runs on a few tiles only: kept rolled (smaller kernel)
    constexpr int KW = MASK ? 32 : TJ;
    XCursor<MASK ? IPT : 1> xs;
    if constexpr (MASK) xs.begin(cx, ig, jt);
    for (int kw = 0; kw < TJ; kw += KW) {
    if constexpr (MASK) xs.window(jt + kw);
#pragma unroll(MASK ? 1 : 8)
    for (int kk = 0; kk < KW; kk++) {
        const int k = kw + kk;
        const typename VT<T>::V4 pj = sp[k];
        const typename VT<T>::V2 qj = sq[k];
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const T dx = pj.x - pi[u].x, dy = pj.y - pi[u].y, dz = pj.z - pi[u].z;
            const T r2 = dx * dx + dy * dy + dz * dz;
            T ri = VT<T>::rsq(r2);
            if (DM == 1) ri = (k == dk[u]) ? T(0) : ri;
            if (DM == 2) ri = (k <= dk[u]) ? T(0) : ri;
            T sc = T(1);
            if constexpr (MASK) sc = (T)xs.scale(u, kk);
            const T ri2 = ri * ri;
            const T e = MASK ? pi[u].w * pj.w * sc * ri : pi[u].w * pj.w * ri;
            const T ri6 = ri2 * ri2 * ri2;
            const T c6 = MASK ? ci[u].x * qj.x * sc : ci[u].x * qj.x;
            const T c12 = MASK ? ci[u].y * qj.y * sc : ci[u].y * qj.y;
            const T t1 = c12 * ri6 - c6;
            ec[u] += e;
            lj[u] += ri6 * t1;
            if (GRAD) {
                const T t2 = c12 * ri6 + t1;
                const T f = (ri6 * t2 + e) * ri2;
                gx[u] += f * dx;
                gy[u] += f * dy;
                gz[u] += f * dz;
            }
        }
    }
    }
}

// FP32 line-search trial as an energy difference from the base point: with
// d = x_j - x_i at the base and dd = the difference of the two atoms'
// displacements, r'^2 - r^2 = dd.(2 d + dd) is formed without cancellation,
// and so are
//   r'^-2 - r^-2 = -(r'^2 - r^2) r^-2 r'^-2,
//   r'^-1 - r^-1 = (r'^-2 - r^-2) / (r^-1 + r'^-1),
//   r'^-6 - r^-6 = (r'^-2 - r^-2)(r'^-4 + r'^-2 r^-2 + r^-4),
//   r'^-12 - r^-12 = (r'^-6 - r^-6)(r'^-6 + r^-6);
// the row then accumulates the exact-difference form of
// e_cul + 6 e_lj, whose rounding error is relative to the difference, not to
// the energies (FP32 coordinates of the trial point would add noise of order
// u |x| |F| per pair, larger than the line search's energy decrements).
template <int IPT, int DM, bool MASK = false>
__device__ __forceinline__ void sweep_delta(const float4 *__restrict__ sp, const float2 *__restrict__ sq,
                                            const float4 *__restrict__ sd, const float4 (&pi)[IPT],
                                            const float2 (&ci)[IPT], const float4 (&di)[IPT],
                                            const int (&dk)[IPT], float (&ec)[IPT], float (&lj)[IPT],
                                            const Ctx *cx = nullptr, const int *ig = nullptr, int jt = 0) {
    constexpr int KW = MASK ? 32 : TJ;
    XCursor<MASK ? IPT : 1> xs;
    if constexpr (MASK) xs.begin(cx, ig, jt);
    for (int kw = 0; kw < TJ; kw += KW) {
    if constexpr (MASK) xs.window(jt + kw);
#pragma unroll(MASK ? 1 : 4)
    for (int kk = 0; kk < KW; kk++) {
        const int k = kw + kk;
        const float4 pj = sp[k];
        const float2 qj = sq[k];
        const float4 dj = sd[k];
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const float dx = pj.x - pi[u].x, dy = pj.y - pi[u].y, dz = pj.z - pi[u].z;
            const float ex = dj.x - di[u].x, ey = dj.y - di[u].y, ez = dj.z - di[u].z;
            float r2 = dx * dx + dy * dy + dz * dz;
            if (DM != 0) r2 = (k == dk[u]) ? 1.f : r2;  // j == i: dd = 0, every difference vanishes
            float D = ex * (2.f * dx + ex) + ey * (2.f * dy + ey) + ez * (2.f * dz + ez);
            if (DM == 2) D = (k <= dk[u]) ? 0.f : D;  // each pair once: j < i contributes nothing
            const float ri = rsqrt_approx(r2), rp = rsqrt_approx(r2 + D);
            const float ri2 = ri * ri, rp2 = rp * rp;
            const float X = -D * ri2 * rp2;
            float inv;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(ri + rp));
            const float d1 = X * inv;
            const float ri4 = ri2 * ri2, rp4 = rp2 * rp2;
            const float d6 = X * (rp4 + rp2 * ri2 + ri4);
            const float d12 = d6 * (rp4 * rp2 + ri4 * ri2);
            float sc = 1.f;
            if constexpr (MASK) sc = xs.scale(u, kk);
            const float c6 = MASK ? ci[u].x * qj.x * sc : ci[u].x * qj.x;
            const float c12 = MASK ? ci[u].y * qj.y * sc : ci[u].y * qj.y;
            ec[u] += MASK ? pi[u].w * pj.w * sc * d1 : pi[u].w * pj.w * d1;
            lj[u] += c12 * d12 - c6 * d6;
        }
    }
    }
}

// Energy-only forms with the i atom's factors outside the sums: per i the
// sums of q'_j X1, c6_j X6 and c12_j X12 (X = r^-1, r^-6, r^-12 for a plain
// energy; the exact differences r'^-1 - r^-1, ... for a difference trial),
// combined with q'_i, c6_i, c12_i once per item.  fa, f6, f12 accumulate
// across the item's j tiles.
template <int IPT, int DM>
__device__ __forceinline__ void sweep_e_factored(const float4 *__restrict__ sp, const float2 *__restrict__ sq,
                                                 const float4 (&pi)[IPT], const int (&dk)[IPT], float (&fa)[IPT],
                                                 float (&f6)[IPT], float (&f12)[IPT]) {
#pragma unroll 8
    for (int k = 0; k < TJ; k++) {
        const float4 pj = sp[k];
        const float2 qj = sq[k];
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const float dx = pj.x - pi[u].x, dy = pj.y - pi[u].y, dz = pj.z - pi[u].z;
            const float r2 = dx * dx + dy * dy + dz * dz;
            float ri = rsqrt_approx(r2);
            if (DM == 1) ri = (k == dk[u]) ? 0.f : ri;
            if (DM == 2) ri = (k <= dk[u]) ? 0.f : ri;
            const float ri2 = ri * ri;
            const float ri6 = ri2 * ri2 * ri2;
            fa[u] = fmaf(pj.w, ri, fa[u]);
            f6[u] = fmaf(qj.x, ri6, f6[u]);
            f12[u] = fmaf(qj.y, ri6 * ri6, f12[u]);
        }
    }
}

template <int IPT, int DM>
__device__ __forceinline__ void sweep_delta_factored(const float4 *__restrict__ sp, const float2 *__restrict__ sq,
                                                     const float4 *__restrict__ sd, const float4 (&pi)[IPT],
                                                     const float4 (&di)[IPT], const int (&dk)[IPT],
                                                     float (&fa)[IPT], float (&f6)[IPT], float (&f12)[IPT]) {
#pragma unroll 4
    for (int k = 0; k < TJ; k++) {
        const float4 pj = sp[k];
        const float2 qj = sq[k];
        const float4 dj = sd[k];
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const float dx = pj.x - pi[u].x, dy = pj.y - pi[u].y, dz = pj.z - pi[u].z;
            const float ex = dj.x - di[u].x, ey = dj.y - di[u].y, ez = dj.z - di[u].z;
            float r2 = dx * dx + dy * dy + dz * dz;
            if (DM != 0) r2 = (k == dk[u]) ? 1.f : r2;  // j == i: dd = 0, every difference vanishes
            float D = ex * (2.f * dx + ex) + ey * (2.f * dy + ey) + ez * (2.f * dz + ez);
            if (DM == 2) D = (k <= dk[u]) ? 0.f : D;  // each pair once: j < i contributes nothing
            const float ri = rsqrt_approx(r2), rp = rsqrt_approx(r2 + D);
            const float ri2 = ri * ri, rp2 = rp * rp;
            const float X = -D * ri2 * rp2;
            float inv;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(ri + rp));
            const float d1 = X * inv;
            const float ri4 = ri2 * ri2, rp4 = rp2 * rp2;
            const float d6 = X * (rp4 + rp2 * ri2 + ri4);
            const float d12 = d6 * (rp4 * rp2 + ri4 * ri2);
            fa[u] = fmaf(pj.w, d1, fa[u]);
            f6[u] = fmaf(qj.x, d6, f6[u]);
            f12[u] = fmaf(qj.y, d12, f12[u]);
        }
    }
}

// Packed forms of the unmasked FP32 sweeps for two i-atoms per thread (i-atom
// u in lane u of every packed register): fma.rn.f32x2 and its kin take one
// issue slot for two lanes of the FMA pipe, which takes issue (25 scalar
// instructions a pair with forces, 39 for a difference trial) off the list of
// bounds.  What bounds them now is the register file: an fma2 of three
// different registers takes 3 cycles of a partition and not 2 (measured in
// isolation), 51 cycles for the two pairs of a step with forces where the FMA
// pipe alone would take 44.  30,000 atoms: E + grad 0.737 -> 0.682 ms, difference
// trial 0.568 -> 0.506 ms, energy 0.237 -> 0.227 ms.  Every lane performs the
// operations of the scalar sweep in its order with its roundings, fused
// multiply-adds included: a minimization amplifies any other rounding of
// these sums (1e-7 in a gradient is 1e-3 A ten steps later), so both forms
// give the same bits.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// a j-atom staged with both lanes equal, so that a packed operand is what a
// 128-bit load returns: building the pairs by moves puts scalar instructions
// between the packed ones, which stalls the FMA pipe (78 % busy instead of
// the 90s, measured)
struct J2 {
    ulonglong2 xy, zq, c;  // (x x, y y), (z z, q' q'), (c6 c6, c12 c12)
};

// r^-1 of a packed r^2; DM as in sweep()
template <int DM>
__device__ __forceinline__ f2 rsqrt2(f2 r2, int k, const int (&dk)[2]) {
    float a, b;
    upk(r2, a, b);
    a = rsqrt_approx(a);
    b = rsqrt_approx(b);
    if (DM == 1) { a = k == dk[0] ? 0.f : a; b = k == dk[1] ? 0.f : b; }
    if (DM == 2) { a = k <= dk[0] ? 0.f : a; b = k <= dk[1] ? 0.f : b; }
    return pk(a, b);
}

// the i-atoms of a thread: negated coordinates, (q', -c6, c12)
struct IPair {
    f2 nx, ny, nz, q, nc6, c12;
};

template <int DM>
__device__ __forceinline__ void sweep2(const J2 *__restrict__ sj, const IPair &A, const int (&dk)[2],
                                       f2 &gx, f2 &gy, f2 &gz, f2 &ec, f2 &lj) {
#pragma unroll 8
    for (int k = 0; k < TJ; k++) {
        const ulonglong2 xy = sj[k].xy, zq = sj[k].zq, cj = sj[k].c;
        const f2 dx = add2(xy.x, A.nx), dy = add2(xy.y, A.ny), dz = add2(zq.x, A.nz);
        const f2 r2 = fma2(dz, dz, fma2(dx, dx, mul2(dy, dy)));
        const f2 ri = rsqrt2<DM>(r2, k, dk);
        const f2 ri2 = mul2(ri, ri);
        const f2 qq = mul2(A.q, zq.y);
        const f2 ri6 = mul2(mul2(ri2, ri2), ri2);
        const f2 p12 = mul2(mul2(A.c12, cj.y), ri6);
        const f2 t1 = fma2(A.nc6, cj.x, p12);
        ec = fma2(qq, ri, ec);
        lj = fma2(ri6, t1, lj);
        const f2 f = mul2(fma2(qq, ri, mul2(ri6, add2(p12, t1))), ri2);
        gx = fma2(f, dx, gx);
        gy = fma2(f, dy, gy);
        gz = fma2(f, dz, gz);
    }
}

template <int DM>
__device__ __forceinline__ void sweep2_e(const J2 *__restrict__ sj, const IPair &A, const int (&dk)[2], f2 &fa, f2 &f6, f2 &f12) {
#pragma unroll 8
    for (int k = 0; k < TJ; k++) {
        const ulonglong2 xy = sj[k].xy, zq = sj[k].zq, cj = sj[k].c;
        const f2 dx = add2(xy.x, A.nx), dy = add2(xy.y, A.ny), dz = add2(zq.x, A.nz);
        const f2 r2 = fma2(dz, dz, fma2(dx, dx, mul2(dy, dy)));
        const f2 ri = rsqrt2<DM>(r2, k, dk);
        const f2 ri2 = mul2(ri, ri);
        const f2 ri6 = mul2(mul2(ri2, ri2), ri2);
        fa = fma2(zq.y, ri, fa);
        f6 = fma2(cj.x, ri6, f6);
        f12 = fma2(cj.y, mul2(ri6, ri6), f12);
    }
}

// the i-atoms' displacements are negated like their coordinates.  The scalar
// form negates D before it multiplies; here the last sums change sign instead
// (exact), so fa, f6, f12 hold the opposite of its sums
template <int DM>
__device__ __forceinline__ void sweep2_delta(const J2 *__restrict__ sj, const ulonglong2 *__restrict__ sexy,
                                             const f2 *__restrict__ sez, const IPair &A, f2 nex, f2 ney, f2 nez,
                                             const int (&dk)[2], f2 &fa, f2 &f6, f2 &f12) {
    const f2 two = pk(2.f, 2.f);
#pragma unroll 4
    for (int k = 0; k < TJ; k++) {
        const ulonglong2 xy = sj[k].xy, zq = sj[k].zq, cj = sj[k].c;
        const ulonglong2 exy = sexy[k];
        const f2 dx = add2(xy.x, A.nx), dy = add2(xy.y, A.ny), dz = add2(zq.x, A.nz);
        const f2 ex = add2(exy.x, nex), ey = add2(exy.y, ney), ez = add2(sez[k], nez);
        f2 r2 = fma2(dz, dz, fma2(dx, dx, mul2(dy, dy)));
        f2 D = fma2(ez, fma2(two, dz, ez), fma2(ex, fma2(two, dx, ex), mul2(ey, fma2(two, dy, ey))));
        float a, b, u, v;
        upk(r2, a, b);
        if (DM != 0) {  // j == i: r = 1 and no displacement, every difference vanishes
            a = k == dk[0] ? 1.f : a;
            b = k == dk[1] ? 1.f : b;
            r2 = pk(a, b);
        }
        if (DM == 2) {  // each pair once: j < i contributes nothing
            upk(D, u, v);
            u = k <= dk[0] ? 0.f : u;
            v = k <= dk[1] ? 0.f : v;
            D = pk(u, v);
        }
        upk(add2(r2, D), u, v);
        const f2 ri = pk(rsqrt_approx(a), rsqrt_approx(b)), rp = pk(rsqrt_approx(u), rsqrt_approx(v));
        upk(add2(ri, rp), a, b);
        const f2 inv = pk(rcp_approx(a), rcp_approx(b));
        const f2 ri2 = mul2(ri, ri), rp2 = mul2(rp, rp);
        const f2 X = mul2(mul2(D, ri2), rp2);
        const f2 ri4 = mul2(ri2, ri2), rp4 = mul2(rp2, rp2);
        const f2 d6 = mul2(X, add2(fma2(rp2, ri2, rp4), ri4));
        const f2 d12 = mul2(d6, fma2(ri4, ri2, mul2(rp4, rp2)));
        fa = fma2(zq.y, mul2(X, inv), fa);
        f6 = fma2(cj.x, d6, f6);
        f12 = fma2(cj.y, d12, f12);
    }
}

// Item of position q of a work queue (the active systems' items in order), -1
// past its end
template <int LIST>
__device__ __forceinline__ int queue_item(const Ctx &c, const int2 *items, int q) {
    const int32_t *A = c.act + LIST * (2 * c.n_sys + 2);
    const int n_act = A[0], total = A[1];
    if (q >= total) return -1;
    if (c.n_sys == 1) return q;
    const int32_t *aoff = A + 2, *asys = A + 2 + c.n_sys;
    int lo = 0, hi = n_act - 1;  // last active system whose first item is <= q
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (aoff[mid] <= q) lo = mid;
        else hi = mid - 1;
    }
    return items[asys[lo]].x + (q - aoff[lo]);
}
// The next item of a block.  Its first position in the queue is its index and
// is found by every thread; the following ones come from the counter, and a
// block whose grid covers the queue takes none.  (Every position through one
// thread and the counter was a chain of nine loads: E + grad kernel with its
// list kernel at 3,334 atoms FP64 165 -> 160 us, energies 77 -> 73 us; MIXED trials of
// 10,000 atoms 82 -> 76 us, of 5,000 with exclusions 54 -> 48 us.)
template <int LIST>
__device__ __forceinline__ int next_item(const Ctx &c, const int2 *items, unsigned *counter, bool first, int &s_item) {
    if (first) return queue_item<LIST>(c, items, blockIdx.x);
    if (threadIdx.x == 0)
        s_item = c.act[LIST * (2 * c.n_sys + 2) + 1] <= (int)gridDim.x
                     ? -1
                     : queue_item<LIST>(c, items, gridDim.x + (int)atomicAdd(counter, 1u));
    __syncthreads();
    const int it = s_item;
    __syncthreads();
    return it;
}

// NT threads per block, IPT i-atoms per thread, NT * IPT == TI (one tile).
// FP32 shapes: two i-atoms per thread (64-thread blocks: every j load from
// shared memory serves two pairs) or one (128-thread blocks: twice the warps
// per work item, which pays when an object has few items); the autotuner
// picks one per object.  Register caps: the FP32 E + grad kernel is compiled
// for 832 threads per SM (13 blocks of 64, whose 72 registers let 14 be
// resident, or 6 of 128 with 80; it spills 148 bytes), the FP32
// energy kernel for 512 (128 registers: a difference trial keeps more values).  At
// 30,000 atoms with 512, 640, 768, 832 threads: E + grad 744, 711, 682, 667
// us (896 is the same kernel in blocks of 64); with 512, 640, 768, 896 difference
// trials 500, 532, 531, 537 us and plain energies 231, 223, 228, 232 us;
// a minimization takes difference trials.  At 3,334 they are within 2 %, but
// trials with 768 are 10 % slower.  With exclusions E + grad runs 640 (1,000
// atoms 3 % faster than with 768, 20,000 the same).  The FP64 kernel runs 8 blocks of 128 (64
// registers); the rarely-run bonded items may spill.  FFMIN_F32_EG_THREADS,
// _XS_THREADS and _E_THREADS override the FP32 caps (registers per thread follow:
// 65536 / threads).
#ifndef FFMIN_F32_EG_THREADS
#define FFMIN_F32_EG_THREADS 832
#endif
#ifndef FFMIN_F32_XS_THREADS
#define FFMIN_F32_XS_THREADS 640
#endif
#ifndef FFMIN_F32_E_THREADS
#define FFMIN_F32_E_THREADS 512
#endif
constexpr int f32_blocks(bool xs, bool eonly, int nt) {
    return (eonly ? FFMIN_F32_E_THREADS : (xs ? FFMIN_F32_XS_THREADS : FFMIN_F32_EG_THREADS)) / nt;
}
// XS: the object carries the exclusion variant (FP32 sweeps scale the listed
// pairs); a separate instantiation keeps the masked code out of the kernel
// every other object runs
// EONLY (FP32): the energy-only kernel (plain energies and difference
// trials, on the symmetric list) with its own work queue; the other FP32
// instantiation runs the E + grad row sweep only.  The FP64 row sweep (the
// fallback of batches too large for the symmetric list) takes both kinds.
template <typename T, int NT, int IPT, bool XS = false, bool EONLY = false>
__global__ void __launch_bounds__(NT, (sizeof(T) == 4 ? f32_blocks(XS, EONLY, NT) : 8)) k_pair(Ctx c);
template <typename T, int NT, int IPT, bool XS, bool EONLY>
__global__ void __launch_bounds__(NT, (sizeof(T) == 4 ? f32_blocks(XS, EONLY, NT) : 8)) k_pair(Ctx c) {
    static_assert(NT * IPT == TI, "a block covers one i-tile");
    using V4 = typename VT<T>::V4;
    using V2 = typename VT<T>::V2;
    constexpr bool PACKED = sizeof(T) == 4 && IPT == 2;  // unmasked tiles
    constexpr bool SCALAR = !PACKED || XS;               // masked tiles and the other shapes
    __shared__ V4 sp[SCALAR ? TJ : 1];
    __shared__ V2 sq[SCALAR ? TJ : 1];
    __shared__ float4 sd[SCALAR && EONLY ? TJ : 1];  // displacements (FP32 difference trials)
    __shared__ J2 sj[PACKED ? TJ : 1];
    __shared__ ulonglong2 sexy[PACKED && EONLY ? TJ : 1];
    __shared__ f2 sez[PACKED && EONLY ? TJ : 1];
    __shared__ int s_item;
    const V4 *__restrict__ pos;
    const V2 *__restrict__ par;
    V4 *__restrict__ out;
    if constexpr (sizeof(T) == 4) {
        pos = c.posf; par = c.parf; out = c.gpf;
    } else {
        pos = c.posd; par = c.pard; out = c.gpd;
    }
    constexpr int MODE = sizeof(T) == 4 ? 0 : 1;
    constexpr int LIST = MODE == 1 ? LIST_F64 : (EONLY ? LIST_F32_E : LIST_F32_EG);
    constexpr int CNT = MODE == 1 ? CNT_PAIR64 : (EONLY ? CNT_PAIR32E : CNT_PAIR);
    // the queue runs over the items of the systems evaluating in this
    // precision and kind only (active list rebuilt before every launch).
    // FP32 energy-only evaluations (plain or difference trials) run on the
    // symmetric list: each pair once, no forces
    const bool sym = MODE == 0 && EONLY && c.sym32;
    const int tid = threadIdx.x;
    for (bool first = true;; first = false) {
        const int it = next_item<LIST>(c, sym ? c.sys_items32 : c.sys_items, &c.counters[CNT], first, s_item);
        if (it < 0) break;
        const Item I = (sym ? c.items32 : c.items)[it];
        if (I.tile < 0) {  // bonded terms (FP64), overlapping the pair items of other warps
            bonded_item(c, I.j0, I.nj, MODE, tid, NT);
            continue;
        }
        const Tile tl = c.tiles[I.tile];
        const SysState &S = c.st[I.sys];
        const int kind = S.ev_kind;
        const bool delta = MODE == 0 && S.ev_delta;
        if (kind == EV_NONE || S.mode != MODE) continue;
        if (MODE == 0 && (kind == EV_E) != EONLY) continue;  // the other FP32 queue's system
        V4 pi[IPT];
        V2 ci[IPT];
        int ig[IPT];
        T gx[IPT], gy[IPT], gz[IPT], ec[IPT], lj[IPT];
        f2 p0 = 0, p1 = 0, p2 = 0, p3 = 0, p4 = 0;  // packed sums
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            const int li = tid + u * NT;
            ig[u] = tl.a0 + li;
            if (li < tl.na) {
                pi[u] = pos[ig[u]];
                ci[u] = par[ig[u]];
            } else {  // padding atom far away with no charge and no LJ
                pi[u].x = T(-1e6); pi[u].y = T(-1e6); pi[u].z = T(-1e6); pi[u].w = T(0);
                ci[u].x = T(0); ci[u].y = T(0);
            }
            gx[u] = gy[u] = gz[u] = ec[u] = lj[u] = T(0);
        }
        float4 di[IPT];
        if constexpr (MODE == 0) {
#pragma unroll
            for (int u = 0; u < IPT; u++)
                di[u] = (delta && tid + u * NT < tl.na) ? c.dispf[ig[u]] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        IPair A{};
        f2 nex = 0, ney = 0, nez = 0;
        if constexpr (PACKED) {
            A.nx = pk(-pi[0].x, -pi[1].x); A.ny = pk(-pi[0].y, -pi[1].y); A.nz = pk(-pi[0].z, -pi[1].z);
            A.q = pk(pi[0].w, pi[1].w);
            A.nc6 = pk(-ci[0].x, -ci[1].x);
            A.c12 = pk(ci[0].y, ci[1].y);
            nex = pk(-di[0].x, -di[1].x); ney = pk(-di[0].y, -di[1].y); nez = pk(-di[0].z, -di[1].z);
        }
        const int jend = I.j0 + I.nj;
        for (int jt = I.j0; jt < jend; jt += TJ) {
#pragma unroll
            for (int q = tid; q < TJ; q += NT) {
                const int jl = jt + q;
                V4 pj;
                V2 cj;
                if (jl < jend) {
                    pj = pos[jl];
                    cj = par[jl];
                } else {
                    pj.x = pj.y = pj.z = T(1e6); pj.w = T(0);
                    cj.x = cj.y = T(0);
                }
                if constexpr (SCALAR) { sp[q] = pj; sq[q] = cj; }
                if constexpr (PACKED) {
                    sj[q].xy = make_ulonglong2(pk(pj.x, pj.x), pk(pj.y, pj.y));
                    sj[q].zq = make_ulonglong2(pk(pj.z, pj.z), pk(pj.w, pj.w));
                    sj[q].c = make_ulonglong2(pk(cj.x, cj.x), pk(cj.y, cj.y));
                }
                if constexpr (MODE == 0 && EONLY) {
                    if (delta) {
                        const float4 d = jl < jend ? c.dispf[jl] : make_float4(0.f, 0.f, 0.f, 0.f);
                        if constexpr (SCALAR) sd[q] = d;
                        if constexpr (PACKED) {
                            sexy[q] = make_ulonglong2(pk(d.x, d.x), pk(d.y, d.y));
                            sez[q] = pk(d.z, d.z);
                        }
                    }
                }
            }
            __syncthreads();
            // the i tile lies inside this j tile when jt == a0 (tiles and
            // chunks are aligned to TJ == TI inside a system)
            const bool diag = I.diag && jt == tl.a0;
            int dk[IPT];
#pragma unroll
            for (int u = 0; u < IPT; u++) dk[u] = ig[u] - jt;
            if constexpr (MODE == 0) {
                // exclusion variant: this j tile holds scaled partners of
                // the i tile (near the diagonal of a chain); -1 marks padding
                const bool masked = XS && tl.xlo <= tl.xhi && tl.xhi >= jt && tl.xlo < jt + TJ;
                int igm[IPT];
#pragma unroll
                for (int u = 0; u < IPT; u++) igm[u] = tid + u * NT < tl.na ? ig[u] : -1;
                if constexpr (EONLY) {  // energy only: plain or difference trial
                    if (XS && masked) {
                        if (delta) {
                            if (diag && sym) sweep_delta<IPT, 2, true>(sp, sq, sd, pi, ci, di, dk, ec, lj, &c, igm, jt);
                            else if (diag) sweep_delta<IPT, 1, true>(sp, sq, sd, pi, ci, di, dk, ec, lj, &c, igm, jt);
                            else sweep_delta<IPT, 0, true>(sp, sq, sd, pi, ci, di, dk, ec, lj, &c, igm, jt);
                        } else {
                            if (diag && sym) sweep<T, IPT, false, 2, true>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj, &c, igm, jt);
                            else if (diag) sweep<T, IPT, false, 1, true>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj, &c, igm, jt);
                            else sweep<T, IPT, false, 0, true>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj, &c, igm, jt);
                        }
                    } else if constexpr (PACKED) {
                        if (delta) {
                            if (diag && sym) sweep2_delta<2>(sj, sexy, sez, A, nex, ney, nez, dk, p0, p1, p2);
                            else if (diag) sweep2_delta<1>(sj, sexy, sez, A, nex, ney, nez, dk, p0, p1, p2);
                            else sweep2_delta<0>(sj, sexy, sez, A, nex, ney, nez, dk, p0, p1, p2);
                        } else {
                            if (diag && sym) sweep2_e<2>(sj, A, dk, p0, p1, p2);
                            else if (diag) sweep2_e<1>(sj, A, dk, p0, p1, p2);
                            else sweep2_e<0>(sj, A, dk, p0, p1, p2);
                        }
                    } else if (delta) {  // factored sums in the (idle) gradient registers
                        if (diag && sym) sweep_delta_factored<IPT, 2>(sp, sq, sd, pi, di, dk, gx, gy, gz);
                        else if (diag) sweep_delta_factored<IPT, 1>(sp, sq, sd, pi, di, dk, gx, gy, gz);
                        else sweep_delta_factored<IPT, 0>(sp, sq, sd, pi, di, dk, gx, gy, gz);
                    } else {
                        if (diag && sym) sweep_e_factored<IPT, 2>(sp, sq, pi, dk, gx, gy, gz);
                        else if (diag) sweep_e_factored<IPT, 1>(sp, sq, pi, dk, gx, gy, gz);
                        else sweep_e_factored<IPT, 0>(sp, sq, pi, dk, gx, gy, gz);
                    }
                } else {  // E + grad row sweep
                    if (XS && masked) {
                        if (diag) sweep<T, IPT, true, 1, true>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj, &c, igm, jt);
                        else sweep<T, IPT, true, 0, true>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj, &c, igm, jt);
                    } else if constexpr (PACKED) {
                        // masked tiles add to the scalar sums in between: both
                        // forms continue the same running sums
                        p0 = pk(gx[0], gx[1]); p1 = pk(gy[0], gy[1]); p2 = pk(gz[0], gz[1]);
                        p3 = pk(ec[0], ec[1]); p4 = pk(lj[0], lj[1]);
                        if (diag) sweep2<1>(sj, A, dk, p0, p1, p2, p3, p4);
                        else sweep2<0>(sj, A, dk, p0, p1, p2, p3, p4);
                        upk(p0, gx[0], gx[1]); upk(p1, gy[0], gy[1]); upk(p2, gz[0], gz[1]);
                        upk(p3, ec[0], ec[1]); upk(p4, lj[0], lj[1]);
                    } else {
                        if (diag) sweep<T, IPT, true, 1>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj);
                        else sweep<T, IPT, true, 0>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj);
                    }
                }
            } else if (kind == EV_EG) {  // FP64 row sweep (fallback of very large batches)
                if (diag) sweep<T, IPT, true, 1>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj);
                else sweep<T, IPT, true, 0>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj);
            } else {
                if (diag) sweep<T, IPT, false, 1>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj);
                else sweep<T, IPT, false, 0>(sp, sq, pi, ci, dk, gx, gy, gz, ec, lj);
            }
            __syncthreads();
        }
        V4 *dst = out + (int64_t)it * TI;
        // FP32 energy only: masked tiles summed the pair terms into ec / lj,
        // the others the factored sums into gx, gy, gz
        constexpr bool factored = MODE == 0 && EONLY;
        if constexpr (factored && PACKED) {
            const f2 sg = delta ? pk(-1.f, -1.f) : pk(1.f, 1.f);
            upk(mul2(p0, sg), gx[0], gx[1]); upk(mul2(p1, sg), gy[0], gy[1]); upk(mul2(p2, sg), gz[0], gz[1]);
        }
#pragma unroll
        for (int u = 0; u < IPT; u++) {
            V4 o;
            if (factored) {
                o.x = T(0); o.y = T(0); o.z = T(0);
                o.w = ec[u] + lj[u] * T(1.0 / 6.0) + pi[u].w * gx[u] +
                      (ci[u].y * gz[u] - ci[u].x * gy[u]) * T(1.0 / 6.0);
            } else {
                o.x = gx[u]; o.y = gy[u]; o.z = gz[u];
                o.w = ec[u] + lj[u] * T(1.0 / 6.0);
            }
            // symmetric list (FP32 energy only): energies alone
            if (MODE == 0 && EONLY && sym) c.gpf_sym[(int64_t)I.slot * TI + tid + u * NT] = (float)o.w;
            else dst[tid + u * NT] = o;
        }
    }
}

// Symmetric FP64 pair kernel: every unordered pair once.  An item (i-tile I,
// chunk of j-tiles at or right of I, or a part of one j-tile) evaluates each
// pair (i, j) once, adds the force to i's registers and its opposite to j's
// entry of a warp-private shared-memory array (lanes of a warp take distinct
// j at every step: thread t pairs with j = (t + k) mod W at step k, W the
// j-atoms of the part).  The diagonal tile runs k = 1 .. TJ/2 and, at
// k = TJ/2, only its first half of the threads, so every pair of the tile
// appears once; in parts it takes the pairs with j > i.  No atomics: after
// each j-tile the four warps' arrays are summed in warp order into the
// tile's j-side partial row, and the i-side row is written once per item; the
// finalize kernel sums an atom's rows in a fixed order.  Row energies count
// each pair once.
//
// Bound: the FP64 pipe at 2 operations per SM and clock, and issue.  Differences
// (in fixed point, when the tile pair's coordinates fit), terms and their sums
// are formed on the integer pipes (pair64.cuh), which leaves 7 FP64
// instructions of 31 a pair with forces and 3 of 18.5 for an energy.  30,000
// atoms, E + grad / E: 24.46 / 14.83 ms in plain FP64, 12.53 / 5.06 ms with FP64
// differences, 10.14 / 3.98 ms with the sum of a pair's terms in FP64 (12
// instructions, pipe 88 % busy), 8.66 / 3.98 ms now.  Blocks per SM: 5 (4: 4 % and
// 7 % slower, 6: 3 % and 1 % faster at 30,000 atoms, 1 % and 2 % slower at 3,334).
constexpr int NT_SYM = 128;
#ifndef FFMIN_SYM_MINBLOCKS
#define FFMIN_SYM_MINBLOCKS 5
#endif

// the plain FP64 terms of a pair (coordinates or parameters outside the
// range of the integer forms): e_cul, C6 r^-6, C12 r^-12, r^-2
__device__ __noinline__ void terms64_plain(double dx, double dy, double dz, double qq, double c6, double c12,
                                           double (&o)[4]) {
    const double ri = rsqrt(dx * dx + dy * dy + dz * dz);
    const double ri2 = ri * ri, ri6 = ri2 * ri2 * ri2;
    o[0] = qq * ri;
    o[1] = c6 * ri6;
    o[2] = c12 * ri6 * ri6;
    o[3] = ri2;
}

// CL: for objects with fewer parts of tile pairs than the SMs hold, a part is
// shared by a cluster of c.cl64 blocks: each takes a run of the part's steps,
// and the blocks' sums are added in order through their shared memory.  A lone
// warp needs about 2,500 cycles for a step (430 dependent instructions) and
// 500 atoms kept every warp busy for 32 of them on 40 SMs.  The grid covers
// every item of the object once, without the queue.
// E + grad with the queue's kernel before it, us: 500 atoms 45 (one block a part)
// and 34 (four times the warps in a block) -> 22, 1,500 atoms 67 -> 51.
template <bool CL>
__global__ void __launch_bounds__(NT_SYM, FFMIN_SYM_MINBLOCKS) k_pair64_sym(Ctx c) {
    // staged j-atoms: x, y | z, then q', c6, c12 as significands with their
    // exponents and the charge's sign (forces), or as they are (energy only)
    __shared__ ulonglong2 s_xy[TJ], s_zq[TJ], s_c[TJ];
    __shared__ int2 s_e[TJ];
    __shared__ double jfx[4 * TJ], jfy[4 * TJ], jfz[4 * TJ];  // opposite forces, [warp][j of the part]
    __shared__ double s_i[CL ? 4 : 1][CL ? TI : 1], s_j[CL ? 3 * TJ : 1];  // this block's sums
    __shared__ int s_item;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    cg::cluster_group cl = cg::this_cluster();
    const int CS = CL ? (int)cl.num_blocks() : 1, rank = CL ? (int)cl.block_rank() : 0;
    for (bool first = true;; first = false) {
        const int it = CL ? (int)blockIdx.x / CS
                          : next_item<LIST_F64>(c, c.sys_items64, &c.counters[CNT_PAIR64], first, s_item);
        if (it < 0) break;
        const Item I = c.items64[it];
        if (I.tile < 0) {
            bonded_item(c, I.j0, I.nj, 1, rank * NT_SYM + tid, CS * NT_SYM);
            if constexpr (CL) return;
            continue;
        }
        const Tile &tl = c.tiles[I.tile];
        const int kind = c.st[I.sys].ev_kind;
        if (kind == EV_NONE || c.st[I.sys].mode != 1) {
            if constexpr (CL) return;  // every block of the cluster
            continue;
        }
        const bool grad = kind == EV_EG;
        const bool part = tl.r64.split > 1;
        const int W = TJ / tl.r64.split;
        double4_32a pi;
        double2 ci;
        if (tid < tl.na) {
            pi = c.posd[tl.a0 + tid];
            ci = c.pard[tl.a0 + tid];
        } else {  // padding atom far away with no charge and no LJ
            pi = make_double4_32a(-1e6, -1e6, -1e6, 0.0);
            ci = make_double2(0.0, 0.0);
        }
        u64 qm, c6m, c12m;
        int qe, c6e, c12e;
        bool in_range = split64(pi.w, qm, qe);
        in_range = split64(ci.x, c6m, c6e) && in_range;
        in_range = split64(ci.y, c12m, c12e) && in_range;
        const int ce = (c6e << 16) | c12e;  // both biased: the sums of two stay below 2^16
        const uint32_t qs = (uint32_t)(bits64(pi.w) >> 32) & 0x80000000u;
        long long xi, yi, zi;
        bool i_fix = fix64(pi.x, xi);
        i_fix = fix64(pi.y, yi) && i_fix;
        i_fix = fix64(pi.z, zi) && i_fix;
        if (tid >= tl.na) {
            xi = yi = zi = -FIX_FAR;
            i_fix = true;
        }
        double gx = 0.0, gy = 0.0, gz = 0.0, e6 = 0.0;  // e6: six times the energy
        double sc1 = 0.0, s6 = 0.0, s12 = 0.0;  // energy-only factored sums
        const int jend = I.j0 + I.nj;
        double *fx = jfx + w * W, *fy = jfy + w * W, *fz = jfz + w * W;
        for (int jt = I.j0; jt < jend; jt += TJ) {
            const int jl = jt + tid;
            double4_32a pj = make_double4_32a(1e6, 1e6, 1e6, 0.0);
            double2 cj0 = make_double2(0.0, 0.0);
            long long xj = FIX_FAR, yj = FIX_FAR, zj = FIX_FAR;
            u64 m1 = 0, m6 = 0, m12 = 0;
            int x1 = P64_ZERO, x6 = P64_ZERO, x12 = P64_ZERO;
            bool j_range = in_range, j_fix = i_fix;
            if (tid < W && jl < jend) {
                pj = c.posd[jl];
                cj0 = c.pard[jl];
                j_range = split64(pj.w, m1, x1) && j_range;
                j_range = split64(cj0.x, m6, x6) && j_range;
                j_range = split64(cj0.y, m12, x12) && j_range;
                j_fix = fix64(pj.x, xj) && j_fix;
                j_fix = fix64(pj.y, yj) && j_fix;
                j_fix = fix64(pj.z, zj) && j_fix;
            }
            // fixed-point coordinates for the tile pair when all of them fit;
            // the integer forms of the terms when every parameter is in range
            const bool fix = __syncthreads_and(j_fix && j_range);
            const bool plain = fix ? false : __syncthreads_or(!j_range);
            if (tid < W) {
                s_xy[tid] = fix ? make_ulonglong2((u64)xj, (u64)yj) : make_ulonglong2(bits64(pj.x), bits64(pj.y));
                s_zq[tid] = make_ulonglong2(fix ? (u64)zj : bits64(pj.z), grad ? m1 : bits64(pj.w));
                s_c[tid] = grad ? make_ulonglong2(m6, m12) : make_ulonglong2(bits64(cj0.x), bits64(cj0.y));
                if (grad)
                    s_e[tid] = make_int2((int)((uint32_t)x1 | ((uint32_t)(bits64(pj.w) >> 32) & 0x80000000u)),
                                         (x6 << 16) | x12);
            }
            if (grad) {
                for (int q = lane; q < W; q += 32) { fx[q] = 0.0; fy[q] = 0.0; fz[q] = 0.0; }
            }
            __syncthreads();
            // the diagonal tile (j-tile == i-tile): whole, thread t pairs with
            // t + k, k = 1 .. TJ/2 (at k = TJ/2 only t < TJ/2); in parts,
            // the pairs with j > i
            const bool diag = I.diag && (part || jt == I.j0);
            const bool half = diag && !part, mask = diag && part;
            const int k0 = half ? 1 : 0;
            const int k1 = half ? (tid < TJ / 2 ? TJ / 2 : TJ / 2 - 1)  // warp-uniform
                                : (mask && I.joff + W <= (w << 5) + 1 ? -1 : W - 1);
            const int ka = CL ? rank * (W / CS) : k0, kb = CL ? min(k1, ka + W / CS - 1) : k1;
            // the FP64 differences of a pair whose fixed-point ones are too small
            auto differences = [&](int j, double &dx, double &dy, double &dz) {
                const double4_32a q = jt + j < jend ? c.posd[jt + j] : make_double4_32a(1e6, 1e6, 1e6, 0.0);
                dx = q.x - pi.x; dy = q.y - pi.y; dz = q.z - pi.z;
            };
            auto energies = [&](auto FIX) {
                // energy only: the i atom's factors leave the sums,
                // E_i = q'_i sum q'_j / r + (c12_i sum c12_j r^-12 - c6_i sum c6_j r^-6) / 6
                for (int k = ka; k <= kb; k++) {
                    const int j = (tid + k) & (W - 1);
                    const ulonglong2 xy = s_xy[j], zq = s_zq[j], cj = s_c[j];
                    const bool on = !mask || I.joff + j > tid;
                    Inv64 v;
                    bool ok;
                    double dx = 1.0, dy = 0.0, dz = 0.0;
                    if constexpr (decltype(FIX)::value) {
                        u64 ax, ay, az;
                        int n;
                        ok = inv64_fix((long long)xy.x - xi, (long long)xy.y - yi, (long long)zq.x - zi, v, ax, ay, az, n) || !on;
                    } else {
                        if (on) {
                            dx = from_bits64(xy.x) - pi.x;
                            dy = from_bits64(xy.y) - pi.y;
                            dz = from_bits64(zq.x) - pi.z;
                        }
                        ok = inv64(dx, dy, dz, v);
                    }
                    double ri = inv64_r1(v), ri6 = inv64_r6(v), ri12 = inv64_r12(v);
                    if (__any_sync(0xffffffffu, !ok)) {
                        if (decltype(FIX)::value && on) differences(j, dx, dy, dz);
                        double o[4];
                        terms64_plain(dx, dy, dz, 1.0, 1.0, 1.0, o);
                        ri = o[0]; ri6 = o[1]; ri12 = o[2];
                    }
                    if (!on) ri = ri6 = ri12 = 0.0;
                    sc1 = fma(from_bits64(zq.y), ri, sc1);
                    s6 = fma(from_bits64(cj.x), ri6, s6);
                    s12 = fma(from_bits64(cj.y), ri12, s12);
                }
            };
            auto forces = [&](auto FIX) {
                for (int k = ka; k <= kb; k++) {
                    const int j = (tid + k) & (W - 1);
                    const ulonglong2 xy = s_xy[j], zq = s_zq[j], cj = s_c[j];
                    const int2 ej = s_e[j];
                    const bool on = !mask || I.joff + j > tid;
                    Inv64 v;
                    bool ok;
                    double dx = 1.0, dy = 0.0, dz = 0.0;
                    if constexpr (decltype(FIX)::value) {
                        const long long fx = (long long)xy.x - xi, fy = (long long)xy.y - yi, fz = (long long)zq.x - zi;
                        u64 ax, ay, az;
                        int n;
                        ok = inv64_fix(fx, fy, fz, v, ax, ay, az, n) || !on;
                        dx = fix_to_double(ax, n, fx);
                        dy = fix_to_double(ay, n, fy);
                        dz = fix_to_double(az, n, fz);
                    } else {
                        if (on) {
                            dx = from_bits64(xy.x) - pi.x;
                            dy = from_bits64(xy.y) - pi.y;
                            dz = from_bits64(zq.x) - pi.z;
                        }
                        ok = inv64(dx, dy, dz, v);
                    }
                    const int es = ce + ej.y;
                    double f, y;
                    inv64_force(v, qm, zq.y, qe + (ej.x & 0xffff), ((uint32_t)ej.x ^ qs) & 0x80000000u, c6m, cj.x,
                                (int)((uint32_t)es >> 16), c12m, cj.y, es & 0xffff, f, y);
                    if (__any_sync(0xffffffffu, !ok) || plain) {
                        if (decltype(FIX)::value) {
                            dx = 1.0; dy = dz = 0.0;
                            if (on) differences(j, dx, dy, dz);
                        }
                        const int jg = jt + j;
                        const double q_j = jg < jend ? c.posd[jg].w : 0.0;
                        const double2 c_j = jg < jend ? c.pard[jg] : make_double2(0.0, 0.0);
                        double o[4];
                        terms64_plain(dx, dy, dz, pi.w * q_j, ci.x * c_j.x, ci.y * c_j.y, o);
                        const double u = o[2] - o[1];
                        f = ((u + o[2]) + o[0]) * o[3];
                        y = fma(6.0, o[0], u);
                    }
                    if (!on) f = y = 0.0;
                    e6 += y;
                    gx = fma(f, dx, gx);
                    gy = fma(f, dy, gy);
                    gz = fma(f, dz, gz);
                    fx[j] = fma(-f, dx, fx[j]);
                    fy[j] = fma(-f, dy, fy[j]);
                    fz[j] = fma(-f, dz, fz[j]);
                    __syncwarp();
                }
            };
            if (!grad) {
                if (fix) energies(std::true_type{});
                else energies(std::false_type{});
                continue;
            }
            if (fix) forces(std::true_type{});
            else forces(std::false_type{});
            __syncthreads();
            // j-side partial row of this j-tile, warps summed in order
            if constexpr (CL) {
                for (int q = tid; q < 3 * W; q += NT_SYM) {
                    const int j = q % W;
                    const double *f = (q < W ? jfx : (q < 2 * W ? jfy : jfz)) + j;
                    s_j[q] = ((f[0] + f[W]) + f[2 * W]) + f[3 * W];
                }
            } else if (tid < W && jl < jend) {
                double4_32a o;
                o.x = jfx[tid]; o.y = jfy[tid]; o.z = jfz[tid];
#pragma unroll
                for (int v = 1; v < 4; v++) { o.x += jfx[v * W + tid]; o.y += jfy[v * W + tid]; o.z += jfz[v * W + tid]; }
                o.w = 0.0;
                c.gpd[(int64_t)(I.jslot + (jt - I.j0) / TJ) * TI + I.joff + tid] = o;
            }
        }
        double4_32a o;
        o.x = gx; o.y = gy; o.z = gz;
        o.w = grad ? e6 * (1.0 / 6.0) : pi.w * sc1 + (ci.y * s12 - ci.x * s6) * (1.0 / 6.0);
        if constexpr (CL) {
            s_i[0][tid] = o.x; s_i[1][tid] = o.y; s_i[2][tid] = o.z; s_i[3][tid] = o.w;
            cl.sync();
            const int n = 4 * TI + (grad ? 3 * W : 0);
            double *irow = reinterpret_cast<double *>(c.gpd + (int64_t)I.slot * TI);
            double *jrow = reinterpret_cast<double *>(c.gpd + (int64_t)I.jslot * TI + I.joff);
            for (int u = rank * NT_SYM + tid; u < n; u += CS * NT_SYM) {
                const int v = u - 4 * TI;
                double *mine = v < 0 ? &s_i[0][u] : &s_j[v];
                double x = *cl.map_shared_rank(mine, 0);
                for (int r = 1; r < CS; r++) x += *cl.map_shared_rank(mine, r);
                if (v < 0) irow[4 * (u % TI) + u / TI] = x;
                else if (v % W < I.nj) jrow[4 * (v % W) + v / W] = x;
            }
            cl.sync();  // no block leaves while its shared memory is read
            return;
        }
        c.gpd[(int64_t)I.slot * TI + tid] = o;
    }
}

// FP64 row sweep: one i-atom per thread (the FP64 pipe, not the loads, is
// the limit)
constexpr int NT_F64 = 128;
#define K_F64 k_pair<double, 128, 1>

int pair_grid_size(int mode, int f32_ipt, bool xs) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool one = f32_ipt == 1;
    if (mode == 0 && xs && one)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pair<float, TI, 1, true>, TI, 0);
    else if (mode == 0 && xs)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pair<float, TI / 2, 2, true>, TI / 2, 0);
    else if (mode == 0 && one)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pair<float, TI, 1>, TI, 0);
    else if (mode == 0)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pair<float, TI / 2, 2>, TI / 2, 0);
    else if (mode == 1)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, K_F64, NT_F64, 0);
    else if (mode == 2)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pair64_sym<false>, NT_SYM, 0);
    else if (one)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pair<float, TI, 1, false, true>, TI, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pair<float, TI / 2, 2, false, true>, TI / 2, 0);
    if (per < 1) per = 1;
    return sms * per;
}

// the FP32 E + grad (eonly false) or energy-only kernel in the object's shape
template <int IPT>
static void launch_f32_shape(const Ctx &c, bool eonly, int grid, cudaStream_t s) {
    constexpr int NT = TI / IPT;
    if (c.xs_off) {
        if (eonly) k_pair<float, NT, IPT, true, true><<<grid, NT, 0, s>>>(c);
        else k_pair<float, NT, IPT, true><<<grid, NT, 0, s>>>(c);
    } else {
        if (eonly) k_pair<float, NT, IPT, false, true><<<grid, NT, 0, s>>>(c);
        else k_pair<float, NT, IPT><<<grid, NT, 0, s>>>(c);
    }
}

static cudaError_t launch_pair64_cl(const Ctx &c, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(c.n_items64 * c.cl64);
    cfg.blockDim = dim3(NT_SYM);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = c.cl64;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_pair64_sym<true>, c);
}

cudaError_t launch_pair_list(const Ctx &c, int list, int grid, cudaStream_t s) {
    if (list == LIST_F64) {
        if (c.sym64 && c.cl64 > 1) return launch_pair64_cl(c, s);
        if (c.sym64) k_pair64_sym<false><<<grid, NT_SYM, 0, s>>>(c);
        else K_F64<<<grid, NT_F64, 0, s>>>(c);
    } else if (c.f32_ipt == 1) {
        launch_f32_shape<1>(c, list == LIST_F32_E, grid, s);
    } else {
        launch_f32_shape<2>(c, list == LIST_F32_E, grid, s);
    }
    return cudaGetLastError();
}

__global__ void __launch_bounds__(32 * N_LISTS) k_activelist(Ctx c) { active_lists(c); }

// The three pair kernels of a MIXED object take disjoint work queues and
// write disjoint outputs, so with side streams the FP32 energy-only and the
// FP64 kernels run beside the FP32 E + grad kernel (parallel graph branches
// when captured): a round waits for the slowest, not for all three in turn.
cudaError_t launch_pair_kernels(const Ctx &c, int grid32, int grid32e, int grid64, cudaStream_t s,
                                const Branches *br) {
    cudaError_t e;
    if (c.prec != FFMIN_MIXED) return launch_pair_list(c, LIST_F64, grid64, s);
    cudaStream_t se = s, s64 = s;
    if (br) {
        if ((e = cudaEventRecord(br->fork, s)) != cudaSuccess) return e;
        for (int k = 0; k < 2; k++)
            if ((e = cudaStreamWaitEvent(br->side[k], br->fork, 0)) != cudaSuccess) return e;
        se = br->side[0];
        s64 = br->side[1];
    }
    if ((e = launch_pair_list(c, LIST_F32_EG, grid32, s)) != cudaSuccess) return e;
    if ((e = launch_pair_list(c, LIST_F32_E, grid32e, se)) != cudaSuccess) return e;
    if ((e = launch_pair_list(c, LIST_F64, grid64, s64)) != cudaSuccess) return e;
    if (br) {
        for (int k = 0; k < 2; k++) {
            if ((e = cudaEventRecord(br->join[k], br->side[k])) != cudaSuccess) return e;
            if ((e = cudaStreamWaitEvent(s, br->join[k], 0)) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_pair(const Ctx &c, int grid32, int grid32e, int grid64, cudaStream_t s) {
    k_activelist<<<1, 32 * N_LISTS, 0, s>>>(c);  // also gives every pair kernel a fresh work queue
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_pair_kernels(c, grid32, grid32e, grid64, s, nullptr);
}

}  // namespace ffm
