// FP64 pair terms with most of their arithmetic on the integer pipes.
//
// GB300 retires 2 FP64 operations per SM and clock, 16 cycles for a warp's
// one, while a 64 x 64 -> high 64-bit product takes about 4 cycles.  A pair with
// forces costs about 31 FP64 instructions (CUDA's rsqrt alone 5.7) when it
// is written in FP64.  Here r^2, its reciprocal square root, the powers of r
// and the products with the atoms' parameters are formed on 64-bit
// significands with separate exponents, the terms of a pair are added as
// integers, and the results rounded once to FP64; FP64 instructions remain for
// the accumulation (7 a pair with forces, 3 for an energy) and, outside the
// fixed-point range, for the coordinate differences (3 more).  The relative
// errors of the significands (largest of millions of differences, host side,
// against long double) are 2^-56.8 for r^-1, 2^-55.8 for r^-2, 2^-54.2 for r^-6 and
// 2^-53.2 for r^-12 (each product's cuts and the power's multiple of r^-1's), and
// a result is rounded to 53 bits once, so a term is within two units of 2^-53,
// where the roundings of the FP64 formula (2^-53 each, raised to the same powers)
// add up to more.
//
// r^-1 from the hardware's approximate FP32 reciprocal square root y and one
// step of the series (1 - h)^(-1/2) = 1 + h/2 + 3 h^2/8 + O(h^3) with
// h = 1 - r^2 y^2, |h| < 2^-20, so that the next term is below 2^-61.
//
// Coordinate differences come in as doubles (any range below) or, for the
// coordinates of an ordinary system, as fixed-point integers.
//
// Ranges: |d|max in [2^-40, 2^41) A and parameters that are zero or within
// 2^-200 .. 2^200; then no intermediate leaves the exponent range of FP64.
// Anything else (coincident atoms, infinities, NaN) takes the FP64 formula.
#pragma once

#include <cstdint>

#ifdef __CUDA_ARCH__
#define FFM_P64 __device__ __forceinline__
#else
#define FFM_P64 __host__ __device__ inline
#endif

namespace ffm {

typedef unsigned long long u64;

// high 64 bits of a * b, at most 2 below; a, b <= 2^63 and not both 2^63
FFM_P64 u64 mulh(u64 a, u64 b) {
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    const u64 mid = (u64)ah * bl + (u64)al * bh;
    return (u64)ah * bh + (mid >> 32);
}
// high 64 bits of a * a, at most 2 below; a <= 2^63
FFM_P64 u64 sqh(u64 a) {
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
    return (u64)ah * ah + (((u64)ah * al) >> 31);
}
FFM_P64 int clz_hi(u64 v) {  // leading zeros of v >= 2^32
#ifdef __CUDA_ARCH__
    return __clz((int)(v >> 32));
#else
    return __builtin_clzll(v);
#endif
}
FFM_P64 u64 bits64(double x) {
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(x);
#else
    u64 u;
    __builtin_memcpy(&u, &x, 8);
    return u;
#endif
}
FFM_P64 double from_bits64(u64 u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    __builtin_memcpy(&x, &u, 8);
    return x;
#endif
}
// y ~ x^-1/2 (relative error below 2^-21), x = xh 2^-30 in [1/4, 3), as an integer times 2^-30
FFM_P64 uint32_t rsqrt_seed(uint32_t xh) {
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint2float_rn(xh)));
    return __float2uint_rz(y * 0x1p45f);  // (xh)^-1/2 2^15 = y, times 2^30
#else
    const float y = 1.0f / __builtin_sqrtf((float)xh);
    return (uint32_t)(y * 0x1p45f);
#endif
}

// v 2^(b - 1023) rounded to FP64 (v in [2^55, 2^64)); ZERO: below the normal
// range it is 0 (the exponent of a zero parameter puts it there)
template <bool ZERO>
FFM_P64 double pack64(u64 v, int b) {
    const int n = clz_hi(v), s = 11 - n;
    const u64 m = (v >> s) + ((uint32_t)((uint32_t)v >> (s - 1)) & 1u);  // 53 bits, or 2^53: carries into the exponent
    const int ex = b + 63 - n;
    const u64 r = m + ((u64)(uint32_t)((ex - 1) << 20) << 32);
    return from_bits64(ZERO && ex < 1 ? 0 : r);
}

// a parameter's significand (top bit 62; value = m 2^(e - 62)) and biased
// exponent e + P64_BIAS; zero: an exponent that every product flushes
constexpr int P64_BIAS = 8192, P64_ZERO = P64_BIAS - 4000;
FFM_P64 bool split64(double x, u64 &m, int &e) {  // |x|; false: out of the range of these forms
    const u64 u = bits64(x);
    const int ex = (int)((u >> 52) & 0x7ff);
    m = ((u & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
    if ((u << 1) == 0) {
        e = P64_ZERO;
        return true;
    }
    e = ex - 1023 + P64_BIAS;
    return ex >= 1023 - 200 && ex <= 1023 + 200;
}

// r^-1 = m 2^(-63 - E), r^-2 = n2 2^(-62 - n - 2 E), r^-6 = n6 2^(-59 - 3 n - k - 6 E),
// with m in [2^61, 2^63], n2 and n6 in [2^62, 2^63)
struct Inv64 {
    u64 m, n2, n6;
    int E, n, k;
};

// from r^2 = R 2^(2 E - 60), R in [2^60, 3 2^62)
FFM_P64 void inv64_back(u64 R, int E, Inv64 &o) {
    o.E = E;
    const uint32_t y = rsqrt_seed((uint32_t)(R >> 32));
    // h = 1 - r^2 y^2 in units of 2^-57, then c = h/2 + 3 h^2/8 in units of 2^-58
    const long long h = (long long)(1ULL << 57) - (long long)mulh(R >> 1, (u64)y * y);
    const int hs = (int)(h >> 10);
    const long long c = h + (((long long)hs * hs * 3) >> 39);
    // m = y (1 + c), 62 fraction bits
    const int ch = (int)(c >> 16);
    const uint32_t cl = (uint32_t)c & 0xffffu;
    o.m = ((u64)y << 32) + (u64)(((long long)((u64)y * cl) >> 26) + (((long long)(int)ch * (long long)y) >> 10));
    const u64 q2 = sqh(o.m);  // 60 fraction bits, [2^58, 2^62]
    o.n = clz_hi(q2) - 1;
    o.n2 = q2 << o.n;
    const u64 q6 = mulh(sqh(o.n2) << 1, o.n2);  // [2^59, 2^62), 53 + 3 n fraction bits
    o.k = clz_hi(q6) - 1;
    o.n6 = q6 << o.k;
}

// from the coordinate differences; false: outside the range
FFM_P64 bool inv64(double dx, double dy, double dz, Inv64 &o) {
    const u64 ux = bits64(dx), uy = bits64(dy), uz = bits64(dz);
    const int ex = (int)((uint32_t)(ux >> 32) >> 20) & 0x7ff, ey = (int)((uint32_t)(uy >> 32) >> 20) & 0x7ff,
              ez = (int)((uint32_t)(uz >> 32) >> 20) & 0x7ff;
    const int em = ex > ey ? (ex > ez ? ex : ez) : (ey > ez ? ey : ez);
    // significands aligned to the largest exponent, top bit 62 (a zero's
    // implicit bit is shifted out with the rest)
    const u64 one = 0x10000000000000ULL, frac = one - 1;
    const int sx = em - ex < 63 ? em - ex : 63, sy = em - ey < 63 ? em - ey : 63, sz = em - ez < 63 ? em - ez : 63;
    const u64 ax = (((ux & frac) | one) << 10) >> sx, ay = (((uy & frac) | one) << 10) >> sy,
              az = (((uz & frac) | one) << 10) >> sz;
    inv64_back(sqh(ax) + sqh(ay) + sqh(az), em - 1023, o);
    return em >= 1023 - 40 && em <= 1023 + 40;
}

// ---- coordinates in fixed point, units of 2^-54 A, for |x| < FIX_MAX A.  A
// double of at least 1/4 A converts exactly (its last place is 2^-54 or more),
// a smaller one with an error of 2^-55 A at most, and differences are exact,
// where an FP64 difference is rounded at 2^-53 of itself.  Pairs closer than
// 1/4 A take the FP64 differences, so the error of a difference, relative to
// the separation, stays below the two units that FP64 coordinates give.
constexpr double FIX_MAX = 224.0;
constexpr long long FIX_FAR = 255LL << 54;  // padding atoms: beyond any real one, differences still fit
FFM_P64 bool fix64(double x, long long &o) {  // false: out of range (or NaN)
#ifdef __CUDA_ARCH__
    o = __double2ll_rn(x * 0x1p54);
#else
    o = (long long)__builtin_rint(x * 0x1p54);
#endif
    return x > -FIX_MAX && x < FIX_MAX;
}
FFM_P64 u64 abs64(long long v) {
    const long long s = v >> 63;
    return (u64)((v ^ s) - s);
}
// from fixed-point differences (|d| < 2^63); a* return |d| shifted left by the
// returned n; false: below 1/4 A in every component
FFM_P64 bool inv64_fix(long long dx, long long dy, long long dz, Inv64 &o, u64 &ax, u64 &ay, u64 &az, int &n) {
    ax = abs64(dx);
    ay = abs64(dy);
    az = abs64(dz);
    const u64 any = (ax | ay | az) | 1ULL << 32;  // at least one bit for the count
    n = clz_hi(any) - 1;
    const bool ok = ((ax | ay | az) >> 52) != 0ULL;
    ax <<= n;
    ay <<= n;
    az <<= n;
    inv64_back(sqh(ax) + sqh(ay) + sqh(az), 8 - n, o);
    return ok;
}
// a 2^-(54 + n) with the sign of v, rounded to FP64
FFM_P64 double fix_to_double(u64 a, int n, long long v) {
    const uint32_t hi = (uint32_t)(a >> 32), lo = (uint32_t)a;
#ifdef __CUDA_ARCH__
    const int z = hi ? __clz((int)hi) : 32 + __clz((int)lo);
#else
    const int z = a ? __builtin_clzll(a) : 64;
#endif
    const u64 m = a << (z & 63);
    const u64 r = ((m >> 11) + ((uint32_t)((uint32_t)m >> 10) & 1u)) +
                  ((u64)(uint32_t)((1023 + 63 - 54 - 1 - n - z) << 20) << 32);
    return from_bits64((a ? r : 0) | ((u64)v & 0x8000000000000000ULL));
}
FFM_P64 double inv64_r1(const Inv64 &v) { return pack64<false>(v.m, 1023 - 63 - v.E); }
FFM_P64 double inv64_r2(const Inv64 &v) { return pack64<false>(v.n2, 1023 - 62 - v.n - 2 * v.E); }
FFM_P64 double inv64_r6(const Inv64 &v) { return pack64<false>(v.n6, 1023 - 59 - 3 * v.n - v.k - 6 * v.E); }
FFM_P64 double inv64_r12(const Inv64 &v) {
    return pack64<false>(sqh(v.n6), 1023 - 54 - 6 * v.n - 2 * v.k - 12 * v.E);
}

// The force over r and six times the energy of a pair,
//   f = (e + 2 p12 - p6) r^-2,  y = 6 e + p12 - p6,
// from the terms' significands (each in [2^58, 2^62)), aligned to the largest
// exponent and added as integers, which leaves one FP64 addition (y) of a
// pair's six besides the accumulation of the forces.  A term is cut at 2^-56
// of the largest or better.  s1, s6, s12: sums of the parameters' biased
// exponents; neg: sign of the charges' product in the top bit.
FFM_P64 int clz64(u64 v) {  // v != 0
#ifdef __CUDA_ARCH__
    const uint32_t hi = (uint32_t)(v >> 32);
    return hi ? __clz((int)hi) : 32 + __clz((int)(uint32_t)v);
#else
    return __builtin_clzll(v);
#endif
}
FFM_P64 void inv64_force(const Inv64 &v, u64 q1, u64 q2, int s1, uint32_t neg, u64 a6, u64 b6, int s6, u64 a12, u64 b12,
                         int s12, double &f, double &y) {
    const u64 ve = mulh(mulh(q1, q2) << 1, v.m), v6 = mulh(mulh(a6, b6) << 1, v.n6),
              v12 = mulh(mulh(a12, b12) << 1, sqh(v.n6) << 1);
    const int k6 = 3 * v.n + v.k + 6 * v.E;
    const int be = s1 - v.E - 60, be6 = s6 - k6 - 56, be12 = s12 - 2 * k6 - 52;
    const int bm = be > be6 ? (be > be12 ? be : be12) : (be6 > be12 ? be6 : be12);
    const int d = bm - be < 61 ? bm - be : 61, d6 = bm - be6 < 61 ? bm - be6 : 61, d12 = bm - be12 < 61 ? bm - be12 : 61;
    const long long sg = (long long)(int)neg >> 63;
    const long long e = ((long long)(ve >> (d + 2)) ^ sg) - sg, x6 = (long long)(v6 >> (d6 + 2)),
                    x12 = (long long)(v12 >> (d12 + 2));
    const long long u = x12 - x6, x = u + x12 + e, z = u + 6 * e;
    const int b = bm + 2 + 1023 - 2 * P64_BIAS;  // biased exponent of a unit
    const u64 ax = abs64(x), az = abs64(z);
    const int n = clz64(ax | 1ULL) - 1, nz = clz64(az | 1ULL);
    const double r = pack64<true>(mulh(ax << n, v.n2), b + 4 - 2 - n - v.n - 2 * v.E);
    f = from_bits64(ax ? bits64(r) | ((u64)x & 0x8000000000000000ULL) : 0);
    const u64 m = az << nz;
    const int ex = b + 63 - nz;
    const u64 w = ((m >> 11) + ((uint32_t)((uint32_t)m >> 10) & 1u)) + ((u64)(uint32_t)((ex - 1) << 20) << 32);
    y = from_bits64(az && ex >= 1 ? w | ((u64)z & 0x8000000000000000ULL) : 0);
}

}  // namespace ffm
