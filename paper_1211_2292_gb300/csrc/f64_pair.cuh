// (dx^2 + dy^2 + dz^2 + eps^2)^(-3/2) in float64 precision on the integer pipe.
//
// sm_103a has two float64 lanes per SM and clock (a warp operation takes 16
// cycles) against 64 integer ones, so of a pair's arithmetic only the
// differences, the product with m and the three sums are left to the float64
// pipe: 7 operations, 112 cycles a warp, where r^2, a refined reciprocal root
// and its cube made 19 and two conversions.  The integer side is some 140
// instructions, 31 % of the issue slots.  16384 bodies: 9.56 ms before, 3.38
// now (float64 pipe 89 % busy), 4097 bodies 703 us before and 238 now; the
// factor's error against 113 bits is 0.59 2^-53 rms and 2 2^-53 at most (1.75
// and 8 before).
#pragma once
#include <stdint.h>

namespace nb {

// eps^2 = b 2^-58 4^(e - 1023), b in [2^58, 2^60); e < 0: eps^2 below 2^-1022.
struct EpsFixed {
    uint64_t b;
    int e;
};

__device__ __forceinline__ EpsFixed eps_fixed(double eps2)
{
    const int hi = __double2hiint(eps2);
    const int ex = ((hi >> 20) & 0x7ff) - 1023;  // eps^2 = f 2^ex, 1 <= f < 2
    if (ex == -1023) return {0, -1};
    const uint64_t f = ((uint64_t)((hi & 0xfffff) | 0x100000) << 32) | (uint32_t)__double2loint(eps2);
    return {f << (6 + (ex & 1)), (ex >> 1) + 1023};
}

// a >> n for any n >= 0 (0 from 64 on)
__device__ __forceinline__ uint64_t shr_clamped(uint64_t a, unsigned n)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
    return r;
#else
    return n < 64 ? a >> n : 0;
#endif
}

// x^(-3/2) of x = X 2^-62 4^h, X in [2^62, 2^64), |h| <= 340: relative error
// below 2^-53 + 2^-57.
//   y = Y 2^-24, the MUFU's root of X's high word: y = x'^(-1/2) (1 + e0) for
//       x' = X 2^-62, |e0| < 2^-22.7
//   e = 1 - x' y^2, |e| < 2^-21.6, to 2^-78: x' y^2 is known to be 1 - e, so
//       the product is formed modulo 2^-14
//   x'^(-3/2) = y^3 (1 - e)^(-3/2) = y^3 (1 + 3e/2 + 15e^2/8 + O(2.2 e^3 < 2^-63))
__device__ __forceinline__ double inv_cube_fixed(uint64_t X, int h)
{
    const uint32_t X1 = (uint32_t)(X >> 32), X0 = (uint32_t)X;
    // y in [2^-16, 2^-15]; as an integer it has 24 bits, 2^24 for y = 2^-15
    const uint32_t Y = (uint32_t)__float_as_int(rsqrt_mufu(__uint2float_rn(X1))) - (110u << 23);
    const uint64_t Q = (uint64_t)Y * Y;  // y^2 2^48
    const uint32_t Q1 = (uint32_t)(Q >> 32), Q0 = (uint32_t)Q;
    // x' y^2 2^78 modulo 2^64
    uint64_t p = (uint64_t)X1 * Q0 + __umulhi(X0, Q0);
    p += (uint64_t)X0 * Q1;
    p += (uint64_t)(X1 * Q1) << 32;
    const int64_t e78 = -(int64_t)p;
    const int64_t e64 = e78 >> 14;                   // e 2^64
    const int e46 = (int)(e78 >> 32);                // e 2^46
    const int e2 = __mulhi(e46 * 16, e46);           // e^2 2^64
    const int64_t g = e64 + (e64 >> 1) + (2 * e2 - (e2 >> 3));  // (3e/2 + 15e^2/8) 2^64
    // y^3 2^62, and times 1 + g
    const uint64_t c = ((uint64_t)((uint64_t)Q1 * Y) << 22) + (((uint64_t)Q0 * Y) >> 10);
    const int c1 = (int)(c >> 32), g1 = (int)(g >> 32);
    int64_t d = (int64_t)c1 * g1 + __umulhi((uint32_t)c1, (uint32_t)g);
    d += 2 * __mulhi((int)((uint32_t)c >> 1), g1);
    const uint64_t r = c + (uint64_t)d;              // in [2^59, 2^62]
    // to float64, rounded at bit 53
    const int lz = __clz((int)(r >> 32));
    const uint64_t s = r << lz;
    const uint64_t b = (s >> 11) + ((s >> 10) & 1);
    const uint64_t bits = b + ((uint64_t)(uint32_t)(1023 - lz - 3 * h) << 52);
    return __longlong_as_double((long long)bits);
}

// The general form, for any x: m x^(-3/2) on the float64 pipe.  With the seed
// y and q = y^2 (exact, y has 24 bits) e = 1 - x q is one operation.
__device__ __forceinline__ double mass_inv_cube(double x, double m)
{
    const double y = rsqrt_seed(x), q = y * y;
    const double e = fma(-x, q, 1.0);
    const double s = (m * y) * q;
    return fma(s * e, fma(e, 1.875, 1.5), s);
}

// (dx^2 + dy^2 + dz^2 + eps2)^(-3/2); false (and no result) where the general
// form is needed.
//
// The squares are summed as integers relative to the largest exponent em of
// the differences and eps: |dx| = A 2^-61 2^(em-1023) with A < 2^62, A^2 2^-64
// from the two upper partial products, so that x = X 2^-58 4^(em-1023) with X
// >= 2^58 off by at most 8: a relative 2^-55, where three float64 operations
// leave up to 3 x 2^-54.  Exponents beyond 2^+-330 (and infinities, NaN) take
// the general form; within them a zero or subnormal difference, read here as a
// power of two, is below 2^-690 of the largest.
template <bool ZEPS>
__device__ __forceinline__ bool pair_inv_cube(double dx, double dy, double dz, const EpsFixed &ef,
                                              double &r)
{
    const uint32_t hx = __double2hiint(dx) & 0x7fffffff, hy = __double2hiint(dy) & 0x7fffffff,
                   hz = __double2hiint(dz) & 0x7fffffff;
    int em = (int)(max(max(hx, hy), hz) >> 20);
    if (!ZEPS) em = max(em, ef.e);
    uint64_t X = ZEPS ? 0 : shr_clamped(ef.b, 2u * (unsigned)(em - ef.e)), cross = 0;
    auto square = [&](uint32_t h, uint32_t l) {
        const uint32_t t = (__funnelshift_l(l, h, 9) & 0x1fffffffu) | 0x20000000u;
        const uint64_t A = shr_clamped(((uint64_t)t << 32) | (l << 9), (unsigned)em - (h >> 20));
        const uint32_t A1 = (uint32_t)(A >> 32), A0 = (uint32_t)A;
        X += (uint64_t)A1 * A1;
        cross += (uint64_t)A1 * A0;
    };
    square(hx, (uint32_t)__double2loint(dx));
    square(hy, (uint32_t)__double2loint(dy));
    square(hz, (uint32_t)__double2loint(dz));
    X += cross >> 31;
    const bool low = X < (1ull << 60);
    r = inv_cube_fixed(low ? X << 4 : X << 2, em - 1023 + (low ? 0 : 1));
    return (unsigned)(em - 693) <= 660u;
}

// The same times m, from the general form; ZEPS (eps2 = 0): 0 where r^2 is 0.
template <bool ZEPS>
__device__ __forceinline__ double pair_factor_general(double dx, double dy, double dz, double m,
                                                      double eps2)
{
    const double x = fma(dz, dz, fma(dy, dy, fma(dx, dx, eps2)));
    const double r = mass_inv_cube(x, m);
    return ZEPS ? (x > 0.0 ? r : 0.0) : r;
}

}  // namespace nb
