// Pair terms of float64 forces on the integer pipe.
//
// sm_103a has two float64 lanes per SM and clock (a warp operation takes 16
// cycles) against 64 integer ones.  So only a pair's three differences are left
// to the float64 pipe; the squares, the -3/2 power, the product with m and the
// sums are fixed-point, some 230 instructions and 92 cycles a warp, where 19
// float64 operations and two conversions took 340.  Bound by the integer pipe
// (ALU 66 % busy at 65536 bodies, issue 65 %, float64 57 %; 63, 63, 55 at 16384).  16384 bodies: 9.56 ms before, 2.47
// now; with only the power in integers and a float64 product and sums 3.38.
// A single term's error against 113 bits is 0.45 x 2^-53 rms and 1.6 x 2^-53 at
// most (1.8 and 8.4 before).
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

// x^(-3/2) of x = X 2^-62 4^h, X in [2^62, 2^64), to a relative 2^-57.
//   y = Y 2^-24, the MUFU's root of X's high word: y = x'^(-1/2) (1 + e0) for
//       x' = X 2^-62, |e0| < 2^-22.7
//   e = 1 - x' y^2, |e| < 2^-21.6, to 2^-78: x' y^2 is known to be 1 - e, so
//       the product is formed modulo 2^-14
//   x'^(-3/2) = y^3 (1 - e)^(-3/2) = y^3 (1 + 3e/2 + 15e^2/8 + O(2.2 e^3 < 2^-63))
// Result: x'^(-3/2) 2^62, in [2^59, 2^62]; x^(-3/2) is 8^-h times as much.
__device__ __forceinline__ uint64_t inv_cube_fixed(uint64_t X)
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
    return c + (uint64_t)d;
}

// A mass in units of 2^-63 2^e, M in [2^63, 2^64) or 0; lim 0: not finite.
struct __align__(16) MassFixed {
    uint32_t lo, hi;
    int e2;        // 2 e + (1 if negative)
    uint32_t lim;  // exponents of the differences below 693 + lim take the integer form
};
constexpr int F64_NO_TERM = -30000;  // below any term's exponent

__device__ __forceinline__ MassFixed mass_fixed(double m)
{
    const int hi = __double2hiint(m), ex = (hi >> 20) & 0x7ff, neg = (int)((unsigned)hi >> 31);
    uint64_t f = ((uint64_t)(hi & 0xfffff) << 32) | (uint32_t)__double2loint(m);
    if (ex == 0x7ff || (ex == 0 && f == 0)) return {0, 0, 2 * F64_NO_TERM, ex ? 0u : 661u};
    int e = ex - 1023;
    if (ex == 0) {
        const int lz = (f >> 32) ? __clz((int)(f >> 32)) : 32 + __clz((int)f);
        f <<= lz;
        e = -1011 - lz;
    } else {
        f = (f | 1ull << 52) << 11;
    }
    return {(uint32_t)f, (uint32_t)(f >> 32), 2 * e + neg, 661};
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

// One pair's term (dx, dy, dz) m (dx^2 + dy^2 + dz^2 + eps2)^(-3/2) in integers:
// coordinate c is +- A[c] S 2^(e[c] - 1145), A in [2^61, 2^62), S in [2^63, 2^64)
// (or 0, or e F64_NO_TERM), the sign that of d[c] times m's.  false (and no
// result) where the general form is needed.
//
// The squares are summed relative to the largest exponent em of the
// differences and eps: |dx| = B 2^-61 2^(em-1023) with B < 2^62, B^2 2^-64 from the two
// upper partial products, so that x = X 2^-58 4^(em-1023) with X >= 2^58 off by
// at most 10: a relative 2^-54.7, where three float64 operations leave up to
// 3 x 2^-54.  Differences beyond 2^+-330 (and infinities, NaN) take the general
// form; beside one within them a subnormal difference, below 2^-690 of it, is
// taken half.
struct PairTerm {
    uint64_t A[3], S;
    int e[3];
};

__device__ __forceinline__ bool in_integer_form(double dx, double dy, double dz, const MassFixed &m)
{
    const uint32_t h = max(max(__double2hiint(dx) & 0x7fffffff, __double2hiint(dy) & 0x7fffffff),
                           __double2hiint(dz) & 0x7fffffff);
    return (h >> 20) - 693u < m.lim;
}

template <bool ZEPS>
__device__ __forceinline__ bool pair_term(double dx, double dy, double dz, const MassFixed &m,
                                          const EpsFixed &ef, PairTerm &t)
{
    const uint32_t h[3] = {__double2hiint(dx) & 0x7fffffffu, __double2hiint(dy) & 0x7fffffffu,
                           __double2hiint(dz) & 0x7fffffffu};
    const uint32_t l[3] = {(uint32_t)__double2loint(dx), (uint32_t)__double2loint(dy),
                           (uint32_t)__double2loint(dz)};
    int em = (int)(max(max(h[0], h[1]), h[2]) >> 20);
    const bool in_range = (unsigned)(em - 693) < m.lim;
    if (!ZEPS) em = max(em, ef.e);
    uint64_t X = ZEPS ? 0 : shr_clamped(ef.b, 2u * (unsigned)(em - ef.e)), cross = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int ex = (int)(h[c] >> 20);
        const uint32_t f = (__funnelshift_l(l[c], h[c], 9) & 0x1fffffffu) | (ex ? 0x20000000u : 0u);
        t.A[c] = ((uint64_t)f << 32) | (l[c] << 9);
        t.e[c] = ex;
        const uint64_t B = shr_clamped(t.A[c], (unsigned)(em - ex));
        const uint32_t B1 = (uint32_t)(B >> 32), B0 = (uint32_t)B;
        X += (uint64_t)B1 * B1;
        cross += (uint64_t)B1 * B0;
    }
    X += cross >> 31;
    const bool low = X < (1ull << 60);
    const uint64_t r = inv_cube_fixed(low ? X << 4 : X << 2);
    // S 2^64 = r M, brought to 64 bits
    const uint32_t r1 = (uint32_t)(r >> 32), r0 = (uint32_t)r;
    uint64_t S = (uint64_t)r1 * m.hi + __umulhi(r1, m.lo);
    S += __umulhi(r0, m.hi);
    const int lz = __clz((int)(S >> 32));
    t.S = S << lz;
    // 3 h for x^(-3/2), h = em - 1023 or one more
    int base = (m.e2 >> 1) - 3 * (em - 1023) - (low ? 0 : 3) - lz;
    if (!in_range) base = F64_NO_TERM;
#pragma unroll
    for (int c = 0; c < 3; ++c) t.e[c] += base;
    return in_range;
}

// One coordinate's fixed-point sum over a tile of J bodies: acc 2^(E - 1075 +
// HEAD - 6), E the largest exponent of a term of this tile so far.  A term is
// rounded to 2^-54 of the largest (J = 128), as a float64 addition would round
// the sum.  E starts again with each tile: kept over the tiles, two close
// bodies on either side, whose terms cancel, left every later term rounded to
// 2^-54 of theirs (1e6 of them: 6.0e-15 of such a term together, 6.2e-17 so).  Each
// step raises E without asking whether it must: in a branch, some lane of a warp
// met a new largest term in most steps (181 us at 4097 bodies, 195; 186 with the
// rounding below).
template <int J>
struct FixedSum {
    static constexpr int HEAD = J <= 128 ? 6 : 7;  // terms below 2^(62 - HEAD), J of them below 2^63
    static_assert(J <= 256, "");
    int64_t acc;
    int E;
    __device__ __forceinline__ void reset()
    {
        acc = 0;
        E = 2 * F64_NO_TERM;
    }
    // to a new largest exponent
    __device__ __forceinline__ void raise(int e)
    {
        acc >>= min(e - E, 63);
        E = e;
    }
    __device__ __forceinline__ void add(uint64_t A, uint64_t S, int e, int sign)
    {
        const uint64_t s = shr_clamped(S, (unsigned)(E - e + HEAD));
        const uint32_t A1 = (uint32_t)(A >> 32), A0 = (uint32_t)A;
        const uint32_t s1 = (uint32_t)(s >> 32), s0 = (uint32_t)s;
        // A (s + 1/2) 2^-64, rounded: s lost half a unit on the mean.  (Without
        // the half, and with A0 s0 taken at its mean, a million terms far below
        // the largest add up to 1e-12 of it.)
        uint64_t p = (uint64_t)A1 * s0 + (0x80000000u + (A1 >> 1));
        p += (uint64_t)A0 * s1;
        p += __umulhi(A0, s0);
        p = (uint64_t)A1 * s1 + (p >> 32);
        acc += (int64_t)(p ^ (uint64_t)(int64_t)sign) - sign;
    }
    __device__ __forceinline__ double take()
    {
        const double v = ldexp((double)acc, E - 1075 + HEAD - 6);
        reset();
        return v;
    }
};

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
