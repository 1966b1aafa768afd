// Device-side building blocks shared by the force, energy and adjoint kernels.
//
// Everything here is arithmetic on values already in registers or shared
// memory; the kernels decide layout and scheduling.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace nb {

// ---------------------------------------------------------------- float32x2
// Blackwell executes one float32x2 instruction (two IEEE round-to-nearest
// float32 operations on a 64-bit register pair) per issue slot, so pairing
// two i-bodies halves the issue cost of the pair arithmetic; the FP32 pipe
// throughput is unchanged.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Hardware reciprocal square root (MUFU), inputs flushed to zero when
// subnormal.  Relative error below 2^-22.
__device__ __forceinline__ float rsqrt_mufu(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Hardware base-2 logarithm and exponential (MUFU), subnormals flushed.
// lg2: absolute error below 2^-22 on [0.5, 2) (relative elsewhere through the
// exact exponent); ex2: relative error below 2^-22.
__device__ __forceinline__ float lg2_mufu(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_mufu(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// log2(m) of a float64 mass as float32: m = 2^e f, 1 <= f < 2; with r about 1/f
// (nine bits, from the top five bits of f) log2 m = e - log2 r + log2(1 + z),
// z = f r - 1 exact, |z| < 1/60.  -log2 r is tabulated as hi (a multiple of
// 2^-12, so that e + hi is exact) and lo, log2(1 + z) a polynomial: the result
// is within half an ulp plus about 2^-29.  Two float64 operations in place of
// the library's logarithm's dozens: on this part (2 float64 lanes per clock per
// SM) those took the packing of 2^20 bodies 75 us.
struct Log2Row {
    double r;
    float hi, lo;
};
static __device__ const Log2Row LOG2_ROWS[32] = {
    {0.984375, 0.02270507812f, 1.49983751e-05f},
    {0.955078125, 0.06640625f, -9.69049522e-05f},
    {0.927734375, 0.1081542969f, 6.19999067e-05f},
    {0.90234375, 0.1481933594f, 5.75992089e-05f},
    {0.876953125, 0.189453125f, -2.47597411e-05f},
    {0.853515625, 0.228515625f, -5.0945006e-06f},
    {0.83203125, 0.2653808594f, -9.04796008e-05f},
    {0.810546875, 0.3029785156f, 5.39581407e-05f},
    {0.791015625, 0.3381347656f, 8.7136603e-05f},
    {0.771484375, 0.3742675781f, 2.35788105e-05f},
    {0.75390625, 0.4074707031f, 7.22596069e-05f},
    {0.736328125, 0.4416503906f, -7.11038937e-05f},
    {0.71875, 0.4763183594f, 0.000119684568f},
    {0.703125, 0.5080566406f, 9.02630453e-05f},
    {0.6875, 0.5405273438f, 4.10376127e-05f},
    {0.673828125, 0.5695800781f, -3.26297905e-05f},
    {0.66015625, 0.5991210938f, -5.30032184e-07f},
    {0.646484375, 0.6293945312f, -8.19380572e-05f},
    {0.6328125, 0.66015625f, -6.25288462e-06f},
    {0.62109375, 0.6870117188f, 0.000105325966f},
    {0.609375, 0.7145996094f, -1.82823725e-06f},
    {0.59765625, 0.7426757812f, -6.36239427e-05f},
    {0.587890625, 0.7663574219f, 2.29013653e-05f},
    {0.576171875, 0.7954101562f, 1.86995008e-05f},
    {0.56640625, 0.8200683594f, 2.25506101e-05f},
    {0.556640625, 0.8452148438f, -3.29528021e-05f},
    {0.546875, 0.8706054688f, 0.000111514305f},
    {0.537109375, 0.8967285156f, -1.6324037e-05f},
    {0.529296875, 0.91796875f, -0.000117791354f},
    {0.51953125, 0.9448242188f, -0.000106654251f},
    {0.51171875, 0.9665527344f, 2.42640875e-05f},
    {0.50390625, 0.9887695312f, 3.21332675e-06f}};
__device__ __forceinline__ float log2_packed(double m)
{
    const int h = __double2hiint(m);
    if ((unsigned)(h >> 20) - 1u >= 2046u) return (float)log2(m);  // 0, < 0, subnormal, inf, NaN
    const Log2Row w = LOG2_ROWS[(h >> 15) & 31];
    const double f = __hiloint2double((h & 0xfffff) | 0x3ff00000, __double2loint(m));
    const float z = (float)fma(f, w.r, -1.0);
    // log2(1 + z) = z (c1 + z (c2 + z (c3 + z (c4 + z c5)))), c_k = (-1)^(k+1) / (k ln 2)
    float q = fmaf(z, 0.288539008f, -0.360673760f);
    q = fmaf(z, q, 0.480898347f);
    q = fmaf(z, q, -0.721347520f);
    q = fmaf(z, q, 1.442695041f);
    return ((float)((h >> 20) - 1023) + w.hi) + fmaf(z, q, w.lo);
}

// x as the float32 pair h = fl(x), l = fl(x - h), bit for bit, from the integer
// pipe: a conversion to or from float64 and a float64 operation take the
// float64 pipe 16 cycles a warp, and the plain form needs four of them per
// value.  Packing 804501 bodies takes 25 us that way, 11 so.  Zero, tiny, huge
// and non-finite values go the plain way.
static __device__ __noinline__ float2 split_f64_plain(double x)  // (a call: else all lanes wait for it)
{
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}
__device__ __forceinline__ void split_f64(double x, float &h, float &l)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu) - 1023;  // |x| = 1.f 2^e
    if ((unsigned)(e + 70) > 190u) {
        const float2 p = split_f64_plain(x);
        h = p.x;
        l = p.y;
        return;
    }
    // the significand's upper 24 bits and the 29 below, rounded to nearest even
    const unsigned q = ((hi & 0xfffffu) | 0x100000u) << 3 | lo >> 29, r = lo & 0x1fffffffu;
    const unsigned up = r + (q & 1u) > 0x10000000u;
    const unsigned sign = hi & 0x80000000u;
    h = __uint_as_float((((unsigned)(e + 126) << 23) + q + up) | sign);  // q holds the hidden bit
    const int rem = (int)r - (int)(up << 29);  // x - h in units of 2^(e - 52)
    l = __int2float_rn(sign ? -rem : rem) * __uint_as_float((unsigned)(e + 75) << 23);
}

// Seed of the float64 reciprocal square root: y0 = x^(-1/2) (1 + e0), |e0| <
// 2^-22, with a 24-bit significand, for any positive normal x.  x is scaled by
// an even power of two into [1, 4), cut to float32 and sent through the MUFU,
// and the result scaled back, all on the integer pipe: a conversion between
// float64 and float32 takes the float64 pipe (2 lanes per clock per SM) as an
// operation would.  (A float32 seed of x itself would overflow or flush to
// zero outside 1.2e-38 .. 3.4e38, e.g. for r^2 = 1e-40 at eps = 0.)
__device__ __forceinline__ double rsqrt_seed(double x)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int ex = (int)(((unsigned)hi >> 20) & 0x7ffu) - 1023;  // x = f 2^ex, 1 <= f < 2
    const unsigned xf = ((unsigned)(127 + (ex & 1)) << 23) | (((unsigned)hi & 0xfffffu) << 3) |
                        ((unsigned)lo >> 29);
    const unsigned yf = __float_as_uint(rsqrt_mufu(__uint_as_float(xf)));  // in (1/2, 1]
    return __hiloint2double((int)(yf >> 3) + (1023 - 127 - (ex >> 1)) * (1 << 20), (int)(yf << 29));
}

// float64 reciprocal square root: the seed y0 refined by one second-order
// Householder step for f(y) = 1/y^2 - x.  With e = 1 - x*y0^2 the exact answer
// is y0*(1-e)^(-1/2) = y0*(1 + e/2 + 3e^2/8 + ...); keeping two terms leaves a
// relative error of about (5/16)e^3 ~ 1e-20, below float64 rounding.  Valid
// for positive normal x; x = 0 gives a large finite value (callers mask the
// self pair).
__device__ __forceinline__ double rsqrt_f64(double x)
{
    const double y = rsqrt_seed(x);
    double h = x * y;
    double e = fma(-h, y, 1.0);
    double p = fma(e, 0.375, 0.5);
    return fma(y * e, p, y);
}

// Exclusive scan of in[0..total) into out[0..total) (in == out allowed) by
// one block of 1024 threads, in index order, starting from carry0; returns
// carry0 plus the sum (every thread).
// Tiles of 8192 entries pass through shared memory (coalesced loads and
// stores), 8 consecutive entries per thread, a two-level warp scan of the
// thread sums and a carry from tile to tile.  tile: 8192 + 256 entries,
// wsum: 32 entries of shared memory.
constexpr int BSCAN_PER = 8, BSCAN_TILE = 1024 * BSCAN_PER;
__device__ __forceinline__ int bscan_pad(int i) { return i + (i >> 5); }  // no bank conflicts

template <typename T>
__device__ T block_scan_exclusive(const T *in, T *out, int total, T *tile, T *wsum, T carry0 = 0)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T carry = carry0;
    for (int base = 0; base < total; base += BSCAN_TILE) {
        for (int q = threadIdx.x; q < BSCAN_TILE; q += 1024)
            tile[bscan_pad(q)] = base + q < total ? in[base + q] : T(0);
        __syncthreads();
        T v[BSCAN_PER], sum = 0;
#pragma unroll
        for (int q = 0; q < BSCAN_PER; ++q) {
            v[q] = tile[bscan_pad(threadIdx.x * BSCAN_PER + q)];
            sum += v[q];
        }
        T incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const T t = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            T w = wsum[lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const T t = __shfl_up_sync(0xffffffffu, w, off);
                if (lane >= off) w += t;
            }
            wsum[lane] = w;
        }
        __syncthreads();
        T run = carry + (warp ? wsum[warp - 1] : T(0)) + incl - sum;
#pragma unroll
        for (int q = 0; q < BSCAN_PER; ++q) {
            tile[bscan_pad(threadIdx.x * BSCAN_PER + q)] = run;
            run += v[q];
        }
        __syncthreads();
        for (int q = threadIdx.x; q < BSCAN_TILE; q += 1024)
            if (base + q < total) out[base + q] = tile[bscan_pad(q)];
        carry += wsum[31];
        __syncthreads();  // tile and wsum are rewritten by the next tile
    }
    return carry;
}

// Kahan-compensated accumulation of a partial sum p into (s, c); the value
// represented is s - c.
__device__ __forceinline__ void kahan_add(float &s, float &c, float p)
{
    float y = p - c;
    float t = s + y;
    c = (t - s) - y;
    s = t;
}

// (s, c) += (so, co) for Kahan pairs holding s - c: the sums' rounding
// error goes into the carry (the two-sum of s and so).
__device__ __forceinline__ void kahan_merge(float &s, float &c, float so, float co)
{
    const float t = s + so;
    const float bp = t - s;
    const float e = (s - (t - bp)) + (so - bp);
    s = t;
    c = (c + co) - e;
}

// (double)x on the integer pipe, where a conversion would take the float64 pipe
// as long as an operation; subnormal and non-finite values go the plain way.
static __device__ __noinline__ double widen_plain(float x) { return (double)x; }
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x), e = b & 0x7f800000u, a = b & 0x7fffffffu;
    if (a != 0u && e - 0x00800000u >= 0x7f000000u) return widen_plain(x);
    const unsigned hi = (a >> 3) + (a ? 0x38000000u : 0u);
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29));
}

// a + b = s + e exactly (s the rounded sum).
__device__ __forceinline__ float two_sum(float a, float b, float &e)
{
    const float s = a + b;
    const float bp = s - a;
    e = (a - (s - bp)) + (b - bp);
    return s;
}

// A sum s - (c + d) of float32 (sum, carry) pairs with what the merged carries
// lost, so that merging rounds no more than float64 additions would: to about
// 2^-70 of the sum, where a carry alone keeps 2^-48.  Some 20 float32 operations
// a merge; a float64 addition takes a warp 16 cycles and a conversion as many.
struct Sum3 {
    float s, c, d;
    __device__ __forceinline__ void merge(float so, float co, float dd = 0.f)
    {
        float e, e1, e2;
        s = two_sum(s, so, e);
        c = two_sum(two_sum(c, co, e1), -e, e2);
        d += dd + (e1 + e2);
    }
    __device__ __forceinline__ double value() const { return widen(s) - (widen(c) + widen(d)); }
};

// n (sum, carry) slots `stride` apart, merged in slot order, 16 slots' loads in
// flight (and four merges in the code: unrolled to 16 their instructions took
// longer to arrive than to run).
__device__ __forceinline__ double merge_slots(const float2 *slot, size_t stride, int n)
{
    const float2 f = __ldcg(slot);
    Sum3 a = {f.x, f.y, 0.f};
    for (int q = 1; q < n; q += 16) {
        float2 b[16];
#pragma unroll
        for (int u = 0; u < 16; ++u)
            b[u] = q + u < n ? __ldcg(slot + (size_t)(q + u) * stride) : make_float2(0.f, 0.f);
        const int m = min(4, (n - q + 3) >> 2);
#pragma unroll 1
        for (int r = 0; r < m; ++r) {
#pragma unroll
            for (int u = 0; u < 4; ++u) a.merge(b[u].x, b[u].y);
#pragma unroll
            for (int u = 0; u < 12; ++u) b[u] = b[u + 4];
        }
    }
    double v = a.value();
    if (!isfinite(v)) {  // past float32's range on the way, or a slot is not finite
        v = (double)f.x - (double)f.y;
        for (int q = 1; q < n; ++q) {
            const float2 b = __ldcg(slot + (size_t)q * stride);
            v += (double)b.x - (double)b.y;
        }
    }
    return v;
}

// Sum of n float64 triples `stride` doubles apart in slot order, 24 loads in
// flight.
__device__ __forceinline__ void sum_slots(const double *slot, size_t stride, int n, double (&a)[3])
{
    a[0] = a[1] = a[2] = 0.0;
    for (int q = 0; q < n; q += 8) {
        double b[8][3];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int d = 0; d < 3; ++d)
                b[u][d] = q + u < n ? __ldcg(slot + (size_t)(q + u) * stride + d) : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (q + u < n)
#pragma unroll
                for (int d = 0; d < 3; ++d) a[d] += b[u][d];
    }
}

// Range of j-tiles [t0, t1) handled by split `js` of `nsplit`.
__device__ __forceinline__ void split_range(int ntiles, int nsplit, int js, int &t0, int &t1)
{
    t0 = (int)(((long long)ntiles * js) / nsplit);
    t1 = (int)(((long long)ntiles * (js + 1)) / nsplit);
}

__device__ __forceinline__ bool finite3(double a, double b, double c)
{
    return isfinite(a) && isfinite(b) && isfinite(c);
}

// Tile-local coordinate of a hi/lo packed component.
__device__ __forceinline__ float rel(float hi, float lo, float c) { return (hi - c) + lo; }

// Centre of the bounding box of the CTA's valid i-bodies (every thread gets
// the same value).  red: shared scratch of 6 x (T/32) floats.
template <int T>
__device__ __forceinline__ float3 block_center(float (&mn)[3], float (&mx)[3], float (*red)[T / 32])
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            mn[c] = fminf(mn[c], __shfl_xor_sync(0xffffffffu, mn[c], off));
            mx[c] = fmaxf(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], off));
        }
    }
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            red[c][warp] = mn[c];
            red[3 + c][warp] = mx[c];
        }
    }
    __syncthreads();
    float a[3], b[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        a[c] = red[c][0];
        b[c] = red[3 + c][0];
#pragma unroll
        for (int w = 1; w < T / 32; ++w) {
            a[c] = fminf(a[c], red[c][w]);
            b[c] = fmaxf(b[c], red[3 + c][w]);
        }
    }
    __syncthreads();  // red may be reused by the caller afterwards
    float3 o;
    o.x = a[0] <= b[0] ? 0.5f * (a[0] + b[0]) : 0.f;
    o.y = a[1] <= b[1] ? 0.5f * (a[1] + b[1]) : 0.f;
    o.z = a[2] <= b[2] ? 0.5f * (a[2] + b[2]) : 0.f;
    return o;
}

}  // namespace nb
