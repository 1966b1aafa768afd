// The float32 pair sum (force_f32.cuh: the same pair terms, tile-local hi/lo
// coordinates and compensated sums) for systems too small to fill the chip
// with one thread per body or two.
//
// What bounds such a call is not arithmetic (4096 bodies are 1.7e7 pairs, 6 us
// of the FP32 pipe; 1000 bodies 0.4 us) but how many warps share it and the
// steps around it.  So a block's eight warps all keep the same 32 I bodies (I
// per lane) and take an eighth of the block's j range each, alone: a warp
// stages 32 j-bodies at a time in its own shared memory, with no block barrier
// in the loop.  Up to eight blocks of a thread-block cluster share one i-tile
// and split the j range further; their sums meet in distributed shared memory
// (added in rank order) instead of global partials, a fence and an arrival
// counter.  For the smallest systems the bodies are read straight from the
// caller's float64 arrays (RAW), packed the same way in registers, which saves
// the packing launch.
#include <cooperative_groups.h>

#include "force_f32.cuh"

namespace nb {
namespace {

namespace cg = cooperative_groups;

constexpr int TEAM_T = 256, TEAM_W = TEAM_T / 32;
constexpr int TEAM_FOLD = 128;  // j-bodies per compensated fold

// Body j as hi/lo pairs, from the packed arrays or (the same values) from float64.
template <bool RAW>
__device__ __forceinline__ void team_load(const ForceParams &p, int j, bool ok, float4 &h, float4 &l)
{
    if (!ok) {
        h = far_body(0.f);
        l = make_float4(0.f, 0.f, 0.f, 0.f);
    } else if (RAW) {
        const double *x = p.pos + 3 * (size_t)j;
        const double a = __ldg(x), b = __ldg(x + 1), c = __ldg(x + 2);
        split_f64(a, h.x, l.x);
        split_f64(b, h.y, l.y);
        split_f64(c, h.z, l.z);
        h.w = (float)__ldg(p.mass + j);
        l.w = 0.f;
    } else {
        h = __ldg(static_cast<const float4 *>(p.P) + j);
        l = __ldg(p.Plo + j);
    }
}

// float32 values as integers in the same order, and back.
__device__ __forceinline__ int ordered(float x)
{
    const int b = __float_as_int(x);
    return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float from_ordered(int b)
{
    return __int_as_float(b ^ ((b >> 31) & 0x7fffffff));
}

// The warps' own sums of one value, `stride` apart, in float64 over the cluster's
// blocks (as in merge_slots: a merged sum that is not finite; rolled up, for its
// instructions, unrolled, made a launch of 256 bodies 0.3 us longer).
__device__ __forceinline__ double sum64(float2 *mine, int stride, int cs)
{
    double t = 0.0;
#pragma unroll 1
    for (int r = 0; r < cs; ++r) {
        const float2 *s = cs > 1 ? cg::this_cluster().map_shared_rank(mine, r) : mine;
#pragma unroll 1
        for (int w = 0; w < TEAM_W; ++w) t += pair_value(s[w * stride]);
    }
    return t;
}

template <int I, bool COMP, bool ZEPS, bool RAW>
__global__ void __launch_bounds__(TEAM_T) force_f32_team_kernel(const ForceParams p)
{
    constexpr int NP = I / 2, TI = 32 * I, NV = 3 * TI;
    __shared__ __align__(16) float4 tile[TEAM_W][2 * 32];
    __shared__ float2 sums[TEAM_W][NV];  // (sum, carry) pairs
    __shared__ float2 total[NV];
    __shared__ int2 box[3][TEAM_W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cs = p.nsplit;  // blocks of the cluster
    const int rank = blockIdx.x % cs, i0 = blockIdx.x / cs * TI;
    const int n = p.n;
    const int part = rank * TEAM_W + warp, parts = cs * TEAM_W;
    const int j0 = (int)((long long)n * part / parts), j1 = (int)((long long)n * (part + 1) / parts);

    // the first j-bodies' loads overlap the i-bodies'
    float4 bh, bl;
    team_load<RAW>(p, j0 + lane, j0 + lane < j1, bh, bl);
    float4 h[I], l[I];
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const int i = i0 + lane + 32 * k;
        team_load<RAW>(p, i, i < n, h[k], l[k]);
    }
    // The origin: the centre of the bounding box of the 256 bodies around the
    // tile (512 from 2048 bodies on with compensated sums), as if they shared a
    // block of one or two bodies per thread.  A pair's term is then bit for bit
    // the same in both kinds of kernel and only the order of the sums differs,
    // so a trajectory does not depend on which of them a size is given.  (The
    // mean of the tile's own bodies is a better origin, 6.4e-7 of |a| where this
    // gives 1.0e-6 at 1000 bodies; the box of 64 bodies a worse one, 1.6e-6.)
    const int around = COMP && n >= 2048 ? 512 : 256;
    const int o0 = i0 & ~(around - 1);
    int lo_[3], hi_[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) lo_[d] = 0x7fffffff, hi_[d] = (int)0x80000000;
    for (int i = o0 + threadIdx.x; i < min(n, o0 + around); i += TEAM_T) {
        float4 a, b;
        team_load<RAW>(p, i, true, a, b);
        const int v[3] = {ordered(a.x), ordered(a.y), ordered(a.z)};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            lo_[d] = min(lo_[d], v[d]);
            hi_[d] = max(hi_[d], v[d]);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        lo_[d] = __reduce_min_sync(0xffffffffu, lo_[d]);
        hi_[d] = __reduce_max_sync(0xffffffffu, hi_[d]);
        if (lane == 0) box[d][warp] = make_int2(lo_[d], hi_[d]);
    }
    __syncthreads();
    float cc[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int2 b = box[d][lane % TEAM_W];
        cc[d] = 0.5f * (from_ordered(__reduce_min_sync(0xffffffffu, b.x)) +
                        from_ordered(__reduce_max_sync(0xffffffffu, b.y)));
    }
    const float3 c = make_float3(cc[0], cc[1], cc[2]);
    float2 nx[NP], ny[NP], nz[NP], ax[NP], ay[NP], az[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const float4 a = h[2 * q], b = h[2 * q + 1], al = l[2 * q], b2 = l[2 * q + 1];
        nx[q] = make_float2(-rel(a.x, al.x, c.x), -rel(b.x, b2.x, c.x));
        ny[q] = make_float2(-rel(a.y, al.y, c.y), -rel(b.y, b2.y, c.y));
        nz[q] = make_float2(-rel(a.z, al.z, c.z), -rel(b.z, b2.z, c.z));
        ax[q] = ay[q] = az[q] = make_float2(0.f, 0.f);
    }
    float s[3][I], e[3][I];
#pragma unroll
    for (int k = 0; k < I; ++k)
#pragma unroll
        for (int d = 0; d < 3; ++d) s[d][k] = e[d][k] = 0.f;
    auto fold = [&]() {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            kahan_add(s[0][2 * q], e[0][2 * q], ax[q].x);
            kahan_add(s[0][2 * q + 1], e[0][2 * q + 1], ax[q].y);
            kahan_add(s[1][2 * q], e[1][2 * q], ay[q].x);
            kahan_add(s[1][2 * q + 1], e[1][2 * q + 1], ay[q].y);
            kahan_add(s[2][2 * q], e[2][2 * q], az[q].x);
            kahan_add(s[2][2 * q + 1], e[2][2 * q + 1], az[q].y);
            ax[q] = ay[q] = az[q] = make_float2(0.f, 0.f);
        }
    };
    const float2 e2 = make_float2(p.eps2f, p.eps2f);
    float4 *t = tile[warp];
    constexpr int UNR = 8;
    int since = 0;  // j-bodies since the last fold
    for (int jb = j0; jb < j1; jb += 32) {
        const float x = rel(bh.x, bl.x, c.x), y = rel(bh.y, bl.y, c.y), z = rel(bh.z, bl.z, c.z);
        __syncwarp();  // the last tile has been read
        t[2 * lane] = make_float4(x, x, y, y);
        t[2 * lane + 1] = make_float4(z, z, bh.w, bh.w);  // past the end: massless
        __syncwarp();
        const int jn = jb + 32 + lane;
        team_load<RAW>(p, jn, jn < j1, bh, bl);
        const int cnt = min(32, j1 - jb);
        for (int q = 0; q < cnt; q += UNR) {
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                const float4 q0 = t[2 * (q + u)], q1 = t[2 * (q + u) + 1];
                const float2 xj = make_float2(q0.x, q0.y), yj = make_float2(q0.z, q0.w);
                const float2 zj = make_float2(q1.x, q1.y), mj = make_float2(q1.z, q1.w);
#pragma unroll
                for (int r = 0; r < NP; ++r)
                    interact2<ZEPS, false>(xj, yj, zj, mj, e2, nx[r], ny[r], nz[r], ax[r], ay[r],
                                           az[r]);
            }
        }
        if (COMP && (since += 32) == TEAM_FOLD) {
            fold();
            since = 0;
        }
    }
    if (COMP) fold();
#pragma unroll
    for (int k = 0; k < I; ++k) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float2 a = d == 0 ? ax[k >> 1] : (d == 1 ? ay[k >> 1] : az[k >> 1]);
            sums[warp][d * TI + 32 * k + lane] =
                COMP ? make_float2(s[d][k], e[d][k]) : make_float2((k & 1) ? a.y : a.x, 0.f);
        }
    }
    __syncthreads();
    // the warps' sums in warp order, then the blocks' in rank order (float32
    // two-sums, to 2^-48 of the sum: eight float64 sums per value held the float64
    // pipe 3000 cycles, and Sum3 made a step of 4096 bodies 0.9 us longer; the
    // errors against float64, 1e-7 from the pair terms, are 1 to 13 % below those
    // of the block kernels with float64 merges at 64 to 8191 bodies)
    for (int v = threadIdx.x; v < NV; v += TEAM_T) {
        float2 a = sums[0][v];
#pragma unroll
        for (int w = 1; w < TEAM_W; ++w) kahan_merge(a.x, a.y, sums[w][v].x, sums[w][v].y);
        total[v] = a;
    }
    cg::cluster_group cluster = cg::this_cluster();
    if (cs > 1)
        cluster.sync();
    else
        __syncthreads();
    const int v0 = NV * rank / cs, v1 = NV * (rank + 1) / cs;
    for (int v = v0 + threadIdx.x; v < v1; v += TEAM_T) {
        float2 b[8];
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (r < cs) b[r] = cs > 1 ? *cluster.map_shared_rank(total + v, r) : total[v];
#pragma unroll
        for (int r = 1; r < 8; ++r)
            if (r < cs) kahan_merge(b[0].x, b[0].y, b[r].x, b[r].y);
        const int d = v / TI, k = i0 + v % TI;
        if (k < n) {
            const int i = p.perm ? p.perm[k] : k;
            double a = p.G * pair_value(b[0]);
            if (!isfinite(a)) {
                a = p.G * sum64(&sums[0][v], NV, cs);
                if (!isfinite(a)) atomicOr(p.err, ERR_NONFINITE);
            }
            p.acc[3 * (size_t)i + d] = a;
            if (p.vel) p.vel[3 * (size_t)i + d] += p.half_dt * a;
        }
    }
    if (cs > 1) cluster.sync();  // no block leaves while its sums are being read
}

// (the block's warps stage 32 j-bodies each)
// (j-tile: 32 bodies staged by each warp)
#define NB_TEAM_KERNEL(I, C, Z)                                                             \
    {TEAM_T, I, 32 * TEAM_W, (const void *)force_f32_team_kernel<I, C, Z, false>, false, 0, \
     (const void *)force_f32_team_kernel<I, C, Z, true>}
#define NB_TEAM_ENTRY(I)                                                                   \
    {{NB_TEAM_KERNEL(I, false, false), NB_TEAM_KERNEL(I, false, true)},                     \
     {NB_TEAM_KERNEL(I, true, false), NB_TEAM_KERNEL(I, true, true)}}

const Quad kTeam[] = {NB_TEAM_ENTRY(2), NB_TEAM_ENTRY(4)};

}  // namespace

int f32_team_variants() { return (int)(sizeof(kTeam) / sizeof(kTeam[0])); }
const KernelEntry &f32_team_kernel(int v, bool comp, bool zeps) { return kTeam[v][comp][zeps]; }

}  // namespace nb
