// Spatial ordering of bodies for the float32 force kernels.
//
// The float32 pair differences d = x_j - x_i are formed in coordinates
// relative to an origin at the centre of the i-tile (see force_f32.cu).  This
// only helps close pairs when an i-tile is spatially compact, so for large N
// the bodies are processed in Morton (Z-curve) order:
//   1. bounding box of all positions (per-block partials, folded by every
//      block of the next kernel: no atomics, deterministic);
//   2. 24-bit Morton key per body (8 bits per axis over the cube that holds
//      the box);
//   3. stable LSD radix sort of (key, body index), 8 bits per pass: tiles of
//      consecutive keys, one block each, ranked per warp with
//      __match_any_sync, ordered in shared memory and written out in runs;
//      each pass also counts the next pass's digits per destination tile;
//   4. packing in sorted order as float32 hi/lo pairs:
//      P_hi = (fl(x), fl(y), fl(z), fl(m)),
//      P_lo = (fl(x - fl(x)), ..., fl(log2 m) for kernels with log-domain pairs,
//      else 0),
//      or as float64 (x, y, z, m), by the sort's last pass.
// Every step is deterministic, so the order and the forces are reproducible.
#include <cuda_runtime.h>
#include <float.h>

#include "nb_device.cuh"
#include "nb_internal.h"

namespace nb {
namespace {

constexpr int OTPB = 256;
constexpr int MAX_BOX_PARTS = 304;  // box partials, each folded by every block of the next kernel

__device__ __forceinline__ unsigned spread8(unsigned v)
{
    v &= 0xffu;
    v = (v | (v << 8)) & 0x00f00fu;
    v = (v | (v << 4)) & 0x0c30c3u;
    v = (v | (v << 2)) & 0x249249u;
    return v;
}

// Order-preserving 64-bit integer image of a float64 (and back): the boxes'
// minima and maxima are taken on the integer pipe (the float64 pipe has 2
// lanes per clock per SM).
__device__ __forceinline__ long long order_image(double v)
{
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double from_image(long long b)
{
    return __longlong_as_double(b ^ ((b >> 63) & 0x7fffffffffffffffLL));
}
constexpr long long IMAGE_INF = 0x7ff0000000000000LL;  // of +infinity; NaNs lie beyond +-it
constexpr long long IMAGE_MAX = 0x7fefffffffffffffLL;  // of DBL_MAX; ~ gives -DBL_MAX's

// Box of the warp's lanes in every lane: mn, mx of each component.
__device__ __forceinline__ void warp_box(long long (&mn)[3], long long (&mx)[3])
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            mn[c] = min(mn[c], __shfl_xor_sync(0xffffffffu, mn[c], off));
            mx[c] = max(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], off));
        }
    }
}

// Per-block min/max of the positions (NaNs left out), as images:
// parts[b] = {minx,miny,minz,maxx,maxy,maxz}.
__global__ void __launch_bounds__(OTPB) bbox_kernel(int n, const double *__restrict__ pos,
                                                     long long *__restrict__ parts)
{
    __shared__ long long sh[OTPB / 32][6];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    long long mn[3], mx[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        mn[c] = IMAGE_MAX;
        mx[c] = ~IMAGE_MAX;
    }
#pragma unroll 2
    for (int i = blockIdx.x * OTPB + threadIdx.x; i < n; i += gridDim.x * OTPB) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long v = order_image(pos[3 * (size_t)i + c]);
            if (v <= IMAGE_INF && v >= ~IMAGE_INF) {
                mn[c] = min(mn[c], v);
                mx[c] = max(mx[c], v);
            }
        }
    }
    warp_box(mn, mx);
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sh[warp][c] = mn[c];
            sh[warp][3 + c] = mx[c];
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        long long v = sh[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < OTPB / 32; ++w)
            v = threadIdx.x < 3 ? min(v, sh[w][threadIdx.x]) : max(v, sh[w][threadIdx.x]);
        parts[6 * (size_t)blockIdx.x + threadIdx.x] = v;
    }
}

// The box {min x,y,z, max x,y,z} of the partials, folded by every block for
// itself (at most MAX_BOX_PARTS x 48 bytes from L2, ~1 us; a launch of its own
// took as long and its gap more).
__device__ __forceinline__ void fold_box(const long long *__restrict__ parts, int nparts,
                                         double (&box)[6])
{
    __shared__ double sh[6];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < 6) {
        const bool is_min = warp < 3;
        long long v = is_min ? IMAGE_MAX : ~IMAGE_MAX;
#pragma unroll 4
        for (int b = lane; b < nparts; b += 32) {
            const long long p = parts[6 * (size_t)b + warp];
            v = is_min ? min(v, p) : max(v, p);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const long long o = __shfl_xor_sync(0xffffffffu, v, off);
            v = is_min ? min(v, o) : max(v, o);
        }
        if (lane == 0) sh[warp] = from_image(v);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 6; ++c) box[c] = sh[c];
}

// Keys of a tile for the sort's first pass: the tile's digit counts into row
// blockIdx.x of the first pass, the later passes' rows zeroed (each pass adds
// the next one's counts).  key(i) gives body i's key; i is its value.
template <class F>
__device__ __forceinline__ void emit_keys(int n, int tile, int rows, int passes,
                                          unsigned *__restrict__ keys,
                                          unsigned *__restrict__ hist, F &&key)
{
    __shared__ unsigned cnt[256];
    cnt[threadIdx.x] = 0u;
    __syncthreads();
    const int base = blockIdx.x * tile, m = min(tile, n - base);
    for (int q = threadIdx.x; q < m; q += OTPB) {
        const unsigned k = key(base + q);
        keys[base + q] = k;
        atomicAdd(&cnt[k & 255u], 1u);
    }
    __syncthreads();
    hist[(size_t)blockIdx.x * 256 + threadIdx.x] = cnt[threadIdx.x];
    for (int p = 1; p < passes; ++p)
        hist[((size_t)p * rows + blockIdx.x) * 256 + threadIdx.x] = 0u;
}

// Morton keys (8 bits per axis) in the folded box.
__global__ void __launch_bounds__(OTPB) morton_kernel(int n, const double *__restrict__ pos,
                                                       const long long *__restrict__ parts,
                                                       int nparts, int tile, int rows,
                                                       unsigned *__restrict__ keys,
                                                       unsigned *__restrict__ hist)
{
    double box[6];
    fold_box(parts, nparts, box);
    const double ext = fmax(fmax(box[3] - box[0], box[4] - box[1]), box[5] - box[2]);
    const double scale = ext > 0.0 ? 256.0 / ext : 0.0;
    emit_keys(n, tile, rows, 3, keys, hist, [&](int i) {
        unsigned q[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double t = (pos[3 * (size_t)i + c] - box[c]) * scale;
            t = fmin(fmax(t, 0.0), 255.0);
            q[c] = (unsigned)t;
        }
        return spread8(q[0]) | (spread8(q[1]) << 1) | (spread8(q[2]) << 2);
    });
}

__device__ __forceinline__ unsigned spread10(unsigned v)
{
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// floor(t) clamped to [0, 1023], 0 for NaN, from t's bits: comparisons and the
// conversion would take the float64 pipe (2 lanes per clock per SM), which
// bounds the key kernel.
__device__ __forceinline__ unsigned cell1024(double t)
{
    const int hi = __double2hiint(t), e = (hi >> 20) - 1023;  // sign bit set: e < 0
    if (e < 0) return 0u;                                     // t < 1, t negative
    if (hi >= 0x408ff800)                                     // t >= 1023, infinity, NaN
        return hi > 0x7ff00000 || (hi == 0x7ff00000 && __double2loint(t) != 0) ? 0u : 1023u;
    return (unsigned)((hi & 0xfffff) | 0x100000) >> (20 - e);
}

// 30-bit Morton keys for the tree code: q = floor((x - lo) * (1024 / ext)),
// clamped to [0, 1023], with lo the box minimum and ext its longest side, all
// in float64 (the same operations as the tree's cell geometry, so a body's
// key and its cells agree exactly).  Block 0 also stores {lo_x, lo_y, lo_z,
// ext} for the tree kernels.
__global__ void __launch_bounds__(OTPB) morton30_kernel(int n, const double *__restrict__ pos,
                                                         const long long *__restrict__ parts,
                                                         int nparts, int tile, int rows,
                                                         unsigned *__restrict__ keys,
                                                         unsigned *__restrict__ hist,
                                                         double *__restrict__ box_out)
{
    double box[6];
    fold_box(parts, nparts, box);
    double ext = box[3] - box[0];
    if (box[4] - box[1] > ext) ext = box[4] - box[1];
    if (box[5] - box[2] > ext) ext = box[5] - box[2];
    if (!(ext > 0.0)) ext = 1.0;
    const double scale = 1024.0 / ext;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        box_out[0] = box[0];
        box_out[1] = box[1];
        box_out[2] = box[2];
        box_out[3] = ext;
    }
    emit_keys(n, tile, rows, 4, keys, hist, [&](int i) {
        unsigned q[3];
#pragma unroll
        for (int c = 0; c < 3; ++c)
            q[c] = cell1024(__dmul_rn(__dsub_rn(pos[3 * (size_t)i + c], box[c]), scale));
        return spread10(q[0]) | (spread10(q[1]) << 1) | (spread10(q[2]) << 2);
    });
}

// Keys of a plain integer sort: k32[i] or k64[i] (values below 2^31).
__global__ void __launch_bounds__(OTPB) key_init_kernel(int n, const int *__restrict__ k32,
                                                         const long long *__restrict__ k64,
                                                         int tile, int rows, int passes,
                                                         unsigned *__restrict__ keys,
                                                         unsigned *__restrict__ hist)
{
    emit_keys(n, tile, rows, passes, keys, hist,
              [&](int i) { return k32 ? (unsigned)k32[i] : (unsigned)k64[i]; });
}

// Per digit: exclusive scan of its counts over the tiles (rows), in place, and
// the digit's total.  A block takes 32 digits (a lane each), its 32 warps a
// range of rows each.
__global__ void __launch_bounds__(1024) radix_rows_kernel(unsigned *__restrict__ hist, int rows,
                                                          unsigned *__restrict__ total)
{
    __shared__ unsigned ws[32][33];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int d = blockIdx.x * 32 + lane;
    const int per = (rows + 31) / 32, r0 = min(rows, warp * per), r1 = min(rows, r0 + per);
    unsigned v = 0u;
#pragma unroll 8
    for (int r = r0; r < r1; ++r) v += hist[(size_t)r * 256 + d];
    ws[warp][lane] = v;
    __syncthreads();
    unsigned run = 0u, all = 0u;
#pragma unroll
    for (int w = 0; w < 32; ++w) {
        if (w == warp) run = all;
        all += ws[w][lane];
    }
    if (warp == 0) total[d] = all;
#pragma unroll 8
    for (int r = r0; r < r1; ++r) {
        const unsigned c = hist[(size_t)r * 256 + d];
        hist[(size_t)r * 256 + d] = run;
        run += c;
    }
}

// Exclusive scan over the block's 256 threads.
__device__ __forceinline__ unsigned scan256(unsigned v, unsigned (&ws)[OTPB / 32])
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    unsigned below = 0u;
#pragma unroll
    for (int w = 0; w < OTPB / 32; ++w)
        if (w < warp) below += ws[w];
    __syncthreads();  // ws may be reused
    return below + incl - v;
}

// Body i packed at slot k: float32 hi/lo pairs, or float64, or not at all.
__device__ __forceinline__ void put_body(const SortedPack &p, size_t k, int i)
{
    if (p.Phi) {
        const double *x = p.pos + 3 * (size_t)i;
        const double m = p.mass[i];
        float4 h, l;
        split_f64(x[0], h.x, l.x);
        split_f64(x[1], h.y, l.y);
        split_f64(x[2], h.z, l.z);
        h.w = (float)m;
        l.w = p.logm ? log2_packed(m) : 0.f;
        p.Phi[k] = h;
        p.Plo[k] = l;
    } else if (p.P64) {
        const double *x = p.pos + 3 * (size_t)i;
        p.P64[k] = make_double4(x[0], x[1], x[2], p.mass[i]);
    }
}

struct SortPass {
    int n, rows, shift;
    const unsigned *kin;
    const int *vin;          // NULL: the value is the index (first pass)
    unsigned *kout;          // NULL: the sorted keys are not wanted
    int *vout;
    const unsigned *hist;    // this pass's counts, [rows][256]
    const unsigned *total;   // digit totals when radix_rows_kernel scanned hist, else NULL
    unsigned *next;          // the next pass's counts, NULL in the last one
    SortedPack pack;         // last pass: the bodies packed in sorted order
};

// One tile of one pass.  What bounds it at a tree's sizes (2^14 to 2^20 keys,
// all in L2) is latency and the number of blocks: a warp ranks 32 keys at a
// time with __match_any_sync against its own counters (stable: warps, rounds
// and lanes are in key order), the tile is put in order in shared memory and
// written in runs.  Up to SORT_SELF_ROWS tiles every block sums the tiles'
// counts for itself; beyond, radix_rows_kernel has.  Against warps that took
// 2048 keys each (2 to 64 blocks; two scan launches per pass, packing in a
// launch of its own) a tree evaluation takes 2413 us instead of 2822 for four
// steps of 20000 bodies, 4282 instead of 4408 at 2^20 bodies; the order itself
// 106 us less at 16384 bodies, all with the same results.
template <int IPT>
__global__ void __launch_bounds__(OTPB) radix_scatter_kernel(const SortPass a)
{
    constexpr int TILE = OTPB * IPT, NW = OTPB / 32;
    __shared__ __align__(16) unsigned cnt[NW][256];
    __shared__ unsigned skey[TILE];
    __shared__ int sval[TILE];
    __shared__ unsigned gofs[256];
    __shared__ unsigned ws[NW];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = threadIdx.x;
    const unsigned lt = (1u << lane) - 1u;
    const int tile0 = blockIdx.x * TILE, m = min(TILE, a.n - tile0);
    const int wbase = warp * 32 * IPT;  // this warp's first key in the tile

    unsigned k[IPT];
    int v[IPT], rank[IPT];
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int q = wbase + 32 * r + lane;
        k[r] = q < m ? a.kin[tile0 + q] : 0u;
        v[r] = q < m ? (a.vin ? a.vin[tile0 + q] : tile0 + q) : 0;
    }
    // counts of digit t before this tile, and in all tiles
    unsigned pre, tot;
    if (a.total) {
        pre = a.hist[(size_t)blockIdx.x * 256 + t];
        tot = a.total[t];
    } else {
        uint4 s4 = make_uint4(0u, 0u, 0u, 0u), p4 = s4;
        const uint4 *h4 = reinterpret_cast<const uint4 *>(a.hist);
#pragma unroll 8
        for (int r = t >> 6; r < a.rows; r += OTPB / 64) {
            const uint4 c = h4[(size_t)r * 64 + (t & 63)];
            s4.x += c.x; s4.y += c.y; s4.z += c.z; s4.w += c.w;
            if (r < (int)blockIdx.x) {
                p4.x += c.x; p4.y += c.y; p4.z += c.z; p4.w += c.w;
            }
        }
        uint4 *c4 = reinterpret_cast<uint4 *>(&cnt[0][0]);  // rows 0..3 all tiles, 4..7 before
        c4[t] = s4;
        c4[OTPB + t] = p4;
        __syncthreads();
        tot = cnt[0][t] + cnt[1][t] + cnt[2][t] + cnt[3][t];
        pre = cnt[4][t] + cnt[5][t] + cnt[6][t] + cnt[7][t];
        __syncthreads();
    }
#pragma unroll
    for (int w = 0; w < NW; ++w) cnt[w][t] = 0u;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const bool valid = wbase + 32 * r + lane < m;
        const unsigned d = valid ? ((k[r] >> a.shift) & 255u) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        rank[r] = valid ? (int)(cnt[warp][d] + __popc(peers & lt)) : 0;
        __syncwarp();
        if (valid && (peers & lt) == 0u) cnt[warp][d] += (unsigned)__popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {  // digit t: each warp's first place in the ordered tile, and the way from there to the output
        unsigned run = 0u;
#pragma unroll
        for (int w = 0; w < NW; ++w) run += cnt[w][t];
        unsigned place = scan256(run, ws);
        gofs[t] = scan256(tot, ws) + pre - place;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const unsigned c = cnt[w][t];
            cnt[w][t] = place;
            place += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        if (wbase + 32 * r + lane < m) {
            const unsigned q = cnt[warp][(k[r] >> a.shift) & 255u] + (unsigned)rank[r];
            skey[q] = k[r];
            sval[q] = v[r];
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int q = t; q < m; q += OTPB) {
        const unsigned key = skey[q];
        const int i = sval[q];
        const unsigned off = gofs[(key >> a.shift) & 255u] + (unsigned)q;
        if (a.kout) a.kout[off] = key;
        a.vout[off] = i;
        if (a.next)
            atomicAdd(a.next + (size_t)(off / TILE) * 256 + ((key >> (a.shift + 8)) & 255u), 1u);
        else
            put_body(a.pack, off, i);
    }
}

__global__ void __launch_bounds__(OTPB) pack_hilo_kernel(int n, const SortedPack p)
{
    for (int k = blockIdx.x * OTPB + threadIdx.x; k < n; k += gridDim.x * OTPB) put_body(p, k, k);
}

inline int grid_for(int n)
{
    int g = (n + OTPB - 1) / OTPB;
    return g < 1 ? 1 : (g > 4096 ? 4096 : g);
}

// Tiles of the sort: small ones up to 2^16 keys, so that a few thousand keys
// still spread over many blocks; up to SORT_SELF_ROWS tiles sum each other's
// counts themselves (a block reads 1 KB per tile: above 64 tiles that costs
// more than the launch that scans them).
constexpr int SORT_SMALL = 4, SORT_LARGE = 16, SORT_SMALL_N = 1 << 16, SORT_SELF_ROWS = 64;
inline int sort_ipt(int n) { return n <= SORT_SMALL_N ? SORT_SMALL : SORT_LARGE; }
inline int sort_rows(int n)
{
    const int tile = OTPB * sort_ipt(n);
    return (n + tile - 1) / tile;
}

// Passes 0..passes-1 over the keys in o.keys[0] (their counts for the first
// pass in o.hist): the order into perm_out, the sorted keys (if wanted) into
// o.keys[passes & 1].
void sort_passes(cudaStream_t s, int n, int passes, OrderScratch &o, int *perm_out, bool want_keys,
                 const SortedPack &pack, int &kernels)
{
    const int rows = sort_rows(n);
    unsigned *total = o.hist + (size_t)passes * rows * 256;
    int cur = 0;
    for (int pass = 0; pass < passes; ++pass) {
        const bool last = pass == passes - 1;
        unsigned *hist = o.hist + (size_t)pass * rows * 256;
        SortPass a;
        a.n = n;
        a.rows = rows;
        a.shift = 8 * pass;
        a.kin = o.keys[cur];
        a.vin = pass == 0 ? nullptr : o.vals[cur];
        a.kout = last && !want_keys ? nullptr : o.keys[cur ^ 1];
        a.vout = last ? perm_out : o.vals[cur ^ 1];
        a.hist = hist;
        a.total = nullptr;
        a.next = last ? nullptr : hist + (size_t)rows * 256;
        a.pack = pack;
        if (rows > SORT_SELF_ROWS) {
            radix_rows_kernel<<<8, 1024, 0, s>>>(hist, rows, total);
            ++kernels;
            a.total = total;
        }
        if (sort_ipt(n) == SORT_SMALL)
            radix_scatter_kernel<SORT_SMALL><<<rows, OTPB, 0, s>>>(a);
        else
            radix_scatter_kernel<SORT_LARGE><<<rows, OTPB, 0, s>>>(a);
        ++kernels;
        cur ^= 1;
    }
}

inline int box_parts(int n)
{
    const int g = grid_for(n);
    return g < MAX_BOX_PARTS ? g : MAX_BOX_PARTS;
}

}  // namespace

size_t sort_hist_entries(int n)
{
    // 256 counts per tile for each of at most 4 passes, then the digit totals;
    // fewer bodies than n may make up to 64 of the small tiles
    const size_t large = ((size_t)n + OTPB * SORT_LARGE - 1) / (OTPB * SORT_LARGE);
    const size_t rows = large > 64 ? large : 64;
    return (4 * rows + 1) * 256;
}

cudaError_t launch_morton_sort(cudaStream_t s, int n, const double *pos, OrderScratch &o,
                               int *perm_out, const SortedPack &pack, int &kernels)
{
    kernels = 0;
    if (n <= 0) return cudaSuccess;
    const int nparts = box_parts(n), rows = sort_rows(n);
    bbox_kernel<<<nparts, OTPB, 0, s>>>(n, pos, o.box);
    morton_kernel<<<rows, OTPB, 0, s>>>(n, pos, o.box, nparts, OTPB * sort_ipt(n), rows, o.keys[0],
                                        o.hist);
    kernels += 2;
    sort_passes(s, n, 3, o, perm_out, false, pack, kernels);
    return cudaGetLastError();
}

cudaError_t launch_tree_sort(cudaStream_t s, int n, const double *pos, OrderScratch &o,
                             int *perm_out, double *box_out, const SortedPack &pack, int &kernels)
{
    kernels = 0;
    if (n <= 0) return cudaSuccess;
    const int nparts = box_parts(n), rows = sort_rows(n);
    bbox_kernel<<<nparts, OTPB, 0, s>>>(n, pos, o.box);
    morton30_kernel<<<rows, OTPB, 0, s>>>(n, pos, o.box, nparts, OTPB * sort_ipt(n), rows,
                                          o.keys[0], o.hist, box_out);
    kernels += 2;
    sort_passes(s, n, 4, o, perm_out, true, pack, kernels);  // sorted keys end in keys[0]
    return cudaGetLastError();
}

cudaError_t launch_key_sort(cudaStream_t s, int n, const int *k32, const long long *k64,
                            int passes, OrderScratch &o, int *perm_out, int &kernels)
{
    kernels = 0;
    if (n <= 0) return cudaSuccess;
    const int rows = sort_rows(n);
    key_init_kernel<<<rows, OTPB, 0, s>>>(n, k32, k64, OTPB * sort_ipt(n), rows, passes, o.keys[0],
                                          o.hist);
    ++kernels;
    sort_passes(s, n, passes, o, perm_out, false, SortedPack{}, kernels);
    return cudaGetLastError();
}

cudaError_t launch_pack_hilo(cudaStream_t s, int n, const double *pos, const double *mass,
                             float4 *Phi, float4 *Plo, bool logm)
{
    if (n <= 0) return cudaSuccess;
    pack_hilo_kernel<<<grid_for(n), OTPB, 0, s>>>(n, SortedPack{pos, mass, Phi, Plo, nullptr, logm});
    return cudaGetLastError();
}

}  // namespace nb
