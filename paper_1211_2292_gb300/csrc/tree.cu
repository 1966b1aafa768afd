// Barnes-Hut tree code on the GPU (paper Sec. IV-A): the bodies are placed
// in an octree by recursive 8-way division of space until a cell holds few
// enough bodies; the force on a body is the sum over the cells that are
// distant enough (as their total mass at their centre of mass) and over the
// bodies of the nearby leaves.
//
// Readings (the paper gives no opening rule, threshold or grouping):
//  * space is the cube at the bodies' box minimum with edge `ext`, the
//    longest box side; a body's cell at level L is the top 3L bits of its
//    30-bit Morton key (order.cu: launch_tree_sort);
//  * a cell is a leaf when it holds at most `leaf_cap` bodies or is at
//    level 10;
//  * bodies are taken 32 or 64 at a time in key order (one warp per
//    group); a cell is used as a monopole only when it is distant enough
//    from every body of the group: distance from the body to the cell's
//    cube >= edge / theta, computed in float32 with the same operations as
//    the oracle (no contraction), so both take the same decisions;
//  * cell moments are float64 (mass, centre of mass).
//
// Build (all on the device, no host synchronisation, so it can be captured
// in a graph): the sorted keys alone say which nodes start at which body; one
// launch counts them per level and block of bodies, one numbers and writes
// them (level by level, children consecutive in octant order), one sums the
// moments bottom-up.
//
// Walk arithmetic: float32 pair terms in coordinates relative to the
// group's centre (hi/lo packed positions and centres of mass, as in the
// direct-sum kernel), float32 partial sums over every NB_WALK_FOLD_EVERY
// flushes of FLUSH listed sources folded into Kahan (sum, carry) pairs.
#include <cuda_runtime.h>
#include <float.h>

#include <algorithm>

#include "nb_device.cuh"
#include "nb_internal.h"

namespace nb {
namespace {

constexpr int TTPB = 256;
// Walk launch shape: warps per block, and the resident blocks per SM the
// register allocation is sized for (one and two bodies per lane).
#ifndef NB_WALK_WARPS
#define NB_WALK_WARPS 4
#endif
#ifndef NB_WALK_MINB1
#define NB_WALK_MINB1 8
#endif
#ifndef NB_WALK_MINB2
#define NB_WALK_MINB2 5
#endif
constexpr int WALK_WARPS = NB_WALK_WARPS;
constexpr int LEVELS = 11;

enum { META_COUNT = 0, META_BASE = 12, META_QUEUE = 25, META_INTS = 32 };
static_assert(META_COUNT == TREE_META_COUNT && META_BASE == TREE_META_BASE &&
                  META_QUEUE == TREE_META_QUEUE, "meta layout shared with nb_internal.h");

inline int grid_cap(int64_t work)
{
    int64_t g = (work + TTPB - 1) / TTPB;
    return (int)(g < 1 ? 1 : (g > 4096 ? 4096 : g));
}

// 2^-L exactly (0 <= L <= 10), from its bit pattern.
__device__ __forceinline__ double pow2_neg(int L)
{
    return __longlong_as_double((long long)(1023 - L) << 52);
}

// Float32 cube of the level-L cell with key prefix `pre`, exactly as the
// oracle forms it (float64 lo + edge * index, rounded).
__device__ __forceinline__ void cube_corners(const double *__restrict__ box, int L, unsigned pre,
                                             float4 &lo4, float4 &hi4)
{
    unsigned ic[3] = {0u, 0u, 0u};
    for (int bb = 0; bb < L; ++bb) {
        const unsigned trip = (pre >> (3 * bb)) & 7u;
#pragma unroll
        for (int c = 0; c < 3; ++c) ic[c] |= ((trip >> c) & 1u) << bb;
    }
    // ext / 2^L: the product with the exact power 2^-L rounds the same real
    // value as the quotient, so it is the same number, without a division
    const double cell = __dmul_rn(box[3], pow2_neg(L));
    float blo[3], bhi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        blo[c] = (float)__dadd_rn(box[c], __dmul_rn(cell, (double)ic[c]));
        bhi[c] = (float)__dadd_rn(box[c], __dmul_rn(cell, (double)(ic[c] + 1u)));
    }
    lo4 = make_float4(blo[0], blo[1], blo[2], 0.f);
    hi4 = make_float4(bhi[0], bhi[1], bhi[2], 0.f);
}

// ------------------------------------------------------------------ build
// The nodes follow from the sorted keys alone.  With lcp(a, b) the number of
// leading octants two keys share (10 when equal), a cell of level L starts at
// body i when L > lcp(key[i-1], key[i]); it is a node when its parent holds
// more than leaf_cap bodies, and a leaf when it does not itself, or L = 10.
// So the nodes that start at body i are those of levels lo..hi:
//   lo = lcp(key[i-1], key[i]) + 1 (0 for i = 0), and with
//   D = lcp(key[i], key[i+leaf_cap]) (the deepest cell from i on that holds
//   more than leaf_cap): hi = min(10, D + 1) when D >= lo, else hi = lo when
//   the cell of level lo - 1 around i holds more than leaf_cap (the root
//   always is a node), else none.
// A node's number is its rank by (level, start), which one scan of the
// (level, block of bodies) counts and ballots within the block give; children
// are consecutive in octant order.  It ends where the next cell of its level
// starts: in the warp's ballot, else at the first one of a later warp, or of a
// later block (searching the keys for it, by doubling steps, was 14 of the
// build's 85 us at 20000 bodies and 64 us at 2^20).
//
// Two launches over the bodies (count, write) took the place of three launches
// per level (octant boundaries by binary search, one block's scan, children
// written), which were 30 launches of 3 to 10 us at any size.  With the moments
// below: four tree steps of 20000 bodies 2413 -> 1939 us, a tree evaluation of
// 2^20 bodies 4282 -> 3911 us, the same results to the bit.
__device__ __forceinline__ int key_lcp(unsigned a, unsigned b)
{
    return (__clz(a ^ b) - 2) / 3;  // 30-bit keys; 10 when equal
}

constexpr int BUILD_BLOCKS = 592;  // blocks of bodies at most: each sums the others' counts

// Per body, lv[i] = lo | hi << 4 (hi < lo: no node starts there; lo is the
// shallowest level whose cell starts at i, 11 for none), and per block and
// level how many nodes start, tab[L * nblk + b], and the first body a cell
// starts at, tab[(LEVELS + L) * nblk + b] (n for none).
__global__ void __launch_bounds__(TTPB) tree_levels_kernel(TreeView t, int n,
                                                           const unsigned *__restrict__ keys,
                                                           int leaf_cap, int chunk,
                                                           unsigned char *__restrict__ lv,
                                                           int *__restrict__ tab)
{
    __shared__ int wsum[TTPB / 32][LEVELS], wfirst[TTPB / 32][LEVELS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (blockIdx.x == 0) {
        if (threadIdx.x < META_INTS) t.meta[threadIdx.x] = 0;
        if (threadIdx.x < 4) t.stats[threadIdx.x] = 0ull;
    }
    const int b0 = blockIdx.x * chunk, b1 = min(n - b0, chunk) + b0;
    int mine = 0, first = n;  // lane L: nodes of level L, the first cell start
    for (int r = b0; r < b1; r += TTPB) {
        const int i = r + threadIdx.x;
        int lo = 11, hi = 0;
        if (i < b1) {
            const unsigned k = keys[i];
            lo = i == 0 ? 0 : key_lcp(keys[i - 1], k) + 1;
            const int D = n - i > leaf_cap ? key_lcp(k, keys[i + leaf_cap]) : -1;
            if (lo > 10) {
                hi = 0;  // the same cell as the body before at every level
            } else if (D >= lo) {
                hi = min(10, D + 1);
            } else if (lo == 0) {
                hi = 0;
            } else {
                // the parent's start, if within leaf_cap bodies before i
                const int sh = 3 * (11 - lo);
                const unsigned pre = k >> sh;
                int a = max(0, i - leaf_cap), b = i;
                while (a < b) {
                    const int mid = (a + b) >> 1;
                    if ((keys[mid] >> sh) < pre)
                        a = mid + 1;
                    else
                        b = mid;
                }
                const bool over = n - a > leaf_cap && (keys[a + leaf_cap] >> sh) == pre;
                hi = over ? lo : lo - 1;
            }
            lv[i] = (unsigned char)(lo | (hi << 4));
        }
#pragma unroll
        for (int L = 0; L < LEVELS; ++L) {
            const unsigned b = __ballot_sync(0xffffffffu, lo <= L && L <= hi);
            const unsigned st = __ballot_sync(0xffffffffu, lo <= L);
            if (lane == L) {
                mine += __popc(b);
                if (st) first = min(first, r + 32 * warp + __ffs(st) - 1);
            }
        }
    }
    if (lane < LEVELS) {
        wsum[warp][lane] = mine;
        wfirst[warp][lane] = first;
    }
    __syncthreads();
    if (threadIdx.x < LEVELS) {
        int s = 0, f = n;
#pragma unroll
        for (int w = 0; w < TTPB / 32; ++w) {
            s += wsum[w][threadIdx.x];
            f = min(f, wfirst[w][threadIdx.x]);
        }
        tab[threadIdx.x * gridDim.x + blockIdx.x] = s;
        tab[(LEVELS + threadIdx.x) * gridDim.x + blockIdx.x] = f;
    }
}

__global__ void __launch_bounds__(TTPB) tree_emit_kernel(TreeView t, int n,
                                                         const unsigned *__restrict__ keys,
                                                         int chunk,
                                                         const unsigned char *__restrict__ lv,
                                                         const int *__restrict__ tab, int *err)
{
    __shared__ int tot[LEVELS], run[LEVELS], nxt[LEVELS], top_s;
    __shared__ int wcnt[TTPB / 32][LEVELS], woff[TTPB / 32][LEVELS], wnext[TTPB / 32][LEVELS];
    __shared__ unsigned bal[TTPB / 32][LEVELS], stt[TTPB / 32][LEVELS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nblk = gridDim.x;
    const unsigned lt = (1u << lane) - 1u;
    for (int L = warp; L < LEVELS; L += TTPB / 32) {
        int all = 0, pre = 0, next = n;  // in all blocks, up to this one's end; the next cell start
#pragma unroll 4
        for (int b = lane; b < nblk; b += 32) {
            const int c = tab[L * nblk + b], f = tab[(LEVELS + L) * nblk + b];
            all += c;
            if (b <= (int)blockIdx.x)
                pre += c;
            else
                next = min(next, f);
        }
        all = __reduce_add_sync(0xffffffffu, all);
        pre = __reduce_add_sync(0xffffffffu, pre);
        next = __reduce_min_sync(0xffffffffu, next);
        if (lane == 0) {
            tot[L] = all;
            run[L] = pre;
            nxt[L] = next;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // The levels' first nodes.  Past the capacity (never, with
        // tree_node_bound) the tree stops a level early: the nodes of the last
        // level that fits become leaves, and the flag is raised.
        int base = 0, top = LEVELS - 1;
        for (int L = 0; L < LEVELS; ++L) {
            if (L <= top && tot[L] > t.cap - base) {
                top = L - 1;
                if (blockIdx.x == 0) atomicOr(err, ERR_TREE);
            }
            const int c = L <= top ? tot[L] : 0;
            if (blockIdx.x == 0) {
                t.meta[META_BASE + L] = base;
                t.meta[META_COUNT + L] = c;
            }
            run[L] += base;
            base += c;
        }
        top_s = top;
    }
    __syncthreads();
    const int top = top_s;
    const int b0 = blockIdx.x * chunk, b1 = min(n - b0, chunk) + b0;
    // from the block's end: run holds the numbers past its nodes, nxt the cell
    // starts past them
    for (int r = b0 + (b1 - b0 - 1) / TTPB * TTPB; r >= b0; r -= TTPB) {
        const int i = r + threadIdx.x;
        int lo = 11, hi = 0;
        if (i < b1) {
            const int q = lv[i];
            lo = q & 15;
            hi = min(q >> 4, top);
        }
#pragma unroll
        for (int L = 0; L < LEVELS; ++L) {
            const unsigned b = __ballot_sync(0xffffffffu, lo <= L && L <= hi);
            const unsigned st = __ballot_sync(0xffffffffu, lo <= L);
            if (lane == L) {
                bal[warp][L] = b;
                wcnt[warp][L] = __popc(b);
                stt[warp][L] = st;
            }
        }
        __syncthreads();
        if (lane < LEVELS) {
            int s = run[lane], next = nxt[lane];
            for (int w = warp; w < TTPB / 32; ++w) s -= wcnt[w][lane];
            for (int w = TTPB / 32 - 1; w > warp; --w)
                if (stt[w][lane]) next = r + 32 * w + __ffs(stt[w][lane]) - 1;
            woff[warp][lane] = s;
            wnext[warp][lane] = next;
        }
        __syncthreads();
        if (threadIdx.x < LEVELS) {
            run[threadIdx.x] = woff[0][threadIdx.x];
            nxt[threadIdx.x] = stt[0][threadIdx.x] ? r + __ffs(stt[0][threadIdx.x]) - 1
                                                   : wnext[0][threadIdx.x];
        }
        if (lo <= hi) {
            const unsigned k = keys[i];
            int child = -1;
            for (int L = hi; L >= lo; --L) {
                const unsigned later = stt[warp][L] & ~(lt | (1u << lane));
                const int node = woff[warp][L] + __popc(bal[warp][L] & lt);
                t.start[node] = i;
                t.end[node] = later ? r + 32 * warp + __ffs(later) - 1 : wnext[warp][L];
                t.prefix[node] = k >> (3 * (10 - L));
                t.level[node] = L;
                t.nchild[node] = L < hi ? -1 : 0;  // counted with the moments
                t.first[node] = child;
                // the last node of the level above that starts at or before i
                t.parent[node] = L == 0 ? -1
                                        : woff[warp][L - 1] +
                                              __popc(bal[warp][L - 1] & (lt | (1u << lane))) - 1;
                t.arrive[node] = 0;
                child = node;
            }
        }
        __syncthreads();  // the shared rows are rewritten
    }
}

// Walk data of a node whose float64 moments are final: mass and centre of
// mass as a float32 hi/lo pair.
__device__ __forceinline__ void put_walk_moments(const TreeView &t, int node, double M, double cx,
                                                 double cy, double cz)
{
    t.M[node] = M;
    t.com[3 * (size_t)node] = cx;
    t.com[3 * (size_t)node + 1] = cy;
    t.com[3 * (size_t)node + 2] = cz;
    const float hx = (float)cx, hy = (float)cy, hz = (float)cz;
    t.chi[node] = make_float4(hx, hy, hz, (float)M);
    t.clo[node] = make_float4((float)(cx - (double)hx), (float)(cy - (double)hy),
                              (float)(cz - (double)hz), 0.f);
}

// Counts v in at p, releasing this thread's writes (and those it has observed)
// to whoever counts in later, and acquiring those of all who did before (one
// instruction, lighter than two sequentially consistent __threadfence()).
__device__ __forceinline__ int arrive_add(int *p, int v)
{
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;"
                 : "=r"(old)
                 : "l"(p), "r"(v)
                 : "memory");
    return old;
}

// Float64 monopoles of every node in one launch, bottom-up without any block waiting
// (and every node's float32 cube).  A thread per leaf sums its bodies; its
// node then counts its bodies in at the parent with an atomic, and only the
// child that completes the parent's count goes on to the parent, whose
// children eight lanes then sum (totalled in a fixed order, so the result does
// not depend on who arrives last); the climbing nodes of a warp are taken four
// at a time.  Fences order the sums before the arrival.
//
// What bounds it is the float64 pipe (2 lanes per clock per SM: a warp
// instruction takes 16 cycles whether one lane needs it or all) and, for small
// trees, the chain of levels.  So the cubes and the leaves' sums keep every
// lane busy, a parent's four sums are reduced over its eight lanes with four
// additions (each lane ends with one of them), and one division per node
// turns each lane's sum into its coordinate.  Blocks of two warps, so that the
// nodes of a small tree spread over the SMs' float64 pipes.  20000 bodies: 42 ->
// 34 us with the parent's tree data loaded beside the arrival and eight bodies'
// loads in flight per leaf; what is left is the chain of levels (arrival,
// children's sums, division).
//
// In a small tree the cells of at most direct_max bodies do not wait for their
// children but are summed from their bodies, a warp each, which leaves two or
// three levels to climb: walk and build of 2000 bodies 123 -> 107 us, 20000
// 182 -> 173 (this kernel 36 -> 29), 40000 244 -> 239, but 60000 319 -> 318,
// 200000 714 -> 731 (each body summed once more per such level).  Cells of up to
// 256, 512, 2048 bodies: 177, 175, 177 us at 20000.
constexpr int MTPB = 64;
constexpr int DIRECT_BODIES = 1024, DIRECT_MAX_N = 50000;
__global__ void __launch_bounds__(MTPB) tree_moments_kernel(TreeView t,
                                                            const double *__restrict__ box,
                                                            const double *__restrict__ pos,
                                                            const double *__restrict__ mass,
                                                            const int *__restrict__ perm,
                                                            int direct_max)
{
    const unsigned FULL = 0xffffffffu;
    const int total = t.meta[META_BASE + 10] + t.meta[META_COUNT + 10];
    if (blockIdx.x == 0 && threadIdx.x == 0) t.stats[0] = (unsigned long long)total;
    const int lane = threadIdx.x & 31, o = lane & 7;
    int leaves = 0;
    // whether node q's sums come from its children's (else from its bodies)
    auto climbed = [&](int q) { return q >= 0 && t.end[q] - t.start[q] > direct_max; };
    // climb: each lane with a node (and the bodies it stands for) counts in; the
    // completed parents are summed and count in themselves
    auto climb = [&](int node, int count) {
        while (__any_sync(FULL, node >= 0)) {
            // (what the parent's sum will need of the tree is loaded beside
            // the arrival, whose fence and atomic are the longest link)
            bool won = false;
            int bodies = 0, up = -1, f0 = 0, nch = 0;
            if (node >= 0) {
                bodies = t.end[node] - t.start[node];
                up = t.parent[node];
                f0 = t.first[node];
#pragma unroll
                for (int q = 0; q < 8; ++q) nch += f0 + q < total && t.parent[f0 + q] == node;
                won = arrive_add(t.arrive + node, count) + count == bodies;
            }
            // The children's sums are read by other lanes than the one that
            // arrived last: what its arrival acquired becomes theirs here (a
            // ballot or shuffle orders no memory).
            __syncwarp();
            unsigned win = __ballot_sync(FULL, won);
            while (win) {
                // group g of eight lanes takes the g-th winner
                const int g = lane >> 3;
                int src = -1;
                unsigned w = win;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q == g && w) src = __ffs(w) - 1;
                    w &= w - 1;  // 0 stays 0
                }
                win = w;
                const int p = __shfl_sync(FULL, node, src & 31);
                const int f = __shfl_sync(FULL, f0, src & 31), nc = __shfl_sync(FULL, nch, src & 31);
                const bool mine = src >= 0;
                const bool child = mine && o < nc;
                double v[4] = {0.0, 0.0, 0.0, 0.0};
                if (child) {
                    v[0] = __ldcg(t.M + f + o);
                    const double *c = t.com + 3 * (size_t)(f + o);
                    v[1] = v[0] * __ldcg(c);
                    v[2] = v[0] * __ldcg(c + 1);
                    v[3] = v[0] * __ldcg(c + 2);
                }
                // lanes with bit 2 keep y and z, the others M and x; then bit 1
                const bool hi2 = lane & 4, hi1 = lane & 2;
                const double r0 = __shfl_xor_sync(FULL, hi2 ? v[0] : v[2], 4);
                const double r1 = __shfl_xor_sync(FULL, hi2 ? v[1] : v[3], 4);
                const double a0 = (hi2 ? v[2] : v[0]) + r0, a1 = (hi2 ? v[3] : v[1]) + r1;
                double s = (hi1 ? a1 : a0) + __shfl_xor_sync(FULL, hi1 ? a0 : a1, 2);
                s += __shfl_xor_sync(FULL, s, 1);  // lane pair o >> 1: M, x, y, z
                const double M = __shfl_sync(FULL, s, lane & 24);
                const double cm = M > 0.0 ? s / M : 0.0;
                const double cx = __shfl_sync(FULL, cm, (lane & 24) + 2);
                const double cy = __shfl_sync(FULL, cm, (lane & 24) + 4);
                const double cz = __shfl_sync(FULL, cm, (lane & 24) + 6);
                if (mine && o == 0) {
                    put_walk_moments(t, p, M, cx, cy, cz);
                    t.nchild[p] = nc;
                    reinterpret_cast<int *>(t.box_lo + p)[3] = nc;  // the walk's child count
                }
                __syncwarp();
            }
            // and the parents' sums, written by other lanes too, are ordered
            // before the next round's releasing arrivals by the loop's __syncwarp
            node = won ? up : -1;
            count = bodies;
        }
    };
    for (int q0 = blockIdx.x * MTPB + (threadIdx.x & ~31); q0 < total; q0 += gridDim.x * MTPB) {
        const int me = q0 + lane;
        int node = -1, count = 0;  // what this lane counts in at its parent
        if (me < total) {
            float4 lo, hi;
            cube_corners(box, t.level[me], t.prefix[me], lo, hi);
            float *bl = reinterpret_cast<float *>(t.box_lo + me);
            *reinterpret_cast<float2 *>(bl) = make_float2(lo.x, lo.y);
            bl[2] = lo.z;  // [3], the child count, belongs to the climb
            hi.w = __int_as_float(t.first[me]);
            t.box_hi[me] = hi;
            // (a climbing warp may be replacing a parent's -1 by its count
            // meanwhile: either is not 0, which only a leaf has, from the start)
            if (t.nchild[me] == 0) {
                ++leaves;
                bl[3] = __int_as_float(0);
                const int s = t.start[me], e = t.end[me];
                double M = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
                for (int k = s; k < e; k += 8) {  // eight bodies' loads in flight
                    double m[8], x[8], y[8], z[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int j = perm[min(k + u, e - 1)];
                        m[u] = mass[j];
                        x[u] = pos[3 * (size_t)j];
                        y[u] = pos[3 * (size_t)j + 1];
                        z[u] = pos[3 * (size_t)j + 2];
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (k + u < e) {
                            M += m[u];
                            sx += m[u] * x[u];
                            sy += m[u] * y[u];
                            sz += m[u] * z[u];
                        }
                    }
                }
                // (three divisions: 1 / M of nearly massless bodies overflows)
                put_walk_moments(t, me, M, M > 0.0 ? sx / M : 0.0, M > 0.0 ? sy / M : 0.0,
                                 M > 0.0 ? sz / M : 0.0);
                node = t.parent[me];
                if (!climbed(node)) node = -1;
                count = e - s;
            }
        }
        climb(node, count);
    }
    // cells of few bodies: a warp each, from the bodies, the first ones by the
    // warps that had no leaves
    const int nw = gridDim.x * (MTPB / 32), busy = min(nw, (total + 31) >> 5);
    const int gw = blockIdx.x * (MTPB / 32) + (threadIdx.x >> 5);
    for (int q = gw < busy ? nw - busy + gw : gw - busy; direct_max > 0 && q < total; q += nw) {
        if (t.nchild[q] == 0 || climbed(q)) continue;
        const int s = t.start[q], e = t.end[q], f = t.first[q];
        const int nc = __popc(__ballot_sync(FULL, lane < 8 && f + o < total && t.parent[f + o] == q));
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int k = s + lane; k < e; k += 128) {
            double m[4], x[4], y[4], z[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = perm[min(k + 32 * u, e - 1)];
                m[u] = k + 32 * u < e ? mass[j] : 0.0;
                x[u] = pos[3 * (size_t)j];
                y[u] = pos[3 * (size_t)j + 1];
                z[u] = pos[3 * (size_t)j + 2];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (k + 32 * u < e) {
                    v[0] += m[u];
                    v[1] += m[u] * x[u];
                    v[2] += m[u] * y[u];
                    v[3] += m[u] * z[u];
                }
            }
        }
        // lanes with bit 4 keep y and z, the others M and x; then bit 3
        const bool hi4 = lane & 16, hi3 = lane & 8;
        const double r0 = __shfl_xor_sync(FULL, hi4 ? v[0] : v[2], 16);
        const double r1 = __shfl_xor_sync(FULL, hi4 ? v[1] : v[3], 16);
        const double a0 = (hi4 ? v[2] : v[0]) + r0, a1 = (hi4 ? v[3] : v[1]) + r1;
        double sum = (hi3 ? a1 : a0) + __shfl_xor_sync(FULL, hi3 ? a0 : a1, 8);
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) sum += __shfl_xor_sync(FULL, sum, off);
        const double M = __shfl_sync(FULL, sum, 0);
        const double cm = M > 0.0 ? sum / M : 0.0;
        const double cx = __shfl_sync(FULL, cm, 8), cy = __shfl_sync(FULL, cm, 16),
                     cz = __shfl_sync(FULL, cm, 24);
        int node = -1;
        if (lane == 0) {
            put_walk_moments(t, q, M, cx, cy, cz);
            t.nchild[q] = nc;
            reinterpret_cast<int *>(t.box_lo + q)[3] = nc;
            node = t.parent[q];
            if (!climbed(node)) node = -1;
        }
        climb(node, e - s);
    }
    leaves = __reduce_add_sync(FULL, leaves);
    if (lane == 0 && leaves) atomicAdd(t.stats + 1, (unsigned long long)leaves);
}

// Squared opening distance of a level, as the oracle computes it.
__device__ __forceinline__ float open_dist2(double ext, int L, float theta)
{
    const float edge = (float)__dmul_rn(ext, pow2_neg(L));  // = ext / 2^L
    const float d = __fdiv_rn(edge, theta);
    return __fmul_rn(d, d);
}

// Squared distance from p to the cube [lo, hi], no contraction.
__device__ __forceinline__ float cube_dist2(float4 lo, float4 hi, float px, float py, float pz)
{
    float d2 = 0.0f;
    const float pl[3] = {lo.x, lo.y, lo.z}, ph[3] = {hi.x, hi.y, hi.z}, pp[3] = {px, py, pz};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float a = __fsub_rn(pl[c], pp[c]);
        const float b = __fsub_rn(pp[c], ph[c]);
        float dd = a > b ? a : b;
        dd = dd > 0.0f ? dd : 0.0f;
        d2 = __fadd_rn(d2, __fmul_rn(dd, dd));
    }
    return d2;
}

// Squared distance from the cube [lo, hi] to the box [mn, mx], written as
// cube_dist2 with the box's far corner in each difference.  Rounding is
// monotonic, so for every p inside the box this value is <= cube_dist2(p):
// when it passes the opening test, every body of the box passes it too.
__device__ __forceinline__ float cube_box_dist2(float4 lo, float4 hi, const float (&mn)[3],
                                                const float (&mx)[3])
{
    float d2 = 0.0f;
    const float pl[3] = {lo.x, lo.y, lo.z}, ph[3] = {hi.x, hi.y, hi.z};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float a = __fsub_rn(pl[c], mx[c]);
        const float b = __fsub_rn(mn[c], ph[c]);
        float dd = a > b ? a : b;
        dd = dd > 0.0f ? dd : 0.0f;
        d2 = __fadd_rn(d2, __fmul_rn(dd, dd));
    }
    return d2;
}

// Interaction list of a warp: a ring of LIST_CAP sources (cells or bodies)
// as (x, y, z, m), coordinates relative to the group's centre, laid out for
// float32x2 arithmetic.  A flush evaluates the FLUSH sources of the half the
// ring's head is in and moves the head to the other half; at most
// FLUSH - 1 + 32 sources are ever listed, so new ones never reach the half
// being evaluated.  Paired layout: two sources share an instruction,
// a pair of sources is {x0, x1, y0, y1}, {z0, z1, m0, m1} (one body per
// lane, or each of a lane's two bodies in turn).  Doubled layout (two
// bodies per lane, NB_WALK_PAIRED 0): one source meets both bodies, stored
// twice over, {x, x, y, y}, {z, z, m, m}.
#ifndef NB_WALK_FLUSH
#define NB_WALK_FLUSH 64
#endif
#ifndef NB_WALK_PAIRED
#define NB_WALK_PAIRED 1
#endif
#ifndef NB_WALK_FOLD_EVERY
#define NB_WALK_FOLD_EVERY 4  // flushes between Kahan folds of the float32 partials
#endif
constexpr int FLUSH = NB_WALK_FLUSH;  // sources evaluated per flush (a multiple of 32)
constexpr int LIST_CAP = 2 * FLUSH;

template <int BPL>
__host__ __device__ constexpr bool paired_list() { return BPL == 1 || NB_WALK_PAIRED; }
// float4 slots of a list of LIST_CAP sources
template <int BPL>
__host__ __device__ constexpr int list_f4() { return paired_list<BPL>() ? LIST_CAP : LIST_CAP * 2; }

template <int BPL>
__device__ __forceinline__ void list_put(float *L, int q, float x, float y, float z, float m)
{
    if (paired_list<BPL>()) {
        float *b = L + 8 * (q >> 1) + (q & 1);
        b[0] = x;
        b[2] = y;
        b[4] = z;
        b[6] = m;
    } else {
        float4 *b = reinterpret_cast<float4 *>(L) + 2 * q;
        b[0] = make_float4(x, x, y, y);
        b[1] = make_float4(z, z, m, m);
    }
}

template <bool ZEPS>
__device__ __forceinline__ void pair_terms(float2 dx, float2 dy, float2 dz, float2 m, float2 e2,
                                           float2 &ax, float2 &ay, float2 &az)
{
    float2 r2 = fma2(dx, dx, e2);
    r2 = fma2(dy, dy, r2);
    r2 = fma2(dz, dz, r2);
    float2 ri = make_float2(rsqrt_mufu(r2.x), rsqrt_mufu(r2.y));
    if (ZEPS) {
        ri.x = r2.x > 0.f ? ri.x : 0.f;
        ri.y = r2.y > 0.f ? ri.y : 0.f;
    }
    const float2 s = mul2(mul2(m, ri), mul2(ri, ri));
    ax = fma2(dx, s, ax);
    ay = fma2(dy, s, ay);
    az = fma2(dz, s, az);
}

// Add the first `cnt` listed sources (cnt even for the paired layout) onto
// this lane's bodies.  Paired layout: nx = (-x_i, -x_i) per body (the second
// body's in nx2, its sums in a2); doubled layout: nx = (-x_i0, -x_i1).
template <bool ZEPS, int BPL>
__device__ __forceinline__ void list_eval(const float4 *L4, int cnt, float2 nx, float2 ny,
                                          float2 nz, float2 e2, float2 &ax, float2 &ay, float2 &az,
                                          float2 nx2, float2 ny2, float2 nz2, float2 &bx,
                                          float2 &by, float2 &bz)
{
    constexpr bool TWO = BPL == 2 && paired_list<BPL>();
    const int steps = paired_list<BPL>() ? cnt >> 1 : cnt;
#pragma unroll 4
    for (int q = 0; q < steps; ++q) {
        const float4 A = L4[2 * q], B = L4[2 * q + 1];
        const float2 sx = make_float2(A.x, A.y), sy = make_float2(A.z, A.w);
        const float2 sz = make_float2(B.x, B.y), sm = make_float2(B.z, B.w);
        pair_terms<ZEPS>(add2(sx, nx), add2(sy, ny), add2(sz, nz), sm, e2, ax, ay, az);
        if constexpr (TWO)
            pair_terms<ZEPS>(add2(sx, nx2), add2(sy, ny2), add2(sz, nz2), sm, e2, bx, by, bz);
    }
}

// Inclusive warp scan of v (lanes in order).
__device__ __forceinline__ int warp_incl_scan(int v, int lane)
{
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += u;
    }
    return v;
}

// Given inclusive prefix sums `incl` of per-lane counts (non-decreasing over
// the lanes), the lane whose span holds position pos: the number of lanes
// with incl <= pos (a binary search over the lanes, five shuffles).
__device__ __forceinline__ int warp_span_of(int incl, int pos)
{
    int lo = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
        const int v = __shfl_sync(0xffffffffu, incl, lo + step - 1);
        if (v <= pos) lo += step;
    }
    return lo;
}

// One warp (or W, below) per group of 32 * BPL consecutive bodies in key order
// (BPL per lane: bodies base + lane and base + 32 + lane).  The warp walks the tree
// level by level, deepest level first, 32 nodes per round (one per lane).
// The opening test against every body of the group decides, per node,
// between the interaction list (accepted cell: its monopole; leaf: its
// bodies) and descending (its children, a contiguous range, go on the next
// level's stack).  The test runs in three exact stages: the group's box
// (passing it implies every body passes), then the group's first and last
// bodies (failing either rejects), then, for the nodes still undecided, every
// body.  Each level's stack holds at most 32 ranges, the children of one
// round's nodes, since a level is refilled only once every deeper level is
// empty.  Whenever FLUSH sources are listed, every lane adds them to its bodies.
//
// W > 1: W warps walk one group together, level by level: the nodes of a level
// (the shared frontier) are dealt to the warps round robin, each warp appends
// the children it opens to its own segment of the next frontier (one that is
// full leaves the rest to its warp's own stacks, which are emptied before the
// next nodes are dealt), and the block meets once per level.  Who tests what
// depends on the tree only, so each warp's sums, and their total in warp
// order, do not depend on timing.
constexpr int FRONT_CAP = 2048;  // nodes of a frontier, over its segments
constexpr int walk_warps(int W) { return W > 1 ? W : WALK_WARPS; }  // per block

template <int BPL, bool MULTI, int W>
struct WalkShared {
    float4 list[walk_warps(W)][list_f4<BPL>()];  // float4 slots of the lists
    int2 ranges[walk_warps(W)][LEVELS][32];
    int lslot[MULTI ? 1 : walk_warps(W)][32];  // a chunk's leaf starts: body index minus position
    float crit2[MULTI ? 1 + WALK_MAX_MORE : 1][LEVELS];  // per walked tree
    int front[W > 1 ? 2 : 1][W > 1 ? W : 1][W > 1 ? FRONT_CAP / W : 1];
    int seg[2][walk_warps(W)];  // nodes per segment; cells and bodies listed per warp at the end
    int task;
};

// The walk of group g (bodies [g * 32 * BPL, ...) in key order) by one warp:
// over the one tree (tq_only = -1), or (MULTI) over span tq_only of the trees
// in p.more, the group's last span then writing the sums of all of them.
template <bool ZEPS, int BPL, bool MULTI, int W>
__device__ __forceinline__ void walk_group(const TreeWalkParams &p, WalkShared<BPL, MULTI, W> &sh,
                                           int g, int tq_only)
{
    constexpr int GROUP = 32 * BPL;
    constexpr int LIST_F4 = list_f4<BPL>();
    constexpr bool TWO = BPL == 2 && paired_list<BPL>();  // a lane's two bodies in turn
    const unsigned FULL = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = p.n;
    const int base = g * GROUP;
    if (base >= n) return;  // whole warp past the end
    const int nvalid = min(GROUP, n - base);
    float4(*list_s)[LIST_F4] = sh.list;

    bool valid[BPL];
    float4 h[BPL];
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    float4 lo_[BPL];
#pragma unroll
    for (int b = 0; b < BPL; ++b) {
        const int k = base + 32 * b + lane;
        valid[b] = k < n;
        h[b] = valid[b] ? __ldg(p.P + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        lo_[b] = valid[b] ? __ldg(p.Plo + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid[b]) {
            mn[0] = fminf(mn[0], h[b].x);
            mn[1] = fminf(mn[1], h[b].y);
            mn[2] = fminf(mn[2], h[b].z);
            mx[0] = fmaxf(mx[0], h[b].x);
            mx[1] = fmaxf(mx[1], h[b].y);
            mx[2] = fmaxf(mx[2], h[b].z);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            mn[c] = fminf(mn[c], __shfl_xor_sync(FULL, mn[c], off));
            mx[c] = fmaxf(mx[c], __shfl_xor_sync(FULL, mx[c], off));
        }
    }
    const float cx = 0.5f * (mn[0] + mx[0]), cy = 0.5f * (mn[1] + mx[1]),
                cz = 0.5f * (mn[2] + mx[2]);
    float xi[BPL], yi[BPL], zi[BPL];
#pragma unroll
    for (int b = 0; b < BPL; ++b) {
        xi[b] = rel(h[b].x, lo_[b].x, cx);
        yi[b] = rel(h[b].y, lo_[b].y, cy);
        zi[b] = rel(h[b].z, lo_[b].z, cz);
    }
    const bool bc = BPL == 1 || TWO;  // the first body broadcast over a source pair
    const float2 nx = bc ? make_float2(-xi[0], -xi[0]) : make_float2(-xi[0], -xi[BPL - 1]);
    const float2 ny = bc ? make_float2(-yi[0], -yi[0]) : make_float2(-yi[0], -yi[BPL - 1]);
    const float2 nz = bc ? make_float2(-zi[0], -zi[0]) : make_float2(-zi[0], -zi[BPL - 1]);
    const float2 nx2 = make_float2(-xi[BPL - 1], -xi[BPL - 1]);
    const float2 ny2 = make_float2(-yi[BPL - 1], -yi[BPL - 1]);
    const float2 nz2 = make_float2(-zi[BPL - 1], -zi[BPL - 1]);
    const float2 e2 = make_float2(p.eps2f, p.eps2f);
    // the group's first and last bodies, for the quick rejection
    const int lastb = (nvalid - 1) >> 5, lastl = (nvalid - 1) & 31;
    float r0[3], r1[3];
    {
        const float4 hl = lastb == 0 ? h[0] : h[BPL - 1];
        r0[0] = __shfl_sync(FULL, h[0].x, 0);
        r0[1] = __shfl_sync(FULL, h[0].y, 0);
        r0[2] = __shfl_sync(FULL, h[0].z, 0);
        r1[0] = __shfl_sync(FULL, hl.x, lastl);
        r1[1] = __shfl_sync(FULL, hl.y, lastl);
        r1[2] = __shfl_sync(FULL, hl.z, lastl);
    }

    float *L = reinterpret_cast<float *>(list_s[warp]);
    const float4 *L4 = list_s[warp];
    int2(*rs)[32] = sh.ranges[warp];
    const unsigned lt = (1u << lane) - 1u;
    int head = 0;  // the list ring's current half (0 or FLUSH)

    // Each tree's sum per body, G (s - c) from its Kahan pair, added in tree
    // order in float64 (as separate accumulating walks would add them).
    double tg[BPL][3];
    int nc = 0, nb = 0;
    const int ntrees = MULTI ? 1 + p.nmore : 1;
    // split mode: this task walks trees [tq_only * tspan, ... + tspan)
    const int tq_lo = MULTI && tq_only >= 0 ? tq_only * p.tspan : 0;
    const int tq_hi = MULTI && tq_only >= 0 ? min(tq_lo + p.tspan, ntrees) : ntrees;
    for (int tq = tq_lo; tq < tq_hi; ++tq) {
    WalkSource t;
    if (!MULTI) {
        t = WalkSource{p.tree.box_lo, p.tree.box_hi, p.tree.chi, p.tree.clo,
                       p.tree.start,  p.tree.end,    p.sP,      p.sPlo,
                       p.box};
    } else {  // every tree of a multi-tree walk, the first included, from `more`
        t = p.more[tq];
    }
    const float *crit2 = sh.crit2[MULTI ? tq : 0];
    float2 ax = make_float2(0.f, 0.f), ay = ax, az = ax, bx = ax, by = ax, bz = ax;
    // Kahan (sum, carry) per body and axis: the paired layout folds both
    // halves of a body's float32x2 accumulators into it (the second body's
    // are bx..bz); the doubled layout keeps .x and .y apart.
    float sx[BPL], sy[BPL], sz[BPL], qx[BPL], qy[BPL], qz[BPL];
#pragma unroll
    for (int b = 0; b < BPL; ++b) sx[b] = sy[b] = sz[b] = qx[b] = qy[b] = qz[b] = 0.f;
    auto fold = [&]() {
        if (paired_list<BPL>()) {
            kahan_add(sx[0], qx[0], ax.x);
            kahan_add(sx[0], qx[0], ax.y);
            kahan_add(sy[0], qy[0], ay.x);
            kahan_add(sy[0], qy[0], ay.y);
            kahan_add(sz[0], qz[0], az.x);
            kahan_add(sz[0], qz[0], az.y);
            if (TWO) {
                kahan_add(sx[BPL - 1], qx[BPL - 1], bx.x);
                kahan_add(sx[BPL - 1], qx[BPL - 1], bx.y);
                kahan_add(sy[BPL - 1], qy[BPL - 1], by.x);
                kahan_add(sy[BPL - 1], qy[BPL - 1], by.y);
                kahan_add(sz[BPL - 1], qz[BPL - 1], bz.x);
                kahan_add(sz[BPL - 1], qz[BPL - 1], bz.y);
            }
        } else {
            kahan_add(sx[0], qx[0], ax.x);
            kahan_add(sy[0], qy[0], ay.x);
            kahan_add(sz[0], qz[0], az.x);
            kahan_add(sx[BPL - 1], qx[BPL - 1], ax.y);
            kahan_add(sy[BPL - 1], qy[BPL - 1], ay.y);
            kahan_add(sz[BPL - 1], qz[BPL - 1], az.y);
        }
        ax = ay = az = bx = by = bz = make_float2(0.f, 0.f);
    };
    int cnt = 0;  // listed sources (warp-uniform)
    int nflush = 0;
    // FLUSH sources listed from the head on: add them, head to the other half
    auto flush = [&]() {
        __syncwarp();
        list_eval<ZEPS, BPL>(L4 + (paired_list<BPL>() ? head : 2 * head), FLUSH, nx, ny, nz, e2,
                             ax, ay, az, nx2, ny2, nz2, bx, by, bz);
        if (++nflush % NB_WALK_FOLD_EVERY == 0) fold();
        head ^= FLUSH;
        cnt -= FLUSH;
        __syncwarp();
    };

    int lsize = 0;  // lane L holds the size of level L's stack
    // the frontier: ftot nodes of level fl, at first the root; its next round;
    // the children this warp appended to the next one
    int fl = 0, ftot = 1, fr = 0, cur = 0, found = 0;
    if (W > 1) {
        if (threadIdx.x < W) sh.seg[0][threadIdx.x] = threadIdx.x == 0;
        if (threadIdx.x == 0) sh.front[0][0][0] = 0;
        __syncthreads();
    }
    for (;;) {
        int node = -1, Lv = fl;
        const unsigned nonempty = __ballot_sync(FULL, lane < LEVELS && lsize > 0);
        const bool shared_round = W > 1 && !nonempty;
        if (shared_round) {
            if (32 * W * fr >= ftot) {  // every warp is done with the level
                if (lane == 0) sh.seg[cur ^ 1][warp] = found;
                __syncthreads();
                cur ^= 1;
                found = fr = ftot = 0;
#pragma unroll
                for (int w = 0; w < W; ++w) ftot += sh.seg[cur][w];
                if (ftot == 0) break;
                Lv = ++fl;
            }
            int at = 32 * W * fr + W * lane + warp, w = 0;
            ++fr;
            if (at < ftot) {
#pragma unroll
                for (int q = 0; q < W - 1; ++q) {
                    const int c = sh.seg[cur][q];
                    if (w == q && at >= c) {
                        at -= c;
                        ++w;
                    }
                }
                node = sh.front[cur][w][at];
            }
        } else if (!nonempty) {
            if (fr > 0) break;
            if (lane == 0) node = 0;
            ++fr;
        } else {
        Lv = 31 - __clz(nonempty);
        const int size = __shfl_sync(FULL, lsize, Lv);
        // take up to 32 nodes from the top ranges of level Lv
        const int R = min(size, 32);
        const int2 r = lane < R ? rs[Lv][size - 1 - lane] : make_int2(0, 0);
        const int incl = warp_incl_scan(r.y, lane);
        const int excl = incl - r.y;
        const int take = min(__shfl_sync(FULL, incl, 31), 32);
        // the range holding this lane's node: the last range starting at or
        // before it (ranges 0..R-1 are non-empty, so their starts increase)
        const unsigned starts = __reduce_or_sync(FULL, lane < R && excl < 32 ? 1u << excl : 0u);
        const int src = __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
        const int first_src = __shfl_sync(FULL, r.x, src), excl_src = __shfl_sync(FULL, excl, src);
        node = lane < take ? first_src + (lane - excl_src) : -1;
        const unsigned done = __ballot_sync(FULL, lane < R && incl <= 32);
        if (lane < R && excl < 32 && incl > 32)
            rs[Lv][size - 1 - lane] = make_int2(r.x + (32 - excl), incl - 32);
        if (lane == Lv) lsize -= __popc(done);
        __syncwarp();
        }

        // opening test
        const bool has = node >= 0;
        float4 blo = make_float4(0.f, 0.f, 0.f, 0.f), bhi = blo;
        if (has) {
            blo = __ldg(t.box_lo + node);
            bhi = __ldg(t.box_hi + node);
        }
        const float cr = crit2[Lv];
        bool accept = has && cube_box_dist2(blo, bhi, mn, mx) >= cr;
        unsigned und = __ballot_sync(FULL, has && !accept);
        if (und) {
            const bool rej = cube_dist2(blo, bhi, r0[0], r0[1], r0[2]) < cr ||
                             cube_dist2(blo, bhi, r1[0], r1[1], r1[2]) < cr;
            und = __ballot_sync(FULL, has && !accept && !rej);
        }
        // undecided nodes one at a time, every lane testing its own bodies
        while (und) {
            const int j = __ffs(und) - 1;
            und &= und - 1;
            const float4 jlo = make_float4(__shfl_sync(FULL, blo.x, j), __shfl_sync(FULL, blo.y, j),
                                           __shfl_sync(FULL, blo.z, j), 0.f);
            const float4 jhi = make_float4(__shfl_sync(FULL, bhi.x, j), __shfl_sync(FULL, bhi.y, j),
                                           __shfl_sync(FULL, bhi.z, j), 0.f);
            bool ok = true;
#pragma unroll
            for (int b = 0; b < BPL; ++b)
                ok = ok && (!valid[b] || cube_dist2(jlo, jhi, h[b].x, h[b].y, h[b].z) >= cr);
            const bool all = __all_sync(FULL, ok);
            if (lane == j) accept = all;
        }
        const int nch = has ? __float_as_int(blo.w) : 0;
        const bool open = has && !accept && nch > 0;
        const bool leaf = has && !accept && nch == 0;

        // children: of a shared node onto the next frontier while this warp's
        // segment has room
        bool own = open;
        if (shared_round) {
            const int c = open ? nch : 0;
            const int incl = warp_incl_scan(c, lane);
            const int at = found + incl - c;
            own = open && at + c > FRONT_CAP / W;  // then the later lanes' do not fit either
            if (!own)
                for (int q = 0; q < c; ++q) sh.front[cur ^ 1][warp][at + q] = __float_as_int(bhi.w) + q;
            const unsigned full = __ballot_sync(FULL, own);
            found = full ? __shfl_sync(FULL, at, __ffs(full) - 1)
                         : found + __shfl_sync(FULL, incl, 31);
        }
        // else their ranges onto the next level (Lv < 10 whenever a node opens)
        const unsigned om = __ballot_sync(FULL, own);
        if (om) {
            const int size1 = __shfl_sync(FULL, lsize, Lv + 1);
            const int slot1 = size1 + __popc(om & lt);
            if (own && slot1 < 32) rs[Lv + 1][slot1] = make_int2(__float_as_int(bhi.w), nch);
            if (lane == Lv + 1) lsize = min(size1 + __popc(om), 32);
            if (lane == 0 && size1 + __popc(om) > 32) atomicOr(p.err, ERR_TREE);  // never: see above
        }
        __syncwarp();
        // accepted cells: their monopoles
        const unsigned am = __ballot_sync(FULL, accept);
        if (am) {
            if (accept) {
                const float4 ch = __ldg(t.chi + node), cl = __ldg(t.clo + node);
                list_put<BPL>(L, (head + cnt + __popc(am & lt)) & (LIST_CAP - 1),
                              rel(ch.x, cl.x, cx), rel(ch.y, cl.y, cy), rel(ch.z, cl.z, cz), ch.w);
            }
            cnt += __popc(am);
            nc += __popc(am);
            if (cnt >= FLUSH) flush();
        }
        // leaves: the bodies of all of this round's leaves, 32 list slots at a
        // time (lane l of a chunk fetches the chunk's l-th body)
        if (__ballot_sync(FULL, leaf)) {
            int ls = 0, lsz = 0;
            if (leaf) {
                ls = t.start[node];
                lsz = t.end[node] - ls;
            }
            const int linc = warp_incl_scan(lsz, lane);
            const int lexc = linc - lsz;
            const int T = __shfl_sync(FULL, linc, 31);
            nb += T;
            int carry = 0;  // the offset of the leaf running into the chunk
            for (int c0 = 0; c0 < T; c0 += 32) {
                const int pos = c0 + lane;
                int body;
                if constexpr (MULTI) {  // (the slots cost this instance spills)
                    const int j = warp_span_of(linc, pos);
                    body = __shfl_sync(FULL, ls, j & 31) + (pos - __shfl_sync(FULL, lexc, j & 31));
                } else {
                    // the leaf holding position pos: the last one starting at
                    // or before it, in this chunk (its slot) or earlier (carry)
                    const bool st = lsz > 0 && lexc >= c0 && lexc < c0 + 32;
                    if (st) sh.lslot[warp][lexc - c0] = ls - lexc;
                    const unsigned S = __reduce_or_sync(FULL, st ? 1u << (lexc - c0) : 0u);
                    __syncwarp();
                    const unsigned below = S & (0xffffffffu >> (31 - lane));
                    const int off = below ? sh.lslot[warp][31 - __clz(below)] : carry;
                    carry = __shfl_sync(FULL, off, 31);
                    body = off + pos;
                }
                const int kk = min(32, T - c0);
                if (lane < kk) {
                    const float4 bh = __ldg(t.sP + body), bl = __ldg(t.sPlo + body);
                    list_put<BPL>(L, (head + cnt + lane) & (LIST_CAP - 1), rel(bh.x, bl.x, cx),
                                  rel(bh.y, bl.y, cy), rel(bh.z, bl.z, cz), bh.w);
                }
                cnt += kk;
                if (cnt >= FLUSH) flush();
                __syncwarp();  // the slots are rewritten for the next chunk
            }
        }
    }
    if (cnt > 0) {  // the rest, within the head's half (paired layout: padded to a
                    // pair with a massless source)
        if (paired_list<BPL>() && lane == 0 && (cnt & 1))
            list_put<BPL>(L, head + cnt, 0.f, 0.f, 0.f, 0.f);
        __syncwarp();
        list_eval<ZEPS, BPL>(L4 + (paired_list<BPL>() ? head : 2 * head),
                             paired_list<BPL>() ? (cnt + 1) & ~1 : cnt, nx, ny, nz, e2, ax, ay,
                             az, nx2, ny2, nz2, bx, by, bz);
    }
    if (nflush % NB_WALK_FOLD_EVERY != 0 || cnt > 0) fold();
    __syncwarp();  // the next tree reuses this warp's list and stacks
#pragma unroll
    for (int b = 0; b < BPL; ++b) {
        const double d[3] = {p.G * ((double)sx[b] - (double)qx[b]),
                             p.G * ((double)sy[b] - (double)qy[b]),
                             p.G * ((double)sz[b] - (double)qz[b])};
#pragma unroll
        for (int c = 0; c < 3; ++c) tg[b][c] = (!MULTI || tq == tq_lo) ? d[c] : __dadd_rn(tg[b][c], d[c]);
    }
    }  // trees
    bool stats_done = false;
    if (W > 1) {  // the warps' sums and counts, added in warp order by the first
        __syncthreads();  // every warp has read the last level's segments
        double *mine = reinterpret_cast<double *>(list_s[warp]);
        static_assert(sizeof(float4) * LIST_F4 >= sizeof(double) * 3 * GROUP, "sums fit the list");
#pragma unroll
        for (int b = 0; b < BPL; ++b)
#pragma unroll
            for (int c = 0; c < 3; ++c) mine[(3 * b + c) * 32 + lane] = tg[b][c];
        if (lane == 0) {
            sh.seg[0][warp] = nc;
            sh.seg[1][warp] = nb;
        }
        __syncthreads();
        if (warp == 0) {
            for (int w = 1; w < W; ++w) {
                const double *o = reinterpret_cast<const double *>(list_s[w]);
#pragma unroll
                for (int b = 0; b < BPL; ++b)
#pragma unroll
                    for (int c = 0; c < 3; ++c) tg[b][c] += o[(3 * b + c) * 32 + lane];
                nc += sh.seg[0][w];
                nb += sh.seg[1][w];
            }
        }
        __syncthreads();
        if (warp != 0) return;
    }
    if (MULTI && tq_only >= 0) {
        // this task's sums and counts; the group's last task adds all tasks'
        // in tree order (with one tree per task, as the walk over every tree
        // in turn does) and writes
        const int ngroups = (n + GROUP - 1) / GROUP;
        const size_t npad = (size_t)ngroups * GROUP;
#pragma unroll
        for (int b = 0; b < BPL; ++b) {
            double *q = p.tpart + ((size_t)tq_only * npad + base + 32 * b + lane) * 3;
            q[0] = tg[b][0];
            q[1] = tg[b][1];
            q[2] = tg[b][2];
        }
        if (lane == 0) {
            p.tcnt[((size_t)tq_only * ngroups + g) * 2] = nc;
            p.tcnt[((size_t)tq_only * ngroups + g) * 2 + 1] = nb;
            atomicAdd(p.tree.stats + 2, (unsigned long long)nc * nvalid);
            atomicAdd(p.tree.stats + 3, (unsigned long long)nb * nvalid);
        }
        stats_done = true;
        __threadfence();
        __syncwarp();
        unsigned last = 0;
        const int nspans = (ntrees + p.tspan - 1) / p.tspan;
        if (lane == 0) last = atomicAdd(p.tctr + g, 1u) == (unsigned)(nspans - 1);
        __syncwarp();  // lane 0's arrival before the other lanes' fences
        if (!__shfl_sync(FULL, last, 0)) return;
        __threadfence();
        nc = nb = 0;
        for (int tq = 0; tq < nspans; ++tq) {
#pragma unroll
            for (int b = 0; b < BPL; ++b) {
                const double *q = p.tpart + ((size_t)tq * npad + base + 32 * b + lane) * 3;
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    tg[b][c] = tq == 0 ? __ldcg(q + c) : __dadd_rn(tg[b][c], __ldcg(q + c));
            }
            nc += __ldcg(p.tcnt + ((size_t)tq * ngroups + g) * 2);
            nb += __ldcg(p.tcnt + ((size_t)tq * ngroups + g) * 2 + 1);
        }
        if (lane == 0) p.tctr[g] = 0u;  // every task of the group has arrived
    }
#pragma unroll
    for (int b = 0; b < BPL; ++b) {
        if (!valid[b]) continue;
        const int i = p.perm[base + 32 * b + lane];
        const double gx = tg[b][0], gy = tg[b][1], gz = tg[b][2];
        double *a = p.acc + 3 * (size_t)i;
        if (p.accumulate) {  // a further tree's share (a received LET)
            a[0] += gx;
            a[1] += gy;
            a[2] += gz;
            if (p.counts) {
                p.counts[2 * (size_t)i] += nc;
                p.counts[2 * (size_t)i + 1] += nb;
            }
        } else {
            a[0] = gx;
            a[1] = gy;
            a[2] = gz;
            if (p.vel) {
                double *v = p.vel + 3 * (size_t)i;
                v[0] += p.half_dt * gx;
                v[1] += p.half_dt * gy;
                v[2] += p.half_dt * gz;
            }
            if (p.counts) {
                p.counts[2 * (size_t)i] = nc;
                p.counts[2 * (size_t)i + 1] = nb;
            }
        }
        if (!finite3(gx, gy, gz)) atomicOr(p.err, ERR_NONFINITE);
    }
    if (lane == 0 && !stats_done) {  // nc, nb are the same for the group's nvalid bodies
        atomicAdd(p.tree.stats + 2, (unsigned long long)nc * nvalid);
        atomicAdd(p.tree.stats + 3, (unsigned long long)nb * nvalid);
    }
    __syncwarp();  // the next group reuses this warp's lists and stacks
}

// Scheduling of the groups over the warps (the paper's OpenMP loop
// schedules, Sec. II, applied to the walk): static, one group per warp of a
// grid covering all groups; dynamic, a grid of resident warps taking `chunk`
// groups at a time from an atomic counter; guided, the same with chunks of
// max(chunk, remaining / (2 x warps)).
// (In units of blocks and groups when a block's W warps walk one group.)
template <bool ZEPS, int BPL, bool MULTI, int W>
__global__ void __launch_bounds__(32 * walk_warps(W),
                                  BPL == 1 ? NB_WALK_MINB1 * WALK_WARPS / walk_warps(W)
                                           : NB_WALK_MINB2 * WALK_WARPS / walk_warps(W))
    tree_walk_kernel(const TreeWalkParams p)
{
    extern __shared__ __align__(16) unsigned char walk_smem[];
    WalkShared<BPL, MULTI, W> &sh = *reinterpret_cast<WalkShared<BPL, MULTI, W> *>(walk_smem);
    for (int q = threadIdx.x; q < (MULTI ? 1 + p.nmore : 1) * LEVELS; q += blockDim.x) {
        const int tq = q / LEVELS, L = q % LEVELS;
        sh.crit2[tq][L] = open_dist2(MULTI ? p.more[tq].box[3] : p.box[3], L, p.theta);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // workers: the warps, or the blocks
    const int gw = W > 1 ? blockIdx.x : blockIdx.x * WALK_WARPS + warp;
    const int ngroups = (p.n + 32 * BPL - 1) / (32 * BPL);
    // tasks: the groups, or with further trees (split mode) the (group,
    // tree) pairs, tree-major
    const int ntasks = MULTI ? ngroups * ((1 + p.nmore + p.tspan - 1) / p.tspan) : ngroups;
    auto task = [&](int t) {
        if constexpr (MULTI)
            walk_group<ZEPS, BPL, MULTI, W>(p, sh, t % ngroups, t / ngroups);
        else
            walk_group<ZEPS, BPL, MULTI, W>(p, sh, t, -1);
    };
    if (p.sched == 0) {
        if (gw < ntasks) task(gw);
        return;
    }
    const int nworkers = W > 1 ? gridDim.x : gridDim.x * WALK_WARPS;
    int *queue = p.queue;
    int seen = 0;
    for (;;) {
        int c = p.chunk;
        if (p.sched == 2) c = max(c, (ntasks - seen) / (2 * nworkers));
        int g0 = 0;
        if (W > 1) {
            if (threadIdx.x == 0) sh.task = atomicAdd(queue, c);
            __syncthreads();
            g0 = sh.task;
            __syncthreads();
        } else {
            if (lane == 0) g0 = atomicAdd(queue, c);
            g0 = __shfl_sync(0xffffffffu, g0, 0);
        }
        if (g0 >= ntasks) break;
        seen = g0 + c;
        const int g1 = min(g0 + c, ntasks);
        for (int g = g0; g < g1; ++g) task(g);
    }
}

// ---------------------------------------------- locally essential trees
// The LET of this tree for a destination whose bodies lie in the float32
// box [dlo, dhi] (paper Sec. IV-B, the influence-ring test from the
// destination's side): the root is sent; a sent node whose cube is distant
// enough from the box (cube_box_dist2, the walk's own first-stage test, so
// every body inside the box accepts it) is sent alone; otherwise a sent
// leaf goes with its bodies and a sent cell with all its children.
// Level by level, parents first.
__global__ void __launch_bounds__(TTPB) let_kind_kernel(TreeView t, const double *__restrict__ box,
                                                        float theta, float3 dlo, float3 dhi, int L,
                                                        int *__restrict__ kind)
{
    const int cnt = t.meta[META_COUNT + L], base = t.meta[META_BASE + L];
    const float crit2 = open_dist2(box[3], L, theta);
    const float mn[3] = {dlo.x, dlo.y, dlo.z}, mx[3] = {dhi.x, dhi.y, dhi.z};
    for (int q = blockIdx.x * TTPB + threadIdx.x; q < cnt; q += gridDim.x * TTPB) {
        const int u = base + q;
        int k = 0;
        if (L == 0 || kind[t.parent[u]] == 2) {
            if (cube_box_dist2(t.box_lo[u], t.box_hi[u], mn, mx) >= crit2)
                k = 1;
            else
                k = t.nchild[u] == 0 ? 3 : 2;
        }
        kind[u] = k;
    }
}

// One block: each sent node's index in the LET and each sent leaf's first
// body there (exclusive scans in node order); totals = {nodes, bodies}.
__global__ void __launch_bounds__(1024) let_scan_kernel(TreeView t, LetScratch sc)
{
    __shared__ int tile[BSCAN_TILE + BSCAN_TILE / 32];
    __shared__ int wsum[32];
    const int total = t.meta[META_BASE + 10] + t.meta[META_COUNT + 10];
    // flags and body counts first go into the output arrays, scanned in place
    for (int u = threadIdx.x; u < total; u += 1024) {
        const int k = sc.kind[u];
        sc.nidx[u] = k != 0;
        sc.boff[u] = k == 3 ? t.end[u] - t.start[u] : 0;
    }
    __syncthreads();
    const int nn = block_scan_exclusive<int>(sc.nidx, sc.nidx, total, tile, wsum);
    const int nb = block_scan_exclusive<int>(sc.boff, sc.boff, total, tile, wsum);
    if (threadIdx.x == 0) {
        sc.totals[0] = nn;
        sc.totals[1] = nb;
    }
}

__global__ void __launch_bounds__(TTPB) let_emit_kernel(TreeView t, const double *__restrict__ box,
                                                        LetScratch sc, const float4 *__restrict__ P,
                                                        const float4 *__restrict__ Plo,
                                                        unsigned char *__restrict__ out)
{
    const int total = t.meta[META_BASE + 10] + t.meta[META_COUNT + 10];
    const long long nn = sc.totals[0], nb = sc.totals[1];
    const LetLayout lay = let_layout(nn, nb);
    float4 *lo = reinterpret_cast<float4 *>(out + lay.lo);
    float4 *hi = reinterpret_cast<float4 *>(out + lay.hi);
    float4 *chi = reinterpret_cast<float4 *>(out + lay.chi);
    float4 *clo = reinterpret_cast<float4 *>(out + lay.clo);
    int *st = reinterpret_cast<int *>(out + lay.start);
    int *en = reinterpret_cast<int *>(out + lay.end);
    float4 *bP = reinterpret_cast<float4 *>(out + lay.P);
    float4 *bPlo = reinterpret_cast<float4 *>(out + lay.Plo);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        LetHeader h;
        h.magic = LET_MAGIC;
        h.n_nodes = nn;
        h.n_bodies = nb;
        h.reserved = 0;
        for (int c = 0; c < 4; ++c) h.box[c] = box[c];
        *reinterpret_cast<LetHeader *>(out) = h;
    }
    for (int u = blockIdx.x * TTPB + threadIdx.x; u < total; u += gridDim.x * TTPB) {
        const int k = sc.kind[u];
        if (k == 0) continue;
        const int v = sc.nidx[u];
        float4 a = t.box_lo[u], b = t.box_hi[u];
        // children are kept only for an opened cell; they are consecutive
        // in both trees, so the first one's LET index locates them all
        a.w = __int_as_float(k == 2 ? t.nchild[u] : 0);
        b.w = __int_as_float(k == 2 ? sc.nidx[t.first[u]] : -1);
        lo[v] = a;
        hi[v] = b;
        chi[v] = t.chi[u];
        clo[v] = t.clo[u];
        const int b0 = sc.boff[u];
        const int len = k == 3 ? t.end[u] - t.start[u] : 0;
        st[v] = b0;
        en[v] = b0 + len;
        for (int q = 0; q < len; ++q) {
            bP[b0 + q] = P[t.start[u] + q];
            bPlo[b0 + q] = Plo[t.start[u] + q];
        }
    }
}

}  // namespace

int tree_meta_ints() { return META_INTS; }

int64_t tree_node_bound(int64_t n, int leaf_cap)
{
    // Nodes of one level are disjoint and non-empty (<= n), at most 8^L, and
    // children of the split nodes of the level above, which hold more than
    // leaf_cap bodies each (<= 8 n / (leaf_cap + 1)).
    if (n <= 0) return 1;
    const int64_t split = leaf_cap >= 1 ? n / ((int64_t)leaf_cap + 1) : n;
    int64_t total = 1, p8 = 1;
    for (int L = 1; L <= 10; ++L) {
        p8 *= 8;
        int64_t c = p8 < n ? p8 : n;
        if (8 * split < c) c = 8 * split;
        total += c;
    }
    return total;
}

cudaError_t launch_tree_build(cudaStream_t s, const TreeView &t, int n, const OrderScratch &o,
                              const double *box, const double *pos, const double *mass,
                              const int *perm, int leaf_cap, bool moments, int num_sms, int *err,
                              int &kernels)
{
    // one block per 256 bodies until the blocks' table of counts, which every
    // block sums, is as large as is cheap (26 KB)
    const unsigned *keys = o.keys[0];
    unsigned char *lv = reinterpret_cast<unsigned char *>(o.vals[0]);
    int *tab = reinterpret_cast<int *>(o.hist);
    const int tiles = (n + TTPB - 1) / TTPB;
    const int chunk = (tiles + BUILD_BLOCKS - 1) / BUILD_BLOCKS * TTPB;
    const int nblk = (n + chunk - 1) / chunk;
    tree_levels_kernel<<<nblk, TTPB, 0, s>>>(t, n, keys, leaf_cap, chunk, lv, tab);
    tree_emit_kernel<<<nblk, TTPB, 0, s>>>(t, n, keys, chunk, lv, tab, err);
    kernels = 2;
    if (!moments) return cudaGetLastError();
    // a thread per node, at most 20 blocks of two warps per SM
    const int64_t blocks = std::min<int64_t>(((int64_t)t.cap + MTPB - 1) / MTPB, 20 * num_sms);
    const int direct_max = n <= DIRECT_MAX_N ? DIRECT_BODIES : 0;
    tree_moments_kernel<<<(int)blocks, MTPB, 0, s>>>(t, box, pos, mass, perm, direct_max);
    kernels = 3;
    return cudaGetLastError();
}

cudaError_t launch_let_select(cudaStream_t s, const TreeView &t, const double *box, float theta,
                              float3 dlo, float3 dhi, const LetScratch &sc, int &kernels)
{
    kernels = 0;
    const int g = grid_cap(t.cap);
    for (int L = 0; L < LEVELS; ++L) {
        let_kind_kernel<<<g, TTPB, 0, s>>>(t, box, theta, dlo, dhi, L, sc.kind);
        ++kernels;
    }
    let_scan_kernel<<<1, 1024, 0, s>>>(t, sc);
    ++kernels;
    return cudaGetLastError();
}

cudaError_t launch_let_emit(cudaStream_t s, const TreeView &t, const double *box,
                            const LetScratch &sc, const float4 *P, const float4 *Plo, void *out,
                            int &kernels)
{
    let_emit_kernel<<<grid_cap(t.cap), TTPB, 0, s>>>(t, box, sc, P, Plo,
                                                     static_cast<unsigned char *>(out));
    kernels = 1;
    return cudaGetLastError();
}

namespace {

// Warps that walk one group together.  One warp per group is the most work per
// instruction, but a launch then lasts as long as its slowest groups' walks,
// and below a few groups per resident warp SMs idle.  Measured (walk alone, us,
// Plummer spheres, theta 0.5, leaves of 16; 1 / 4 / 8 warps per group):
//   groups of 64: 2000 bodies 108 / 58 / 39, 20000 389 / 163 / 101,
//     60000 516 / 314 / 280, 100000 627 / 442 / 463, 200000 893 / 774 / 870,
//     400000 1496 / 1497 / 1737, 800000 2746 / 3003 / 3570;
//   groups of 32: 20000 318 / 146 / 112, 60000 430 / 313 / 306,
//     100000 538 / 527 / 513, 200000 870 / 971 / 991.
// (2 warps per group were slower than 4 up to 400000 bodies, 16 than 8 from
// 20000 on.)  So 8 warps up to 8 groups per SM (20 of the smaller ones), 4 up
// to 40, then one.
int walk_split(int groups, int bodies_per_lane, int num_sms)
{
    if (bodies_per_lane == 1) return groups < 20 * num_sms ? 8 : 1;
    return groups < 8 * num_sms ? 8 : (groups < 40 * num_sms ? 4 : 1);
}

// The same for a walk over `trees` trees (a process's own and the LETs it
// received) in one launch, whose tasks are the (group, tree) pairs: what fills
// the SMs is their number.  Measured (walk alone, us, two Plummer spheres over P
// processes, theta 0.5, leaves of 16; 1 / 4 / 8 warps per task):
//   groups of 64: 1024 tasks (P = 4) 466 / 189 / 147, 2048 (P = 2) 720 / 388 /
//     360, (P = 8) 436 / 177 / 187, 4096 (P = 8) 578 / 246 / 348, 8192 (P = 2)
//     1294 / 1206 / 1436, (P = 8) 652 / 450 / 662, 16384 (P = 8) 779 / 882 / 1297;
//   groups of 32: 1024 (P = 2) 363 / 155 / 129, 2048 (P = 4) 386 / 172 / 186,
//     4096 (P = 2) 591 / 457 / 486, 8192 (P = 2) 723 / 884 / 1006, (P = 8) 423 /
//     362 / 487, 16384 (P = 8) 503 / 693 / 939.
// (By the groups alone, as for one tree, 8 x 65536 bodies in groups of 32 took
// 939 us, 8 x 131072 in groups of 64 882.)  Above 16 trees they are counted as
// 16 for the step from 8 to 4 warps: most are remote and walked in a few rounds.
int walk_split_trees(int groups, int trees, int bodies_per_lane, int num_sms)
{
    if (trees <= 1) return walk_split(groups, bodies_per_lane, num_sms);
    if (groups * (int64_t)min(trees, 16) < 12 * num_sms) return 8;
    return groups * (int64_t)trees < (bodies_per_lane == 1 ? 40 : 56) * num_sms ? 4 : 1;
}

template <int BPL, bool MULTI, int W>
cudaError_t walk_launch(cudaStream_t s, const TreeWalkParams &p, bool zeps, int tasks, int &kernels)
{
    void (*fn)(const TreeWalkParams) = zeps ? tree_walk_kernel<true, BPL, MULTI, W>
                                            : tree_walk_kernel<false, BPL, MULTI, W>;
    constexpr int threads = 32 * walk_warps(W);
    constexpr int smem = (int)sizeof(WalkShared<BPL, MULTI, W>);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    int blocks = W > 1 ? tasks : (tasks + WALK_WARPS - 1) / WALK_WARPS;
    if (p.sched != 0) {  // resident blocks only
        int per_sm = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
        if (e != cudaSuccess) return e;
        blocks = min(blocks, max(per_sm, 1) * p.num_sms);
    }
    fn<<<blocks, threads, smem, s>>>(p);
    kernels = 1;
    return cudaGetLastError();
}

template <int BPL, bool MULTI>
cudaError_t walk_launch_split(cudaStream_t s, const TreeWalkParams &p, bool zeps, int W, int tasks,
                              int &kernels)
{
    if (W == 8) return walk_launch<BPL, MULTI, 8>(s, p, zeps, tasks, kernels);
    if constexpr (BPL == 2 || MULTI)
        if (W == 4) return walk_launch<BPL, MULTI, 4>(s, p, zeps, tasks, kernels);
    return walk_launch<BPL, MULTI, 1>(s, p, zeps, tasks, kernels);
}

}  // namespace

cudaError_t launch_tree_walk(cudaStream_t s, const TreeWalkParams &p, bool zeps, int &kernels)
{
    kernels = 0;
    if (p.n <= 0) return cudaSuccess;
    if (p.nmore > 0 && (!p.tpart || !p.tcnt || !p.tctr || p.tspan < 1))
        return cudaErrorInvalidValue;
    const int bpl = p.group / 32;
    const int groups = (p.n + p.group - 1) / p.group;
    const int tasks = groups * (p.nmore > 0 ? (1 + p.nmore + p.tspan - 1) / p.tspan : 1);
    // (a task of several trees is one warp's)
    const int W = p.nmore > 0 && p.tspan > 1 ? 1 : walk_split_trees(groups, p.trees, bpl, p.num_sms);
    if (p.nmore > 0)  // a separate instance: the single-tree walk keeps its own registers
        return bpl == 1 ? walk_launch_split<1, true>(s, p, zeps, W, tasks, kernels)
                        : walk_launch_split<2, true>(s, p, zeps, W, tasks, kernels);
    return bpl == 1 ? walk_launch_split<1, false>(s, p, zeps, W, tasks, kernels)
                    : walk_launch_split<2, false>(s, p, zeps, W, tasks, kernels);
}

}  // namespace nb
