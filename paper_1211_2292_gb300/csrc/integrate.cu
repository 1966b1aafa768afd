// O(n) kernels around the pair kernels: packing the caller's float64
// (n,3)+(n) arrays into the internal (x,y,z,m) layout, the leapfrog's
// kick+drift (the reading of the paper's "Move_bodies", Sec. IV-B), the
// adjoint's drift/cotangent packing, and the final energy reduction.
//
// All are memory-bound one-thread-per-body kernels (grid-stride loops).
#include <cuda_runtime.h>

#include "nb_device.cuh"
#include "nb_internal.h"

namespace nb {
namespace {

constexpr int TPB = 256;

inline int grid_for(int n)
{
    int g = (n + TPB - 1) / TPB;
    return g < 1 ? 1 : (g > 65535 * 8 ? 65535 * 8 : g);
}

__device__ __forceinline__ void put(float4 *P, int i, double x, double y, double z, double m)
{
    P[i] = make_float4((float)x, (float)y, (float)z, (float)m);
}
__device__ __forceinline__ void put(double4 *P, int i, double x, double y, double z, double m)
{
    P[i] = make_double4(x, y, z, m);
}
// float32 hi/lo pair: x = hi + lo with hi = fl(x), lo = fl(x - hi); the lo
// slot's w carries log2 m for the log-domain pair factor (logm), else 0.
__device__ __forceinline__ void put_hilo(float4 *P, float4 *Plo, int i, double x, double y,
                                         double z, double m, bool logm)
{
    float4 h, l;
    split_f64(x, h.x, l.x);
    split_f64(y, h.y, l.y);
    split_f64(z, h.z, l.z);
    h.w = (float)m;
    l.w = logm ? log2_packed(m) : 0.f;
    P[i] = h;
    Plo[i] = l;
}

__global__ void pack_kernel(int n, const double *__restrict__ pos, const double *__restrict__ mass,
                            double4 *__restrict__ P)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const double *x = pos + 3 * (size_t)k;
        put(P, k, x[0], x[1], x[2], mass[k]);
    }
}

// One coordinate (index i = 3 body + axis, in packed order) of the force from a
// float32 force kernel's j-split slots: G * (slots merged in order).
__device__ __forceinline__ double merged_force(const MergeParams &g, size_t i)
{
    const double a = g.G * merge_slots(g.slots + i, (size_t)g.n * 3, g.nslots);
    if (!isfinite(a)) atomicOr(g.err, (int)ERR_NONFINITE);
    return a;
}

// The end of a split force evaluation: a thread per coordinate merges the
// slots, writes acc and applies the closing half-kick.  A launch of its own
// rather than the last CTA of each i-tile, whose 128 threads went through
// nslots x 6 bodies alone at the end of the launch; a thread per body took
// 9.2 us at 16384 bodies and 19 slots (dependent batches of loads).
__global__ void __launch_bounds__(128) merge_kernel(const MergeParams g, double *__restrict__ vel,
                                                    double half_dt)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3ll * g.n) return;
    const double a = merged_force(g, (size_t)i);
    const size_t b = g.perm ? 3 * (size_t)g.perm[i / 3] + (size_t)(i % 3) : (size_t)i;
    g.acc[b] = a;
    if (vel) vel[b] += half_dt * a;
}

// Opening half-kick and drift of one leapfrog step, then repack:
//   v += half_dt * a;  x += dt * v.
// (x, v) before the update are copied to rec_pos/rec_vel when given.  MERGE:
// first the end of the step before, whose force is still in its slots:
// a = G (slots merged), v += half_dt * a.
// MERGE takes 96 threads (32 bodies) a block, a thread per coordinate, whose
// new positions meet in shared memory for the packing.
constexpr int KM_T = 96;
__global__ void __launch_bounds__(KM_T)
    kdp_merge_kernel(int n, double *__restrict__ pos, double *__restrict__ vel,
                     const double *__restrict__ mass, double half_dt, double dt,
                     float4 *__restrict__ P, float4 *__restrict__ Plo, bool logm,
                     double *__restrict__ rec_pos, double *__restrict__ rec_vel,
                     const MergeParams g)
{
    __shared__ double xs[KM_T];
    const size_t i = (size_t)blockIdx.x * KM_T + threadIdx.x;
    if (i < 3 * (size_t)n) {
        double x = pos[i], v = vel[i];
        const double a = merged_force(g, i);
        g.acc[i] = a;
        v += half_dt * a;
        if (rec_pos) rec_pos[i] = x;
        if (rec_vel) rec_vel[i] = v;
        v += half_dt * a;
        x += dt * v;
        vel[i] = v;
        pos[i] = x;
        xs[threadIdx.x] = x;
    }
    __syncthreads();
    const int b = blockIdx.x * (KM_T / 3) + threadIdx.x;
    if (threadIdx.x < KM_T / 3 && b < n && P)
        put_hilo(P, Plo, b, xs[3 * threadIdx.x], xs[3 * threadIdx.x + 1], xs[3 * threadIdx.x + 2],
                 mass[b], logm);
}

template <typename V>
__global__ void kdp_kernel(int n, double *__restrict__ pos, double *__restrict__ vel,
                           const double *__restrict__ acc, const double *__restrict__ mass,
                           double half_dt, double dt, V *__restrict__ P, float4 *__restrict__ Plo,
                           bool logm, double *__restrict__ rec_pos, double *__restrict__ rec_vel)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double *x = pos + 3 * (size_t)i;
        double *v = vel + 3 * (size_t)i;
        const double *a = acc + 3 * (size_t)i;
        double xx = x[0], xy = x[1], xz = x[2];
        double vx = v[0], vy = v[1], vz = v[2];
        if (rec_pos) {
            double *r = rec_pos + 3 * (size_t)i;
            r[0] = xx; r[1] = xy; r[2] = xz;
        }
        if (rec_vel) {
            double *r = rec_vel + 3 * (size_t)i;
            r[0] = vx; r[1] = vy; r[2] = vz;
        }
        vx += half_dt * a[0];
        vy += half_dt * a[1];
        vz += half_dt * a[2];
        xx += dt * vx;
        xy += dt * vy;
        xz += dt * vz;
        v[0] = vx; v[1] = vy; v[2] = vz;
        x[0] = xx; x[1] = xy; x[2] = xz;
        if (Plo)
            put_hilo((float4 *)P, Plo, i, xx, xy, xz, mass[i], logm);
        else if (P)
            put(P, i, xx, xy, xz, mass[i]);
    }
}

// Adjoint packing: optional drift adjoint lam_v += drift * lam_x, then
// cotangent mu = coef * lam (lam = lam_v when given, else `lam`), packed as
// (x,y,z,m),(mu_x,mu_y,mu_z,0) in float64, or as hi/lo float32 positions plus
// mu in three arrays `stride` float4 apart.
template <typename V>
__global__ void pack_vjp_kernel(int n, const double *__restrict__ pos,
                                const double *__restrict__ mass, const double *__restrict__ lam,
                                double *__restrict__ lam_v, const double *__restrict__ lam_x,
                                double drift, double coef, V *__restrict__ PV, size_t stride)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double *x = pos + 3 * (size_t)i;
        double l0, l1, l2;
        if (lam_v) {
            double *lv = lam_v + 3 * (size_t)i;
            l0 = lv[0]; l1 = lv[1]; l2 = lv[2];
            if (lam_x) {
                const double *lx = lam_x + 3 * (size_t)i;
                l0 += drift * lx[0];
                l1 += drift * lx[1];
                l2 += drift * lx[2];
                lv[0] = l0; lv[1] = l1; lv[2] = l2;
            }
        } else {
            const double *l = lam + 3 * (size_t)i;
            l0 = l[0]; l1 = l[1]; l2 = l[2];
        }
        if (sizeof(V) == sizeof(double4)) {
            put(PV, 2 * i, x[0], x[1], x[2], mass[i]);
            put(PV, 2 * i + 1, coef * l0, coef * l1, coef * l2, 0.0);
        } else {
            float4 *F = reinterpret_cast<float4 *>(PV);
            put_hilo(F, F + stride, i, x[0], x[1], x[2], mass[i], false);
            put(F + 2 * stride, i, coef * l0, coef * l1, coef * l2, 0.0);
        }
    }
}

// out[0..8] = {E_kin, E_pot, E_tot, P_x, P_y, P_z, F_x, F_y, F_z} from the
// per-CTA partials, added in a fixed order by one CTA.
__global__ void energy_final_kernel(const double *__restrict__ red, int nparts, double G,
                                    double *__restrict__ out)
{
    __shared__ double sh[8][TPB];
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < nparts; b += TPB) {
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] += red[8 * (size_t)b + c];
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) sh[c][threadIdx.x] = v[c];
    __syncthreads();
    for (int w = TPB / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
#pragma unroll
            for (int c = 0; c < 8; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double ek = sh[0][0];
        const double ep = -0.5 * G * sh[1][0];
        out[0] = ek;
        out[1] = ep;
        out[2] = ek + ep;
        out[3] = sh[2][0];
        out[4] = sh[3][0];
        out[5] = sh[4][0];
        out[6] = G * sh[5][0];
        out[7] = G * sh[6][0];
        out[8] = G * sh[7][0];
    }
}

}  // namespace


cudaError_t launch_pack_f64(cudaStream_t s, int n, const double *pos, const double *mass,
                            double4 *P)
{
    pack_kernel<<<grid_for(n), TPB, 0, s>>>(n, pos, mass, P);
    return cudaGetLastError();
}

cudaError_t launch_kdp(cudaStream_t s, bool f64, int n, double *pos, double *vel,
                       const double *acc, const double *mass, double half_dt, double dt, void *P,
                       float4 *Plo, bool logm, double *rec_pos, double *rec_vel,
                       const MergeParams *merge)
{
    if (merge)
        kdp_merge_kernel<<<(unsigned)((3 * (int64_t)n + KM_T - 1) / KM_T), KM_T, 0, s>>>(
            n, pos, vel, mass, half_dt, dt, (float4 *)P, Plo, logm, rec_pos, rec_vel, *merge);
    else if (f64)
        kdp_kernel<double4><<<grid_for(n), TPB, 0, s>>>(n, pos, vel, acc, mass, half_dt, dt,
                                                         (double4 *)P, nullptr, false, rec_pos,
                                                         rec_vel);
    else
        kdp_kernel<float4><<<grid_for(n), TPB, 0, s>>>(n, pos, vel, acc, mass, half_dt, dt,
                                                        (float4 *)P, P ? Plo : nullptr, logm,
                                                        rec_pos, rec_vel);
    return cudaGetLastError();
}

cudaError_t launch_merge(cudaStream_t s, const MergeParams &g, double *vel, double half_dt)
{
    merge_kernel<<<(unsigned)((3 * (int64_t)g.n + 127) / 128), 128, 0, s>>>(g, vel, half_dt);
    return cudaGetLastError();
}

cudaError_t launch_pack_vjp(cudaStream_t s, bool f64, int n, const double *pos, const double *mass,
                            const double *lam, double *lam_v, const double *lam_x, double drift,
                            double coef, void *PV, size_t stride)
{
    if (f64)
        pack_vjp_kernel<double4><<<grid_for(n), TPB, 0, s>>>(n, pos, mass, lam, lam_v, lam_x,
                                                              drift, coef, (double4 *)PV, stride);
    else
        pack_vjp_kernel<float4><<<grid_for(n), TPB, 0, s>>>(n, pos, mass, lam, lam_v, lam_x,
                                                             drift, coef, (float4 *)PV, stride);
    return cudaGetLastError();
}

cudaError_t launch_energy_final(cudaStream_t s, const double *red, int nparts, double G,
                                double *out)
{
    energy_final_kernel<<<1, TPB, 0, s>>>(red, nparts, G, out);
    return cudaGetLastError();
}

}  // namespace nb
