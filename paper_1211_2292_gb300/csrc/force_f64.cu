// float64 force and energy kernels (paper Sec. IV-A/IV-B force calculation
// as the exact all-pairs sum, every operation in float64).
//
// An i-tile of T*I bodies per CTA in registers, j-bodies streamed through a
// double-buffered shared tile of J double4 (x,y,z,m), the grid split over j in
// equal body counts with the last arriving CTA adding the float64 partials in
// split order.  The force kernel's pair factor is formed on the integer pipe
// (f64_pair.cuh); the energy kernel, which also needs the potential, refines a
// float32 MUFU seed of the reciprocal root by one second-order Householder
// step (nb_device.cuh).
//
// The energy kernel also accumulates the softened potential
// phi_i = sum_{j != i} m_j / s_ij (self pair skipped by index) and reduces,
// per CTA, E_pot = -G/2 sum m_i phi_i, F = G sum m_i a_i and (split 0 only)
// E_kin and P; a single-CTA kernel adds the per-CTA values in order.
#include <cuda_runtime.h>

#include "nb_device.cuh"
#include "f64_pair.cuh"
#include "nb_internal.h"

namespace nb {
namespace {

constexpr int UNROLL_F64 = 2;

template <int T, int J>
__device__ __forceinline__ void stage_load64(double4 (&buf)[J / T], const double4 *__restrict__ P,
                                             int jbase, int jend)
{
#pragma unroll
    for (int l = 0; l < J / T; ++l) {
        const int j = jbase + l * T + threadIdx.x;
        buf[l] = j < jend ? P[j] : make_double4(0.0, 0.0, 0.0, 0.0);
    }
}

template <int T, int J>
__device__ __forceinline__ void stage_store64(double4 *tile, const double4 (&buf)[J / T])
{
#pragma unroll
    for (int l = 0; l < J / T; ++l) tile[l * T + threadIdx.x] = buf[l];
}

template <bool ZEPS>
__device__ __forceinline__ double pair_rinv(double r2)
{
    double ri = rsqrt_f64(r2);
    if (ZEPS) ri = r2 > 0.0 ? ri : 0.0;
    return ri;
}

template <int T, int I, int J, bool ZEPS, bool ENERGY>
__device__ __forceinline__ void sweep64(const double4 *__restrict__ P, int jlo, int jhi,
                                        double eps2, const double (&xi)[I], const double (&yi)[I],
                                        const double (&zi)[I], const int (&ii)[I], double (&ax)[I],
                                        double (&ay)[I], double (&az)[I], double (&ph)[I],
                                        double4 (*tile)[J])
{
    const EpsFixed ef = eps_fixed(eps2);
    // j-bodies [jlo, jhi) in tiles of J from jlo on; the last tile stops at the
    // next multiple of the unrolling (massless bodies, which add nothing)
    double4 buf[J / T];
    if (jlo < jhi) {
        stage_load64<T, J>(buf, P, jlo, jhi);
        stage_store64<T, J>(tile[0], buf);
    }
    __syncthreads();
    int b = 0;
    for (int j0 = jlo; j0 < jhi; j0 += J, b ^= 1) {
        if (j0 + J < jhi) stage_load64<T, J>(buf, P, j0 + J, jhi);
        const double4 *s = tile[b];
        const int jn = min(J, jhi - j0);
        for (int jj = 0; jj < jn; jj += UNROLL_F64) {
            if (ENERGY) {
#pragma unroll
                for (int u = 0; u < UNROLL_F64; ++u) {
                    const double4 q = s[jj + u];
#pragma unroll
                    for (int k = 0; k < I; ++k) {
                        const double dx = q.x - xi[k], dy = q.y - yi[k], dz = q.z - zi[k];
                        const double ri = pair_rinv<ZEPS>(fma(dz, dz, fma(dy, dy, fma(dx, dx, eps2))));
                        const double mri = q.w * ri;
                        const double sc = mri * (ri * ri);
                        ax[k] = fma(dx, sc, ax[k]);
                        ay[k] = fma(dy, sc, ay[k]);
                        az[k] = fma(dz, sc, az[k]);
                        ph[k] += (j0 + jj + u == ii[k]) ? 0.0 : mri;
                    }
                }
            } else {
                // all of a step's factors first (independent chains), then the
                // rare ones that need the general form in one branch
                double dx[UNROLL_F64][I], dy[UNROLL_F64][I], dz[UNROLL_F64][I], sc[UNROLL_F64][I];
                unsigned general = 0;
#pragma unroll
                for (int u = 0; u < UNROLL_F64; ++u) {
                    const double4 q = s[jj + u];
#pragma unroll
                    for (int k = 0; k < I; ++k) {
                        dx[u][k] = q.x - xi[k];
                        dy[u][k] = q.y - yi[k];
                        dz[u][k] = q.z - zi[k];
                        double r;
                        if (!pair_inv_cube<ZEPS>(dx[u][k], dy[u][k], dz[u][k], ef, r))
                            general |= 1u << (u * I + k);
                        sc[u][k] = q.w * r;
                    }
                }
                if (general) {
#pragma unroll
                    for (int u = 0; u < UNROLL_F64; ++u)
#pragma unroll
                        for (int k = 0; k < I; ++k)
                            if (general >> (u * I + k) & 1)
                                sc[u][k] = pair_factor_general<ZEPS>(dx[u][k], dy[u][k], dz[u][k],
                                                                     s[jj + u].w, eps2);
                }
#pragma unroll
                for (int u = 0; u < UNROLL_F64; ++u)
#pragma unroll
                    for (int k = 0; k < I; ++k) {
                        ax[k] = fma(dx[u][k], sc[u][k], ax[k]);
                        ay[k] = fma(dy[u][k], sc[u][k], ay[k]);
                        az[k] = fma(dz[u][k], sc[u][k], az[k]);
                    }
            }
        }
        if (j0 + J < jhi) stage_store64<T, J>(tile[b ^ 1], buf);
        __syncthreads();
    }
}

template <int T, int I, int J, bool ZEPS>
__global__ void __launch_bounds__(T) force_f64_kernel(const ForceParams p)
{
    constexpr int TILE_I = T * I;
    __shared__ __align__(16) double4 tile[2][J];
    __shared__ int s_last;
    const double4 *P = static_cast<const double4 *>(p.P);
    const int n = p.n;
    const int n_itiles = (n + TILE_I - 1) / TILE_I;
    const int it = blockIdx.x % n_itiles;
    const int js = blockIdx.x / n_itiles;
    const int i0 = it * TILE_I;
    const int jlo = (int)((long long)n * js / p.nsplit);  // an equal share of the bodies
    const int jhi = (int)((long long)n * (js + 1) / p.nsplit);

    double xi[I], yi[I], zi[I], ax[I], ay[I], az[I], ph[I];
    int ii[I];
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const int i = i0 + threadIdx.x + k * T;
        const double4 b = i < n ? P[i] : make_double4(0.0, 0.0, 0.0, 0.0);
        xi[k] = b.x;
        yi[k] = b.y;
        zi[k] = b.z;
        ii[k] = i;
        ax[k] = ay[k] = az[k] = ph[k] = 0.0;
    }
    sweep64<T, I, J, ZEPS, false>(P, jlo, jhi, p.eps2, xi, yi, zi, ii, ax, ay, az, ph, tile);

    if (p.nsplit == 1) {
#pragma unroll
        for (int k = 0; k < I; ++k) {
            const int i = i0 + threadIdx.x + k * T;
            if (i < n) {
                double *a = p.acc + 3 * (size_t)i;
                const double gx = p.G * ax[k], gy = p.G * ay[k], gz = p.G * az[k];
                a[0] = gx;
                a[1] = gy;
                a[2] = gz;
                if (p.vel) {
                    double *v = p.vel + 3 * (size_t)i;
                    v[0] += p.half_dt * gx;
                    v[1] += p.half_dt * gy;
                    v[2] += p.half_dt * gz;
                }
                if (!finite3(gx, gy, gz)) atomicOr(p.err, ERR_NONFINITE);
            }
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const int i = i0 + threadIdx.x + k * T;
        if (i < n) {
            double *q = p.partial + ((size_t)js * n + i) * 3;
            q[0] = ax[k];
            q[1] = ay[k];
            q[2] = az[k];
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(p.counters + it, 1u) == (unsigned)(p.nsplit - 1));
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const int i = i0 + threadIdx.x + k * T;
        if (i < n) {
            double t[3];
            sum_slots(p.partial + (size_t)i * 3, (size_t)n * 3, p.nsplit, t);
            double *a = p.acc + 3 * (size_t)i;
            const double gx = p.G * t[0], gy = p.G * t[1], gz = p.G * t[2];
            a[0] = gx;
            a[1] = gy;
            a[2] = gz;
            if (p.vel) {
                double *v = p.vel + 3 * (size_t)i;
                v[0] += p.half_dt * gx;
                v[1] += p.half_dt * gy;
                v[2] += p.half_dt * gz;
            }
            if (!finite3(gx, gy, gz)) atomicOr(p.err, ERR_NONFINITE);
        }
    }
    if (threadIdx.x == 0) p.counters[it] = 0u;
}

// Fixed-order CTA sum of NV doubles per thread (tree over shared memory).
template <int T, int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double (*sh)[T])
{
#pragma unroll
    for (int c = 0; c < NV; ++c) sh[c][threadIdx.x] = v[c];
    __syncthreads();
    for (int w = T / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
#pragma unroll
            for (int c = 0; c < NV; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < NV; ++c) v[c] = sh[c][0];
}

// Energy/momentum partials.  red[block][0..7] =
// {E_kin, sum m_i phi_i, P_x, P_y, P_z, sum m_i a_x, sum m_i a_y, sum m_i a_z}
// (G and the -1/2 are applied by the final kernel).
template <int T, int I, int J, bool ZEPS>
__global__ void __launch_bounds__(T) energy_f64_kernel(const EnergyParams p)
{
    constexpr int TILE_I = T * I;
    __shared__ __align__(16) double4 tile[2][J];
    __shared__ double sh[8][T];
    const double4 *P = p.P;
    const int n = p.n;
    const int n_itiles = (n + TILE_I - 1) / TILE_I;
    const int it = blockIdx.x % n_itiles;
    const int js = blockIdx.x / n_itiles;
    const int i0 = it * TILE_I;
    int t0, t1;
    split_range((n + J - 1) / J, p.nsplit, js, t0, t1);

    double xi[I], yi[I], zi[I], mi[I], ax[I], ay[I], az[I], ph[I];
    int ii[I];
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const int i = i0 + threadIdx.x + k * T;
        const double4 b = i < n ? P[i] : make_double4(0.0, 0.0, 0.0, 0.0);
        xi[k] = b.x;
        yi[k] = b.y;
        zi[k] = b.z;
        mi[k] = b.w;  // zero for padding bodies, so they add nothing
        ii[k] = i;
        ax[k] = ay[k] = az[k] = ph[k] = 0.0;
    }
    sweep64<T, I, J, ZEPS, true>(P, t0 * J, min(t1 * J, n), p.eps2, xi, yi, zi, ii, ax, ay, az, ph, tile);

    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const int i = i0 + threadIdx.x + k * T;
        v[1] += mi[k] * ph[k];
        v[5] += mi[k] * ax[k];
        v[6] += mi[k] * ay[k];
        v[7] += mi[k] * az[k];
        if (js == 0 && i < n) {
            const double *vi = p.vel + 3 * (size_t)i;
            const double vx = vi[0], vy = vi[1], vz = vi[2];
            v[0] += 0.5 * mi[k] * (vx * vx + vy * vy + vz * vz);
            v[2] += mi[k] * vx;
            v[3] += mi[k] * vy;
            v[4] += mi[k] * vz;
        }
    }
    block_sum<T, 8>(v, sh);
    if (threadIdx.x == 0) {
        double *r = p.red + 8 * (size_t)blockIdx.x;
#pragma unroll
        for (int c = 0; c < 8; ++c) r[c] = v[c];
    }
}

#define NB_F64_ENTRY(T, I, J)                                            \
    {{T, I, J, (const void *)force_f64_kernel<T, I, J, false>},          \
     {T, I, J, (const void *)force_f64_kernel<T, I, J, true>}}

typedef KernelEntry Pair[2];
const Pair kF64[] = {
    NB_F64_ENTRY(128, 1, 128),
    NB_F64_ENTRY(128, 2, 128),
    NB_F64_ENTRY(256, 2, 256),
    NB_F64_ENTRY(64, 2, 128),
};
const Pair kEnergy = {{128, 1, 128, (const void *)energy_f64_kernel<128, 1, 128, false>},
                      {128, 1, 128, (const void *)energy_f64_kernel<128, 1, 128, true>}};

}  // namespace

int f64_force_variants() { return (int)(sizeof(kF64) / sizeof(kF64[0])); }
const KernelEntry &f64_force_kernel(int v, bool zeps) { return kF64[v][zeps]; }
const KernelEntry &f64_energy_kernel(bool zeps) { return kEnergy[zeps]; }

}  // namespace nb
