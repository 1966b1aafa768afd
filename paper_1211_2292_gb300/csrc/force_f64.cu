// float64 force and energy kernels (paper Sec. IV-A/IV-B force calculation
// as the exact all-pairs sum, every operation in float64).
//
// An i-tile of T*I bodies per CTA in registers, j-bodies streamed through a
// double-buffered shared tile of J double4 (x,y,z,m), the grid split over j in
// equal body counts with the last arriving CTA adding the float64 partials in
// split order.  The force kernel's pair terms and sums are integers
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

constexpr int UNROLL_F64 = 2;  // pairs in flight: 2.47 ms at 16384 bodies (1: 2.54, 4: 2.61)

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

// Sums over the j-bodies [jlo, jhi) for the energy kernel.
template <int T, int I, int J, bool ZEPS>
__device__ __forceinline__ void energy_sweep(const double4 *__restrict__ P, int jlo, int jhi,
                                             double eps2, const double (&xi)[I],
                                             const double (&yi)[I], const double (&zi)[I],
                                             const int (&ii)[I], double (&ax)[I], double (&ay)[I],
                                             double (&az)[I], double (&ph)[I], double4 (*tile)[J])
{
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
#pragma unroll 4
        for (int jj = 0; jj < J; ++jj) {
            const double4 q = s[jj];
#pragma unroll
            for (int k = 0; k < I; ++k) {
                const double dx = q.x - xi[k], dy = q.y - yi[k], dz = q.z - zi[k];
                const double ri = pair_rinv<ZEPS>(fma(dz, dz, fma(dy, dy, fma(dx, dx, eps2))));
                const double mri = q.w * ri;
                const double sc = mri * (ri * ri);
                ax[k] = fma(dx, sc, ax[k]);
                ay[k] = fma(dy, sc, ay[k]);
                az[k] = fma(dz, sc, az[k]);
                ph[k] += (j0 + jj == ii[k]) ? 0.0 : mri;
            }
        }
        if (j0 + J < jhi) stage_store64<T, J>(tile[b ^ 1], buf);
        __syncthreads();
    }
}

// Sums over the j-bodies [jlo, jhi), in tiles of J from jlo on; the last tile
// stops at the next multiple of the step (massless bodies, which add nothing).
// Masses are brought into their integer form once per tile.
template <int T, int I, int J, bool ZEPS>
__device__ __forceinline__ void force_sweep(const double4 *__restrict__ P, int jlo, int jhi,
                                            double eps2, const double (&xi)[I],
                                            const double (&yi)[I], const double (&zi)[I],
                                            double (&a)[I][3], double4 (*tile)[J],
                                            MassFixed (*mtile)[J])
{
    const EpsFixed ef = eps_fixed(eps2);
    double4 buf[J / T];
    auto store = [&](int b) {
        stage_store64<T, J>(tile[b], buf);
#pragma unroll
        for (int l = 0; l < J / T; ++l) mtile[b][l * T + threadIdx.x] = mass_fixed(buf[l].w);
    };
    FixedSum<J> sum[I][3];
#pragma unroll
    for (int k = 0; k < I; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) sum[k][c].reset();
    if (jlo < jhi) {
        stage_load64<T, J>(buf, P, jlo, jhi);
        store(0);
    }
    __syncthreads();
    int b = 0;
    for (int j0 = jlo; j0 < jhi; j0 += J, b ^= 1) {
        if (j0 + J < jhi) stage_load64<T, J>(buf, P, j0 + J, jhi);
        const double4 *s = tile[b];
        const MassFixed *ms = mtile[b];
        const int jn = min(J, jhi - j0);
        for (int jj = 0; jj < jn; jj += UNROLL_F64) {
#pragma unroll
            for (int k = 0; k < I; ++k) {
                // a step's terms first (independent chains), then in one branch
                // the rare pairs of the general form
                PairTerm t[UNROLL_F64];
                int sign[UNROLL_F64][3];
                bool general = false;
#pragma unroll
                for (int u = 0; u < UNROLL_F64; ++u) {
                    const double4 q = s[jj + u];
                    const MassFixed m = ms[jj + u];
                    const double dx = q.x - xi[k], dy = q.y - yi[k], dz = q.z - zi[k];
                    general |= !pair_term<ZEPS>(dx, dy, dz, m, ef, t[u]);
                    sign[u][0] = (__double2hiint(dx) ^ (m.e2 << 31)) >> 31;
                    sign[u][1] = (__double2hiint(dy) ^ (m.e2 << 31)) >> 31;
                    sign[u][2] = (__double2hiint(dz) ^ (m.e2 << 31)) >> 31;
                }
                if (general) {
#pragma unroll
                    for (int u = 0; u < UNROLL_F64; ++u) {
                        const double4 q = s[jj + u];
                        const MassFixed m = ms[jj + u];
                        const double dx = q.x - xi[k], dy = q.y - yi[k], dz = q.z - zi[k];
                        // a body and itself: no force, unless its factor overflows
                        if (in_integer_form(dx, dy, dz, m) ||
                            (dx == 0.0 && dy == 0.0 && dz == 0.0 && m.lim && m.e2 < 1000 &&
                             (ZEPS || ef.e > 863)))
                            continue;
                        const double sc = pair_factor_general<ZEPS>(dx, dy, dz, q.w, eps2);
                        a[k][0] = fma(dx, sc, a[k][0]);
                        a[k][1] = fma(dy, sc, a[k][1]);
                        a[k][2] = fma(dz, sc, a[k][2]);
                    }
                }
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    int e = sum[k][c].E;
#pragma unroll
                    for (int u = 0; u < UNROLL_F64; ++u) e = max(e, t[u].e[c]);
                    sum[k][c].raise(e);
                }
#pragma unroll
                for (int u = 0; u < UNROLL_F64; ++u)
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        sum[k][c].add(t[u].A[c], t[u].S, t[u].e[c], sign[u][c]);
            }
        }
#pragma unroll
        for (int k = 0; k < I; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) a[k][c] += sum[k][c].take();
        if (j0 + J < jhi) store(b ^ 1);
        __syncthreads();
    }
}

template <int T, int I, int J, bool ZEPS>
__global__ void __launch_bounds__(T) force_f64_kernel(const ForceParams p)
{
    constexpr int TILE_I = T * I;
    __shared__ __align__(16) double4 tile[2][J];
    __shared__ __align__(16) MassFixed mtile[2][J];
    __shared__ int s_last;
    const double4 *P = static_cast<const double4 *>(p.P);
    const int n = p.n;
    const int n_itiles = (n + TILE_I - 1) / TILE_I;
    const int it = blockIdx.x % n_itiles;
    const int js = blockIdx.x / n_itiles;
    const int i0 = it * TILE_I;
    const int jlo = (int)((long long)n * js / p.nsplit);  // an equal share of the bodies
    const int jhi = (int)((long long)n * (js + 1) / p.nsplit);

    double xi[I], yi[I], zi[I], a[I][3];
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const int i = i0 + threadIdx.x + k * T;
        const double4 b = i < n ? P[i] : make_double4(0.0, 0.0, 0.0, 0.0);
        xi[k] = b.x;
        yi[k] = b.y;
        zi[k] = b.z;
        a[k][0] = a[k][1] = a[k][2] = 0.0;
    }
    force_sweep<T, I, J, ZEPS>(P, jlo, jhi, p.eps2, xi, yi, zi, a, tile, mtile);

    if (p.nsplit == 1) {
#pragma unroll
        for (int k = 0; k < I; ++k) {
            const int i = i0 + threadIdx.x + k * T;
            if (i < n) {
                double *o = p.acc + 3 * (size_t)i;
                const double gx = p.G * a[k][0], gy = p.G * a[k][1], gz = p.G * a[k][2];
                o[0] = gx;
                o[1] = gy;
                o[2] = gz;
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
            q[0] = a[k][0];
            q[1] = a[k][1];
            q[2] = a[k][2];
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
            double *o = p.acc + 3 * (size_t)i;
            const double gx = p.G * t[0], gy = p.G * t[1], gz = p.G * t[2];
            o[0] = gx;
            o[1] = gy;
            o[2] = gz;
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
    energy_sweep<T, I, J, ZEPS>(P, t0 * J, min(t1 * J, n), p.eps2, xi, yi, zi, ii, ax, ay, az, ph, tile);

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
