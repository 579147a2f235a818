// kt_ray.cu -- ray tracing on a Cartesian mesh with Beer-Lambert deposition (Sec. 3 of
// the paper: Eqs. cart-dl, method-rt-ph-num, method-rad-equiv-flux, method-rt-abs).
//
// One thread per ray.  The ray walks the cells it crosses by incremental face stepping
// (the exit length of a cell is the smallest root of the axis-plane equations of Eq.
// cart-dl; here an axis's next crossing distance is computed from the ray origin,
// t_a = (face_a - x0_a)/d_a, so no position error accumulates along the ray; only the axis
// just crossed has a new one).  In each cell it deposits, per energy bin, the path-averaged
// effective flux N dl/(dV dt) (1 - e^-tau)/tau and the absorbed photons N (1 - e^-tau),
// tau = kappa dl, into per-cell accumulators (FP64 atomics: rays cross shared cells), and
// carries N e^-tau on.  A walk crosses at most nx + ny + nz cells, which bounds the loop.
//
// What bounds it: the FP64 pipe (a warp instruction holds a scheduler's for 64 cycles), so a
// crossing's FP64 work is kept small: one face division instead of three, and e^-tau and
// 1 - e^-tau together from one table-driven exponential (13 operations; exp and expm1 took
// about 40) with the quotient by tau as a reciprocal (seed and one cubic step).  160^3 cells,
// two bins, 262,144 rays from one source: 15.7 ms before, 8.9 ms now.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "kt_internal.h"

namespace kt {
namespace {

constexpr int kRayMaxBins = 8;

struct RayArgs {
    int nx, ny, nz, nb;
    double hx, hy, hz, dt;
    long long nrays;
    const double *kappa, *org, *dir, *n0;
    double *feff, *absorbed, *escaped;
};

// 2^(j/256) and what its rounding to double leaves (kt_exp.cuh).
struct RayExpTable {
    double hi[kExpTable], lo[kExpTable];

    RayExpTable()
    {
        for (int j = 0; j < kExpTable; ++j) {
            hi[j] = exp2_table(j);
            lo[j] = static_cast<double>(std::exp2(static_cast<long double>(j) / static_cast<long double>(kExpTable)) -
                                        static_cast<long double>(hi[j]));
        }
    }
};

// Formed by the first call of the process: 512 long double powers take an Arm host, where that
// type is software, about 250 us (a trace of 64 rays through 4^3 cells: 78 us).
const RayExpTable &ray_exp_table()
{
    static const RayExpTable table;
    return table;
}

// e^-tau and 1 - e^-tau for 0 <= tau < 700: -tau = (256 m + j) ln2/256 + r, e^-tau =
// S (1 + p) with S = 2^(j/256) 2^m and p = e^r - 1 (kt_exp.cuh); 1 - e^-tau is summed as
// (1 - S) - S's rounding residue - S p, so it keeps its relative accuracy for small tau.
__device__ __forceinline__ void decay(double tau, const double2 *tab, double &att, double &gone)
{
    const double shift = 6755399441055744.0;            // 1.5 * 2^52
    const double t = fma(-tau, 369.3299304675746, shift);
    const int n = __double2loint(t), j = n & (kExpTable - 1), m = (n - j) >> 8;
    const double nd = t - shift;
    const double r = fma(-nd, 0x1.a39ef35793c76p-41, fma(-nd, 0x1.62e42fee00000p-9, -tau));
    // degree 5: the truncation (r^6/720 < 9e-21) stays below 1 - e^-tau's last bit
    double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    q = fma(r, q, 1.0 / 6.0);
    q = fma(r, q, 0.5);
    const double p = fma(r * r, q, r);
    const double2 e = tab[j];
    const double two_m = __hiloint2double((1023 + m) << 20, 0);
    const double S = __longlong_as_double(__double_as_longlong(e.x) + (static_cast<long long>(m) << 52));
    att = fma(S, p, S);
    gone = fma(-S, p, fma(-e.y, two_m, 1.0 - S));
}

// NB: energy bins held in registers (a.nb of them are there).
template <int NB>
__global__ void __launch_bounds__(128) ray_kernel(const RayArgs a, const __grid_constant__ RayExpTable table)
{
    __shared__ double2 tab[kExpTable];
    for (int j = threadIdx.x; j < kExpTable; j += blockDim.x) tab[j] = make_double2(table.hi[j], table.lo[j]);
    __syncthreads();
    const long long q = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q >= a.nrays) return;
    const double x0[3] = {a.org[3 * q], a.org[3 * q + 1], a.org[3 * q + 2]};
    const double d[3] = {a.dir[3 * q], a.dir[3 * q + 1], a.dir[3 * q + 2]};
    const double h[3] = {a.hx, a.hy, a.hz};
    const int n[3] = {a.nx, a.ny, a.nz};
    const long long jump[3] = {static_cast<long long>(a.ny) * a.nz, a.nz, 1};
    double N[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) N[b] = b < a.nb ? a.n0[q * a.nb + b] : 0.0;
    int c[3];
    bool inside = true;
    double tn[3];   // next face crossing of each axis, from the origin
    long long cell = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        c[k] = static_cast<int>(floor(x0[k] / h[k]));
        inside = inside && c[k] >= 0 && c[k] < n[k] && x0[k] >= 0.0;
        cell += c[k] * jump[k];
        if (d[k] > 0.0) tn[k] = ((c[k] + 1) * h[k] - x0[k]) / d[k];
        else if (d[k] < 0.0) tn[k] = (c[k] * h[k] - x0[k]) / d[k];
        else tn[k] = INFINITY;
    }
    const double dV = a.hx * a.hy * a.hz, inv_dVdt = 1.0 / (dV * a.dt);
    const long long ncell = static_cast<long long>(a.nx) * a.ny * a.nz;
    double t = 0.0;
    const int max_steps = a.nx + a.ny + a.nz + 3;
    for (int it = 0; inside && it < max_steps; ++it) {
        int ax = 0;
        double te = tn[0];
        if (tn[1] < te) {
            ax = 1;
            te = tn[1];
        }
        if (tn[2] < te) {
            ax = 2;
            te = tn[2];
        }
        double dl = te - t;
        if (dl < 0.0) dl = 0.0;
        const double path = dl * inv_dVdt;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if (b >= a.nb) break;
            const double tau = a.kappa[b * ncell + cell] * dl;
            double att, gone, phi;
            if (tau >= 0.0 && tau < 700.0) {
                decay(tau, tab, att, gone);
                // phi = (1 - e^-tau)/tau; 1 to the last bit below 2^-60.  1/tau by the third-order
                // (Chebyshev) iteration on the hardware's seed: r / (1 - e) ~ r (1 + e + e^2)
                double r;
                asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(tau));
                double e = fma(-tau, r, 1.0);
                e = fma(e, e, e);
                phi = tau > 0x1p-60 ? gone * fma(r, e, r) : 1.0;
            } else {
                att = exp(-tau);
                gone = 1.0 - att;
                phi = tau > 0.0 ? -expm1(-tau) / tau : 1.0;
            }
            atomicAdd(&a.feff[b * ncell + cell], N[b] * path * phi);
            atomicAdd(&a.absorbed[b * ncell + cell], N[b] * gone);
            N[b] *= att;
        }
        t = te;
        // step across the face; only that axis has a new crossing
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (k == ax) {
                const bool up = d[k] > 0.0;
                c[k] += up ? 1 : -1;
                cell += up ? jump[k] : -jump[k];
                inside = c[k] >= 0 && c[k] < n[k];
            }
        const double da = ax == 0 ? d[0] : (ax == 1 ? d[1] : d[2]), xa = ax == 0 ? x0[0] : (ax == 1 ? x0[1] : x0[2]);
        const double ha = ax == 0 ? h[0] : (ax == 1 ? h[1] : h[2]);
        const int ca = (ax == 0 ? c[0] : (ax == 1 ? c[1] : c[2])) + (da > 0.0 ? 1 : 0);
        const double tx = (ca * ha - xa) / da;
        if (ax == 0) tn[0] = tx;
        else if (ax == 1) tn[1] = tx;
        else tn[2] = tx;
    }
    if (a.escaped)
#pragma unroll
        for (int b = 0; b < NB; ++b)
            if (b < a.nb) a.escaped[q * a.nb + b] = N[b];
}

// Isotropic point source: Fibonacci-lattice directions (z_k = 1 - (2k+1)/n, azimuth
// k times the golden angle), solid angle 4 pi / n each, N = L dOmega/(4 pi) dt per bin.
constexpr double kPi = 3.141592653589793;

__device__ __forceinline__ void point_source_ray(long long k, double sx, double sy, double sz,
                                                 const double *lum_dt_over_n, int nb, long long nrays, double *org,
                                                 double *dir, double *n0)
{
    const double golden = kPi * (3.0 - sqrt(5.0));
    const double z = 1.0 - (2.0 * static_cast<double>(k) + 1.0) / static_cast<double>(nrays);
    const double r = sqrt(fmax(0.0, 1.0 - z * z));
    const double ph = static_cast<double>(k) * golden;
    double s, c;
    sincos(ph, &s, &c);
    org[3 * k] = sx;
    org[3 * k + 1] = sy;
    org[3 * k + 2] = sz;
    dir[3 * k] = r * c;
    dir[3 * k + 1] = r * s;
    dir[3 * k + 2] = z;
    for (int b = 0; b < nb; ++b) n0[k * nb + b] = lum_dt_over_n[b];
}

struct LumArg {
    double v[kRayMaxBins];
};

__global__ void point_source_kernel(double sx, double sy, double sz, const LumArg lum, int nb, long long nrays,
                                    double *org, double *dir, double *n0)
{
    const long long k = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (k < nrays) point_source_ray(k, sx, sy, sz, lum.v, nb, nrays, org, dir, n0);
}

}  // namespace
}  // namespace kt

extern "C" KT_API int kt_raytrace(int nx, int ny, int nz, double hx, double hy, double hz, int nbins,
                                  const double *kappa, int64_t nrays, const double *origins,
                                  const double *dirs, const double *n0, double dt, double *feff,
                                  double *absorbed, double *escaped, void *cuda_stream)
{
    if (nx < 1 || ny < 1 || nz < 1 || !(hx > 0) || !(hy > 0) || !(hz > 0) || nbins < 1 ||
        nbins > kt::kRayMaxBins || nrays < 0 || !(dt > 0)) {
        kt::set_error("kt_raytrace: bad grid, bins, ray count or dt");
        return KT_EINVAL;
    }
    if (nrays == 0) return KT_OK;
    if (!kappa || !origins || !dirs || !n0 || !feff || !absorbed) {
        kt::set_error("kt_raytrace: NULL device buffer");
        return KT_EINVAL;
    }
    kt::RayArgs a{nx, ny, nz, nbins, hx, hy, hz, dt, nrays, kappa, origins, dirs, n0, feff, absorbed, escaped};
    const kt::RayExpTable &tab = kt::ray_exp_table();
    const int threads = 128;
    const unsigned blocks = static_cast<unsigned>((nrays + threads - 1) / threads);
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (nbins == 1) kt::ray_kernel<1><<<blocks, threads, 0, s>>>(a, tab);
    else if (nbins == 2) kt::ray_kernel<2><<<blocks, threads, 0, s>>>(a, tab);
    else if (nbins <= 4) kt::ray_kernel<4><<<blocks, threads, 0, s>>>(a, tab);
    else kt::ray_kernel<kt::kRayMaxBins><<<blocks, threads, 0, s>>>(a, tab);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        kt::set_error(cudaGetErrorString(e));
        return KT_ECUDA;
    }
    return KT_OK;
}

extern "C" KT_API int kt_rays_point_source(const double *src, const double *lum, int nbins, double dt,
                                           int64_t nrays, double *origins, double *dirs, double *n0,
                                           void *cuda_stream)
{
    if (!src || !lum || nbins < 1 || nbins > kt::kRayMaxBins || nrays < 1 || !(dt > 0) || !origins || !dirs ||
        !n0) {
        kt::set_error("kt_rays_point_source: bad argument");
        return KT_EINVAL;
    }
    kt::LumArg l{};
    for (int b = 0; b < nbins; ++b) l.v[b] = lum[b] * dt / static_cast<double>(nrays);
    const int threads = 128;
    kt::point_source_kernel<<<static_cast<unsigned>((nrays + threads - 1) / threads), threads, 0,
                                static_cast<cudaStream_t>(cuda_stream)>>>(src[0], src[1], src[2], l, nbins, nrays,
                                                                          origins, dirs, n0);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        kt::set_error(cudaGetErrorString(e));
        return KT_ECUDA;
    }
    return KT_OK;
}
