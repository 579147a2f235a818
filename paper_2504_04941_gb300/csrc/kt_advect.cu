// kt_advect.cu -- stoichiometry-compatible species advection (Sec. 2.1.3 of the paper):
// one directional sweep of piecewise-linear reconstruction with the slope corrections
// projected onto the null space of the element matrix, upwind species fluxes
// F^s = x^s F^rho (Eq. method-flux-sp) and the conservative update, fused in one pass.
//
// The correction of a cell at its two interfaces is chi = +-dx/2 s (s: the limited
// slopes of x^s = n^s/rho), so projecting chi onto the stoichiometric space S = null(N)
// is projecting s once: s' = s - V_r (V_r^T s), with V_r an orthonormal basis of N's row
// space (rank <= 8).  That costs O(N_species N_elements) per cell instead of a dense
// N_species^2 product, and leaves N s' = 0 exactly up to rounding.
//
// Layout: lines of L cells, periodic; n[s][line][j] (species-major SoA), rho and the mass
// flux [line][j] (mass_flux[j] at the interface j-1/2).
//
// What bounds it: the FP64 pipe (2 lanes per clock per SM), not HBM: at ten species and two
// elements a cell and species costs 17 FP64 operations here, 1.1 ms of pipe time per sweep
// of 160^3 cells against 0.13 ms of traffic.  So the operations are what is saved: slopes
// are kept as half slopes times dx (no division by dx), the limiter's quotient is one
// reciprocal (a 20-bit seed and one cubic step) and two products, comparisons and the halving
// run on the bit patterns, dt/dx is folded into the mass flux once per cell, each interface's
// flux is formed once, and nothing is computed twice but x = n / rho in the second pass.
// A group of W lanes owns a window of 2 W cells, two per lane, of which the two at either
// end are halo; neighbours are exchanged by shuffles, so there is no block barrier, and
// only the half slopes wait in shared memory (a lane reads back its own) for the sum over
// species that the projection needs.  The first version (a block per 128 cells, slopes,
// fluxes and states through shared memory, ~35 operations, 8 of them the division) took
// 9.17 ms for the two stages of a step on 160^3 cells and ten species; this one 3.81 ms.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "kt_internal.h"

namespace kt {
namespace {

constexpr int kAdvMaxRank = kMaxElements;
constexpr int kAdvWarps = 4;

// NV: room for V_r [ns][rank]; the arguments travel as a kernel parameter, so a small
// network does not pay for a large one's table.
template <int NV>
struct AdvArgs {
    long long nlines, L, nseg;
    int ns, rank, W, vec;
    const double *n_in, *rho, *mflux, *n_base;
    double *n_out;
    double dtdx, alpha;
    double vr[NV];
};

// a b / s for sums whose reciprocal is subnormal.  Out of line: the division inlined under its
// branch is computed for every slope (one sweep of 160^3 cells, ten species: 1.8 -> 3.1 ms).
__device__ __noinline__ double large_quotient(double a, double b, double s) { return a / s * b; }

// dx / 2 times the slope of the modified van Leer limiter from the forward and backward
// differences a and b: min(a b / (a + b), b / 2) in magnitude (the first when |a| <= |b|),
// zero at extrema; the uniform-grid geometric factor 2c/(c+d) is 1.
// 1/s from the hardware's seed r by the geometric series of 1/(1 - e), e = 1 - s r, cut after
// e^2: the third-order (Chebyshev) iteration for a reciprocal.
__device__ __forceinline__ double half_slope(double a, double b)
{
    const double s = a + b;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(s));
    double e = fma(-s, r, 1.0);
    e = fma(e, e, e);
    r = fma(r, e, r);
    double q = (a * r) * b;
    const long long m = 0x7fffffffffffffffLL, inf = 0x7ff0000000000000LL, bit = 1LL << 52;
    const long long ba = __double_as_longlong(a), bb = __double_as_longlong(b), ia = ba & m, ib = bb & m;
    // b / 2: one less in the exponent; below 2^-1021, where a double is the integer of its bits
    // times 2^-1074, half of that integer (ties to even)
    const double half = __longlong_as_double(ib >= 2 * bit ? bb - bit : (bb & ~m) | ((ib + ((ib >> 1) & 1)) >> 1));
    if (__builtin_expect((__double_as_longlong(s) & m) >= 2045 * bit, 0)) q = large_quotient(a, b, s);
    // zero: signs differ, a zero or a NaN, or so small (2^-959) that a b underflows.  (|s|'s bits
    // are written out twice: kept in a variable, the compiler compares |s| on the FP64 pipe, one
    // operation more per slope, 1.81 -> 1.91 ms.)
    const bool zero = (ba ^ bb) < 0 || ia == 0 || ib == 0 || ia > inf || ib > inf ||
                      (__double_as_longlong(s) & m) < (64LL << 52);
    return zero ? 0.0 : (ia <= ib || ia == inf ? q : half);
}

template <int RK, int NV>
__global__ void __launch_bounds__(kAdvWarps * 32) advect_kernel(const __grid_constant__ AdvArgs<NV> p)
{
    extern __shared__ double2 adv_sm[];
    const int lane = threadIdx.x & 31, W = p.W, gl = lane & (W - 1), ns = p.ns;
    double2 *H = adv_sm + static_cast<size_t>(threadIdx.x >> 5) * ns * 32 + lane;
    const long long L = p.L;
    const long long unit = (static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (32 / W) +
                           (lane / W);
    const bool on = unit < p.nlines * p.nseg;
    const long long line = on ? unit / p.nseg : 0, seg = on ? unit - line * p.nseg : 0;
    const long long c0 = seg * (2 * W - 4) - 2 + 2 * gl;   // the lane's cells: c0, c0 + 1
    auto wrap = [&](long long j) { return j >= 0 && j < L ? j : ((j %= L) < 0 ? j + L : j); };
    const long long j0 = wrap(c0), j1 = wrap(c0 + 1), row = line * L, stride = p.nlines * L;
    const bool pair = p.vec && j1 == j0 + 1 && (j0 & 1) == 0;   // one 16-byte access
    const double inv0 = 1.0 / p.rho[row + j0], inv1 = 1.0 / p.rho[row + j1];
    // (the flux's own sign decides the upwind side: dt/dx may be negative)
    const double g0 = p.mflux[row + j0], g1 = p.mflux[row + j1], m0 = g0 * p.dtdx, m1 = g1 * p.dtdx;
    const bool up0 = g0 > 0.0, up1 = g1 > 0.0;
    auto load = [&](const double *a, int s) {
        const double *q = a + s * stride + row;
        if (pair) return *reinterpret_cast<const double2 *>(q + j0);
        return make_double2(q[j0], q[j1]);
    };
    double ca[RK], cb[RK];   // V_r^T times the half slopes of the two cells
#pragma unroll
    for (int k = 0; k < RK; ++k) ca[k] = cb[k] = 0.0;
#pragma unroll 2
    for (int s = 0; s < ns; ++s) {
        const double2 n = load(p.n_in, s);
        const double x0 = n.x * inv0, x1 = n.y * inv1;
        const double xn = __shfl_down_sync(0xffffffffu, x0, 1, W);
        const double d0 = x1 - x0, d1 = xn - x1;
        const double dp = __shfl_up_sync(0xffffffffu, d1, 1, W);
        const double2 h = make_double2(half_slope(d0, dp), half_slope(d1, d0));
        H[s * 32] = h;
#pragma unroll
        for (int k = 0; k < RK; ++k)
            if (k < p.rank) {
                const double v = p.vr[s * p.rank + k];
                ca[k] = fma(v, h.x, ca[k]);
                cb[k] = fma(v, h.y, cb[k]);
            }
    }
    const bool store = on && gl >= 1 && gl <= W - 2 && c0 < L, store1 = store && c0 + 1 < L;
    const double beta = 1.0 - p.alpha;
#pragma unroll 2
    for (int s = 0; s < ns; ++s) {
        double2 h = H[s * 32];
#pragma unroll
        for (int k = 0; k < RK; ++k)
            if (k < p.rank) {
                const double v = -p.vr[s * p.rank + k];
                h.x = fma(v, ca[k], h.x);
                h.y = fma(v, cb[k], h.y);
            }
        const double2 n = load(p.n_in, s);
        const double x0 = n.x * inv0, x1 = n.y * inv1;
        const double xp = __shfl_up_sync(0xffffffffu, x1, 1, W), hp = __shfl_up_sync(0xffffffffu, h.y, 1, W);
        // upwind states at the lower interfaces of the two cells, then dt/dx times the fluxes
        const double f0 = ((up0 ? xp : x0) + (up0 ? hp : -h.x)) * m0;
        const double f1 = ((up1 ? x0 : x1) + (up1 ? h.x : -h.y)) * m1;
        const double f2 = __shfl_down_sync(0xffffffffu, f0, 1, W);
        double v0 = n.x + (f0 - f1), v1 = n.y + (f1 - f2);
        if (p.n_base) {
            const double2 b = load(p.n_base, s);
            v0 = fma(p.alpha, b.x, beta * v0);
            v1 = fma(p.alpha, b.y, beta * v1);
        }
        if (store) {
            double *q = p.n_out + s * stride + row + c0;
            if (pair && store1) {
                *reinterpret_cast<double2 *>(q) = make_double2(v0, v1);
            } else {
                q[0] = v0;
                if (store1) q[1] = v1;
            }
        }
    }
}

template <int RK, int NV>
int launch_advect(const AdvArgs<kAdvMaxRank * 256> &h, const double *vr, cudaStream_t s)
{
    AdvArgs<NV> a{};
    a.nlines = h.nlines;
    a.L = h.L;
    a.nseg = h.nseg;
    a.ns = h.ns;
    a.rank = h.rank;
    a.W = h.W;
    a.vec = h.vec;
    a.n_in = h.n_in;
    a.rho = h.rho;
    a.mflux = h.mflux;
    a.n_base = h.n_base;
    a.n_out = h.n_out;
    a.dtdx = h.dtdx;
    a.alpha = h.alpha;
    for (int q = 0; q < h.ns * h.rank; ++q) a.vr[q] = vr[q];
    const size_t per_warp = static_cast<size_t>(h.ns) * 32 * sizeof(double2);
    int warps = kAdvWarps;
    while (warps > 1 && warps * per_warp > 64 * 1024) --warps;
    const size_t smem = warps * per_warp;
    cudaError_t e = cudaFuncSetAttribute(advect_kernel<RK, NV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    const long long units = h.nlines * h.nseg, per_block = static_cast<long long>(warps) * (32 / h.W);
    const long long blocks = (units + per_block - 1) / per_block;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    advect_kernel<RK, NV><<<static_cast<unsigned>(blocks), warps * 32, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace
}  // namespace kt

extern "C" KT_API int kt_advect_sweep(const kt_network *net, int64_t nlines, int64_t L, const double *n_in,
                                      const double *rho, const double *mass_flux, double dx, double dtdx,
                                      double alpha, const double *n_base, double *n_out, int project,
                                      void *scratch, void *cuda_stream)
{
    using namespace kt;
    int ns = 0, rank = 0;
    double vr[kAdvMaxRank * 256];
    int rc = network_element_basis(net, vr, &ns, &rank);
    if (rc) return rc;
    if (nlines < 0 || L < 0 || !(dx > 0) || !std::isfinite(dtdx) || ns > 256) {
        set_error("kt_advect_sweep: bad sizes or dx");
        return KT_EINVAL;
    }
    if (nlines == 0 || L == 0) return KT_OK;
    if (L < 3) {
        set_error("kt_advect_sweep: a periodic line needs at least 3 cells");
        return KT_EINVAL;
    }
    if (!n_in || !rho || !mass_flux || !n_out || !scratch || nlines > 65535) {
        set_error("kt_advect_sweep: NULL device buffer or more than 65535 lines");
        return KT_EINVAL;
    }
    if (n_out == n_in) {
        set_error("kt_advect_sweep: n_out must not alias n_in (neighbouring blocks read it)");
        return KT_EINVAL;
    }
    if (reinterpret_cast<uintptr_t>(scratch) % 16) {
        set_error("kt_advect_sweep: scratch not 16-B aligned");
        return KT_EINVAL;
    }
    // lanes per window: the width whose windows cover a line with the fewest lanes (wide
    // windows lose less to their halo, narrow ones pack several short lines into a warp)
    AdvArgs<kAdvMaxRank * 256> h{};
    long long best = -1;
    for (int W = 4; W <= 32; W *= 2) {
        const long long nseg = (L + 2 * W - 5) / (2 * W - 4);
        if (best < 0 || nseg * W < best) {
            best = nseg * W;
            h.W = W;
            h.nseg = nseg;
        }
    }
    auto aligned = [](const double *q) { return reinterpret_cast<uintptr_t>(q) % 16 == 0; };
    h.nlines = nlines;
    h.L = L;
    h.ns = ns;
    h.rank = project ? rank : 0;
    h.vec = L % 2 == 0 && aligned(n_in) && aligned(n_out) && (!n_base || aligned(n_base));
    h.n_in = n_in;
    h.rho = rho;
    h.mflux = mass_flux;
    h.n_base = n_base;
    h.n_out = n_out;
    h.dtdx = dtdx;
    h.alpha = alpha;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const int nv = ns * h.rank;
    const int e = h.rank <= 2 && nv <= 64 ? launch_advect<2, 64>(h, vr, s)
                  : h.rank <= 4 && nv <= 256 ? launch_advect<4, 256>(h, vr, s)
                                             : launch_advect<kAdvMaxRank, kAdvMaxRank * 256>(h, vr, s);
    if (e != cudaSuccess) {
        set_error(cudaGetErrorString(static_cast<cudaError_t>(e)));
        return KT_ECUDA;
    }
    return KT_OK;
}

// The kernel's arguments travel as parameters; the scratch of earlier callers is accepted
// and left untouched.
extern "C" KT_API size_t kt_advect_scratch_bytes(void) { return 16; }
