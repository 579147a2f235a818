// kt_warp.cuh -- one to four warps per cell, for larger networks (N <= 96 unknowns).
//
// What bounds it: every FP64 instruction of a warp holds its scheduler's pipe for 64 cycles,
// and a launch lasts at least as long as its longest cell, so what counts is the number of
// FP64 instructions in one Newton iteration of one cell.  A team of NW warps owns a cell
// (the paper's Sec. 2.3 gives it a thread block): with four, each on a scheduler of its own,
// four FP64 pipes work on the cell.  Inside the team:
//   rates          threads over reactions (modified Arrhenius, Sec. 2.2.1): the rate w_r and,
//                  when a Jacobian is wanted, its partial derivatives, each formed once in
//                  FP64 and rounded once (the rows below only add them);
//   f and J rows   threads over species rows of f, each walking its own list of (reaction,
//                  +-1) entries; threads over the entries of J, each entry's terms summed by
//                  one thread in the same order (a program the host lays out once): fixed
//                  orders, no atomics (Eq. method-jacobian);
//   T row          threads over columns: J_T,m = -sum_s h_s J_s,m / C_V, and I - h J of the
//                  column in the same pass;
//   LU             right-looking with the implicit-scaled row pivoting of Algorithm
//                  lu-decomp (same factors as Crout's ordering, other rounding) on a
//                  column-major matrix: every warp finds the pivot by itself (integer
//                  reductions on the bit patterns, ties to the smaller row), threads over
//                  columns exchange the rows and update 16 bytes at a time; two team
//                  barriers per step;
//   solve          warp 0, the right-hand side in registers, NQ rows per lane, each finished
//                  entry broadcast by a shuffle.
// Sums over species go through the same 32 partial sums and shuffle tree whatever the team's
// size, so every team size gives the same bits.  The sub-step control (step doubling or
// TR-BDF2, Newton, retry / revert, projection) is the same sequence as the FP64 oracle, run
// team-uniformly.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "kt_exp.cuh"
#include "kt_internal.h"
#include "kt_tma.cuh"
#include "kt_trbdf2.cuh"

namespace kt {
namespace {

constexpr unsigned kFull = 0xffffffffu;

struct NetS {
    const double *A, *b, *th, *h, *cv, *cnt, *ex;
    const unsigned long long *idx;
    const int *rp, *re;
};

__device__ __forceinline__ double wsum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return __shfl_sync(kFull, v, 0);
}

// x < -700 decided on the bit pattern (integer compare; same result as the FP64 compare
// for every non-NaN x): negative and |x| > 700.0 (0x4085E00000000000).
__device__ __forceinline__ bool below_m700(double x)
{
    const long long b = __double_as_longlong(x);
    return b < 0 && (b & 0x7fffffffffffffffLL) > 0x4085E00000000000LL;
}

// log(T / T_ref), skipping the division when T_ref is 1 (the same value bit for bit).
__device__ __forceinline__ double log_t(double T, double t_ref)
{
    return log(t_ref == 1.0 ? T : T / t_ref);
}

__device__ __forceinline__ void arrhenius(const NetS &t, int r, double lt, double invT, double &k, double &dk)
{
    const double b = t.b[r], th = t.th[r];
    // (no branch: the exponentials of two reactions run interleaved)
    const double arg = fma(b, lt, -__dmul_rn(th, invT));
    const bool zero = below_m700(arg);
    const double v = __dmul_rn(t.A[r], tang_exp(zero ? -700.0 : arg, t.ex));
    k = zero ? 0.0 : v;
    dk = __dmul_rn(__dmul_rn(k, fma(th, invT, b)), invT);
}

// phi(tau) = (1 - e^-tau)/tau of Eq. photo-reaction-single and its derivative; below
// tau = 0.1 by their Taylor series (8 terms), where the closed forms cancel.
__device__ __forceinline__ void photo_phi(double tau, double &phi, double &dphi)
{
    if (tau < 0.1) {
        double p = 0.0, d = 0.0, pw = 1.0, pwm = 0.0, fact = 1.0;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            fact *= (k + 1);
            const double sg = (k & 1) ? -1.0 : 1.0;
            p += sg * pw / fact;
            if (k >= 1) d += sg * k * pwm / fact;
            pwm = pw;
            pw *= tau;
        }
        phi = p;
        dphi = d;
    } else {
        const double e = exp(-tau);
        phi = (1.0 - e) / tau;
        dphi = (e * (1.0 + tau) - 1.0) / (tau * tau);
    }
}

// Tabulated rate (Sec. 2.2.1 item 3) of table row tr at T (lT = ln T) for a cell whose
// density sits at weight w between density nodes iR and iR + 1: ln k linear in ln rho
// between those rows (the per-cell reduction of Sec. 2.2.2), then linear in ln T between
// the T nodes; dk/dT from that slope; constant beyond the grid.  Tables are in global
// memory (read-only path).
__device__ __forceinline__ void table_rate(const NetView &nv, const double *tab, int tr, int iR, double w,
                                           double T, double lT, double &k, double &dk)
{
    const int nT = nv.tab_nT;
    const double *r0 = tab + (static_cast<size_t>(tr) * nv.tab_nR + iR) * nT;
    const bool two = nv.tab_nR > 1;
    auto L = [&](int j) { return two ? (1.0 - w) * __ldg(r0 + j) + w * __ldg(r0 + nT + j) : __ldg(r0 + j); };
    const double v = (lT - nv.tab_lt0) / nv.tab_dlt;
    if (!(v > 0.0)) {
        k = exp(L(0));
        dk = 0.0;
        return;
    }
    if (v >= nT - 1) {
        k = exp(L(nT - 1));
        dk = 0.0;
        return;
    }
    int j = static_cast<int>(floor(v));
    if (j > nT - 2) j = nT - 2;
    const double fr = v - j, a = L(j), b = L(j + 1);
    k = exp(a + fr * (b - a));
    dk = k * ((b - a) / nv.tab_dlt) / T;
}

// Barrier of one team: T threads on the named barrier `id`.
template <int T>
__device__ __forceinline__ void team_sync(int id)
{
    if constexpr (T == 32) __syncwarp();
    else asm volatile("barrier.sync %0, %1;" ::"r"(id), "n"(T) : "memory");
}

// float -> double on the integer pipes (exact for normal values and zeros); subnormals,
// infinities and NaNs take the conversion instruction, which occupies the FP64 pipe.
__device__ __forceinline__ double widen(float f)
{
    const unsigned u = __float_as_uint(f), m = u & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u || m == 0u)
        return __hiloint2double(static_cast<int>((u & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)),
                                static_cast<int>(u << 29));
    return static_cast<double>(f);
}

__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }

// Pivot of column j: argmax_{i >= j} |M_ij| V_i over the warp's candidates c[q] (row
// lane + 32 q, NaN already 0), ties to the smaller row; -1 if none is positive.
template <int NQW>
__device__ __forceinline__ int pivot_row(const float (&c)[NQW], int lane)
{
    unsigned k = 0;
#pragma unroll
    for (int q = 0; q < NQW; ++q) k = max(k, __float_as_uint(c[q]));
    const unsigned best = __reduce_max_sync(kFull, k);
    unsigned row = 0xffffu;
#pragma unroll
    for (int q = NQW - 1; q >= 0; --q)
        if (__float_as_uint(c[q]) == best) row = static_cast<unsigned>(lane + 32 * q);
    row = __reduce_min_sync(kFull, row);
    return best == 0u ? -1 : static_cast<int>(row);
}

template <int NQW>
__device__ __forceinline__ int pivot_row(const double (&c)[NQW], int lane)
{
    unsigned hi = 0;
#pragma unroll
    for (int q = 0; q < NQW; ++q) hi = max(hi, static_cast<unsigned>(__double2hiint(c[q])));
    const unsigned bh = __reduce_max_sync(kFull, hi);
    unsigned lo = 0;
#pragma unroll
    for (int q = 0; q < NQW; ++q)
        if (static_cast<unsigned>(__double2hiint(c[q])) == bh)
            lo = max(lo, static_cast<unsigned>(__double2loint(c[q])));
    const unsigned bl = __reduce_max_sync(kFull, lo);
    unsigned row = 0xffffu;
#pragma unroll
    for (int q = NQW - 1; q >= 0; --q)
        if (static_cast<unsigned>(__double2hiint(c[q])) == bh && static_cast<unsigned>(__double2loint(c[q])) == bl)
            row = static_cast<unsigned>(lane + 32 * q);
    row = __reduce_min_sync(kFull, row);
    return (bh | bl) == 0u ? -1 : static_cast<int>(row);
}

// NW warps per cell, NQ components per thread (thread t owns t, t + 32 NW, ...), NQW rows
// per lane of one warp (N <= 32 NQW).  Twelve single-warp teams per SM with 168 registers
// rather than sixteen with 128 (32 species, dt 1e8 s: 1,000 cells 111 | 116 ms, 2,049 cells
// 120 | 122, 4,096 cells 135 | 139, 8,192 cells 203 | 196).
template <int NW, int NQ, int NQW, bool ENERGY, bool F32>
__global__ void __launch_bounds__(NW == 1 ? 128 : 512, NW == 1 ? 3 : 1) warp_kernel(const LaunchArgs a, const WarpLayout L)
{
    using R = typename std::conditional<F32, float, double>::type;
    constexpr int T = 32 * NW, VW = 16 / sizeof(R);
    union Vec {   // 16 bytes of a column
        typename std::conditional<F32, float4, double2>::type q;
        R v[VW];
    };
    auto ld16 = [](const R *p) {
        Vec x;
        x.q = *reinterpret_cast<const decltype(x.q) *>(p);
        return x;
    };
    auto st16 = [](R *p, const Vec &x) { *reinterpret_cast<decltype(Vec::q) *>(p) = x.q; };
    extern __shared__ __align__(16) unsigned char sm[];
    const NetView nv = a.nv;
    if (!stage_table(sm, a.blob, static_cast<unsigned>(nv.bytes_warp),
                     reinterpret_cast<uint64_t *>(sm + nv.bytes_warp), &a.scratch->error, kDevErrTma))
        return;
    NetS t;
    t.A = reinterpret_cast<const double *>(sm + nv.off_A);
    t.b = reinterpret_cast<const double *>(sm + nv.off_b);
    t.th = reinterpret_cast<const double *>(sm + nv.off_th);
    t.h = reinterpret_cast<const double *>(sm + nv.off_h);
    t.cv = reinterpret_cast<const double *>(sm + nv.off_cv);
    t.cnt = reinterpret_cast<const double *>(sm + nv.off_cnt);
    t.idx = reinterpret_cast<const unsigned long long *>(sm + nv.off_idx);
    t.rp = reinterpret_cast<const int *>(sm + nv.off_rp);
    t.re = reinterpret_cast<const int *>(sm + nv.off_re);
    t.ex = reinterpret_cast<const double *>(sm + nv.off_exp);
    const DevOpts o = a.o;
    const int N = nv.N, ns = nv.ns, ne = nv.ne, nr = nv.nr, LD = L.LD;
    const long long nc = a.ncells;
    const int lane = threadIdx.x & 31, team = threadIdx.x / T, tid = threadIdx.x % T, wrp = tid >> 5;
    auto sync = [&]() { team_sync<T>(1 + team); };
    unsigned char *wb = sm + L.base + team * L.warp_bytes;
    R *J = reinterpret_cast<R *>(wb + L.off_J);     // Jacobian; in M's storage when not kept apart
    R *M = reinterpret_cast<R *>(wb + L.off_M);     // iteration matrix, then its factors
    R *V = reinterpret_cast<R *>(wb + L.off_V);     // inverse pivots
    R *LC = reinterpret_cast<R *>(wb + L.off_X);    // right-hand side; FP64 elimination column
    R *D = reinterpret_cast<R *>(wb + L.off_D);     // partial derivatives [kind][reaction]
    int *G = reinterpret_cast<int *>(wb + L.off_G); // row order of the factors
    double *ys = reinterpret_cast<double *>(wb + L.off_Y);    // current iterate
    double *fs = reinterpret_cast<double *>(wb + L.off_W);    // f; error terms; state being finished
    double *ws = reinterpret_cast<double *>(wb + L.off_RW);   // reaction rates
    double *K = reinterpret_cast<double *>(wb + L.off_K);     // rate coefficients (isothermal)
    float *mon = reinterpret_cast<float *>(wb + L.off_C);     // per-warp convergence monitors, 2 sets

    long long cell = 0;
    double T_iso = 0.0, invCV = 0.0, atol_s = 0.0, dtc = a.dt;
    // C_V(T) of polynomial networks (Sec. 4.2): the cell's coefficients sum_s n0_s c_s,k
    // (five below t_mid, five from t_mid), and C_V'/C_V at the current iterate
    const bool CVP = ENERGY && nv.cvpoly != 0;
    const double *cvp = reinterpret_cast<const double *>(sm + nv.off_cvp);
    double *cvc = reinterpret_cast<double *>(wb + L.off_CV);
    double dcvr = 0.0;
    // tabulated and photo rates: rate types, the cell's density weight in the tables,
    // its photo flux factor and path length, and phi'(tau) at the current iterate
    const int *rtype = reinterpret_cast<const int *>(sm + nv.off_rtype);
    const double *sigr = reinterpret_cast<const double *>(sm + nv.off_sigr);
    const double *sigs = reinterpret_cast<const double *>(sm + nv.off_sigs);
    const double *tabs = reinterpret_cast<const double *>(a.blob + nv.off_tab);
    int tab_iR = 0;
    double tab_w = 0.0, ph_F = 1.0, ph_dl = 0.0, ph_phi = 1.0, ph_dphi = 0.0;
    const int nin_max = nv.nin_max, kT = nin_max;   // kinds of partials: reactants, then T
    const bool slim = L.off_D < 0;                  // no room for partials: K and dk/dT (in ws) instead
    if (!slim && tid == 0) D[nr * (nin_max + (ENERGY ? 1 : 0))] = R(0);   // the partial of padding terms

    // k and dk/dT of reaction r at T (lt = ln(T/T_ref), lT = ln T); photo-reactions take
    // the current phi(tau) (dk/dT = 0)
    auto rate = [&](int r, double Tc, double lt, double lT, double invT, double &k, double &dk) {
        const int ty = nv.special ? rtype[r] : 0;
        if (ty == 0) {
            arrhenius(t, r, lt, invT, k, dk);
        } else if (ty == 2) {
            k = ph_F * sigr[r] * ph_phi;
            dk = 0.0;
        } else {
            table_rate(nv, tabs, ty >> 8, tab_iR, tab_w, Tc, lT, k, dk);
        }
    };
    int nnew = 0, flip = 0;

    double Y[NQ], F0[NQ], YF[NQ], YH[NQ], CUR[NQ], W[NQ];   // own components
    auto own = [&](int q) { return tid + T * q; };
    auto yin = [&](int s) { return a.y_in[static_cast<long long>(s) * nc + cell]; };

    auto load_pre = [&]() {
        const double Tin = a.T_in[cell];
        T_iso = Tin < nv.t_min ? nv.t_min : (Tin > nv.t_max ? nv.t_max : Tin);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int i = own(q);
            Y[q] = 0.0;
            if (i < ns) {
                const double v = yin(i);
                Y[q] = v > 0.0 ? v : 0.0;
            } else if (ENERGY && i == ns) {
                Y[q] = T_iso;
            }
        }
    };

    auto put = [&](double *to, const double (&v)[NQ]) {
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            if (own(q) < N) to[own(q)] = v[q];
    };

    // Rates at the state in ys (written and synchronised by the caller): w_r into ws and,
    // when wantJ, the partials into D; then the species rows of f into fs / W and, when
    // wantJ, of J; the temperature row of f.  hph is only read when the iteration matrix
    // replaces J in place (L.off_J == L.off_M with fuse).
    auto rates_rows = [&](bool wantJ) {
        const double Tc = ENERGY ? ys[ns] : T_iso;
        if (nv.nphoto) {
            // optical depth tau = dl sum_s n_s sigma_s of the iterate, then phi(tau)
            double sg = 0.0;
            for (int s = lane; s < ns; s += 32) sg = fma(ys[s], sigs[s], sg);
            photo_phi(ph_dl * wsum(sg), ph_phi, ph_dphi);
        }
        if (CVP) {
            const int o5 = Tc < nv.t_mid ? 0 : 5;
            const double cv = (((cvc[o5 + 4] * Tc + cvc[o5 + 3]) * Tc + cvc[o5 + 2]) * Tc + cvc[o5 + 1]) * Tc + cvc[o5];
            const double dcv = ((4.0 * cvc[o5 + 4] * Tc + 3.0 * cvc[o5 + 3]) * Tc + 2.0 * cvc[o5 + 2]) * Tc + cvc[o5 + 1];
            invCV = 1.0 / cv;
            dcvr = dcv * invCV;
        }
        double lt = 0.0, invT = 0.0, lT = 0.0;
        if (ENERGY) {
            lt = log_t(Tc, nv.t_ref);
            invT = 1.0 / Tc;
            lT = nv.ntab ? log(Tc) : 0.0;
        }
        auto reaction = [&](int r, bool on) {   // rate (and partials) of reaction r, kept if on
            double k, dk = 0.0;
            if (ENERGY) rate(r, Tc, lt, lT, invT, k, dk);
            else k = nv.nphoto && rtype[r] == 2 ? ph_F * sigr[r] * ph_phi : K[r];
            const unsigned long long ix = t.idx[r];
            const int nin = static_cast<int>(ix & 0x7f);
            const double y0 = ys[(ix >> 16) & 0xff];
            const double y1 = nin > 1 ? ys[(ix >> 24) & 0xff] : 1.0;
            const double p01 = __dmul_rn(y0, y1);
            double w = __dmul_rn(k, p01), y2 = 1.0;
            if (nin_max > 2) {
                y2 = nin > 2 ? ys[(ix >> 32) & 0xff] : 1.0;
                w = __dmul_rn(w, y2);
            }
            if (!on) return;
            ws[r] = w;
            if (wantJ && slim) {
                if (ENERGY) {
                    K[r] = k;
                    ws[r] = dk;
                } else {
                    K[r] = k;   // (a photo rate at this iterate)
                }
            } else if (wantJ) {
                double d0 = __dmul_rn(k, y1), d1 = __dmul_rn(k, y0);
                if (nin_max > 2) {
                    d0 = __dmul_rn(d0, y2);
                    d1 = __dmul_rn(d1, y2);
                    D[2 * nr + r] = static_cast<R>(__dmul_rn(k, p01));
                }
                D[r] = static_cast<R>(d0);
                if (nin_max > 1) D[nr + r] = static_cast<R>(d1);
                if (ENERGY) {
                    double dT = __dmul_rn(dk, p01);
                    if (nin_max > 2) dT = __dmul_rn(dT, y2);
                    D[kT * nr + r] = static_cast<R>(dT);
                }
            }
        };
        if (ENERGY && !nv.special) {
            // two reactions at a time: the second's loads and integer work hide behind the
            // first's FP64 instructions
            for (int r = tid; r < nr; r += 2 * T) {
                const bool two = r + T < nr;
                reaction(r, true);
                reaction(two ? r + T : r, two);
            }
        } else {
            for (int r = tid; r < nr; r += T) reaction(r, true);
        }
        sync();
        // f: every species row adds +-w_r per list entry (every entry has a coefficient of
        // +-1, the sign applied on the bit pattern), the next entry's rate loaded ahead
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int s = own(q);
            double f = 0.0;
            if (s < ns && !(wantJ && slim)) {
                const int e0 = t.rp[s], e1 = t.rp[s + 1];
                int n0 = e0 < e1 ? t.re[e0] : 0, n1 = e0 + 1 < e1 ? t.re[e0 + 1] : 0;
                double w0 = e0 < e1 ? ws[n0 >> 8] : 0.0;
                for (int e = e0; e < e1; ++e) {
                    const int n2 = e + 2 < e1 ? t.re[e + 2] : 0;
                    const double w1 = ws[n1 >> 8];
                    // -1 is stored as 0xff: its bit 7 becomes the sign bit of w_r
                    f += __longlong_as_double(__double_as_longlong(w0) ^ (static_cast<long long>(n0 & 0x80) << 56));
                    n0 = n1;
                    n1 = n2;
                    w0 = w1;
                }
                fs[s] = f;
            }
            W[q] = f;
        }
        if (wantJ && !slim) {
            // every entry of the species rows is the sum of its terms +-D in list order, formed by
            // one thread (kt_coop_tables.cu); the program streams from L2, eight steps ahead.  (Rows
            // walking their lists, read-modify-write: 65 unknowns 13.0k cycles per iteration,
            // this 6.8k; 32 unknowns 3.8k | 2.5k.)
            const unsigned *prog = a.jac + tid;
            R v = R(0);
            unsigned u[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) u[e] = __ldg(prog + e * T);
            for (int e0 = 0; e0 < a.jac_steps; e0 += 8) {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const unsigned c = u[e];
                    u[e] = __ldg(prog + (e0 + 8 + e) * T);
                    const R d = D[c & kTermIndex];
                    if constexpr (F32) v += __uint_as_float(__float_as_uint(d) ^ (c & kTermMinus));
                    else v += __hiloint2double(__double2hiint(d) ^ static_cast<int>(c & kTermMinus), __double2loint(d));
                    if (c & kTermEnd) {
                        J[(c >> kTermPlace) & kTermIndex] = v;
                        v = R(0);
                    }
                }
            }
            if (nv.nphoto) {
                // dw/dn_m of a photo rate through tau: + (sum) sigma_m for every absorber m, the
                // sum over the row's photo reactions of nu F sigma_r n_i phi' dl
                sync();
                for (int s = tid; s < ns; s += T) {
                    double gph = 0.0;
                    const int e1 = t.rp[s + 1];
                    for (int e = t.rp[s]; e < e1; ++e) {
                        const int ent = t.re[e], r = ent >> 8;
                        if (rtype[r] == 2) {
                            const int i0 = static_cast<int>((t.idx[r] >> 16) & 0xff);
                            const double g = ph_F * sigr[r] * ys[i0] * ph_dphi * ph_dl;
                            gph += (ent & 0x80) ? -g : g;
                        }
                    }
                    if (gph != 0.0)
                        for (int m = 0; m < ns; ++m) {
                            if constexpr (F32) J[m * LD + s] += static_cast<float>(__dmul_rn(gph, sigs[m]));
                            else J[m * LD + s] = fma(gph, sigs[m], J[m * LD + s]);
                        }
                }
            }
        } else if (wantJ) {
            for (int s = tid; s < ns; s += T) {
                R *row = J + s;   // entry m of the row at m * LD
                for (int m = 0; m < N; ++m) row[m * LD] = R(0);
                const int e1 = t.rp[s + 1];
                double gph = 0.0, f = 0.0;
                R aT = R(0);
                for (int e = t.rp[s]; e < e1; ++e) {
                    const int ent = t.re[e], r = ent >> 8;
                    const unsigned long long ix = t.idx[r];
                    const int nin = static_cast<int>(ix & 0x7f);
                    const int i0 = static_cast<int>((ix >> 16) & 0xff), i1 = static_cast<int>((ix >> 24) & 0xff),
                              i2 = static_cast<int>((ix >> 32) & 0xff);
                    const R sg = (ent & 0x80) ? R(-1) : R(1);   // fma(+-1, d, a) = a +- d
                    const double k = K[r], y0 = ys[i0], y1 = nin > 1 ? ys[i1] : 1.0, y2 = nin > 2 ? ys[i2] : 1.0;
                    const double p01 = __dmul_rn(y0, y1), w = __dmul_rn(__dmul_rn(k, p01), y2);
                    f += (ent & 0x80) ? -w : w;
                    row[i0 * LD] = fma_t(sg, static_cast<R>(__dmul_rn(__dmul_rn(k, y1), y2)), row[i0 * LD]);
                    if (nin > 1) row[i1 * LD] = fma_t(sg, static_cast<R>(__dmul_rn(__dmul_rn(k, y0), y2)), row[i1 * LD]);
                    if (nin > 2) row[i2 * LD] = fma_t(sg, static_cast<R>(__dmul_rn(k, p01)), row[i2 * LD]);
                    if (ENERGY) aT = fma_t(sg, static_cast<R>(__dmul_rn(__dmul_rn(ws[r], p01), y2)), aT);
                    if (nv.nphoto && rtype[r] == 2) {
                        const double g = ph_F * sigr[r] * y0 * ph_dphi * ph_dl;
                        gph += (ent & 0x80) ? -g : g;
                    }
                }
                if (ENERGY) row[ns * LD] = aT;
                fs[s] = f;
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (own(q) == s) W[q] = f;
                if (gph != 0.0)
                    for (int m = 0; m < ns; ++m) {
                        if constexpr (F32) row[m * LD] += static_cast<float>(__dmul_rn(gph, sigs[m]));
                        else row[m * LD] = fma(gph, sigs[m], row[m * LD]);
                    }
            }
        }
        if (ENERGY) {
            sync();
            if (wrp == ((ns % T) >> 5)) {   // the warp that owns the temperature
                double qs = 0.0;
                for (int s = lane; s < ns; s += 32) qs = fma(t.h[s], fs[s], qs);
                qs = wsum(qs);
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (own(q) == ns) W[q] = -qs * invCV;
            }
        }
    };

    // temperature row of J (threads over columns) and, when hph > 0, I - hph J into M in the
    // same pass over the column
    auto t_row = [&](double hph) {
        const R hr = static_cast<R>(hph);
        sync();
        for (int m = tid; m < N; m += T) {
            double c = 0.0;
            const R *jm = J + m * LD;
            R *mm = M + m * LD;
            int s = 0;
            for (; s + VW <= ns; s += VW) {
                const Vec j = ld16(jm + s);
                Vec x;
#pragma unroll
                for (int e = 0; e < VW; ++e) {
                    if (ENERGY) {
                        if constexpr (F32) c = fma(t.h[s + e], widen(j.v[e]), c);
                        else c = fma(t.h[s + e], j.v[e], c);
                    }
                    x.v[e] = fma_t(-hr, j.v[e], s + e == m ? R(1) : R(0));
                }
                if (hph > 0.0) st16(mm + s, x);
            }
            for (; s < ns; ++s) {
                const R j = jm[s];
                if (ENERGY) {
                    if constexpr (F32) c = fma(t.h[s], widen(j), c);
                    else c = fma(t.h[s], j, c);
                }
                if (hph > 0.0) mm[s] = fma_t(-hr, j, s == m ? R(1) : R(0));
            }
            if (ENERGY) {
                R jt = static_cast<R>(-c * invCV);
                // d f_T / d T of C_V(T): -f_T C_V'/C_V
                if (CVP && m == ns) {
                    if constexpr (F32) jt -= static_cast<float>(__dmul_rn(fs[ns], dcvr));
                    else jt = fma(-fs[ns], dcvr, jt);
                }
                J[m * LD + ns] = jt;
                if (hph > 0.0) mm[ns] = fma_t(-hr, jt, m == ns ? R(1) : R(0));
            }
        }
    };

    // Right-looking LU of M; G: composed gather index of the right-hand side, V: inverse
    // pivots.  Columns are contiguous, so a thread updates a column 16 bytes at a time
    // (measured on 65 unknowns: 260k cycles per factorisation row-major, one value at a
    // time).  Team-uniform result.
    auto lu = [&]() -> bool {
        constexpr int H = NW > 1 ? 2 : 1;   // threads per column
        sync();
        R v[NQW];   // inverse row maxima of rows lane + 32 q, the same in every warp
        bool ok = true;
#pragma unroll
        for (int q = 0; q < NQW; ++q) {
            const int i = lane + 32 * q;
            v[q] = R(1);
            if (i < N) {
                R big = R(0);
#pragma unroll 4
                for (int m = 0; m < N; ++m) {
                    const R x = fabs(M[m * LD + i]);
                    big = x > big ? x : big;
                }
                ok = ok && big > R(0);
                if (big > R(0)) v[q] = R(1) / big;
            }
        }
        ok = __all_sync(kFull, ok) != 0;
        for (int i = tid; i < N; i += T) G[i] = i;
        for (int j = 0; j < N; ++j) {
            sync();   // the previous step's update is complete
            R *mj = M + j * LD;
            R c[NQW];
#pragma unroll
            for (int q = 0; q < NQW; ++q) {
                const int i = lane + 32 * q;
                R x = R(0);
                if (i >= j && i < N) {
                    x = fabs(mj[i]) * v[q];
                    if (!(x == x)) x = R(0);
                }
                c[q] = x;
            }
            const int p = pivot_row(c, lane);
            if (p < 0) return false;
            const R piv = mj[p], mjj = mj[j], rinv = R(1) / piv;
            // the multipliers of the rows below, as they stand after rows j and p exchange
            for (int i = j + 1 + tid; i < N; i += T) {
                const R x = i == p ? mjj : mj[i];
                LC[i] = x * rinv;
            }
            if (p != j) {
                for (int k = tid; k < N; k += T)
                    if (k != j) {
                        R *mk = M + k * LD;
                        const R x = mk[j];
                        mk[j] = mk[p];
                        mk[p] = x;
                    }
                // row scales follow their rows
                R vj = R(0);
#pragma unroll
                for (int q = 0; q < NQW; ++q)
                    if (j >> 5 == q) vj = v[q];
                vj = __shfl_sync(kFull, vj, j & 31);
#pragma unroll
                for (int q = 0; q < NQW; ++q)
                    if (lane + 32 * q == p) v[q] = vj;
            }
            if (tid == T - 1) {
                const int g = G[j];
                G[j] = G[p];
                G[p] = g;
                V[j] = rinv;
            }
            sync();
            for (int i = j + tid; i < N; i += T) mj[i] = i == j ? piv : LC[i];
            // rows j + 1 .. of the columns to the right, VW rows at a time from the chunk that
            // holds row j + 1 (its rows up to j stay)
            const int i0 = (j + 1) & ~(VW - 1);
            for (int k = j + 1 + tid / H; k < N; k += T / H) {
                R *mk = M + k * LD;
                const R u = mk[j];
                int i = i0 + (tid % H) * VW;
                if (H == 1 || tid % H == 0) {
                    const Vec l = ld16(LC + i);
                    Vec x = ld16(mk + i);
#pragma unroll
                    for (int e = 0; e < VW; ++e) {
                        const R y = fma_t(-l.v[e], u, x.v[e]);
                        if (i + e > j) x.v[e] = y;
                    }
                    st16(mk + i, x);
                    i += H * VW;
                }
#pragma unroll 2
                for (; i < N; i += H * VW) {
                    const Vec l = ld16(LC + i);
                    Vec x = ld16(mk + i);
#pragma unroll
                    for (int e = 0; e < VW; ++e) x.v[e] = fma_t(-l.v[e], u, x.v[e]);
                    st16(mk + i, x);
                }
            }
        }
        sync();
        return ok;
    };

    // x <- M^-1 b for the factors of lu(): b gathered from LC by G, the solution left in LC.
    // Each step is a shuffle and an update; the factors of eight steps are loaded ahead.
    auto solve = [&]() {
        sync();
        if (wrp == 0) {
            R x[NQW];
            int at[NQW];   // row of the lane, the last row where there is none (not stored)
#pragma unroll
            for (int q = 0; q < NQW; ++q) {
                const int i = lane + 32 * q;
                at[q] = i < N ? i : N - 1;
                x[q] = LC[G[at[q]]];
            }
            __syncwarp();
#pragma unroll
            for (int jq = 0; jq < NQW; ++jq) {
                const int n = N - 1 - 32 * jq < 32 ? N - 1 - 32 * jq : 32;
                auto steps = [&](int jj, auto count) {
                    constexpr int B = decltype(count)::value;
                    R m[B][NQW];
#pragma unroll
                    for (int e = 0; e < B; ++e)
#pragma unroll
                        for (int q = jq; q < NQW; ++q) m[e][q] = M[(32 * jq + jj + e) * LD + at[q]];
#pragma unroll
                    for (int e = 0; e < B; ++e) {
                        const R xj = __shfl_sync(kFull, x[jq], jj + e);
#pragma unroll
                        for (int q = jq; q < NQW; ++q) {
                            const R y = fma_t(-m[e][q], xj, x[q]);
                            x[q] = q > jq || lane > jj + e ? y : x[q];
                        }
                    }
                };
                int jj = 0;
                for (; jj + 8 <= n; jj += 8) steps(jj, std::integral_constant<int, 8>());
                for (; jj < n; ++jj) steps(jj, std::integral_constant<int, 1>());
            }
#pragma unroll
            for (int jq = NQW - 1; jq >= 0; --jq) {
                const int n = N - 32 * jq < 32 ? N - 32 * jq : 32;
                auto steps = [&](int top, auto count) {   // columns top, top - 1, ..
                    constexpr int B = decltype(count)::value;
                    R m[B][NQW], vi[B];
#pragma unroll
                    for (int e = 0; e < B; ++e) {
                        vi[e] = V[32 * jq + top - e];
#pragma unroll
                        for (int q = 0; q <= jq; ++q) m[e][q] = M[(32 * jq + top - e) * LD + at[q]];
                    }
#pragma unroll
                    for (int e = 0; e < B; ++e) {
                        const R xj = __shfl_sync(kFull, x[jq], top - e) * vi[e];
#pragma unroll
                        for (int q = 0; q <= jq; ++q) {
                            const R y = fma_t(-m[e][q], xj, x[q]);
                            if (q < jq) x[q] = y;
                            else x[q] = lane < top - e ? y : (lane == top - e ? xj : x[q]);
                        }
                    }
                };
                int top = n - 1;
                for (; top >= 7; top -= 8) steps(top, std::integral_constant<int, 8>());
                for (; top >= 0; --top) steps(top, std::integral_constant<int, 1>());
            }
#pragma unroll
            for (int q = 0; q < NQW; ++q)
                if (lane + 32 * q < N) LC[lane + 32 * q] = x[q];
        }
        sync();
    };

    bool luok = false;
    const double natol_f = F32 ? o.newton_atol_frac * kF32NewtonAtolScale : o.newton_atol_frac;

    // One solve y = b + hph f(y) by Newton from the guess in CUR (ys holds it too), b in YB.
    // fmode (FP32 form): 2 assemble J at the guess and factor; 1 factor from the stored J;
    // 0 reuse the current factor.
    auto be_solve = [&](const double (&yb)[NQ], double hph, int fmode) -> bool {
        int refresh = 0;
        bool doJ = !F32 || fmode == 2, doF = !F32 || fmode >= 1;
        float dprev = 0.0f, dprevr = 0.0f;
        const double natol = __dmul_rn(natol_f, atol_s);
        for (int it = 0;; ++it) {
            ++nnew;
            sync();
            const double Tc = ENERGY ? ys[ns] : T_iso;
            if (!(Tc > 0.0)) return false;
            rates_rows(doJ);
            if (CVP && doJ) {
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (own(q) == ns) fs[ns] = W[q];
            }
            if (doJ) t_row(doF ? hph : 0.0);
            else if (doF) {   // a new h with the stored J
                const R hr = static_cast<R>(hph);
                for (int m = tid; m < N; m += T)
                    for (int s = 0; s < N; ++s) M[m * LD + s] = fma_t(-hr, J[m * LD + s], s == m ? R(1) : R(0));
            }
            if (doF) luok = lu();
            if (F32) doJ = doF = false;
            if (!luok) return false;
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (own(q) < N)
                    LC[own(q)] = static_cast<R>(-fma(-hph, W[q], __dadd_rn(CUR[q], -yb[q])));
            solve();
            bool conv = true;
            // contraction monitors (FP32 is plenty): dmax = max |delta|/tol, dmaxr =
            // max |delta| / (newton_rtol |y|), the purely relative part of the tolerance
            float dmax = 0.0f, dmaxr = 0.0f;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int i = own(q);
                if (i < N) {
                    const double x = static_cast<double>(LC[i]);
                    const double y = __dadd_rn(CUR[q], x);
                    CUR[q] = y;
                    ys[i] = y;
                    const double ny = __dmul_rn(o.newton_rtol, fabs(y));
                    const double tol = fma(o.newton_rtol, fabs(y), i < ns ? natol : 0.0);
                    if (!(fabs(x) <= tol)) conv = false;
                    if constexpr (F32) {
                        const float ad = fabsf(LC[i]), tf = static_cast<float>(tol);
                        const float r = __fdiv_rn(ad, fmaxf(tf, 1e-37f));
                        // the relative part newton_rtol |y| formed directly: as a difference
                        // tf - natol in FP32 it rounds to an ulp of natol for trace species
                        const float trl = static_cast<float>(ny);
                        const float rr = __fdiv_rn(ad, fmaxf(trl, 1e-37f));
                        dmax = r > dmax ? r : dmax;
                        dmaxr = rr > dmaxr ? rr : dmaxr;
                    }
                }
            }
            conv = __all_sync(kFull, conv) != 0;
            if constexpr (F32) {   // non-negative: ordered like their bit patterns
                dmax = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(dmax)));
                dmaxr = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(dmaxr)));
            }
            if constexpr (NW > 1) {
                float *slot = mon + 3 * NW * flip;
                flip ^= 1;
                if (lane == 0) {
                    slot[3 * wrp] = conv ? 1.0f : 0.0f;
                    slot[3 * wrp + 1] = dmax;
                    slot[3 * wrp + 2] = dmaxr;
                }
                sync();
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    conv = conv && slot[3 * w] != 0.0f;
                    dmax = fmaxf(dmax, slot[3 * w + 1]);
                    dmaxr = fmaxf(dmaxr, slot[3 * w + 2]);
                }
            }
            if (conv) return true;
            if (!F32) {
                if (it + 1 >= o.max_newton) return false;
            } else {
                if (!isfinite(dmax)) return false;
                // stop on the contraction rate (Hairer & Wanner, Solving ODEs II, Sec. IV.8):
                // with theta = dmaxr / dprevr < 1/2 the error left after this update is about
                // theta / (1 - theta) * |delta|; accept when that is within newton_rtol |y_i|
                // for every component (the relative part only: species below the absolute
                // tolerance end as close to the root as the plain test leaves them)
                if (it > 0) {
                    const float th = dmaxr / dprevr;
                    if (th < 0.5f && th / (1.0f - th) * dmaxr <= 1.0f) return true;
                }
                const bool stalled = it > 0 && !(dmax < 0.5f * dprev);
                if (stalled || it + 1 >= o.max_newton) {
                    if (refresh >= 2) return false;
                    ++refresh;
                    doJ = true;
                    doF = true;
                    it = -1;
                }
                dprev = dmax;
                dprevr = dmaxr;
            }
        }
    };

    // Sub-steps over [0, dtc] in either scheme; every Newton solve goes through the one
    // call of be_solve below (one inlined copy of the solver per kernel).
    //   backward Euler with step doubling: stage 0 the full step h from Y (-> YF),
    //     stage 1 the first half step from Y (-> YH), stage 2 the second from YH
    //   TR-BDF2 (o.scheme == KT_SCHEME_TRBDF2): stage 0 trapezoidal, r = Y + d h f_n in
    //     YH (-> YF), stage 1 BDF2, r = w1 YF - w0 Y in YH; one FP32 factor of
    //     I - d h J serves both stages.  F0 holds f_n: f(Y) on the cell's first step,
    //     afterwards the previous step's stage relation (y_{n+1} - r)/(d h), which keeps
    //     the rounding of an evaluated rate (amplified by h k in the error estimate) out
    //     of the accept decision
    auto advance = [&](double h0, double fgrow, int &nacc) -> bool {
        const bool trs = o.scheme == KT_SCHEME_TRBDF2;
        const TrCoef tr = tr_coef();
        const int nst = trs ? 2 : 3;
        double tt = 0.0, h = h0;
        int natt = 0;
        bool f0ok = false;
        nacc = 0;
        for (;;) {
            if (natt >= o.max_substeps) return false;
            ++natt;
            bool last = false;
            if (tt + h >= dtc * (1.0 - 1e-12)) {
                h = dtc - tt;
                last = true;
            }
            const double dh = tr.d * h;
            bool ok = true;
            if (trs && !f0ok) {
                sync();
                put(ys, Y);
                sync();
                const double Tc = ENERGY ? ys[ns] : T_iso;
                ok = Tc > 0.0;
                if (ok) {
                    rates_rows(false);
#pragma unroll
                    for (int q = 0; q < NQ; ++q) F0[q] = W[q];
                    f0ok = true;
                }
            }
            for (int stg = 0; ok && stg < nst; ++stg) {
                double YB[NQ];
                double hph;
                int fmode;
                if (trs) {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        if (stg == 0) {
                            YH[q] = fma(dh, F0[q], Y[q]);
                            CUR[q] = Y[q];
                        } else {
                            YF[q] = CUR[q];
                            YH[q] = fma(tr.w1, CUR[q], -__dmul_rn(tr.w0, Y[q]));
                        }
                        YB[q] = YH[q];
                    }
                    hph = dh;
                    fmode = stg == 0 ? 2 : 0;
                } else {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        if (stg == 0) {
                            CUR[q] = Y[q];
                        } else if (stg == 1) {
                            YF[q] = CUR[q];
                            CUR[q] = Y[q];
                        } else {
                            YH[q] = CUR[q];
                            if (o.guess != KT_GUESS_PREV) CUR[q] = YF[q];
                        }
                        YB[q] = stg == 2 ? YH[q] : Y[q];
                    }
                    hph = stg == 0 ? h : 0.5 * h;
                    fmode = 2 - stg;
                }
                sync();
                put(ys, CUR);
                ok = be_solve(YB, hph, fmode);
            }
            if (!ok) {
                h *= 0.5;
                if (h < o.h_min) return false;
                continue;
            }
            // local error: 2 C h (a0 f_n + a1 f_g + a2 f_{n+1}) with the stage rates taken from
            // the stage equations, or the step-doubling difference; its weighted RMS
            const double inv = trs ? 1.0 / dh : 0.0, ce = __dmul_rn(__dmul_rn(2.0, tr.C), h);
            sync();
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int i = own(q);
                if (i >= N) continue;
                const double yn = Y[q], y1 = CUR[q];
                const double sc = fma(o.rtol, fmax(fabs(yn), fabs(y1)), i < ns ? atol_s : 0.0);
                double est;
                if (trs) {
                    const double f0 = F0[q];
                    const double fg = fma(__dadd_rn(YF[q], -yn), inv, -f0);
                    const double f1 = __dmul_rn(__dadd_rn(y1, -YH[q]), inv);
                    est = __dmul_rn(ce, fma(tr.a2, f1, fma(tr.a0, f0, __dmul_rn(tr.a1, fg))));
                } else {
                    est = __dadd_rn(y1, -YF[q]);
                }
                fs[i] = est / sc;
            }
            sync();
            double s2 = 0.0;
            for (int i = lane; i < N; i += 32) s2 = fma(fs[i], fs[i], s2);
            const double err = sqrt(wsum(s2) / N);
            if (err <= 1.0) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    if (trs) F0[q] = __dmul_rn(__dadd_rn(CUR[q], -YH[q]), inv);    // first same as last
                    Y[q] = CUR[q];
                }
                ++nacc;
                if (last) return true;
                tt += h;
                double fac = err > 0.0 ? 0.9 / (trs ? cbrt(err) : sqrt(err)) : fgrow;
                if (fac > fgrow) fac = fgrow;
                if (fac < 0.2) fac = 0.2;
                h *= fac;
            } else {
                double fac = 0.9 / (trs ? cbrt(err) : sqrt(err));
                if (!(fac >= 0.2)) fac = 0.2;
                h *= fac;
                if (h < o.h_min) return false;
            }
        }
    };

    // clip, then restore the element totals of the pre-processed input (Sec. 2.2.3); the
    // state goes through fs, every warp forms the same sums
    auto post_process = [&]() -> bool {
        double b0[kMaxElements], r[kMaxElements], Mp[kMaxElements * kMaxElements];
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            if (own(q) < ns && Y[q] < 0.0) Y[q] = 0.0;
        sync();
        put(fs, Y);
        sync();
        for (int e = 0; e < ne; ++e) {
            double pb = 0.0, pt = 0.0;
            for (int s = lane; s < ns; s += 32) {
                const double v = yin(s);
                pb = fma(t.cnt[s * ne + e], v > 0.0 ? v : 0.0, pb);
                pt = fma(t.cnt[s * ne + e], fs[s], pt);
            }
            b0[e] = wsum(pb);
            r[e] = wsum(pt) - b0[e];
            for (int f = 0; f < ne; ++f) {
                double pm = 0.0;
                for (int s = lane; s < ns; s += 32)
                    pm = fma(__dmul_rn(t.cnt[s * ne + e], t.cnt[s * ne + f]), fs[s], pm);
                Mp[e * ne + f] = wsum(pm);
            }
        }
        for (int e = 0; e < ne; ++e) {
            if (Mp[e * ne + e] == 0.0) {
                if (r[e] != 0.0) return false;
                for (int f = 0; f < ne; ++f) Mp[e * ne + f] = Mp[f * ne + e] = 0.0;
                Mp[e * ne + e] = 1.0;
            }
        }
        for (int k = 0; k < ne; ++k) {
            int p = k;
            for (int i = k + 1; i < ne; ++i)
                if (fabs(Mp[i * ne + k]) > fabs(Mp[p * ne + k])) p = i;
            if (!(fabs(Mp[p * ne + k]) > 0.0)) return false;
            if (p != k) {
                for (int j = 0; j < ne; ++j) {
                    const double xx = Mp[k * ne + j];
                    Mp[k * ne + j] = Mp[p * ne + j];
                    Mp[p * ne + j] = xx;
                }
                const double xx = r[k];
                r[k] = r[p];
                r[p] = xx;
            }
            for (int i = k + 1; i < ne; ++i) {
                const double l = Mp[i * ne + k] / Mp[k * ne + k];
                for (int j = k; j < ne; ++j) Mp[i * ne + j] -= l * Mp[k * ne + j];
                r[i] -= l * r[k];
            }
        }
        for (int i = ne - 1; i >= 0; --i) {
            double s = r[i];
            for (int j = i + 1; j < ne; ++j) s -= Mp[i * ne + j] * r[j];
            r[i] = s / Mp[i * ne + i];
        }
        bool ok = !ENERGY || isfinite(fs[ns]);
        for (int s = lane; s < ns; s += 32) {
            double corr = 0.0;
            for (int e = 0; e < ne; ++e) corr = fma(t.cnt[s * ne + e], r[e], corr);
            ok = ok && corr < 1.0 && isfinite(fma(-fs[s], corr, fs[s]));
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            if (own(q) < ns) {
                double corr = 0.0;
                for (int e = 0; e < ne; ++e) corr = fma(t.cnt[own(q) * ne + e], r[e], corr);
                Y[q] = fma(-Y[q], corr, Y[q]);
            }
        return __all_sync(kFull, ok) != 0;
    };

    auto write_out = [&](int st, int nsub) {
        sync();   // every thread has read its inputs (in-place calls)
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int i = own(q);
            if (i < ns) a.y_out[static_cast<long long>(i) * nc + cell] = Y[q];
            else if (ENERGY && i == ns) a.T_out[cell] = Y[q];
        }
        if (tid == 0) {
            if (!ENERGY) a.T_out[cell] = T_iso;
            if (a.status) a.status[cell] = st;
            if (a.nsub) a.nsub[cell] = nsub;
            if (a.nnew) a.nnew[cell] = nnew;
        }
    };

    auto process_cell = [&]() {
        dtc = a.dt_cell ? a.dt_cell[cell] : a.dt;
        bool fin = isfinite(a.T_in[cell]) && dtc > 0.0 && isfinite(dtc);
        for (int s = lane; s < ns; s += 32) fin = fin && isfinite(yin(s));
        fin = __all_sync(kFull, fin) != 0;
        if (!fin) {
            sync();
            for (int s = tid; s < ns; s += T) a.y_out[static_cast<long long>(s) * nc + cell] = yin(s);
            if (tid == 0) {
                a.T_out[cell] = a.T_in[cell];
                if (a.status) a.status[cell] = KT_STATUS_NONFINITE;
                if (a.nsub) a.nsub[cell] = 0;
                if (a.nnew) a.nnew[cell] = 0;
            }
            return;
        }
        load_pre();
        sync();
        put(fs, Y);
        sync();
        double cvt = 0.0, b00 = 0.0;
        for (int s = lane; s < ns; s += 32) {
            cvt = fma(t.cv[s], fs[s], cvt);
            b00 = fma(t.cnt[s * ne], fs[s], b00);
        }
        cvt = wsum(cvt);
        b00 = wsum(b00);
        invCV = ENERGY ? 1.0 / cvt : 0.0;
        if (CVP) {
            for (int k = 0; k < 10; ++k) {
                double c = 0.0;
                for (int s = lane; s < ns; s += 32) c = fma(fs[s], cvp[s * 10 + k], c);
                c = wsum(c);
                if (tid == 0) cvc[k] = c;
            }
        }
        atol_s = (o.atol_mode == 1 && b00 > 0.0) ? o.atol * b00 : o.atol;
        // pre-processing of tabulated and photo rates (Sec. 2.2.2): the cell's weight in
        // the density nodes of the tables, its flux factor and path length
        if (nv.special) {
            ph_F = a.flux ? a.flux[cell] : 1.0;
            ph_dl = a.path ? a.path[cell] : 0.0;
            ph_phi = 1.0;
            ph_dphi = 0.0;
            tab_iR = 0;
            tab_w = 0.0;
            if (nv.ntab && nv.tab_nR > 1) {
                const double rho_c = a.rho ? a.rho[cell] : 1.0;
                double u = (log(rho_c) - nv.tab_lr0) / nv.tab_dlr * (nv.tab_nR - 1);
                if (!(u > 0.0)) u = 0.0;
                if (u > nv.tab_nR - 1) u = nv.tab_nR - 1;
                tab_iR = static_cast<int>(floor(u));
                if (tab_iR > nv.tab_nR - 2) tab_iR = nv.tab_nR - 2;
                tab_w = u - tab_iR;
            }
        }
        if (!ENERGY) {
            const double lt = log_t(T_iso, nv.t_ref), invT = 1.0 / T_iso;
            const double lT = nv.ntab ? log(T_iso) : 0.0;
            for (int r = tid; r < nr; r += T) {
                double k, dk;
                rate(r, T_iso, lt, lT, invT, k, dk);
                K[r] = k;
            }
        }
        nnew = 0;
        int nacc = 0;
        bool ok = advance(o.h_init, o.facmax, nacc) && post_process();
        int st = KT_STATUS_OK;
        if (!ok && o.retry) {
            st = KT_STATUS_RETRIED;
            load_pre();
            ok = advance(o.h_init * o.retry_h_factor, o.retry_facmax, nacc) && post_process();
        }
        if (!ok) {
            load_pre();
            write_out(KT_STATUS_REVERTED, 0);
        } else {
            write_out(st, nacc);
        }
    };

    if (a.persistent) {
        for (;;) {
            unsigned long long c = 0;
            if constexpr (NW == 1) {
                if (lane == 0) c = atomicAdd(&a.scratch->queue, 1ULL);
                c = __shfl_sync(kFull, c, 0);
            } else {
                unsigned long long *next = reinterpret_cast<unsigned long long *>(wb + L.off_C);
                sync();
                if (tid == 0) *next = atomicAdd(&a.scratch->queue, 1ULL);
                sync();
                c = *next;
                sync();
            }
            if (c >= static_cast<unsigned long long>(nc)) break;
            cell = a.order ? static_cast<long long>(a.order[c]) : static_cast<long long>(c);
            process_cell();
        }
    } else {
        cell = static_cast<long long>(blockIdx.x) * (blockDim.x / T) + team;
        if (cell < nc) process_cell();
    }
}

// Teams per block: one up to an SM's worth of cells, so that a small batch spreads over all
// SMs, then as many as share the staged network within an SM's shared memory.
template <int NW, int NQW, bool ENERGY, bool F32>
int launch_t(const LaunchArgs &a, const LaunchCfg &c, cudaStream_t s)
{
    constexpr int NQ = NW == 1 ? NQW : 1, max_teams = kMaxTeams;
    auto layout = [&](bool slim) {
        return warp_layout(a.nv.N, a.nv.nr, a.nv.energy, F32 ? 1 : 0, a.nv.bytes_warp,
                           !F32 || a.o.scheme == KT_SCHEME_TRBDF2, a.nv.nin_max, a.nv.cvpoly, slim);
    };
    WarpLayout L = layout(false);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int smem_optin = 0, nsm = 0;
    cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (L.base + L.warp_bytes > smem_optin || !a.jac) L = layout(true);
    const long long per_sm = (a.ncells + nsm - 1) / nsm;
    int teams = c.block_warps > 0 ? c.block_warps / NW : max_teams;
    if (c.block_warps <= 0 && teams > per_sm) teams = static_cast<int>(per_sm);
    if (teams > max_teams) teams = max_teams;
    if (teams < 1) teams = 1;
    while (teams > 1 && L.base + teams * L.warp_bytes > smem_optin) --teams;
    const size_t smem = static_cast<size_t>(L.base) + static_cast<size_t>(teams) * L.warp_bytes;
    if (smem > static_cast<size_t>(smem_optin)) return cudaErrorInvalidConfiguration;
    auto kern = warp_kernel<NW, NQ, NQW, ENERGY, F32>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    const int threads = teams * NW * 32;
    long long blocks = (a.ncells + teams - 1) / teams;
    if (a.persistent) {
        int fit = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, threads, smem);
        if (e != cudaSuccess) return e;
        if (fit < 1) fit = 1;
        if (c.blocks_per_sm > 0 && c.blocks_per_sm < fit) fit = c.blocks_per_sm;
        if (blocks > static_cast<long long>(fit) * nsm) blocks = static_cast<long long>(fit) * nsm;
    }
    if (blocks < 1) return cudaSuccess;
    kern<<<static_cast<unsigned>(blocks), threads, smem, s>>>(a, L);
    return cudaGetLastError();
}

// Dispatch over the compile-time options for one form of the iteration matrix.  Up to 32
// unknowns one warp holds a row per lane and four would mostly wait for each other
// (32 species, dt 1e8 s, one | four warps, before the Jacobian program: 300 cells
// 163 | 159 ms, 2,049 cells 134 | 189, 8,192 cells 207 | 475); beyond, the team is faster at
// every size (65 unknowns, dt 1e-9 s: 1,024 cells 546 | 291 ms, with the program 258; 8,192
// cells at 1e-10 s 615 | 405).
template <bool F32, bool ENERGY>
int launch_warp_size(const LaunchArgs &a, const LaunchCfg &c, cudaStream_t s)
{
    return team_warps(a.nv.N) == 1 ? launch_t<1, 1, ENERGY, F32>(a, c, s) : launch_t<4, 3, ENERGY, F32>(a, c, s);
}

template <bool F32>
int launch_warp_form(const LaunchArgs &a, const LaunchCfg &c, cudaStream_t s)
{
    return a.nv.energy ? launch_warp_size<F32, true>(a, c, s) : launch_warp_size<F32, false>(a, c, s);
}

}  // namespace

// One translation unit per form (compile time).
int launch_warp_f64(const LaunchArgs &a, const LaunchCfg &c, void *stream);
int launch_warp_f32(const LaunchArgs &a, const LaunchCfg &c, void *stream);

}  // namespace kt
