// kt_coop.cuh -- several lanes per cell for small networks (N <= 16 unknowns).
//
// What bounds it: GB300's FP64 pipe.  A warp's FP64 instruction occupies its scheduler's
// pipe for 64 cycles however many of its lanes are active (measured: 32, 16 and 2 lanes
// cost the same; DSETP and the conversions too), so one cell per lane makes a cell's
// Newton iteration a serial chain of ~2,400 such instructions (74..127 us measured), and a
// launch lasts as long as its longest cell.  Here a group of G lanes owns a cell: the
// reactions' rates go over the lanes, every row of f is summed by one lane, the vectors
// are held one component per lane, and the Jacobian's entries and the elimination go over
// the lanes too, so the chain shrinks to 165 FP64 instructions (G = 32, counted) and a
// warp's 32 / G cells share each of them.  Combustion network, dt 1e-6 s, FP32-LU: 250 cells
// 808 -> 55 ms (G = 32), 65,536 cells end to end 1,040 -> 722 ms (G = 8).
//
// The results are bit for bit those of the lane-per-cell kernels (kt_lane.cuh): every
// rate, every sum (same terms, same order, one lane per sum), every matrix entry (its
// updates in reaction order), every elimination step (right-looking: the updates of an
// entry come in the same order as in Crout's) and every decision is the same sequence of
// rounded operations; products that the lane kernels' compiled code fuses are written as
// fma() here and the others with explicit rounding.
//
// Control flow is warp-converged: every phase is computed by the whole warp with the
// groups it does not concern masked at their stores (idle lanes cost nothing), and only
// cheap per-group decisions diverge.  Exchanges inside a group go through the cell's
// shared memory; the row sums and the matrix assembly follow small per-lane programs that
// the host lays out once per network and group size (kt_coop_tables.cu).
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

enum CoopState : int { kNeed = 0, kRun = 1, kDone = 2 };

// x < -700 decided on the bit pattern (kt_lane.cuh)
__device__ __forceinline__ bool below_m700(double x)
{
    const long long b = __double_as_longlong(x);
    return b < 0 && (b & 0x7fffffffffffffffLL) > 0x4085E00000000000LL;
}

// Comparisons on bit patterns, exact for every operand, so that they run on the integer
// pipes: a > 0; |a| <= b for b >= 0 or NaN; the larger magnitude.
__device__ __forceinline__ bool positive(double a)
{
    const long long b = __double_as_longlong(a);
    return b > 0 && b <= 0x7ff0000000000000LL;
}

__device__ __forceinline__ bool abs_le(double a, double b)
{
    const long long x = __double_as_longlong(a) & 0x7fffffffffffffffLL, y = __double_as_longlong(b);
    return x <= y && y <= 0x7ff0000000000000LL;
}

__device__ __forceinline__ double max_abs(double a, double b)
{
    const long long m = 0x7fffffffffffffffLL, x = __double_as_longlong(a) & m, y = __double_as_longlong(b) & m;
    return __longlong_as_double(x > y ? x : y);
}

template <typename T>
__device__ __forceinline__ T at_byte(const T *p, unsigned off)
{
    return *reinterpret_cast<const T *>(reinterpret_cast<const unsigned char *>(p) + off);
}

__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float abs_t(float a) { return fabsf(a); }
__device__ __forceinline__ double abs_t(double a) { return fabs(a); }

template <int NM, int G, bool ENERGY, bool F32>
__global__ void __launch_bounds__(kCoopMaxWarps * 32, 3) coop_kernel(const LaunchArgs a, const CoopLayout L)
{
    using R = typename std::conditional<F32, float, double>::type;   // matrix, solve
    constexpr int C = 32 / G, NC = (NM + G - 1) / G, LD = coop_ld(NM);
    extern __shared__ __align__(16) unsigned char sm[];
    const NetView nv = a.nv;
    if (!stage_table(sm, a.blob, static_cast<unsigned>(nv.bytes),
                     reinterpret_cast<uint64_t *>(sm + L.off_bar), &a.scratch->error, kDevErrTma))
        return;
    if (!stage_table(sm + L.off_tab, a.coop, static_cast<unsigned>(L.tab.bytes),
                     reinterpret_cast<uint64_t *>(sm + L.off_bar + 8), &a.scratch->error, kDevErrTma))
        return;
    const double *tA = reinterpret_cast<const double *>(sm + nv.off_A);
    const double *tb = reinterpret_cast<const double *>(sm + nv.off_b);
    const double *tth = reinterpret_cast<const double *>(sm + nv.off_th);
    const double *tdH = reinterpret_cast<const double *>(sm + nv.off_dH);
    const double *tcv = reinterpret_cast<const double *>(sm + nv.off_cv);
    const double *tcnt = reinterpret_cast<const double *>(sm + nv.off_cnt);
    const double *tex = reinterpret_cast<const double *>(sm + nv.off_exp);
    const double *cvp = reinterpret_cast<const double *>(sm + nv.off_cvp);
    const unsigned long long *tidx = reinterpret_cast<const unsigned long long *>(sm + nv.off_idx);
    const float *tbf = reinterpret_cast<const float *>(sm + nv.off_f32), *tthf = tbf + nv.nr, *tdHf = tthf + nv.nr;
    const DevOpts o = a.o;
    const int N = NM < kLaneMaxN ? NM : nv.N, ns = N - (ENERGY ? 1 : 0), ne = nv.ne, nr = nv.nr;
    const long long nc = a.ncells;
    const int lane = threadIdx.x & 31, g = lane / G, gl = lane % G, wid = threadIdx.x >> 5;
    const unsigned gmask = (G == 32 ? kFull : ((1u << (G & 31)) - 1u) << (g * G));
    // per-lane programs
    const unsigned *rowp = reinterpret_cast<const unsigned *>(sm + L.off_tab + L.tab.off_row) + gl;
    const unsigned *jacp = reinterpret_cast<const unsigned *>(sm + L.off_tab + L.tab.off_jac) + gl;
    const unsigned char *jact = sm + L.off_tab + L.tab.off_to + gl;
    const double *coef = reinterpret_cast<const double *>(sm + L.off_tab + L.tab.off_coef);
    int own[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) own[q] = reinterpret_cast<const signed char *>(sm + L.off_tab)[gl * NC + q];
    // the cell's shared memory
    unsigned char *cb = sm + L.base + (wid * C + g) * L.cell_bytes;
    double *ys = reinterpret_cast<double *>(cb);                // current iterate
    float *yf = reinterpret_cast<float *>(cb + L.off_YF);       // current iterate in FP32
    double *fs = reinterpret_cast<double *>(cb + L.off_F);      // f rows; error terms; FP64 solve
    double *ws = reinterpret_cast<double *>(cb + L.off_W);      // reaction rates
    double *K = reinterpret_cast<double *>(cb + L.off_K);       // rate coefficients (isothermal)
    double *CV = reinterpret_cast<double *>(cb + L.off_CV);     // C_V(T) coefficients
    R *part = reinterpret_cast<R *>(cb + L.off_P);              // rate partials [kind][reaction]
    R *M = reinterpret_cast<R *>(cb + L.off_M);                 // matrix, then factors
    R *V = reinterpret_cast<R *>(cb + L.off_V);                 // row scales
    R *xs = reinterpret_cast<R *>(cb + L.off_X);                // right-hand side
    const bool CVP = ENERGY && nv.cvpoly != 0;
    const int nin_max = L.tab.nin_max, kT = nin_max, kq = nin_max + 1;   // kinds: 0.. reactants, T, heat

    // operands of padding and of +-1 coefficients (part's kinds start after them)
    if (gl == 0) {
        ws[nr] = 0.0;
        part[0] = R(0);
        part[1] = R(1);
        part[2] = R(-1);
    }
    const R *part0 = part;
    part += kCoopConst;

    int state = g < L.groups ? kNeed : kDone;
    long long cell = -1;
    if (!a.persistent) {
        cell = (static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + wid) * L.groups + g;
        if (cell >= nc) state = kDone;
    }
    double tt = 0.0, h = 0.0, facmax = 0.0, T_iso = 1.0, invCV = 0.0, atol_s = 0.0, dtc = a.dt;
    int phase = 0, it = 0, natt = 0, nacc = 0, nnew = 0, attempt = 0, refresh = 0;
    bool last = false, needF = false, luok = true, atY = false, fyok = false;
    float dprev = 0.0f, dprevr = 0.0f;
    int pos[NC];                   // where the factors' row order puts the own components
    double Y[NC], FY[NC], YF[NC], YH[NC], CUR[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        Y[q] = FY[q] = YF[q] = YH[q] = CUR[q] = 0.0;
        pos[q] = 0;
    }

    const bool TR = F32 || o.scheme == KT_SCHEME_TRBDF2;
    const TrCoef tr = tr_coef();

    const double natol_f = F32 ? o.newton_atol_frac * kF32NewtonAtolScale : o.newton_atol_frac;
    const float rtol_f = static_cast<float>(o.newton_rtol);
    double natol = 0.0;
    const double inv_n = 1.0 / N;

    auto finish = [&]() { state = a.persistent ? kNeed : kDone; };
    auto y_pre = [&](int s) {
        const double v = a.y_in[static_cast<long long>(s) * nc + cell];
        return v > 0.0 ? v : 0.0;
    };

    // Pre-processing (Sec. 2.2.2), own components
    auto load_pre = [&]() {
        fyok = false;
        const double Tin = a.T_in[cell];
        T_iso = Tin < nv.t_min ? nv.t_min : (Tin > nv.t_max ? nv.t_max : Tin);
#pragma unroll
        for (int q = 0; q < NC; ++q)
            if (own[q] >= 0) Y[q] = ENERGY && own[q] == ns ? T_iso : y_pre(own[q]);
    };

    auto write_out = [&](int st) {
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            if (own[q] < 0) continue;
            if (ENERGY && own[q] == ns) a.T_out[cell] = Y[q];
            else a.y_out[static_cast<long long>(own[q]) * nc + cell] = Y[q];
        }
        if (gl == 0) {
            if (!ENERGY) a.T_out[cell] = T_iso;
            if (a.status) a.status[cell] = st;
            if (a.nsub) a.nsub[cell] = st == KT_STATUS_REVERTED ? 0 : nacc;
            if (a.nnew) a.nnew[cell] = nnew;
        }
    };

    auto begin_attempt = [&]() -> bool {
        if (natt >= o.max_substeps) return false;
        ++natt;
        last = false;
        if (tt + h >= dtc * (1.0 - 1e-12)) {
            h = dtc - tt;
            last = true;
        }
        phase = 0;
        it = 0;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            CUR[q] = Y[q];
            if (own[q] >= 0) {
                ys[own[q]] = Y[q];
                if (F32) yf[own[q]] = static_cast<float>(Y[q]);
            }
        }
        atY = true;
        needF = true;
        refresh = 0;
        return true;
    };

    auto start_run = [&](double h0, double fmax) -> bool {
        tt = 0.0;
        h = h0;
        facmax = fmax;
        natt = 0;
        nacc = 0;
        return begin_attempt();
    };

    // A failed run: one retry from the pre-processed input, else revert (Sec. 2.2.3)
    auto run_fail = [&]() {
        if (attempt == 0 && o.retry) {
            attempt = 1;
            load_pre();
            if (start_run(o.h_init * o.retry_h_factor, o.retry_facmax)) return;
        }
        load_pre();
        __syncwarp(gmask);   // every lane has read T_in before T_out is written (in-place calls)
        write_out(KT_STATUS_REVERTED);
        finish();
    };

    // Post-processing (Sec. 2.2.3) of the state in ys; every lane of the group computes the
    // same correction and applies it to its own components.
    auto post_process = [&]() -> bool {
        double b0[kMaxElements], r[kMaxElements], Mp[kMaxElements * kMaxElements];
        auto yc = [&](int s) { return ys[s] < 0.0 ? 0.0 : ys[s]; };
        for (int e = 0; e < ne; ++e) b0[e] = 0.0;
        for (int s = 0; s < ns; ++s) {
            const double y0 = y_pre(s);
            for (int e = 0; e < ne; ++e) b0[e] = fma(tcnt[s * ne + e], y0, b0[e]);
        }
        for (int e = 0; e < ne; ++e) {
            double tot = 0.0;
            for (int s = 0; s < ns; ++s) tot = fma(tcnt[s * ne + e], yc(s), tot);
            r[e] = tot - b0[e];
            for (int f = 0; f < ne; ++f) {
                double m = 0.0;
                for (int s = 0; s < ns; ++s) m = fma(__dmul_rn(tcnt[s * ne + e], tcnt[s * ne + f]), yc(s), m);
                Mp[e * ne + f] = m;
            }
        }
        for (int e = 0; e < ne; ++e) {
            if (Mp[e * ne + e] == 0.0) {
                if (r[e] != 0.0) return false;
                for (int f = 0; f < ne; ++f) Mp[e * ne + f] = Mp[f * ne + e] = 0.0;
                Mp[e * ne + e] = 1.0;
            }
        }
        for (int k = 0; k < ne; ++k) {   // Gaussian elimination, partial pivoting
            int p = k;
            for (int i = k + 1; i < ne; ++i)
                if (fabs(Mp[i * ne + k]) > fabs(Mp[p * ne + k])) p = i;
            if (!(fabs(Mp[p * ne + k]) > 0.0)) return false;
            if (p != k) {
                for (int j = 0; j < ne; ++j) {
                    const double x = Mp[k * ne + j];
                    Mp[k * ne + j] = Mp[p * ne + j];
                    Mp[p * ne + j] = x;
                }
                const double x = r[k];
                r[k] = r[p];
                r[p] = x;
            }
            for (int i = k + 1; i < ne; ++i) {
                const double l = Mp[i * ne + k] / Mp[k * ne + k];
                for (int j = k; j < ne; ++j) Mp[i * ne + j] = fma(-l, Mp[k * ne + j], Mp[i * ne + j]);
                r[i] = fma(-l, r[k], r[i]);
            }
        }
        for (int i = ne - 1; i >= 0; --i) {
            double s = r[i];
            for (int j = i + 1; j < ne; ++j) s = fma(-Mp[i * ne + j], r[j], s);
            r[i] = s / Mp[i * ne + i];
        }
        auto corrected = [&](int s, double y, bool &ok) {
            double corr = 0.0;
            for (int e = 0; e < ne; ++e) corr = fma(tcnt[s * ne + e], r[e], corr);
            ok = ok && corr < 1.0;
            return fma(-y, corr, y);
        };
        bool ok = !ENERGY || isfinite(ys[ns]);
        for (int s = 0; s < ns; ++s) {
            const double v = corrected(s, yc(s), ok);
            ok = ok && isfinite(v);
        }
#pragma unroll
        for (int q = 0; q < NC; ++q)
            if (own[q] >= 0 && own[q] < ns) {
                bool dummy = true;
                Y[q] = corrected(own[q], yc(own[q]), dummy);
            }
        return ok;
    };

    auto arrhenius_k = [&](int r, double lt, double invT) {
        const double arg = fma(tb[r], lt, -__dmul_rn(tth[r], invT));
        return below_m700(arg) ? 0.0 : __dmul_rn(tA[r], tang_exp(arg, tex));
    };

    auto log_t = [&](double T) { return log(nv.t_ref == 1.0 ? T : T / nv.t_ref); };

    auto begin_cell = [&]() {
        dtc = a.dt_cell ? a.dt_cell[cell] : a.dt;
        bool fin = isfinite(a.T_in[cell]) && dtc > 0.0 && isfinite(dtc);
        for (int s = 0; s < ns; ++s) fin = fin && isfinite(a.y_in[static_cast<long long>(s) * nc + cell]);
        if (!fin) {
            // every read of the input precedes the first write (in-place calls)
            __syncwarp(gmask);
            for (int s = gl; s < ns; s += G)
                a.y_out[static_cast<long long>(s) * nc + cell] = a.y_in[static_cast<long long>(s) * nc + cell];
            if (gl == 0) {
                a.T_out[cell] = a.T_in[cell];
                if (a.status) a.status[cell] = KT_STATUS_NONFINITE;
                if (a.nsub) a.nsub[cell] = 0;
                if (a.nnew) a.nnew[cell] = 0;
            }
            finish();
            return;
        }
        load_pre();
        double cvt = 0.0, b00 = 0.0;
        for (int s = 0; s < ns; ++s) {
            const double y = y_pre(s);
            cvt = fma(tcv[s], y, cvt);
            b00 = fma(tcnt[s * ne], y, b00);
        }
        invCV = ENERGY ? 1.0 / cvt : 0.0;
        if (CVP) {
            for (int k = gl; k < 10; k += G) {
                double c = 0.0;
                for (int s = 0; s < ns; ++s) c = fma(y_pre(s), cvp[s * 10 + k], c);
                CV[k] = c;
            }
        }
        atol_s = (o.atol_mode == 1 && b00 > 0.0) ? __dmul_rn(o.atol, b00) : o.atol;
        natol = __dmul_rn(natol_f, atol_s);
        if (!ENERGY) {
            const double lt = log_t(T_iso), invT = 1.0 / T_iso;
            for (int r = gl; r < nr; r += G) K[r] = arrhenius_k(r, lt, invT);
        }
        attempt = 0;
        nnew = 0;
        state = kRun;
        if (!start_run(o.h_init, o.facmax)) run_fail();
    };

    for (;;) {
        // ---- give every idle group a cell
        for (;;) {
            const bool want = state == kNeed;
            const unsigned m = __ballot_sync(kFull, want && gl == 0);
            if (!m) break;
            if (a.persistent) {
                const int leader = __ffs(m) - 1;
                unsigned long long base = 0;
                if (lane == leader) base = atomicAdd(&a.scratch->queue, static_cast<unsigned long long>(__popc(m)));
                base = __shfl_sync(kFull, base, leader);
                if (want) {
                    const long long q = static_cast<long long>(base + __popc(m & ((1u << (g * G)) - 1u)));
                    if (q >= nc) {
                        state = kDone;
                    } else {
                        cell = a.order ? static_cast<long long>(a.order[q]) : q;
                        begin_cell();
                    }
                }
            } else if (want) {
                begin_cell();
            }
        }
        if (__all_sync(kFull, state == kDone)) break;
        __syncwarp();
        const bool run = state == kRun;

        // ---- one Newton iteration of every running group's current solve
        const double hph = TR ? __dmul_rn(tr.d, h) : (phase == 0 ? h : 0.5 * h);
        const bool trF0 = TR && phase == 0 && atY;
        if (run) ++nnew;
        const bool need = run && (!F32 || needF);
        const bool any_need = __any_sync(kFull, need);
        const double T = ENERGY ? ys[ns] : T_iso;
        const bool bad = !positive(T);
        double lt = 0.0, invT = 0.0, invCVi = invCV, dcvr = 0.0;
        if (ENERGY) {
            // (idle groups take 1: an FP64 division or root of arbitrary bits would send the
            // whole warp through its slow path; the same at a step's end below)
            const double Ts = bad || !run ? 1.0 : T;
            lt = log_t(Ts);
            invT = 1.0 / Ts;
            if (CVP) {
                const int o5 = Ts < nv.t_mid ? 0 : 5;
                const double c0 = CV[o5], c1 = CV[o5 + 1], c2 = CV[o5 + 2], c3 = CV[o5 + 3], c4 = CV[o5 + 4];
                const double cv = (((c4 * Ts + c3) * Ts + c2) * Ts + c1) * Ts + c0;
                const double dcv = ((4.0 * c4 * Ts + 3.0 * c3) * Ts + 2.0 * c2) * Ts + c1;
                invCVi = 1.0 / cv;
                dcvr = dcv * invCVi;
            }
        }
        float hf = 0.0f, invTf = 0.0f, invCVf = 0.0f;
        if (F32 && any_need) {
            hf = static_cast<float>(hph);
            invTf = static_cast<float>(invT);
            invCVf = static_cast<float>(invCVi);
        }
        for (int r = gl; r < nr; r += G) {
            const unsigned long long ix = tidx[r];
            const int nin = static_cast<int>(ix & 0x7f);
            const int i0 = static_cast<int>((ix >> 16) & 0xff), i1 = static_cast<int>((ix >> 24) & 0xff),
                      i2 = static_cast<int>((ix >> 32) & 0xff);
            const double k = ENERGY ? arrhenius_k(r, lt, invT) : K[r];
            const double y0 = ys[i0];
            const double y1 = nin > 1 ? ys[i1] : 1.0;
            const double p01 = __dmul_rn(y0, y1);
            double w = __dmul_rn(k, p01), y2 = 1.0;
            if (nin_max > 2) {
                y2 = nin > 2 ? ys[i2] : 1.0;
                w = __dmul_rn(w, y2);
            }
            ws[r] = w;
            if (any_need) {
                if constexpr (F32) {
                    const float hk = __fmul_rn(hf, static_cast<float>(k));
                    const float f0 = yf[i0], f1 = nin > 1 ? yf[i1] : 1.0f, f2 = nin > 2 ? yf[i2] : 1.0f;
                    part[r] = __fmul_rn(__fmul_rn(hk, f1), f2);
                    if (nin_max > 1) part[nr + r] = __fmul_rn(__fmul_rn(hk, f0), f2);
                    if (nin_max > 2) part[2 * nr + r] = __fmul_rn(__fmul_rn(hk, f0), f1);
                    if (ENERGY) {
                        const float dk = __fmul_rn(__fmul_rn(hk, fmaf(tthf[r], invTf, tbf[r])), invTf);
                        part[kT * nr + r] = __fmul_rn(__fmul_rn(dk, __fmul_rn(f0, f1)), f2);
                        part[kq * nr + r] = __fmul_rn(tdHf[r], invCVf);
                    }
                } else {
                    const double hk = __dmul_rn(hph, k);
                    double d0 = __dmul_rn(hk, y1), d1 = __dmul_rn(hk, y0);
                    if (nin_max > 2) {
                        d0 = __dmul_rn(d0, y2);
                        d1 = __dmul_rn(d1, y2);
                        part[2 * nr + r] = __dmul_rn(hk, p01);
                    }
                    part[r] = d0;
                    if (nin_max > 1) part[nr + r] = d1;
                    if (ENERGY) {
                        double dT = __dmul_rn(hph, __dmul_rn(__dmul_rn(k, fma(tth[r], invT, tb[r])), invT));
                        dT = __dmul_rn(dT, p01);
                        if (nin_max > 2) dT = __dmul_rn(dT, y2);
                        part[kT * nr + r] = dT;
                        part[kq * nr + r] = __dmul_rn(tdH[r], invCVi);
                    }
                }
            }
        }
        __syncwarp();
        // rows of f: each lane sums its rows' +-w_r (the T row -dH_r w_r) in reaction order,
        // as fma(+-1, w, f); a term's operands are loaded one step ahead of its FP64 add, and
        // padding terms add 0 * 0
        double W[NC];
        {
            double f = 0.0;
            const signed char *next = reinterpret_cast<const signed char *>(sm + L.off_tab) + gl * NC;
            unsigned u0 = rowp[0], u1 = rowp[G];
            double w0 = at_byte(ws, u0 & kCoopOffset), c0 = at_byte(coef, u0 >> 16);
#pragma unroll 4
            for (int e = 0; e < L.tab.n_row; ++e) {
                const unsigned u2 = rowp[(e + 2) * G];   // padding steps end the program
                const double w1 = at_byte(ws, u1 & kCoopOffset), c1 = at_byte(coef, u1 >> 16);
                f = fma(c0, w0, f);
                if constexpr (NC > 1) {
                    if (u0 & kCoopEnd) {
                        fs[*next++] = f;
                        f = 0.0;
                    }
                }
                u0 = u1;
                u1 = u2;
                w0 = w1;
                c0 = c1;
            }
            if constexpr (NC == 1) W[0] = f;
        }
        // residual of the own components
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            if constexpr (NC > 1) W[q] = own[q] >= 0 ? fs[own[q]] : 0.0;
            if (ENERGY && own[q] == ns) W[q] = __dmul_rn(W[q], invCVi);
        }
        if (run && TR && atY && !fyok) {
#pragma unroll
            for (int q = 0; q < NC; ++q) FY[q] = W[q];
            fyok = true;
        }
        if (run && trF0) {
#pragma unroll
            for (int q = 0; q < NC; ++q) YH[q] = fma(hph, FY[q], Y[q]);
        }
        R res[NC];
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            const double yb = TR ? YH[q] : (phase == 2 ? YH[q] : Y[q]);
            res[q] = static_cast<R>(-fma(-hph, W[q], __dadd_rn(CUR[q], -yb)));
        }
        // iteration matrix I - h J: each lane sums its entries' updates in reaction order
        if (any_need) {
            R v = R(0);
            const unsigned char *next = jact;
            unsigned u0 = jacp[0], u1 = jacp[G];
            R d0 = at_byte(part0, u0 & kCoopOffset), c0 = at_byte(part0, (u0 >> 16) & kCoopOffset);
#pragma unroll 4
            for (int e = 0; e < L.tab.n_jac; ++e) {
                const unsigned u2 = jacp[(e + 2) * G];
                const R d1 = at_byte(part0, u1 & kCoopOffset), c1 = at_byte(part0, (u1 >> 16) & kCoopOffset);
                v = fma_t(c0, d0, v);
                if (u0 & kCoopEnd) {
                    const unsigned to = *next;
                    next += G;
                    if (need) M[to] = v;
                    v = R(0);
                }
                u0 = u1;
                u1 = u2;
                d0 = d1;
                c0 = c1;
            }
            __syncwarp();
            if (CVP) {
#pragma unroll
                for (int q = 0; q < NC; ++q)
                    if (need && own[q] == ns) {
                        if constexpr (F32)
                            M[ns * LD + ns] += static_cast<float>(__dmul_rn(__dmul_rn(hph, W[q]), dcvr));
                        else
                            M[ns * LD + ns] = fma(__dmul_rn(hph, W[q]), dcvr, M[ns * LD + ns]);
                    }
                __syncwarp();
            }
            // ---- LU with implicit-scaled row pivoting (Algorithm lu-decomp), right-looking
            bool ok = true;
            for (int i = gl; i < N; i += G) {
                R big = R(0);
                for (int j = 0; j < N; ++j) {
                    const R m = abs_t(M[i * LD + j]);
                    big = m > big ? m : big;
                }
                ok = ok && big > R(0);
                const R inv = R(1) / (need && big > R(0) ? big : R(1));
                if (need) V[i] = inv;
            }
            unsigned long long pm = 0xfedcba9876543210ULL;
            __syncwarp();
            ok = (__ballot_sync(kFull, ok) & gmask) == gmask;
#pragma unroll(NM < kLaneMaxN ? NM : 1)
            for (int j = 0; j < (NM < kLaneMaxN ? NM : N); ++j) {
                int imax = j;
                if constexpr (F32) {
                    float tmax = fabsf(M[j * LD + j]) * V[j];
#pragma unroll
                    for (int i = j + 1; i < (NM < kLaneMaxN ? NM : N); ++i) {
                        const float t = fabsf(M[i * LD + j]) * V[i];
                        if (t > tmax) {
                            tmax = t;
                            imax = i;
                        }
                    }
                    ok = ok && tmax > 0.0f;
                } else {
                    // one product per lane, compared as integers (non-negative; a NaN is
                    // never larger, and a NaN on the diagonal fails the factorisation)
                    for (int i = j + gl; i < N; i += G)
                        if (need) fs[i] = __dmul_rn(fabs(M[i * LD + j]), V[i]);
                    __syncwarp();
                    const long long nan0 = 0x7ff0000000000000LL;
                    long long tmax = __double_as_longlong(fs[j]);
                    const bool nand = tmax > nan0;
#pragma unroll(NM < kLaneMaxN ? NM : 1)
                    for (int i = j + 1; i < (NM < kLaneMaxN ? NM : N); ++i) {
                        const long long t = __double_as_longlong(fs[i]);
                        if (t > tmax && t <= nan0) {
                            tmax = t;
                            imax = i;
                        }
                    }
                    ok = ok && tmax > 0 && !nand;
                }
                __syncwarp();
                if (need && imax != j) {
                    for (int k = gl; k < N; k += G) {
                        const R x = M[imax * LD + k];
                        M[imax * LD + k] = M[j * LD + k];
                        M[j * LD + k] = x;
                    }
                    if (gl == 0) V[imax] = V[j];
                }
                const unsigned long long df = ((pm >> (4 * j)) ^ (pm >> (4 * imax))) & 15ULL;
                pm ^= (df << (4 * j)) ^ (df << (4 * imax));
                __syncwarp();
                const R rinv = R(1) / (need ? M[j * LD + j] : R(1));
                __syncwarp();
                for (int i = j + 1 + gl; i < N; i += G)
                    if (need) M[i * LD + j] *= rinv;
                if (need && gl == 0) M[j * LD + j] = rinv;
                __syncwarp();
                const int n1 = (NM < kLaneMaxN ? NM : N) - 1 - j;
                for (int e = gl; e < n1 * n1; e += G) {
                    const int ii = e / n1, kk = e - ii * n1;
                    const int i = j + 1 + ii, k = j + 1 + kk;
                    if (need) M[i * LD + k] = fma_t(-M[i * LD + j], M[j * LD + k], M[i * LD + k]);
                }
                __syncwarp();
            }
            if (need) {
                luok = ok;
                needF = false;
#pragma unroll
                for (int i = 0; i < NM; ++i)
#pragma unroll
                    for (int q = 0; q < NC; ++q)
                        if (i < N && static_cast<int>((pm >> (4 * i)) & 15ULL) == own[q]) pos[q] = i;
            }
        }
        // ---- solve with the factors: right-hand side in pivot order, unit-lower forward, upper
        // backward (terms of a row in ascending column order) times the stored inverse pivot
#pragma unroll
        for (int q = 0; q < NC; ++q)
            if (own[q] >= 0) xs[pos[q]] = res[q];
        __syncwarp();
        double d[NC];
        float df[NC];
        if constexpr (F32) {
            // FP32 costs little beside the FP64 pipe: every lane solves for all unknowns
            // (factors read four at a time, the same for all lanes of the group)
            constexpr int NV = LD / 4;
            float x[LD];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const float4 t = reinterpret_cast<const float4 *>(xs)[v];
                x[4 * v] = t.x;
                x[4 * v + 1] = t.y;
                x[4 * v + 2] = t.z;
                x[4 * v + 3] = t.w;
            }
            const float4 *M4 = reinterpret_cast<const float4 *>(M);
#pragma unroll
            for (int i = 1; i < NM; ++i)
                if (i < N) {
                    float s = x[i];
#pragma unroll
                    for (int v = 0; v < NV; ++v)
                        if (4 * v < i) {
                            const float4 t = M4[i * NV + v];
                            const float m[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (4 * v + k < i) s = fmaf(-m[k], x[4 * v + k], s);
                        }
                    x[i] = s;
                }
#pragma unroll
            for (int i = NM - 1; i >= 0; --i)
                if (i < N) {
                    float s = x[i], inv = 0.0f;
#pragma unroll
                    for (int v = 0; v < NV; ++v)
                        if (4 * v + 3 >= i) {
                            const float4 t = M4[i * NV + v];
                            const float m[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                if (4 * v + k == i) inv = m[k];
                                if (4 * v + k > i && 4 * v + k < NM && 4 * v + k < N) s = fmaf(-m[k], x[4 * v + k], s);
                            }
                        }
                    x[i] = __fmul_rn(s, inv);
                }
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                df[q] = 0.0f;
#pragma unroll
                for (int i = 0; i < NM; ++i)
                    if (own[q] == i) df[q] = x[i];
                d[q] = static_cast<double>(df[q]);
            }
        } else {
            // forward over the lanes (row i of lane i mod G), backward on every lane
            double x[NC];
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                const int i = gl + G * q;
                x[q] = i < N ? xs[i] : 0.0;
            }
#pragma unroll
            for (int k = 0; k < NM - 1; ++k) {
                if (k >= N - 1) break;
                const double xk = __shfl_sync(kFull, x[k / G], g * G + k % G);
#pragma unroll
                for (int q = 0; q < NC; ++q) {
                    const int i = gl + G * q;
                    if (i > k && i < N) x[q] = fma(-M[i * LD + k], xk, x[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < NC; ++q)
                if (gl + G * q < N) fs[gl + G * q] = x[q];
            __syncwarp();
            double z[NM];
#pragma unroll
            for (int i = NM - 1; i >= 0; --i)
                if (i < N) {
                    double s = fs[i];
#pragma unroll
                    for (int k = i + 1; k < NM; ++k)
                        if (k < N) s = fma(-M[i * LD + k], z[k], s);
                    z[i] = __dmul_rn(s, M[i * LD + i]);
                }
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                d[q] = 0.0;
#pragma unroll
                for (int i = 0; i < NM; ++i)
                    if (own[q] == i) d[q] = z[i];
            }
        }
        // ---- update and convergence (the monitors of kt_lane.cuh)
        bool convl = true;
        float dmax = 0.0f, dmaxr = 0.0f;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            if (own[q] < 0) continue;
            const double y = __dadd_rn(CUR[q], d[q]);
            const float y32 = F32 ? static_cast<float>(y) : 0.0f;
            if (run) {
                CUR[q] = y;
                ys[own[q]] = y;
                if (F32) yf[own[q]] = y32;
            }
            const double tol = fma(o.newton_rtol, fabs(y), own[q] < ns ? natol : 0.0);
            if (!abs_le(d[q], tol)) convl = false;
            if constexpr (F32) {
                // (idle groups divide by 1, see above)
                const float ad = run ? fabsf(df[q]) : 0.0f, tf = run ? static_cast<float>(tol) : 1.0f;
                const float e = __fdiv_rn(ad, fmaxf(tf, 1e-37f));
                const float trl = run ? __fmul_rn(rtol_f, fabsf(y32)) : 1.0f;
                const float er = __fdiv_rn(ad, fmaxf(trl, 1e-37f));
                dmax = e > dmax ? e : dmax;
                dmaxr = er > dmaxr ? er : dmaxr;
            }
        }
        atY = false;
        const bool all_small = (__ballot_sync(kFull, convl) & gmask) == gmask;
        bool conv = !bad && luok && all_small;
        if constexpr (F32) {
            if constexpr (G == 32) {   // non-negative: ordered like their bit patterns
                dmax = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(dmax)));
                dmaxr = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(dmaxr)));
            } else {
#pragma unroll
                for (int s = G / 2; s > 0; s >>= 1) {
                    dmax = fmaxf(dmax, __shfl_xor_sync(kFull, dmax, s));
                    dmaxr = fmaxf(dmaxr, __shfl_xor_sync(kFull, dmaxr, s));
                }
            }
            if (!conv && !bad && luok && it > 0 && run) {
                const float th = dmaxr / dprevr;
                if (th < 0.5f && th / (1.0f - th) * dmaxr <= 1.0f) conv = true;
            }
        }

        // ---- control (per group)
        bool step = false, failed = false;
        if (run) {
            bool nfail = false;
            if (conv) {
                if (TR) {
                    if (phase == 0) {   // BDF2 stage: r = w1 y_g - w0 y_n, start from y_g
                        phase = 1;
                        it = 0;
#pragma unroll
                        for (int q = 0; q < NC; ++q) {
                            YF[q] = CUR[q];
                            YH[q] = fma(tr.w1, CUR[q], -__dmul_rn(tr.w0, Y[q]));
                        }
                    } else {
                        step = true;
                    }
                } else if (phase == 0) {
                    phase = 1;
                    it = 0;
#pragma unroll
                    for (int q = 0; q < NC; ++q) {
                        YF[q] = CUR[q];
                        CUR[q] = Y[q];
                        if (own[q] >= 0) ys[own[q]] = Y[q];
                    }
                } else if (phase == 1) {
                    phase = 2;
                    it = 0;
#pragma unroll
                    for (int q = 0; q < NC; ++q) {
                        YH[q] = CUR[q];
                        if (o.guess != KT_GUESS_PREV) CUR[q] = YF[q];
                        if (own[q] >= 0) ys[own[q]] = CUR[q];
                    }
                } else {
                    step = true;
                }
            } else if (!F32) {
                if (bad || !luok || it + 1 >= o.max_newton) nfail = true;
                else ++it;
            } else {
                const bool stalled = it > 0 && !(dmax < 0.5f * dprev);
                if (bad || !luok || !isfinite(dmax)) {
                    nfail = true;
                } else if (stalled || it + 1 >= o.max_newton) {
                    if (refresh < 2) {
                        ++refresh;
                        needF = true;
                        it = 0;
                    } else {
                        nfail = true;
                    }
                } else {
                    ++it;
                }
                dprev = dmax;
                dprevr = dmaxr;
            }
            if (nfail) {
                h *= 0.5;
                failed = h < o.h_min || !begin_attempt();
            }
        }
        // ---- end of a step: weighted RMS of the error estimate, then accept or reject
        if (__any_sync(kFull, step)) {
            const double inv = TR ? 1.0 / (step ? hph : 1.0) : 0.0, ce = __dmul_rn(__dmul_rn(2.0, tr.C), h);
            __syncwarp();
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                const double yn = Y[q], y1 = CUR[q];
                const double mx = max_abs(yn, y1), at = own[q] < ns ? atol_s : 0.0;
                const double sc = fma(o.rtol, mx, at);
                double est;
                if (TR) {
                    const double f0 = FY[q];
                    const double fg = fma(__dadd_rn(YF[q], -yn), inv, -f0);
                    const double f1 = __dmul_rn(__dadd_rn(y1, -YH[q]), inv);
                    est = __dmul_rn(ce, fma(tr.a2, f1, fma(tr.a0, f0, __dmul_rn(tr.a1, fg))));
                } else {
                    est = __dadd_rn(y1, -YF[q]);
                }
                const bool on = step && own[q] >= 0;
                const double e = (on ? est : 1.0) / (on ? sc : 1.0);
                if (on) fs[own[q]] = e;
            }
            __syncwarp();
            // (compiled for a fixed size, the lane kernels' sum starts e0^2 + RN(e1^2))
            double s2;
            if constexpr (NM < kLaneMaxN) {
                s2 = fma(fs[0], fs[0], __dmul_rn(fs[1], fs[1]));
#pragma unroll
                for (int i = 2; i < NM; ++i) s2 = fma(fs[i], fs[i], s2);
            } else {
                const bool fixed = lane_fixed(N);
                s2 = fixed ? fma(fs[0], fs[0], __dmul_rn(fs[1], fs[1])) : 0.0;
                for (int i = fixed ? 2 : 0; i < N; ++i) s2 = fma(fs[i], fs[i], s2);
            }
            // s2 / N rounded once: quotient by the reciprocal of the small integer N, then one
            // correction step (Markstein 1990: correctly rounded while nothing under- or
            // overflows; where it does, both give the same decision)
            double ms = __dmul_rn(s2, inv_n);
            ms = fma(fma(-static_cast<double>(N), ms, s2), inv_n, ms);
            const double err = sqrt(step ? ms : 1.0);
            const bool acc = err <= 1.0;
            double fac = 0.9 / (TR ? cbrt(err) : sqrt(err));
            if (acc && !(err > 0.0)) fac = facmax;
            bool fin = false;
            if (step) {
                if (acc) {
#pragma unroll
                    for (int q = 0; q < NC; ++q) {
                        if (TR) FY[q] = __dmul_rn(__dadd_rn(CUR[q], -YH[q]), inv);   // first same as last
                        Y[q] = CUR[q];
                    }
                    fyok = TR;
                    ++nacc;
                    fin = last;
                    if (!fin) {
                        tt += h;
                        if (fac > facmax) fac = facmax;
                        if (fac < 0.2) fac = 0.2;
                        h *= fac;
                        failed = !begin_attempt();
                    }
                } else {
                    if (!(fac >= 0.2)) fac = 0.2;
                    h *= fac;
                    failed = h < o.h_min || !begin_attempt();
                }
            }
            if (__any_sync(kFull, fin)) {
                if (fin) {   // ys holds the accepted state
                    if (post_process()) {
                        __syncwarp(gmask);
                        write_out(attempt == 0 ? KT_STATUS_OK : KT_STATUS_RETRIED);
                        finish();
                    } else {
                        failed = true;
                    }
                }
                __syncwarp();
            }
        }
        if (failed) run_fail();
    }
}

// One warp per block up to an SM's worth of warps, so that a small batch spreads over all
// SMs; then four (one per scheduler), which share the staged tables.
template <int NM, int G, bool ENERGY, bool F32>
int launch_t(const LaunchArgs &a, const LaunchCfg &c, cudaStream_t s)
{
    // (programs laid out for another size class would place the matrix by another row stride)
    if (coop_nm(a.nv.N, a.nv.energy) != NM || a.coop_tab.ld != coop_ld(NM)) return cudaErrorInvalidConfiguration;
    CoopLayout L = coop_layout(a.nv.N, a.nv.nr, a.nv.energy, F32 ? 1 : 0, a.nv.bytes, a.nv.cvpoly, a.coop_tab);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int smem_optin = 0, nsm = 0;
    cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    constexpr int C = 32 / G;
    // fewer cells than cells the schedulers' warps could hold: leave groups idle rather
    // than schedulers (a warp's groups share its FP64 instructions, but each also adds its
    // step ends and factorisations to the warp's path)
    const long long per_warp = (a.ncells + 4LL * nsm - 1) / (4LL * nsm);
    L.groups = per_warp < C ? static_cast<int>(per_warp) : C;
    const long long want = (a.ncells + L.groups - 1) / L.groups;   // warps
    const long long per_sm = (want + nsm - 1) / nsm;
    int warps = c.block_warps > 0 ? c.block_warps : (per_sm < kCoopMaxWarps ? static_cast<int>(per_sm) : kCoopMaxWarps);
    if (warps > kCoopMaxWarps) warps = kCoopMaxWarps;
    const int warp_bytes = C * L.cell_bytes;
    while (warps > 1 && L.base + warps * warp_bytes > smem_optin) --warps;
    const size_t smem = static_cast<size_t>(L.base) + static_cast<size_t>(warps) * warp_bytes;
    if (smem > static_cast<size_t>(smem_optin)) return cudaErrorInvalidConfiguration;
    auto kern = coop_kernel<NM, G, ENERGY, F32>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    const int threads = warps * 32;
    long long blocks = (want + warps - 1) / warps;
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

template <int NM, bool ENERGY, bool F32>
int launch_g(const LaunchArgs &a, const LaunchCfg &c, cudaStream_t s)
{
    switch (a.coop_g) {
    case 8: return launch_t<NM, 8, ENERGY, F32>(a, c, s);
    case 16: return launch_t<NM, 16, ENERGY, F32>(a, c, s);
    default: return launch_t<NM, 32, ENERGY, F32>(a, c, s);
    }
}

}  // namespace

// One size and form each, every one in its own translation unit (compile time).
int launch_coop_n3(const LaunchArgs &a, const LaunchCfg &c, void *stream);
int launch_coop_n11_f32(const LaunchArgs &a, const LaunchCfg &c, void *stream);
int launch_coop_n11_f64(const LaunchArgs &a, const LaunchCfg &c, void *stream);
int launch_coop_any_f64(const LaunchArgs &a, const LaunchCfg &c, void *stream);

}  // namespace kt
