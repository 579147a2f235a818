// kt_coop.cu -- when a cell of a small network gets several lanes, and how many.
//
// Where the lines lie (GB300, ms, one cell per lane | group).  With few cells per scheduler a
// launch lasts as long as its longest cell, so the shortest chain wins; with many, the FP64 pipe
// is full and the fewest instructions per cell win, and of calls of a few steps each, whose
// lanes hardly diverge, the kernels with one cell per lane need the fewest.
// Eleven unknowns with temperature, FP32-LU TR-BDF2, dt 1e-8 s, G = 8 | 16 | 32:
//   2,048 cells    305 |  51 |  33 |  28
//   8,192          308 |  60 |  44 |  50
//   32,768         348 | 105 | 104 | 139
//   131,072        485 | 285 | 333 | 503
//   (4 measured the same as 8 and is not built).  Short intervals, dt in first steps h_init:
//              dt 0.1 h_init     1 h_init        10 h_init      100 h_init
//   20,000     0.78 | 0.93      3.1 | 1.2
//   48,000     1.27 | 1.67      3.6 | 2.3
//   131,072    2.6  | 4.7       5.0 | 5.6      21.1 | 15.1     76.7 | 36.3
//   1,048,576  20.7 | 39.6     24.7 | 42.8    103   | 108     289   | 232
//   FP64: 131,072 6.3 | 7.6, 12.7 | 9.7, 47.6 | 30.5; 1,048,576 47.1 | 62.4, 60.5 | 71.5,
//   216 | 209.  Backward Euler's step doubling takes enough iterations for the groups at every
//   size (1,048,576 cells, dt 0.1 h_init: 126 | 102).
// Three isothermal unknowns (G = 4): without exponentials a cell's chain is short and the
// exchanges of a group cost more than the rates once the chip is full (65,536 cells, FP64 over
// 1e-6 s: 0.28 | 0.43); up to 9,727 cells the groups are ahead at every interval (9,700 cells:
// 1e-7 s 0.156 | 0.104, 100 s 26.6 | 10.5).
// Any other size, FP64, G = 16, whose idle lanes cost more the fewer the unknowns:
//                          one or two steps              longer
//   7, with temperature    5,000 cells 0.42 | 0.35       50,000 cells 87.8 | 37.5
//                          9,700       0.42 | 0.52       200,000      27.8 | 33.4 (dt 1e-11 s)
//   8                                                    9,700       447 | 253
//                                                        20,000      428 | 485, 200,000 1,571 | 4,407
//   10                     9,700       1.02 | 0.87       25,000      647 | 529
//                          14,500      1.02 | 1.28       50,000      486 | 556
//   13                     25,000      2.2 | 2.2         200,000     384 | 183
//                          50,000      4.0 | 4.3
//   16                     200,000     27.9 | 22.6       200,000   8,104 | 4,823
//   6 isothermal           5,000       0.29 | 0.30       9,700      10.8 | 4.8
//   9                      5,000       0.61 | 0.47, 9,700 0.61 | 0.67
//   11                     6,000       0.56 | 0.60       9,700      26.2 | 9.4
//   12                     9,700       0.90 | 0.80       9,700       185 | 50
#include "kt_coop.cuh"

namespace kt {

namespace {

// Cells per scheduler up to which the 16-lane FP64 kernel of any size is the faster one, by the
// figures above (sizes between two measured ones take the smaller one's); few: the interval
// takes no more than two steps that are accepted and grow by facmax, so that the lanes of a
// warp can stay together.
long long any_size_line(int N, bool energy, bool few)
{
    constexpr long long all = 1LL << 62;
    if (!energy) return few ? (N < 9 ? 8 : (N < 12 ? 9 : 16)) : 16;
    if (few) return N < 10 ? 10 : (N < 13 ? 18 : (N < 16 ? 40 : all));
    return N < 10 ? 26 : (N < 13 ? 50 : (N < 16 ? 300 : all));
}

}  // namespace

int coop_group(const LaunchArgs &a, const LaunchCfg &c)
{
    const bool f32 = c.form == KT_FORM_FP32LU;
    // the Jacobian cache, the learned guess and FP32-LU under backward Euler (whose failed
    // solves are redone in FP64) run one cell per lane
    if (a.mlp || (f32 && (a.o.scheme != KT_SCHEME_TRBDF2 || c.lane_variant == KT_LANE_JCACHE))) return 0;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long per = a.ncells / (4LL * nsm);   // cells per scheduler
    // first steps that the interval holds (steps of each cell's own are not known here)
    const double steps = a.dt_cell ? 1e300 : a.dt / a.o.h_init;
    switch (coop_nm(a.nv.N, a.nv.energy)) {
    case 3: return per < 16 ? 4 : 0;
    case 11:
        // the interval below which one cell per lane is ahead grows with the batch
        if (a.o.scheme == KT_SCHEME_TRBDF2 && per >= 25 && steps <= per / (f32 ? 100.0 : 250.0)) return 0;
        return per < 10 ? 32 : (per < 54 ? 16 : 8);
    default: return !f32 && per < any_size_line(a.nv.N, a.nv.energy != 0, steps <= 1.0 + a.o.facmax) ? 16 : 0;
    }
}

bool coop_fits(const LaunchArgs &a, const LaunchCfg &c)
{
    const CoopLayout L = coop_layout(a.nv.N, a.nv.nr, a.nv.energy, c.form == KT_FORM_FP32LU, a.nv.bytes, a.nv.cvpoly,
                                     a.coop_tab);
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return L.base + 32 / a.coop_g * L.cell_bytes <= optin;
}

int launch_coop(const LaunchArgs &a, const LaunchCfg &c, void *stream)
{
    switch (coop_nm(a.nv.N, a.nv.energy)) {
    case 3: return launch_coop_n3(a, c, stream);
    case 11: return c.form == KT_FORM_FP32LU ? launch_coop_n11_f32(a, c, stream) : launch_coop_n11_f64(a, c, stream);
    default: return launch_coop_any_f64(a, c, stream);
    }
}

}  // namespace kt
