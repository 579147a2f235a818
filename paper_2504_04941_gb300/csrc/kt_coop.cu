// kt_coop.cu -- when a cell of a small network gets several lanes, and how many.
//
// Where the lines lie (GB300, ms, combustion network, FP32-LU TR-BDF2; one cell per lane |
// G = 8 | 16 | 32):
//   2,048 cells, dt 1e-8 s:    305 |  51 |  33 |  28
//   8,192:                     308 |  60 |  44 |  50
//   32,768:                    348 | 105 | 104 | 139
//   131,072:                   485 | 285 | 333 | 503
//   262,144, dt 1e-9 s:        269 | 176 | 210 |
// With few cells per scheduler a launch lasts as long as its longest cell, so the shortest
// chain (G = 32) wins; with many, the FP64 pipe is full and the fewest instructions per
// cell win (G = 8; 4 measured the same and is not built).  One cell per lane stays for the
// large isothermal batches: without exponentials a cell's chain is short and the exchanges
// of a group cost more than the rates (Robertson, 65,536 cells, FP64 over 1e-6 s: 0.28 ms
// against 0.43; 16,384 cells over 100 s: 21.7 against 16.0).
#include "kt_coop.cuh"

namespace kt {

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
    if (!a.nv.energy && per >= 16) return 0;
    switch (coop_nm(a.nv.N, a.nv.energy)) {
    case 3: return 4;
    case 11: return per < 10 ? 32 : (per < 54 ? 16 : 8);
    default: return f32 ? 0 : 16;
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
