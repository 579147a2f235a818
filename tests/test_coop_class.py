"""The size class that a network's group programs are laid out for is the one of the kernel
that reads them (csrc/kt_coop.cu, csrc/kt_coop_tables.cu, csrc/kt_internal.h).

The dispatch is compiled as it stands against launchers that record which kernel they are;
for every number of unknowns, with and without temperature, in both forms and at batch
sizes on both sides of every line, the row stride of the programs' matrix places must be
that kernel's, and its matrix must end inside its part of the cell.  Host compiler only.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2504_04941_gb300", "csrc")

# stands in for the kernels' header: what the dispatch sees of CUDA, and launchers that
# return the size they are compiled for
STUB = r"""
#include <cstdint>
#include "kt_internal.h"
using cudaError_t = int;
constexpr int cudaSuccess = 0, cudaDevAttrMultiProcessorCount = 1, cudaDevAttrMaxSharedMemoryPerBlockOptin = 2,
              cudaErrorInvalidValue = 1;
inline int cudaGetDevice(int *d) { return *d = 0; }
inline int cudaDeviceGetAttribute(int *v, int a, int) { return *v = a == 1 ? 152 : 232448, 0; }
namespace kt {
int launch_coop_n3(const LaunchArgs &, const LaunchCfg &, void *) { return 3; }
int launch_coop_n11_f32(const LaunchArgs &, const LaunchCfg &, void *) { return 11; }
int launch_coop_n11_f64(const LaunchArgs &, const LaunchCfg &, void *) { return 11; }
int launch_coop_any_f64(const LaunchArgs &, const LaunchCfg &, void *) { return kLaneMaxN; }
}
"""
PROBE = r"""
#include "kt_coop.cu"
#include "kt_coop_tables.cu"
// out: lanes per cell (0: one cell per lane), size of the kernel, largest matrix place
// written, first byte of the matrix, first byte behind it, element size, whether the programs
// of that many lanes are laid out
// (dt in first steps; negative: one per cell)
extern "C" int route_dt(int N, int energy, int form, int scheme, long long ncells, double dt, int nr, const int *nin,
                        const int *in, int *out)
{
    kt::LaunchArgs a{};
    const double dt_cell = dt;
    a.dt = dt;
    a.dt_cell = dt < 0.0 ? &dt_cell : nullptr;
    a.o.h_init = 1.0;
    a.o.facmax = 4.0;
    a.nv.N = N;
    a.nv.ns = N - energy;
    a.nv.nr = nr;
    a.nv.energy = energy;
    a.ncells = ncells;
    a.o.scheme = scheme;
    const kt::LaunchCfg c{form, 1, 0, 0, 32, 0};
    a.coop_g = out[0] = kt::coop_group(a, c);
    if (!a.coop_g) return 0;
    std::vector<unsigned char> b;
    std::vector<double> dH(nr, 1.0);
    const int f32 = form == KT_FORM_FP32LU;
    if (!kt::coop_tables(N, N - energy, nr, energy, nin, nin, reinterpret_cast<const int(*)[3]>(in),
                         reinterpret_cast<const int(*)[3]>(in), dH.data(), f32, a.coop_g, &a.coop_tab, &b))
        return -1;
    out[1] = kt::launch_coop(a, c, nullptr);
    out[2] = 0;
    for (int i = a.coop_tab.off_to; i < a.coop_tab.off_coef; ++i) out[2] = std::max(out[2], static_cast<int>(b[i]));
    const kt::CoopLayout L = kt::coop_layout(N, nr, energy, f32, 0, 0, a.coop_tab);
    out[3] = L.off_M;
    out[4] = L.off_V;
    out[5] = f32 ? 4 : 8;
    out[6] = kt::coop_sizes(kt::coop_nm(N, energy), f32) * 4 & a.coop_g;
    return 1;
}
extern "C" int route(int N, int energy, int form, int scheme, long long ncells, int nr, const int *nin, const int *in,
                     int *out)
{
    for (double dt : {1e-3, 1.0, 1e6}) {
        const int got = route_dt(N, energy, form, scheme, ncells, dt, nr, nin, in, out);
        if (got) return got;
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("coopclass")
    shutil.copy(os.path.join(CSRC, "kt_coop.cu"), d)      # finds the stub beside it first
    (d / "kt_coop.cuh").write_text(STUB)
    src, so = d / "probe.cpp", d / "probe.so"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(src), "-o", str(so)], check=True, capture_output=True)
    lib = ctypes.CDLL(str(so))
    lib.route_dt.argtypes = [ctypes.c_int] * 4 + [ctypes.c_longlong, ctypes.c_double, ctypes.c_int] + [ctypes.c_void_p] * 3
    lib.route.argtypes = [ctypes.c_int] * 4 + [ctypes.c_longlong, ctypes.c_int] + [ctypes.c_void_p] * 3
    return lib


@pytest.mark.parametrize("form", [0, 1], ids=["fp64", "fp32lu"])
@pytest.mark.parametrize("energy", [0, 1])
@pytest.mark.parametrize("N", range(1, 17))
def test_programs_and_kernel_agree_on_the_row_stride(probe, N, energy, form):
    ns = N - energy
    if ns < 1:
        pytest.skip("no species")
    nr = 20
    nin = np.full(nr, 2, np.int32)
    pin = np.array([[r % ns, (r + 1) % ns, -1] for r in range(nr)], np.int32)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    for scheme in (0, 1):
        for ncells in (1, 250, 6079, 6080, 9727, 9728, 32832, 65536, 10**6):
            out = np.zeros(7, np.int32)
            got = probe.route(N, energy, form, scheme, ncells, nr, p(nin), p(pin), p(out))
            assert got >= 0
            if got == 0:
                continue
            NM, written, begin, end, size, laid_out = (int(v) for v in out[1:])
            assert laid_out
            assert N <= NM
            ld = (NM + 3) & ~3                       # rows of the kernel's matrix
            assert written == (N - 1) * ld + N - 1   # the last entry lies where the kernel reads it
            assert begin + ((N - 1) * ld + N) * size <= end
