"""Shared memory of the larger-network kernels (csrc/kt_internal.h warp_layout).

Whatever network ran before the per-reaction partials were kept still runs: the slim layout
(no partials) needs no more than the earlier one, six FP64 vectors, two FP64 values per
reaction and a row-major matrix (two under FP32 backward Euler).  Host compiler only.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_04941_gb300", "csrc")
PROBE = r"""
#include "kt_internal.h"
extern "C" int probe(int N, int nr, int energy, int fp32, int share, int nin_max, int cvpoly, int slim, int *out)
{
    const kt::WarpLayout L = kt::warp_layout(N, nr, energy, fp32, 0, share != 0, nin_max, cvpoly, slim != 0);
    const int v[12] = {L.off_J, L.off_M, L.off_V, L.off_G, L.off_X, L.off_Y, L.off_W, L.off_RW, L.off_K, L.off_D, L.off_CV, L.off_C};
    for (int i = 0; i < 12; ++i) out[i] = v[i];
    out[12] = L.LD;
    return L.warp_bytes;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("team")
    src, so = d / "probe.cpp", d / "probe.so"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True,
                   capture_output=True)
    return ctypes.CDLL(str(so)).probe


def _earlier(N, nr, fp32, share):
    a = lambda b: (b + 15) & ~15
    r, nn = (4 if fp32 else 8), N * (N | 1)
    o = a(nn * r) * (1 if share or not fp32 else 2) + a(N * r) + 2 * a(N * 4) + 6 * a(N * 8) + 2 * a(nr * 8)
    return (o + 127) & ~127


@pytest.mark.parametrize("fp32,share", [(0, 1), (1, 1), (1, 0)])
def test_slim_layout_needs_no_more_than_before(probe, fp32, share):
    out = (ctypes.c_int * 13)()
    for N in range(1, 97):
        for nr in (1, 200, 1001, 2500):
            for energy in (0, 1):
                for cvpoly in ((0, 1) if energy else (0,)):
                    got = probe(N, nr, energy, fp32, share, 3, cvpoly, 1, out)
                    # the coefficients of polynomial heat capacities moved here from registers
                    assert got <= _earlier(N, nr, fp32, share) + 128 * cvpoly, (N, nr, energy, cvpoly)
                    assert out[9] == -1 and out[12] >= N


def test_columns_start_on_16_bytes_an_odd_number_of_units_apart(probe):
    out = (ctypes.c_int * 13)()
    for N in range(1, 97):
        for fp32, unit in ((1, 4), (0, 2)):
            probe(N, 100, 1, fp32, 1, 2, 0, 0, out)
            assert out[12] % unit == 0 and (out[12] // unit) % 2 == 1 and all(o % 16 == 0 for o in out[:9])
