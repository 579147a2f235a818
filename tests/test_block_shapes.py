"""The launch tuner's block sizes (csrc/kt_internal.h block_shapes): every value launches a block of
another shape, up to the largest the kernel takes, so no candidate is timed twice and a tuned
value is the number of warps that run.  Host compiler only."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2504_04941_gb300", "csrc")

PROBE = r"""
#include "kt_internal.h"
extern "C" int shapes(int N, int cpw, int groups, int *w)
{
    int v[4];
    const int n = kt::block_shapes(N, cpw, groups != 0, v);
    for (int i = 0; i < n; ++i) w[i] = v[i];
    return n;
}
"""


@pytest.mark.parametrize("N,cpw,groups,unit,most", [(3, 32, 0, 1, 8), (16, 32, 0, 1, 8), (11, 32, 1, 1, 4), (11, 1, 0, 1, 4),
                                                    (32, 1, 0, 1, 4), (33, 1, 0, 4, 16), (96, 1, 0, 4, 16)])
def test_every_value_is_another_launch(tmp_path, N, cpw, groups, unit, most):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, so = tmp_path / "probe.cpp", tmp_path / "probe.so"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True,
                   capture_output=True)
    w = np.zeros(4, np.int32)
    n = ctypes.CDLL(str(so)).shapes(N, cpw, groups, ctypes.c_void_p(w.ctypes.data))
    w = w[:n].tolist()
    # what the launchers make of a value: whole units, at least one, at most `most` warps
    run = [min(max(v // unit, 1) * unit, most) for v in w]
    assert run == w and len(set(w)) == n and w[0] == unit and w[-1] == most
