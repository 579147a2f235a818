"""The ray tracer's table of powers is formed once per process, not per call, and holds
2^(j/256) to both its parts' precision (csrc/kt_ray.cu).  Host compiler only."""
import ctypes
import os
import re
import shutil
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_04941_gb300", "csrc")

PROBE = r"""
#include <cmath>
#include "kt_internal.h"
static int calls = 0;
namespace kt {
double exp2_table(int j)
{
    ++calls;
    return static_cast<double>(std::exp2(static_cast<long double>(j) / static_cast<long double>(kExpTable)));
}
%s
}
extern "C" int powers(double *hi, double *lo)
{
    const kt::RayExpTable &t = kt::ray_exp_table();
    for (int j = 0; j < kt::kExpTable; ++j) hi[j] = t.hi[j], lo[j] = t.lo[j];
    return calls;
}
"""


def test_table_is_formed_once_and_exact(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    with open(os.path.join(CSRC, "kt_ray.cu")) as f:
        code = f.read()
    entry = code[code.index("KT_API int kt_raytrace("):]
    assert "exp2" not in entry[:entry.index("\n}\n")].replace("ray_exp_table", "")   # no power in the entry itself
    part = re.search(r"struct RayExpTable \{.*?\n\};\n.*?\n\}\n", code, re.S).group(0)
    src, so = tmp_path / "probe.cpp", tmp_path / "probe.so"
    src.write_text(PROBE % part)
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True,
                   capture_output=True)
    lib = ctypes.CDLL(str(so))
    hi, lo = np.zeros(256), np.zeros(256)
    got = [lib.powers(ctypes.c_void_p(hi.ctypes.data), ctypes.c_void_p(lo.ctypes.data)) for _ in range(3)]
    assert got == [256, 256, 256]
    getcontext().prec = 60
    for j in range(256):
        v = Decimal(2) ** (Decimal(j) / 256)
        # hi to half an ulp; the residue as exactly as the host's long double (64 bits or more) has it
        assert abs(v - Decimal(float(hi[j]))) <= Decimal(2) ** -53
        assert abs(v - Decimal(float(hi[j])) - Decimal(float(lo[j]))) <= Decimal(2) ** -63
