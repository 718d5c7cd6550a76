"""Constants of the odd half of the FP32/FP64 collision (odd_constants.h, compiled
here for the CPU) in exact rational arithmetic: 3ca and 3cb against 1 - k1 and
1 - (1 - k1)/2.  Rounding leaves each candidate residuals of up to 2^-24 of
these two numbers (whose halved first and second sum to 1); the least sum of
1024 candidates is expected near 2^-27, and one above 2^-25 has a probability of e^-16."""

import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_1601_00704_gb300", "csrc")
SHIM = """
#include "odd_constants.h"
extern "C" void f32(float w, float *o) { const auto r = odd_constants(w); o[0] = r.c; o[1] = r.a; o[2] = r.b; }
extern "C" void f64(double w, double *o) { const auto r = odd_constants(w); o[0] = r.c; o[1] = r.a; o[2] = r.b; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("odd")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", SRC, str(d / "shim.cpp"), "-o",
                    str(d / "shim.so")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("name,dtype,ctype,bits", [("f32", np.float32, ctypes.c_float, 24),
                                                   ("f64", np.float64, ctypes.c_double, 53)])
def test_no_momentum_is_lost(lib, name, dtype, ctype, bits):
    out, off = (ctype * 3)(), []
    for tau in [0.5 + 1e-6, 0.501, 0.51] + [0.52 + 0.013 * i for i in range(200)] + [10.0, 333.3, 1e6]:
        w = dtype(1.0 / tau)
        getattr(lib, name)(ctype(w), out)
        c, a, b = (Fraction(float(v)) for v in out)
        om = Fraction(float(dtype(1) - (dtype(1) - w)))
        assert Fraction(1, 8) <= c < Fraction(1, 7)
        off.append(float(abs(3 * c * a - om) + abs(3 * c * b - (1 - om / 2))))
    assert max(off) <= 2.0 ** -(bits + 1) and np.mean(off) <= 2.0 ** -(bits + 3)
