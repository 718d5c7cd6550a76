"""The integer-unit exponential, product and reciprocal of the EM kernel
(fixed.cuh, compiled here for the CPU) against 60-digit decimal arithmetic: at
the edges of table entries, of the integer part and of the significand.  Bound:
the sum of the truncations, at most 8 units of 2^-63 before rounding to FP64."""

import ctypes
import decimal
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_1601_00704_gb300", "csrc")
SHIM = """
#include "fixed.cuh"
static constexpr fx::Table table = fx::make_table();
extern "C" void exp2_neg(uint64_t m, int e, uint64_t *om, int *oe) {
    const fx::Num r = fx::exp2_neg(fx::Num{m, e}, table.t); *om = r.m; *oe = r.e; }
extern "C" void reciprocal(uint64_t m, int e, uint64_t *om, int *oe) {
    const fx::Num r = fx::reciprocal(fx::Num{m, e}); *om = r.m; *oe = r.e; }
extern "C" double product(double a, double b) { return fx::pack(fx::mul(fx::unpack(a), fx::unpack(b))); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", SRC, str(d / "shim.cpp"), "-o",
                    str(d / "shim.so")], check=True)
    lib = ctypes.CDLL(str(d / "shim.so"))
    lib.product.restype = ctypes.c_double
    lib.product.argtypes = [ctypes.c_double] * 2
    return lib


def call(fn, m, e):
    om, oe = ctypes.c_uint64(), ctypes.c_int()
    fn(ctypes.c_uint64(m), ctypes.c_int(e), ctypes.byref(om), ctypes.byref(oe))
    assert om.value >> 63 == 1
    return decimal.Decimal(om.value) * decimal.Decimal(2) ** (oe.value - 63)


def significands(rng, n):
    top = 1 << 63
    edge = [top, top + 1, 2 * top - 1, top + (top >> 1), top + (top >> 7), top + (top >> 7) - 1, 2 * top - (top >> 23)]
    return edge + [int(a) | top for a in rng.integers(0, 1 << 63, n, dtype=np.uint64)]


@pytest.mark.parametrize("e", [-200, -66, -64, -40, -8, -7, -1, 0, 1, 5, 9])
def test_exponential(lib, e):
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        for m in significands(np.random.default_rng(e + 300), 60):
            t = decimal.Decimal(m) * decimal.Decimal(2) ** (e - 63)
            got, want = call(lib.exp2_neg, m, e), decimal.Decimal(2) ** (-t)
            assert abs(got / want - 1) <= 8 * decimal.Decimal(2) ** -63, (m, e)


def test_reciprocal(lib):
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        for m in significands(np.random.default_rng(1), 500):
            x = decimal.Decimal(m) * decimal.Decimal(2) ** (17 - 63)
            assert abs(call(lib.reciprocal, m, 17) * x - 1) <= 8 * decimal.Decimal(2) ** -63, m


def test_product(lib):
    rng = np.random.default_rng(2)
    a = np.ldexp(1 + rng.random(2000), rng.integers(-400, 400, 2000))
    b = np.ldexp(1 + rng.random(2000), rng.integers(-400, 400, 2000))
    got = np.array([lib.product(x, y) for x, y in zip(a, b)])
    assert np.all(np.abs(got - a * b) <= np.spacing(a * b))
