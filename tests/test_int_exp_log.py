"""im_exp and im_log (csrc/intf.cuh) on the CPU: g++ compiles the header behind
a small shim of the device types with the tables of csrc/int_tables.h, and the
results are compared with exp and ln in 50 decimal digits."""
import ctypes
import decimal
import shutil
import subprocess
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_1309_2710_gb300" / "csrc"

SHIM = r"""
#include <algorithm>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
static inline long long dbits(double v) { long long b; std::memcpy(&b, &v, 8); return b; }
static inline int __double2hiint(double v) { return (int)(dbits(v) >> 32); }
static inline int __double2loint(double v) { return (int)dbits(v); }
static inline double __longlong_as_double(long long b) { double v; std::memcpy(&v, &b, 8); return v; }
static inline unsigned __float_as_uint(float v) { unsigned b; std::memcpy(&b, &v, 4); return b; }
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
struct ulonglong2 { unsigned long long x, y; };
#include "int_tables.h"
#include "intf.cuh"
static uint64_t ex2[64], lnc[128];
extern "C" int f_exp(double a, unsigned long long* m, unsigned* e)
{
    if (!ex2[0]) kin::int_exp_log_tables(ex2, lnc);
    kin::im_u64 v;
    uint32_t w;
    const bool ok = kin::im_exp((const kin::im_u64*)ex2, a, v, w);
    *m = v;
    *e = w;
    return ok;
}
extern "C" double f_log(double T)
{
    if (!ex2[0]) kin::int_exp_log_tables(ex2, lnc);
    return kin::im_log((const ulonglong2*)lnc, T);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("explog")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "f.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", str(CSRC), "-o", so, str(d / "shim.cpp")],
                   check=True, capture_output=True)
    L = ctypes.CDLL(so)
    L.f_exp.argtypes = [ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p]
    L.f_log.argtypes = [ctypes.c_double]
    L.f_log.restype = ctypes.c_double
    return L


def test_exp(lib):
    decimal.getcontext().prec = 50
    D = decimal.Decimal
    rng = np.random.default_rng(2)
    ln2 = float(np.log(2.0))
    a = np.concatenate([rng.uniform(-80, 80, 2000), rng.uniform(-700, 700, 1000), rng.uniform(-1, 1, 500) * 1e-9,
                        np.arange(-640, 640) * ln2 / 64.0, [0.0, -0.0, 1e-300, 709.0, -708.0]])
    m, e = ctypes.c_ulonglong(), ctypes.c_uint()
    worst = 0.0
    for v in a:
        assert lib.f_exp(float(v), ctypes.byref(m), ctypes.byref(e))
        assert 2 ** 62 - 64 <= m.value < 2 ** 63
        ref = D(float(v)).exp()
        got = D(m.value) * D(2) ** (int(e.value) - 1085)
        worst = max(worst, float(abs(got / ref - 1)))
    # the argument's 52 fractional bits after log2(e): ln2 (2^-53 + |y| 2^-60)
    assert worst <= 0.6931472 * (2.0 ** -53 + 1024 * 2.0 ** -60) + 2.0 ** -58, worst * 2.0 ** 53


def test_exp_range(lib):
    m, e = ctypes.c_ulonglong(), ctypes.c_uint()
    for v in (710.0, 1100.0, 1e9, np.inf, np.nan):  # overflow, or not a number
        assert not lib.f_exp(v, ctypes.byref(m), ctypes.byref(e))
    for v in (-709.0, -1100.0, -1e300, -np.inf):    # below the normal range
        assert lib.f_exp(v, ctypes.byref(m), ctypes.byref(e)) and m.value == 0


def test_log(lib):
    decimal.getcontext().prec = 50
    D = decimal.Decimal
    rng = np.random.default_rng(3)
    T = np.concatenate([rng.uniform(200, 5000, 3000), np.exp(rng.uniform(0, np.log(65535.0), 1000)),
                        [1.0, 2.0, 1024.0, 298.15, 65535.9]])
    T = np.concatenate([T, 2.0 ** 10 * (1 + np.arange(64) / 64.0), np.nextafter(2.0 ** 10 * (1 + np.arange(64) / 64.0), 0)])
    for t in T:
        ref = D(float(t)).ln()
        got = lib.f_log(float(t))
        # half an ulp of the result, and 2^-57 of the fixed point
        assert abs(D(got) - ref) <= D(0.5 * np.spacing(got)) + D(2) ** -57, t
