"""The records of the lane layout's integer f (build_lane_int of
csrc/int_tables.h), built on the CPU and read back: every reaction with a net
effect once, third bodies and falloffs first, with its reactants, net
coefficients, power of rho and rate-constant index, and every place in range."""
import ctypes
import shutil
import subprocess
from pathlib import Path

import numpy as np
import pytest

from paper_1309_2710_gb300 import synth

HEADER = Path(__file__).resolve().parents[1] / "paper_1309_2710_gb300" / "csrc" / "int_tables.h"

SHIM = r"""
#include "int_tables.h"
#include <cstring>
extern "C" int lane_int(int nS, int nR, const int* reac, const int* prod, const signed char* type, const double* eff,
                        int* tb, unsigned* rx, int* e, int* ex)
{
    kin::LaneInt t = kin::build_lane_int(nS, nR, reac, prod, type, eff);
    *tb = t.tb;
    std::memcpy(rx, t.rx.data(), 4 * t.rx.size());
    std::memcpy(e, t.eff.data(), 4 * t.eff.size());
    std::memcpy(ex, t.effx.data(), 4 * t.effx.size());
    return t.rx.size() == 4 * (size_t)(t.n + 1) && t.effx.size() == (size_t)t.tb ? t.n : -1;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("lane_int")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "lane_int.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", str(HEADER.parent), "-o", so,
                    str(d / "shim.cpp")], check=True, capture_output=True)
    return ctypes.CDLL(so)


def mechanism(name):
    if name in synth.WORKLOADS:
        m = synth.workload_mechanism(name)
        return m.n_species, m.reac, m.prod, m.rtype, m.eff
    rng = np.random.default_rng(5)  # random, with empty slots, repeated and cancelling species
    nS, nR = (32, 90) if name == "random" else (2, 0)
    r = rng.integers(-1, nS, (nR, 2))
    p = np.where(rng.uniform(size=(nR, 2)) < 0.3, r, rng.integers(-1, nS, (nR, 2)))
    r[::7, 1], p[::5, 1] = r[::7, 0], p[::5, 0]
    t = rng.choice([0, 0, 1, 2], nR)
    return nS, r, p, t, rng.uniform(0.5, 3.0, (int((t > 0).sum()), nS))


@pytest.mark.parametrize("name", ["h2_9sp_rkck", "h2co_13sp_rkc", "random", "none"])
def test_records(lib, name):
    nS, reac, prod, typ, eff = mechanism(name)
    nR = len(reac)
    reac, prod = np.ascontiguousarray(reac, np.int32), np.ascontiguousarray(prod, np.int32)
    typ, eff = np.ascontiguousarray(typ, np.int8), np.ascontiguousarray(eff, np.float64)
    rows = len(eff)
    rx, e, ex = np.zeros((nR + 1, 4), np.uint32), np.zeros((rows + 1, nS, 2), np.int32), np.zeros(rows + 1, np.int32)
    tb = np.zeros(1, np.int32)
    q = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    n = lib.lane_int(nS, nR, q(reac), q(prod), q(typ), q(eff), q(tb), q(rx), q(e), q(ex))
    nu = np.zeros((nR, nS), int)
    for j in range(nR):
        for k in reac[j]:
            nu[j, k] -= k >= 0
        for k in prod[j]:
            nu[j, k] += k >= 0
    live = [j for j in range(nR) if nu[j].any()]
    assert n == len(live) and sorted(int(j) for j in rx[:n, 2]) == live
    assert tb[0] == sum(typ[j] != 0 for j in live) and (rx[n] == rx[n - 1]).all()
    row = np.cumsum(typ != 0) - 1
    for r in range(n):
        x, y, j, fo = (int(v) for v in rx[r])
        assert (typ[j] != 0) == (r < tb[0]) and bool(y >> 23 & 1) == (typ[j] == 2)
        if typ[j] == 2:
            assert fo == (typ[:j] == 2).sum()
        assert sorted((x & 255, x >> 8 & 255)) == sorted(nS if k < 0 else int(k) for k in reac[j])
        got = np.zeros(nS + 1, int)
        for place, sign, two in ((x >> 16 & 255, 1, 16), (x >> 24, 1, 17), (y & 255, -1, 18), (y >> 8 & 255, -1, 19)):
            assert place <= nS
            got[place] += sign * (1 + (y >> two & 1))
        assert (got[:nS] == nu[j]).all()
        assert (y >> 20 & 7) == (reac[j] >= 0).sum() + (typ[j] == 1)   # power of rho, less two, plus two
        if r < tb[0]:
            back = e[r, :, 0].astype(np.float64) * 2.0 ** 25 + e[r, :, 1]
            assert np.allclose(back * 2.0 ** (float(ex[r]) - 54), eff[row[j]], rtol=2.0 ** -50, atol=0)
