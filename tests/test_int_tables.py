"""The tables of the warp layout's integer FP64 f (csrc/int_tables.h), built
on the CPU: g++ compiles the header behind a small C shim, and the tests replay
the gather and the third-body sums in Python integers from the tables alone.
This checks the index logic (every nonzero visited as often as its coefficient
says, every place and slot in range) before a GPU runs the tables."""
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
extern "C" int gather(int nS, int nR, const int* ptr, const int* pos, const double* nu, int chunk, int G,
                      int* dims, int* step0, unsigned* ent, int* slot0, int* part)
{
    kin::IntGather t = kin::build_int_gather(nS, nR, ptr, pos, nu, chunk, G);
    dims[0] = t.nchunk; dims[1] = t.nslots;
    std::memcpy(step0, t.step0.data(), 4 * t.step0.size());
    std::memcpy(ent, t.ent.data(), 4 * t.ent.size());
    std::memcpy(slot0, t.slot0.data(), 4 * t.slot0.size());
    std::memcpy(part, t.part.data(), 4 * t.part.size());
    return (int)t.ent.size();
}
extern "C" int effs(int nS, const double* e, int* hi, int* lo) { return kin::int_efficiencies(nS, e, hi, lo); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("int")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "int.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", str(HEADER.parent), "-o", so,
                    str(d / "shim.cpp")], check=True, capture_output=True)
    return ctypes.CDLL(so)


def rows(reac, prod, nS, seed):
    """Species-major rows of net coefficients over permuted reaction positions."""
    nR = len(reac)
    nu = np.zeros((nR, nS), int)
    for j in range(nR):
        for k in reac[j]:
            if k >= 0:
                nu[j, k] -= 1
        for k in prod[j]:
            if k >= 0:
                nu[j, k] += 1
    nu = nu[np.random.default_rng(seed).permutation(nR)]
    ptr, pos, val = [0], [], []
    for i in range(nS):
        at = np.flatnonzero(nu[:, i])
        pos += list(at)
        val += list(nu[at, i])
        ptr.append(len(pos))
    return np.array(ptr, np.int32), np.array(pos, np.int32), np.array(val, np.float64), nu


def mechanism(name):
    if name in synth.WORKLOADS:
        m = synth.workload_mechanism(name)
        return m.reac, m.prod, m.n_species
    if name == "one":          # a single reaction, coefficients of 2, a species that never changes
        return np.array([[0, 0]]), np.array([[1, 1]]), 3
    if name == "none":
        return np.zeros((0, 2), int), np.zeros((0, 2), int), 2
    if name == "hub":          # one species in every reaction: its row spans every lane
        n = 300
        return np.array([[0, 1 + j % 5] for j in range(n)]), np.array([[6 + j % 2, -1] for j in range(n)]), 8
    rng = np.random.default_rng(7)  # random, with empty slots and cancelling reactions
    r = rng.integers(-1, 17, (97, 2))
    p = np.where(rng.uniform(size=(97, 2)) < 0.2, r, rng.integers(-1, 17, (97, 2)))
    return r, p, 17


@pytest.mark.parametrize("G", [8, 16, 32, 128])
@pytest.mark.parametrize("chunk", [32, 128, 256])
@pytest.mark.parametrize("name", ["h2_9sp_rkck", "h2co_13sp_rkc", "ch4_53sp_rkc_mixed", "one", "none", "hub",
                                  "random"])
def test_gather_replay(lib, name, chunk, G):
    reac, prod, nS = mechanism(name)
    ptr, pos, val, nu = rows(reac, prod, nS, 3)
    nR = len(reac)
    cap = 2 * len(pos) + 2 * G * (nR // chunk + 1) + G
    nch = (nR + chunk - 1) // chunk
    dims, step0, ent = np.zeros(2, np.int32), np.zeros(nch + 1, np.int32), np.zeros(cap, np.uint32)
    slot0, part = np.zeros(nch * G + 1, np.int32), np.zeros(nch * nS + 1, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    n = lib.gather(nS, nR, p(ptr), p(pos), p(val), chunk, G, p(dims), p(step0), p(ent), p(slot0), p(part))
    assert dims[0] == nch and n == step0[nch] * G and n <= cap and dims[1] <= 2 * nS + G
    om = [int(v) for v in np.random.default_rng(1).integers(-2 ** 60, 2 ** 60, nR)]
    out = [0] * nS
    for c in range(nch):
        words = om[c * chunk:(c + 1) * chunk] + [0] * (chunk + 1)
        words[chunk] = 0
        P = {}
        for lane in range(G):
            w, slot = 0, int(slot0[c * G + lane])
            for k in range(step0[c], step0[c + 1]):
                e = int(ent[k * G + lane])
                at = e & 0xffff
                assert at == chunk or (at < chunk and c * chunk + at < nR)
                w += words[at]
                if e & 0x10000:
                    assert slot not in P and slot < dims[1]
                    P[slot] = w
                    w, slot = 0, slot + 1
            assert w == 0
        used = 0
        for i in range(nS):
            q = int(part[c * nS + i])
            for k in range(((q >> 8) & 0xff) + (q & 0xff)):
                out[i] += P[(q >> 16) + k] * (1 if k < (q >> 8) & 0xff else -1)
                used += 1
        assert used == len(P)
    assert out == [sum(int(v) * o for v, o in zip(nu[:, i], om)) for i in range(nS)]


@pytest.mark.parametrize("eff", [[1.0] * 4, [0.5, 3.0, 2.999999, 0.75], [0.0, 15.4, 1e-3, 0.0, 6.0], [0.0, 0.0],
                                 [-1.5, 2.0, 1e-30], list(np.linspace(0.5, 3, 200))])
def test_efficiencies(lib, eff):
    e = np.array(eff, np.float64)
    hi, lo = np.zeros(len(e), np.int32), np.zeros(len(e), np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    x = lib.effs(len(e), p(e), p(hi), p(lo))
    assert (np.abs(hi.astype(np.int64)) <= 2 ** 30).all() and (lo >= 0).all() and (lo < 2 ** 25).all()
    back = (hi.astype(object) * 2 ** 25 + lo.astype(object))
    top = np.abs(e).max()
    for b, v in zip(back, e):
        # within half a unit, 2^-54 (2^-53 above 128 species) of the row's largest
        assert abs(b - v * 2.0 ** (54 - x)) <= 0.5
    assert len(e) * 2 ** 55 * (2.0 ** (x - 54) * (np.abs(hi).max() + 1.0) * 2 ** 25 / top if top else 0) <= 2 ** 64
