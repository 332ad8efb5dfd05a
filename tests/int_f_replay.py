"""The integer FP64 f of the warp layout (csrc/warp_int.cuh, as a group of eight
lanes) and of the lane layout (csrc/lane_int.cuh, as a block of one lane) on the
CPU: g++ compiles the headers behind stand-ins for the CUDA types, the warp
collectives (the lanes are threads that meet at barriers) and the few helpers
of csrc/kernels.cuh that they use. Also the
same rates in extended precision, with each species' sum of |terms|."""
import ctypes
import shutil
import subprocess
from pathlib import Path

import numpy as np

ROOT = Path(__file__).resolve().parents[1]
CSRC = ROOT / "paper_1309_2710_gb300" / "csrc"

CUDA = r"""
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <thread>
#include <pthread.h>
#define __CUDACC_RTC__
#define __device__
#define __host__
#define __noinline__
#define __forceinline__ inline
#define __restrict__
using std::max;
using std::min;
using std::isfinite;
static inline long long dbits(double v) { long long b; std::memcpy(&b, &v, 8); return b; }
static inline int __double2hiint(double v) { return (int)(dbits(v) >> 32); }
static inline int __double2loint(double v) { return (int)dbits(v); }
static inline double __longlong_as_double(long long b) { double v; std::memcpy(&v, &b, 8); return v; }
static inline long long __double_as_longlong(double v) { return dbits(v); }
static inline unsigned __float_as_uint(float v) { unsigned b; std::memcpy(&b, &v, 4); return b; }
static inline float __uint_as_float(unsigned b) { float v; std::memcpy(&v, &b, 4); return v; }
static inline int __ffs(unsigned v) { return __builtin_ffs((int)v); }
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double int_inv(double a) { return 1.0 / a; }
struct ulonglong2 { unsigned long long x, y; };
struct int2 { int x, y; };
struct int4 { int x, y, z, w; };
struct uint4 { unsigned x, y, z, w; };
struct double2 { double x, y; };
static inline ulonglong2 make_ulonglong2(unsigned long long x, unsigned long long y) { return {x, y}; }
static inline int2 make_int2(int x, int y) { return {x, y}; }
struct Dim { unsigned x; };
static thread_local Dim threadIdx = {0};
static Dim blockDim = {1};
constexpr int LANES = 8;
static pthread_barrier_t meeting;
static long long word[LANES];
static inline void __syncwarp(unsigned) { pthread_barrier_wait(&meeting); }
template <typename T, typename F> static inline T collect(T v, F f)
{
    std::memcpy(&word[threadIdx.x], &v, sizeof(T));
    __syncwarp(0);
    const T r = f([](int k) { T t; std::memcpy(&t, &word[k], sizeof(T)); return t; });
    __syncwarp(0);
    return r;
}
static inline int __reduce_max_sync(unsigned, int v)
{
    return collect(v, [](auto at) { int m = at(0); for (int k = 1; k < LANES; ++k) m = std::max(m, at(k)); return m; });
}
static inline bool __any_sync(unsigned m, bool v) { return __reduce_max_sync(m, v) != 0; }
static inline bool __all_sync(unsigned m, bool v) { return !__any_sync(m, !v); }
template <typename T> static inline T __shfl_sync(unsigned, T v, int k, int) { return collect(v, [=](auto at) { return at(k); }); }
template <typename T> static inline T __shfl_xor_sync(unsigned, T v, int o)
{
    const int l = threadIdx.x;
    return collect(v, [=](auto at) { return at(l ^ o); });
}
alignas(16) static double kin_smem[1 << 16];
static int general = 0;  // evaluations that took plain FP64
"""

KERNELS = r"""
#pragma once
#include "kin_dev.cuh"
namespace kin {
inline double ddiv(double a, double b) { return a / b; }
inline double quot(double a, double b) { return a / b; }
template <typename R> struct Tab;
template <> struct Tab<double> { static double inv(double a) { return int_inv(a); } };
template <typename T> struct Lane { T* p; int32_t s; T& operator[](int i) const { return p[(int64_t)i * s]; } };
template <typename F> struct IntegerF { static constexpr bool value = false; };
template <typename R, typename KT>
void feval(const MechDev&, double, double, Lane<KT>, Lane<KT>, Lane<R>, Lane<R>, Lane<double>, Lane<double>) { ++general; }
}
"""

SHIM = r"""
#include <vector>
#include "cuda_stubs.h"
#include "int_tables.h"
#include "warp_int.cuh"
#include "lane_int.cuh"
using namespace kin;
struct Mech {
    MechDev M{};
    IntDev I{};
    IntGather g;
    LaneInt li;
    std::vector<double> W, invW, arr, arr0, effV64, nu, nuq;
    std::vector<uint32_t> rxw, scl;
    std::vector<int> perm, ptr, pos, posq;
    std::vector<int32_t> effI, effX, imWe, liE;
    std::vector<uint64_t> imW, ex2, lnc;
};
TABLES
extern "C" void* mech_new(int nS, int nR, const double* W, const double* lnA, const double* beta, const double* EaR,
                          const double* lnA0, const double* beta0, const double* EaR0, const int* reac, const int* prod,
                          const signed char* type, const double* eff)
{
    Mech* m = new Mech();
    std::vector<int> row(nR, -1), pos(nR);
    int nM = 0, nFO = 0;
    for (int j = 0; j < nR; ++j) if (type[j]) row[j] = nM++;
    for (int t = 0; t < 3; ++t)
        for (int j = 0; j < nR; ++j) if (type[j] == t) m->perm.push_back(j), nFO += t == 2;
    m->W.assign(W, W + nS);
    m->arr.resize(3 * nR + 1);
    m->arr0.resize(3 * nFO + 1);
    m->rxw.resize(nR + 1);
    m->effV64.assign((size_t)(nS + 1) / 2 * nM * 2 + 2, 0.0);
    for (int q = 0; q < nR; ++q) {
        const int j = m->perm[q];
        pos[j] = q;
        m->rxw[q] = (uint32_t)(reac[2 * j] + 1) | (uint32_t)(reac[2 * j + 1] + 1) << 16;
        m->arr[q] = lnA[j]; m->arr[nR + q] = beta[j]; m->arr[2 * nR + q] = EaR[j];
        if (type[j] == 2) {
            const int fo = q - (nR - nFO);
            m->arr0[fo] = lnA0[j]; m->arr0[nFO + fo] = beta0[j]; m->arr0[2 * nFO + fo] = EaR0[j];
        }
        for (int k = 0; type[j] && k < nS; ++k)
            m->effV64[((size_t)(k / 2) * nM + q - (nR - nM)) * 2 + k % 2] = eff[(size_t)row[j] * nS + k];
    }
    m->ptr.push_back(0);
    for (int i = 0; i < nS; ++i) {
        for (int j = 0; j < nR; ++j) {
            int c = 0;
            for (int k = 0; k < 2; ++k) c += (prod[2 * j + k] == i) - (reac[2 * j + k] == i);
            if (c) m->pos.push_back(pos[j]), m->nu.push_back(c);
        }
        m->ptr.push_back((int)m->pos.size());
        m->invW.push_back(1.0 / W[i]);
    }
    for (int i = 0; i < nS; ++i) {
        std::vector<std::pair<int, double>> row;
        for (int k = m->ptr[i]; k < m->ptr[i + 1]; ++k) row.push_back({m->pos[k], m->nu[k]});
        std::sort(row.begin(), row.end());
        for (auto& e : row) m->posq.push_back(e.first << 3 | ((int)e.second + 4)), m->nuq.push_back(e.second);
    }
    m->posq.push_back(0);
    m->M.csrq = m->posq.data();
    m->M.csrq_nu = m->nuq.data();
    const int chunk = std::max(32, std::min((nR + 31) / 32 * 32, 256));
    m->g = build_int_gather(nS, nR, m->ptr.data(), m->pos.data(), m->nu.data(), chunk, LANES);
    m->I = IntDev{m->g.nchunk, chunk, m->g.nslots, m->g.step0.data(), m->g.ent.data(), m->g.slot0.data(), m->g.part.data()};
    m->imW.resize(2 * nS);
    m->imWe.resize(2 * nS);
    for (int i = 0; i < nS; ++i) {
        m->imW[2 * i] = int_split(1.0L / W[i], &m->imWe[2 * i]);
        m->imW[2 * i + 1] = int_split(W[i], &m->imWe[2 * i + 1]);
        if (m->ptr[i + 1] == m->ptr[i]) m->imW[2 * i + 1] = 0;
    }
    m->ex2.resize(64);
    m->lnc.resize(128);
    int_exp_log_tables(m->ex2.data(), m->lnc.data());
    m->effI.assign((size_t)(nS + 1) / 2 * nM * 4 + 4, 0);
    m->effX.assign(nM + 1, 0);
    m->li = build_lane_int(nS, nR, reac, prod, (const int8_t*)type, eff);
    MechDev& M = m->M;
    M.nS = nS; M.nR = nR; M.nM = nM; M.nFO = nFO;
    for (int j = 0; j < nR; ++j) if ((reac[2 * j] >= 0) + (reac[2 * j + 1] >= 0) + (type[j] == 1) < 2) M.imLow = 1;
    tables(*m, eff, row.data(), reac, type);
    M.W = m->W.data(); M.invW = m->invW.data();
    M.csr_ptr = m->ptr.data(); M.csrp_rxn = m->pos.data(); M.csr_nu = m->nu.data();
    M.rxw = m->rxw.data(); M.arr = m->arr.data(); M.arr0 = m->arr0.data(); M.effV64 = m->effV64.data();
    M.effI = (const int4*)m->effI.data(); M.effX = m->effX.data();
    M.ex2 = (const unsigned long long*)m->ex2.data(); M.lnc = (const ulonglong2*)m->lnc.data();
    M.imW = (const ulonglong2*)m->imW.data(); M.imWe = (const int2*)m->imWe.data();
    M.li_n = m->li.n; M.li_tb = m->li.tb; M.li_rx = (const uint4*)m->li.rx.data();
    M.li_eff = (const int2*)m->liE.data(); M.li_effx = (const int32_t*)m->li.effx.data();
    return m;
}
template <int NR>
static void warp_nr(Mech* m, double T, double p, const double* Y, double* out, int* scale)
{
    const MechDev& M = m->M;
    const IntSmem S(M, m->I, kin_smem);
    std::vector<std::thread> lanes;
    pthread_barrier_init(&meeting, nullptr, LANES);
    const int scale0 = *scale;
    for (int l = 0; l < LANES; ++l)
        lanes.emplace_back([&, l] {
            threadIdx.x = l;
            Group<LANES> grp(nullptr, 0);
            double x[NR], o[NR];
            for (int r = 0; r < NR; ++r) x[r] = l + LANES * r < M.nS ? Y[l + LANES * r] : 0.0;
            const double pR = p * (1e-6 / R_GAS), invT = 1.0 / T;
            int s = scale0;
            warp_feval_int<NR, LANES, true>(M, m->I, S, rates_at(M, T, invT), true, pR * invT, T / pR, s, x, o, l, grp);
            for (int r = 0; r < NR; ++r)
                if (l + LANES * r < M.nS) out[l + LANES * r] = o[r];
            if (l == 0) *scale = s;
        });
    for (auto& t : lanes) t.join();
    pthread_barrier_destroy(&meeting);
}
extern "C" void f_warp(Mech* m, double T, double p, const double* Y, double* out, int* scale)
{
    if (m->M.nS <= 16) warp_nr<2>(m, T, p, Y, out, scale);
    else if (m->M.nS <= 64) warp_nr<8>(m, T, p, Y, out, scale);
    else warp_nr<32>(m, T, p, Y, out, scale);
}
// K: [nR] rate constants, KR: [nFO] k0 / kinf, both in reaction order
extern "C" int f_lane(Mech* m, double Ctot, double* K, double* KR, double* Y, double* out, int* scale)
{
    Lane<double> k{K, 1}, kr{KR, 1}, x{Y, 1}, o{out, 1};
    general = 0;
    if (*scale == -2) *scale = IntF::scale0(m->M, k, kr);
    IntF::eval<double, double>(m->M, Ctot, 1.0 / Ctot, k, kr, Lane<double>{nullptr, 1}, Lane<double>{nullptr, 1}, x, o, *scale);
    return general;
}
"""

# The tables of abi.cu beside those that the headers build.
TABLES = r"""
static void tables(Mech& m, const double* eff, const int* row, const int* reac, const signed char* type)
{
    const int nS = m.M.nS, nR = m.M.nR, nM = m.M.nM;
    for (int r = 0; r < nM; ++r) {
        std::vector<int32_t> hi(nS), lo(nS);
        const double* e = eff + (size_t)row[m.perm[nR - nM + r]] * nS;
        m.effX[r] = int_efficiencies(nS, e, hi.data(), lo.data());
        int_eff_limbs(nS, e, m.effX[r], 1, hi.data(), lo.data());
        for (int k = 0; k < nS; ++k) {
            m.effI[((size_t)(k / 2) * nM + r) * 4 + 2 * (k % 2)] = hi[k];
            m.effI[((size_t)(k / 2) * nM + r) * 4 + 2 * (k % 2) + 1] = lo[k];
        }
    }
    m.liE = m.li.eff;
    for (int r = 0; r < m.li.tb; ++r)
        int_eff_limbs(nS, eff + (size_t)m.li.row[r] * nS, m.li.effx[r], 2, &m.liE[2 * r * nS], &m.liE[2 * r * nS + 1]);
    m.scl.resize(4 * nR + 4);
    for (int q = 0; q < nR; ++q) {
        const int j = m.perm[q];
        int_scale_table(m.arr[q], m.arr[nR + q], m.arr[2 * nR + q], reac + 2 * j, type[j],
                        q >= nR - nM ? m.effX[q - (nR - nM)] : 0, &m.scl[4 * q]);
    }
    m.M.scl = (const uint4*)m.scl.data();
    int_word_bits(nS, m.ptr.data(), m.nu.data(), &m.M.imUp, &m.M.imShort);
}
"""


def build(tmp):
    """The library, from copies of the headers in tmp (None without g++)."""
    if shutil.which("g++") is None:
        return None
    d = Path(tmp) / "a" / "csrc"
    d.mkdir(parents=True)
    (Path(tmp) / "include").mkdir()
    shutil.copy(ROOT / "include" / "kin.h", Path(tmp) / "include")
    for f in ("intf.cuh", "warp_int.cuh", "lane_int.cuh", "int_tables.h", "kin_dev.cuh"):
        shutil.copy(CSRC / f, d)
    (d / "cuda_stubs.h").write_text(CUDA)
    (d / "kernels.cuh").write_text(KERNELS)
    (d / "shim.cpp").write_text(SHIM.replace("TABLES", TABLES))
    so = str(d / "f.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-pthread", "-o", so, str(d / "shim.cpp")],
                   check=True, capture_output=True)
    L = ctypes.CDLL(so)
    L.mech_new.restype = ctypes.c_void_p
    return L


class Mech:
    """A mechanism (the attributes of synth.Mechanism) in the library L (None:
    its reference only)."""

    def __init__(self, L, m):
        from paper_1309_2710_gb300 import synth
        self.L, self.m = L, m
        c = lambda a, t=np.float64: np.ascontiguousarray(np.zeros(0) if a is None else a, t)
        n0 = np.zeros(m.n_reactions)
        self.a = [c(m.W), c(m.lnA), c(m.beta), c(m.Ea) / synth.R_GAS, c(n0 if m.lnA0 is None else m.lnA0),
                  c(n0 if m.beta0 is None else m.beta0), c(n0 if m.Ea0 is None else m.Ea0) / synth.R_GAS,
                  c(m.reac, np.int32), c(m.prod, np.int32), c(m.rtype, np.int8), c(m.eff)]
        q = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        self.h = L and ctypes.c_void_p(L.mech_new(m.n_species, m.n_reactions, *map(q, self.a)))
        self.type = self.a[9]
        self.nu = np.zeros((m.n_species, m.n_reactions), np.longdouble)
        for j in range(m.n_reactions):
            for k in range(2):
                if m.prod[j, k] >= 0:
                    self.nu[m.prod[j, k], j] += 1
                if m.reac[j, k] >= 0:
                    self.nu[m.reac[j, k], j] -= 1
        self.eff = self.a[10].reshape(int((self.type > 0).sum()), m.n_species)

    def warp(self, T, p, Y, scale):
        """dY/dt of one cell and the scale that it leaves."""
        Y, out, s = np.ascontiguousarray(Y), np.zeros(self.m.n_species), ctypes.c_int(scale)
        self.L.f_warp(self.h, ctypes.c_double(T), ctypes.c_double(p), Y.ctypes.data_as(ctypes.c_void_p),
                      out.ctypes.data_as(ctypes.c_void_p), ctypes.byref(s))
        return out, s.value

    def constants(self, T, t=np.float64):
        """k and k0 / kinf in reaction order."""
        a = [x.astype(t) for x in self.a[1:7]]
        T = t(T)
        e, e0 = a[0] + a[1] * np.log(T) - a[2] / T, a[3] + a[4] * np.log(T) - a[5] / T
        fo = self.type == 2
        return np.exp(e), np.exp(e0[fo] - e[fo])

    def lane(self, T, p, Y, scale=-2):
        """(dY/dt, whether f took the plain FP64 code instead) of one cell."""
        from paper_1309_2710_gb300 import synth
        K, KR = self.constants(T)
        KR = np.append(KR, 1.0)
        Y, out, s = np.ascontiguousarray(Y), np.zeros(self.m.n_species), ctypes.c_int(scale)
        q = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        n = self.L.f_lane(self.h, ctypes.c_double(p * 1e-6 / (synth.R_GAS * T)), q(K), q(KR), q(Y), q(out), ctypes.byref(s))
        return out, n

    def reference(self, T, p, Y, t=np.longdouble, k=None):
        """dY/dt and sum_j |nu_ij Omega_j| W_i / rho of one cell in type t."""
        from paper_1309_2710_gb300 import synth
        m = self.m
        Y, W = Y.astype(t), self.a[0].astype(t)
        k, k0 = self.constants(T, t) if k is None else (a.astype(t) for a in k)
        rho = t(p) * t(1e-6) / (t(synth.R_GAS) * t(T) * (Y / W).sum())
        C = np.append(rho * Y / W, t(1.0))
        q = k * C[self.a[7][:, 0]] * C[self.a[7][:, 1]]
        if len(self.eff):
            M = (self.eff.astype(t) * C[:-1]).sum(1)
            non = np.flatnonzero(self.type)
            fo = self.type[non] == 2
            q[non[~fo]] *= M[~fo]
            pr = k0 * M[fo]
            q[non[fo]] *= pr / (1 + pr)
        out, mag = (self.nu.astype(t) * q).sum(1), np.abs(self.nu.astype(t) * q).sum(1)
        return out * W / rho, mag * W / abs(rho)
