// warp.cuh -- warp-per-cell RKC for large mechanisms (templates; instantiated
// in inst_warp_*.cu).
//
// With one lane per cell, every lane keeps its own concentrations, rates of
// progress and rate constants: ~(2 n_R + n_S) words per cell, which for
// hundreds of reactions spills out of L1/L2 and turns every f evaluation into
// a stream from HBM. Here a group of G lanes integrates one cell (a warp; in
// FP64 a quarter of a warp to four warps, cell_lanes in abi.cu):
//  * the lanes split the reactions (rates of progress, rounds of G) and
//    the species (state vectors in registers: species l + G r in slot r of
//    lane l);
//  * f in FP64 runs on the integer pipes (warp_int.cuh); in mixed precision
//    its concentrations and rates of progress live in
//    shared memory (n_S + n_R words per warp). A cell's rate constants, computed
//    once per call since T is fixed, live in the workspace cell-major and are
//    read coalesced (the working set of the resident cells stays in L2);
//  * reactions are visited in a fixed permutation (plain, then third-body,
//    then falloff) so that a round of 32 lanes mixes the dense efficiency dot
//    products with plain reactions at most once; the efficiency rows are
//    stored transposed ([species][row]) so that the lanes of a round read
//    consecutive words;
//  * all lanes follow the same cell, so the method's control flow is uniform
//    and is written as straight-line code; reductions (mixture sum, error
//    norms, spectral-radius bounds) are butterfly shuffles, which leave every
//    lane with the same bits.
// The method, its decisions and the statistics are those of the lane-per-cell
// kernel (Section 2.3 and the readings listed with it).
#pragma once
#include "int_tables.h"
#include "kernels.cuh"
#include "seg_tables.h"
#include "warp_int.cuh"

namespace kin {

template <typename R>
struct EllT;
template <>
struct EllT<double> {
    __device__ static const CsrW64* tab(const MechDev& M) { return M.ell64; }
};
template <>
struct EllT<float> {
    __device__ static const CsrW32* tab(const MechDev& M) { return M.ell32; }
};

// The third-body concentration of efficiency row `row`, [M] = sum_k eff_k C_k
// (Eq. (E:rxn-rate)), summed as two interleaved partial sums (even k, odd k).
// The rows are stored 16 bytes per species group, [k / V][row][k % V] with V =
// 4 (FP32) or 2 (FP64), so that a lane reads V efficiencies with one load and
// the warp's broadcast concentrations with another; lanes of a round take
// consecutive rows, so a warp's efficiency load is one contiguous span.
template <typename R>
__device__ __forceinline__ R eff_dot(const MechDev& M, int row, const R* C);

template <>
__device__ __forceinline__ float eff_dot<float>(const MechDev& M, int row, const float* C)
{
    const int nS = M.nS, nM = M.nM, n4 = nS >> 2;
    const float4* __restrict__ a = reinterpret_cast<const float4*>(M.effV32) + row;
    const float4* c = reinterpret_cast<const float4*>(C);
    float m0 = 0.0f, m1 = 0.0f;
#pragma unroll 4
    for (int k = 0; k < n4; ++k) {
        const float4 e = a[(int64_t)k * nM], x = c[k];
        m0 += e.x * x.x;
        m1 += e.y * x.y;
        m0 += e.z * x.z;
        m1 += e.w * x.w;
    }
    if (nS & 3) {
        const float4 e = a[(int64_t)n4 * nM];
        const int k = n4 << 2, t = nS & 3;
        m0 += e.x * C[k];
        if (t > 1) m1 += e.y * C[k + 1];
        if (t > 2) m0 += e.z * C[k + 2];
    }
    return m0 + m1;
}

template <>
__device__ __forceinline__ double eff_dot<double>(const MechDev& M, int row, const double* C)
{
    const int nS = M.nS, nM = M.nM, n2 = nS >> 1;
    const double2* __restrict__ a = reinterpret_cast<const double2*>(M.effV64) + row;
    const double2* c = reinterpret_cast<const double2*>(C);
    double m0 = 0.0, m1 = 0.0;
#pragma unroll 4
    for (int k = 0; k < n2; ++k) {
        const double2 e = a[(int64_t)k * nM], x = c[k];
        m0 += e.x * x.x;
        m1 += e.y * x.y;
    }
    if (nS & 1) m0 += a[(int64_t)n2 * nM].x * C[nS - 1];
    return m0 + m1;
}

// The FP64 f's tables for groups of G lanes.
template <int G>
__host__ __device__ __forceinline__ const IntDev& int_tab(const MechDev& M)
{
    return M.ig[G == 4 ? INT_G4 : G == 8 ? INT_G8 : G == 16 ? INT_G16 : G == 32 ? INT_G32 : G == 64 ? INT_G64 : INT_G128];
}

// Shared FP64 words of C [nS] and Omega [nR] in the energy and FP32 forms of
// f, padded to 4.
__host__ __device__ __forceinline__ int warp_smem_elems(const MechDev& M)
{
    return (M.nS + M.nR + 3) & ~3;
}

// Shared FP64 words of a group's f: the integer arrays of the FP64 f, or C and
// Omega (the mixed-precision path evaluates f in FP32 for its RK stages and in
// FP64 for its spectral-radius estimates, over the same words).
template <typename R, bool EN, int G>
__host__ __device__ __forceinline__ int warp_f_words(const MechDev& M)
{
    return sizeof(R) == 4 ? warp_smem_elems(M) : int_smem_words(M, int_tab<G>(M));
}

// The cell's rate constants in shared memory too: f reads every k_j once per
// evaluation, and staged behind C and Omega that read is a shared load instead
// of an L2 round trip on the f's critical path. Isothermal only (with the
// energy equation k follows T inside f), and only for small mechanisms, whose
// group words stay within WARP_K_SMEM_MAX_BYTES: shared memory comes out of
// the same on-chip array as L1, and for 53 species / 634 reactions the larger
// carve-out cost more in L1 misses (tables, spills) than the staged k saved
// (163 K vs 174 K cells/s on GB300), while 9 species / 38 reactions gained.
constexpr int WARP_K_SMEM_MAX_BYTES = 2048;

template <typename R, bool EN>
__host__ __device__ __forceinline__ int warp_k_words(const MechDev& M)
{
    if (EN) return 0;
    const int kw = ((M.nR + M.nFO) * (int)sizeof(R) + 7) / 8;
    return (warp_smem_elems(M) + kw) * 8 <= WARP_K_SMEM_MAX_BYTES ? kw : 0;
}

// Shared FP64 words per cell group: f's, the staged k (if any), the reductions'.
template <typename R, int NR, bool EN, int G>
__host__ __device__ __forceinline__ int warp_group_words(const MechDev& M)
{
    return (warp_f_words<R, EN, G>(M) + warp_k_words<R, EN>(M) + 2 * group_set_words<NR, G>() + 1) & ~1;
}

// f for the mixed-precision path's cell (Eqs. (E:mass), (E:spec-rate),
// (E:rxn-rate)) in arithmetic type R: FP32 for the RK stages, FP64 for the
// spectral-radius estimates. (The FP64 path's f is warp_feval_int. The mixed
// path keeps this one for both: its FP32 f turns any change of rounding in an
// estimate into differences of 3e-8 in the result.) Kc are the cell's rate constants (stored as KT) in
// reaction-permutation order followed by k0/kinf per falloff ordinal (written
// earlier in the same pre-pass kernel, so not read through the read-only
// cache); C and OM are the warp's shared arrays. Ctot and invCtot (the total
// concentration p / (R T) and its reciprocal) come in the arithmetic type, so
// that the FP32 evaluation's scalar work stays off the FP64 pipe: only the
// state's conversions in and the rates' conversions out are FP64 operations.
template <typename R, typename KT, int NR, int G = 32>
__device__ __forceinline__ void warp_feval(const MechDev& M, const KT* Kc, R* C, R* OM,
                                           R Ctot, R invCtot, const double (&x)[NR],
                                           double (&out)[NR], int lane, unsigned mask = 0xffffffffu)
{
    const int nS = M.nS, nR = M.nR, nM = M.nM;
    const R* __restrict__ invW = Tab<R>::invW(M);
    R s = R(0);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        if (i < nS) {
            const R m = (R)x[r] * invW[i];
            C[i] = m;
            s += m;
        }
    }
    s = group_sum<G>(s, mask);
    const R rho = Ctot * Tab<R>::inv(s);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        if (i < nS) C[i] = C[i] * rho;
    }
    __syncwarp(mask);
    // permutation order: plain reactions, then third-body (efficiency row
    // q - nP), then falloff (ordinal q - nF)
    const int nP = nR - nM, nF = nR - M.nFO;
    const uint32_t* __restrict__ rxw = M.rxw;
    // The evaluation waits on L1, L2 and shared-memory round trips (53 species
    // / 634 reactions, FP32: FP64 pipe 68 %, load/store 67 %, issue 57 %), so the
    // loads of four rounds of plain reactions are in flight together, and so
    // are four steps of the gathers below. GB300, 1,024 cells 10.7 -> 8.5 ms, 65,536
    // 235 -> 199 ms, the same bits.
    int q = lane;
#pragma unroll 1
    for (; q - lane + 4 * G <= nP; q += 4 * G) {
        uint32_t w[4];
        R v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            w[u] = rxw[q + u * G];
            v[u] = (R)Kc[q + u * G];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r0 = (int)(w[u] & 0xffffu) - 1, r1 = (int)(w[u] >> 16) - 1;
            const R a = C[max(r0, 0)], b = C[max(r1, 0)];
            v[u] *= r0 >= 0 ? a : R(1);
            v[u] *= r1 >= 0 ? b : R(1);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) OM[q + u * G] = v[u];
    }
#pragma unroll 1
    for (; q < nR; q += G) {
        const uint32_t w = rxw[q];
        R v = (R)Kc[q];
        const int r0 = (int)(w & 0xffffu) - 1, r1 = (int)(w >> 16) - 1;
        if (r0 >= 0) v *= C[r0];
        if (r1 >= 0) v *= C[r1];
        if (q >= nP) {
            const R Mc = eff_dot<R>(M, q - nP, C);
            if (q < nF) {
                v *= Mc;
            } else {
                const R Pr = (R)Kc[nR + (q - nF)] * Mc;
                v *= rdiv<R>(Pr, R(1) + Pr);
            }
        }
        OM[q] = v;
    }
    __syncwarp(mask);
    const R invrho = s * invCtot;
    if constexpr (G == 32 && sizeof(R) == 4) {
        if (M.seg_ent) {
            // omega over equal chunks of the nonzeros (seg_tables.h); the
            // partial sums land past Omega, in the FP32 half of the warp's
            // words that only the FP64 evaluations use. Four entries per load, the
            // next four on their way
            float* P = reinterpret_cast<float*>(OM) + nR;
            const uint4* __restrict__ ent = M.seg_ent + lane;
            int slot = M.seg_slot0[lane];
            float w = 0.0f;
            const int K4 = M.seg_K4;
            uint4 e4 = ent[0];
#pragma unroll 2
            for (int k = 0; k < K4; ++k) {
                const uint32_t e[4] = {e4.x, e4.y, e4.z, e4.w};
                e4 = ent[32 * min(k + 1, K4 - 1)];
                float o[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) o[u] = OM[e[u] & SEG_POS_MASK];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    w = fmaf(__uint_as_float(e[u] & SEG_NU_MASK), o[u], w);
                    if (e[u] & SEG_FLUSH) {
                        P[slot++] = w;
                        w = 0.0f;
                    }
                }
            }
            __syncwarp(mask);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int i = lane + 32 * r;
                double o = 0.0;
                if (i < nS) {
                    const int pt = M.seg_part[i];
                    if (pt >= 0) {
                        const float* pp = P + (pt >> 8);
                        float v = pp[0];
                        for (int c = 1; c < (pt & 0xff); ++c) v += pp[c];
                        o = (double)(v * (M.W32[i] * invrho));
                    }
                }
                out[r] = o;
            }
            __syncwarp(mask);  // C, OM and P are rewritten by the next evaluation
            return;
        }
    }
    // W_i omega_i over the species' row (W_i folded into its coefficients).
    // With 32 lanes per cell the row is read from the ELL copy, where the
    // lanes of a step read consecutive entries (one or two cache lines per
    // load instead of one line per lane); the entries and their order are
    // those of the species-major rows.
    const R* __restrict__ nuW = Tab<R>::nuW(M);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        double o = 0.0;
        if (i < nS) {
            R w0 = R(0), w1 = R(0);
            if constexpr (G == 32) {
                const int len = M.csr_ptr[i + 1] - M.csr_ptr[i];
                const auto* __restrict__ p = EllT<R>::tab(M) + M.ell_base[r] + lane;
                int k = 0;
                for (; k + 3 < len; k += 4) {
                    const auto a = p[32 * k], b = p[32 * (k + 1)], c = p[32 * (k + 2)], e = p[32 * (k + 3)];
                    const R oa = OM[a.pos], ob = OM[b.pos], oc = OM[c.pos], oe = OM[e.pos];
                    w0 += a.nuW * oa;
                    w1 += b.nuW * ob;
                    w0 += c.nuW * oc;
                    w1 += e.nuW * oe;
                }
                for (; k + 1 < len; k += 2) {
                    const auto a = p[32 * k], b = p[32 * (k + 1)];
                    w0 += a.nuW * OM[a.pos];
                    w1 += b.nuW * OM[b.pos];
                }
                if (k < len) {
                    const auto a = p[32 * k];
                    w0 += a.nuW * OM[a.pos];
                }
            } else {
                const int e1 = M.csr_ptr[i + 1];
                int e = M.csr_ptr[i];
                for (; e + 1 < e1; e += 2) {
                    w0 += nuW[e] * OM[M.csrp_rxn[e]];
                    w1 += nuW[e + 1] * OM[M.csrp_rxn[e + 1]];
                }
                if (e < e1) w0 += nuW[e] * OM[M.csrp_rxn[e]];
            }
            o = (double)((w0 + w1) * invrho);
        }
        out[r] = o;
    }
    __syncwarp(mask);  // C and OM are rewritten by the next evaluation
}

// f with the energy equation (Eqs. (E:mass), (E:energy)) for the warp's cell:
// state component nS is T (lane nS % 32, slot nS / 32). Each lane computes the
// rate constants of its reactions from T (they follow T at every
// evaluation); the enthalpy sum and the mixture heat capacity are FP64 warp
// sums, and dT/dt lands in T's slot.
template <typename R, int NR, int G = 32>
__device__ __forceinline__ void warp_feval_energy(const MechDev& M, double p, R* C, R* OM,
                                                  const double (&x)[NR], double (&out)[NR], int lane,
                                                  unsigned mask = 0xffffffffu)
{
    const int nS = M.nS, nR = M.nR, nM = M.nM;
    const double T = __shfl_sync(mask, reg_get(x, nS / G), nS % G, G);
    const double lnT = log(T), invT = ddiv(1.0, T);
    const double Ctot = p * 1e-6 * invT * (1.0 / R_GAS), invCtot = ddiv(1.0, Ctot);
    const R* __restrict__ invW = Tab<R>::invW(M);
    R s = R(0);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        if (i < nS) {
            const R m = (R)x[r] * invW[i];
            C[i] = m;
            s += m;
        }
    }
    s = group_sum<G>(s, mask);
    const R rho = (R)Ctot * Tab<R>::inv(s);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        if (i < nS) C[i] = C[i] * rho;
    }
    __syncwarp(mask);
    const int nP = nR - nM, nF = nR - M.nFO;
    const uint32_t* __restrict__ rxw = M.rxw;
    for (int q = lane; q < nR; q += G) {
        const uint32_t w = rxw[q];
        const int j = M.rxn_perm[q];
        const double a = M.lnA[j] + M.beta[j] * lnT - M.EaR[j] * invT;
        R v = Tab<R>::ex(a);
        const int r0 = (int)(w & 0xffffu) - 1, r1 = (int)(w >> 16) - 1;
        if (r0 >= 0) v *= C[r0];
        if (r1 >= 0) v *= C[r1];
        if (q >= nP) {
            const R Mc = eff_dot<R>(M, q - nP, C);
            if (q < nF) {
                v *= Mc;
            } else {
                const double a0 = M.lnA0[j] + M.beta0[j] * lnT - M.Ea0R[j] * invT;
                const R Pr = Tab<R>::ex(a0 - a) * Mc;
                v *= rdiv<R>(Pr, R(1) + Pr);
            }
        }
        OM[q] = v;
    }
    __syncwarp(mask);
    const R* __restrict__ nu = Tab<R>::nu(M);
    const double invrho = (double)s * invCtot, dT = T - T_REF;
    double hw = 0.0, cpm = 0.0;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        double o = 0.0;
        if (i < nS) {
            R w0 = R(0), w1 = R(0);
            const int e1 = M.csr_ptr[i + 1];
            int e = M.csr_ptr[i];
            for (; e + 1 < e1; e += 2) {
                w0 += nu[e] * OM[M.csrp_rxn[e]];
                w1 += nu[e + 1] * OM[M.csrp_rxn[e + 1]];
            }
            if (e < e1) w0 += nu[e] * OM[M.csrp_rxn[e]];
            const double om = (double)(w0 + w1);
            o = om * (M.W[i] * invrho);
            hw += (M.Hf[i] + M.cp[i] * dT) * om;
            cpm += x[r] * M.cpW[i];
        }
        out[r] = o;
    }
    hw = group_sum<G>(hw, mask);
    cpm = group_sum<G>(cpm, mask);
    const double dTdt = ddiv(-hw * invrho, cpm);
#pragma unroll
    for (int r = 0; r < NR; ++r)
        if (lane + G * r == nS) out[r] = dTdt;
    __syncwarp(mask);  // C and OM are rewritten by the next evaluation
}

template <typename R, int NR, bool EN, int G>
struct WarpRKC {
    const Launch& L;
    const MechDev& M;
    R* C;
    R* OM;
    double* C64;   // the same shared words as C and OM, for the FP64 evaluations
    double* OM64;
    R* Ks;         // the group's staged rate constants, or null
    const R* Kc;
    int lane, nV;  // nV: state length, nS + 1 with the energy equation
    Group<G> grp;
    unsigned mask; // the group's lanes in this warp
    int scale;     // of the integer FP64 f, kept from one evaluation of a cell to the next
    bool kfin;     // the cell's rate constants are finite
    double Ctot, invCtot, atol, rtol, p;
    R CtotR, invCtotR;   // the same in the rate type
    int nfe, nsig, nfs;  // f evaluations, sigma estimates, f evaluations inside them
    double y[NR], f0[NR], w1[NR], w2[NR], fx[NR], x[NR], ev[NR];  // (x: sigma() only)

    __device__ explicit WarpRKC(const Launch& l)
        : L(l), M(l.M), Kc(nullptr), lane(threadIdx.x & (G - 1)), nV(l.nV), grp(nullptr, group_set_words<NR, G>()), mask(group_mask<G>()), scale(0), kfin(true)
    {
        C64 = reinterpret_cast<double*>(kin_smem) + (size_t)(threadIdx.x / G) * warp_group_words<R, NR, EN, G>(M);
        grp.red = C64 + warp_f_words<R, EN, G>(M) + warp_k_words<R, EN>(M);
        OM64 = C64 + M.nS;
        C = reinterpret_cast<R*>(C64);
        OM = C + M.nS;
        Ks = warp_k_words<R, EN>(M) ? reinterpret_cast<R*>(C64 + warp_f_words<R, EN, G>(M)) : nullptr;
    }

    __device__ __forceinline__ bool valid(int r) const { return lane + G * r < nV; }

    __device__ __forceinline__ static unsigned long long bits(double v)
    {
        return (unsigned long long)__double_as_longlong(v);
    }
    // max(|a|, |b|) by the bits (a NaN wins): no comparison on the FP64 pipe
    __device__ __forceinline__ static double max_abs(double a, double b)
    {
        const unsigned long long m = 0x7fffffffffffffffull, u = bits(a) & m, v = bits(b) & m;
        return __longlong_as_double((long long)(u > v ? u : v));
    }
    // a * b + c and a * b of the state vectors. In the FP64 path the fused and
    // the separate operations are named, so that every group size rounds alike;
    // the mixed path leaves the choice to the compiler.
    __device__ __forceinline__ static double mul_add(double a, double b, double c)
    {
        if constexpr (sizeof(R) == 8) return fma(a, b, c);
        else return c + a * b;
    }
    __device__ __forceinline__ static double mul(double a, double b)
    {
        if constexpr (sizeof(R) == 8) return __dmul_rn(a, b);
        else return a * b;
    }

    __device__ __forceinline__ void f(const double (&in)[NR], double (&o)[NR])
    {
        if constexpr (sizeof(R) == 8) f64(in, o);
        else if constexpr (EN) warp_feval_energy<R, NR, G>(M, p, C, OM, in, o, lane, mask);
        else warp_feval<R, R, NR, G>(M, Kc, C, OM, CtotR, invCtotR, in, o, lane, mask);
        nfe++;
    }

    // f of the FP64 path (with the energy equation Ctot and invCtot hold p / R and
    // its reciprocal).
    __device__ __forceinline__ void f64(const double (&in)[NR], double (&o)[NR])
    {
        const IntDev& I = int_tab<G>(M);
        const IntSmem S(M, I, C64);
        if constexpr (EN) warp_feval_int_energy<NR, G>(M, I, S, Ctot, invCtot, scale, in, o, lane, grp);
        else
            warp_feval_int<NR, G, false>(M, I, S, RateSource{reinterpret_cast<const double*>(Kc), 0.0, 0.0}, kfin, Ctot,
                                         invCtot, scale, in, o, lane, grp);
    }

    // f in FP64 for the spectral-radius estimates (FP32 rounding noise in
    // f(y + v) - f(y) would swamp the difference; see SIG_SQRT_U).
    __device__ __forceinline__ void fs(const double (&in)[NR], double (&o)[NR])
    {
        if constexpr (sizeof(R) == 8) f64(in, o);
        else if constexpr (EN) warp_feval_energy<double, NR, G>(M, p, C64, OM64, in, o, lane, mask);
        else warp_feval<double, R, NR, G>(M, Kc, C64, OM64, Ctot, invCtot, in, o, lane, mask);
        nfe++;
        nfs++;
    }

    // Weighted RMS norm, Eq. (E:rmsE), of d with T_i = atol + rtol max(|a_i|, |b_i|).
    __device__ double rms(const double (&d)[NR], const double (&a)[NR], const double (&b)[NR])
    {
        double acc = 0.0;
        if constexpr (sizeof(R) == 8) {
            double q[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r)
                q[r] = valid(r) ? ddiv(d[r], fma(rtol, max_abs(a[r], b[r]), atol)) : 0.0;
            acc = grp.sum_sq(q);
        } else {
#pragma unroll
            for (int r = 0; r < NR; ++r)
                if (valid(r)) {
                    const double sc = atol + rtol * fmax(fabs(a[r]), fabs(b[r]));
                    const double q = ddiv(d[r], sc);
                    acc += q * q;
                }
            acc = group_sum<G>(acc, mask);
        }
        return dsqrt(ddiv(acc, (double)nV));
    }

    // FP64 f(y), the base of the spectral-radius differences: f0 in the FP64
    // path; in the mixed-precision path w2, which the estimate evaluates first.
    __device__ __forceinline__ double sig_base(int r) const
    {
        if constexpr (sizeof(R) == 4) return w2[r];
        else return f0[r];
    }

    // Start of the nonlinear power method, warm-started from ev: scales ev to
    // the difference length sqrt(u) |y| and returns that length.
    __device__ double power_setup()
    {
        double yn = 0.0, vn = 0.0;
        if constexpr (sizeof(R) == 8) {
            yn = grp.sum_sq(y);
            vn = grp.sum_sq(ev);
        } else {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                yn += y[r] * y[r];
                vn += ev[r] * ev[r];
            }
            yn = group_sum<G>(yn, mask);
            vn = group_sum<G>(vn, mask);
        }
        yn = dsqrt(yn);
        vn = dsqrt(vn);
        const double dyn = yn > 0.0 ? SIG_SQRT_U * yn : SIG_SQRT_U;
        if (!(vn > 0.0) || !isfinite(vn)) {
#pragma unroll
            for (int r = 0; r < NR; ++r) ev[r] = valid(r) ? 1.0 : 0.0;
            vn = dsqrt((double)nV);
        }
        const double sc0 = ddiv(dyn, vn);
#pragma unroll
        for (int r = 0; r < NR; ++r) ev[r] = mul(ev[r], sc0);
        return dyn;
    }

    // Spectral radius at y: the Gershgorin bound on the finite-difference
    // Jacobian (one column per evaluation) or the nonlinear power method
    // warm-started from ev (at most 20 products, stopping when two estimates
    // agree to 1 %; returns 1.2 times the last), Section 2.3. The mixed-
    // precision path first re-evaluates f(y) in FP64 into w2. `first` starts
    // the power method from f(y). Every FP64 evaluation of the estimate goes
    // through the one call of fs below, so the kernel holds one inlined copy
    // of the FP64 f.
    __device__ double sigma(bool first)
    {
        constexpr bool MIX = sizeof(R) == 4;
        const bool pw = L.sigma_method == KIN_SIGMA_POWER;
        double rs[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) rs[r] = 0.0;
        double dyn = 0.0, sig = 0.0, prev = 0.0, eps = 0.0;
        if constexpr (!MIX) {
            if (first)
#pragma unroll
                for (int r = 0; r < NR; ++r) ev[r] = f0[r];
            if (pw) dyn = power_setup();
        }
        for (int k = MIX ? -1 : 0;; ++k) {  // k = -1: the base f(y)
            if (k < 0) {
#pragma unroll
                for (int r = 0; r < NR; ++r) x[r] = y[r];
            } else if (pw) {
#pragma unroll
                for (int r = 0; r < NR; ++r) x[r] = y[r] + ev[r];
            } else {  // Gershgorin column k
                const int kr = k / G, kl = k % G;
                const double yk = grp.from(reg_get(y, kr), kl);
                eps = SIG_SQRT_U * fmax(fabs(yk), atol);
#pragma unroll
                for (int r = 0; r < NR; ++r) x[r] = (r == kr && lane == kl) ? yk + eps : y[r];
            }
            fs(x, fx);
            if (k < 0) {
#pragma unroll
                for (int r = 0; r < NR; ++r) w2[r] = fx[r];
                if (first)
#pragma unroll
                    for (int r = 0; r < NR; ++r) ev[r] = w2[r];
                if (pw) dyn = power_setup();
                continue;
            }
            if (pw) {
                double wn = 0.0;
                if constexpr (sizeof(R) == 8) {
#pragma unroll
                    for (int r = 0; r < NR; ++r) fx[r] = fx[r] - sig_base(r);
                    wn = grp.sum_sq(fx);
                } else {
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        fx[r] = fx[r] - sig_base(r);
                        wn += fx[r] * fx[r];
                    }
                    wn = group_sum<G>(wn, mask);
                }
                wn = dsqrt(wn);
                sig = ddiv(wn, dyn);
                if (!(wn > 0.0) || !isfinite(wn)) break;
                const double sc = ddiv(dyn, wn);
#pragma unroll
                for (int r = 0; r < NR; ++r) ev[r] = mul(fx[r], sc);
                if (k >= 1 && fabs(sig - prev) <= 0.01 * sig) break;
                prev = sig;
                if (k + 1 >= 20) break;
            } else {
                const double ie = rcp_newton(eps);
#pragma unroll
                for (int r = 0; r < NR; ++r)
                    if (valid(r)) rs[r] += fabs((fx[r] - sig_base(r)) * ie);
                if (k + 1 >= nV) {
                    double m = 0.0;
#pragma unroll
                    for (int r = 0; r < NR; ++r) m = fmax(m, rs[r]);
                    return grp.max(m);
                }
            }
        }
        return 1.2 * sig;
    }

    __device__ __forceinline__ const double* coef(int s, int j) const
    {
        return M.rkc + ((int64_t)s * RKC_TAB_S + j) * RKC_TAB_W;
    }

    // Stages of a step of hh at spectral radius sig (SMAX + 1: more than the
    // cap). The mixed-precision path takes the square root in FP32: s is an
    // integer, which the FP32 root changes only where 1 + sqrt(1 + 1.54 h sigma)
    // lies within FP32 rounding of an integer, and the FP64 root is a dozen
    // instructions on the FP64 pipe that all lanes repeat. The FP64 path takes
    // it in FP32 too unless that lands within 5e-4 of an integer (or above the
    // cap), where the FP64 root decides.
    __device__ __forceinline__ static int stages(double hh, double sig)
    {
        if constexpr (sizeof(R) == 4) {
            const double sr = (double)floorf(1.0f + sqrtf(1.0f + (float)(1.54 * hh * sig)));
            return sr < 2.0 ? 2 : sr > (double)SMAX ? SMAX + 1 : (int)sr;
        } else {
            const double v = fma(__dmul_rn(1.54, hh), sig, 1.0);
            const float u = 1.0f + sqrtf((float)v), k = floorf(u);
            if (u < SMAX + 0.5f && u - k >= 5e-4f && u - k <= 1.0f - 5e-4f) return max(2, (int)k);
            const double sr = floor(1.0 + dsqrt(v));
            return sr < 2.0 ? 2 : sr > (double)SMAX ? SMAX + 1 : (int)sr;
        }
    }

    // w_1 = y + mu~_1 h f_0 of a step of s stages; w_0 = y.
    __device__ __forceinline__ void first_stage(int s, double hh)
    {
        const double m1 = coef(s, 1)[2] * hh;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            w2[r] = y[r];
            w1[r] = mul_add(m1, f0[r], y[r]);
        }
    }

    // w_j from f(w_{j-1}) in fx (the three-term recursion).
    __device__ __forceinline__ void stage(int s, int j, double hh)
    {
        const double* c = coef(s, j);
        const double mu = c[0], nu = c[1], mt = c[2] * hh, gt = c[3] * hh, c0 = c[4];
        if (sizeof(R) == 8 && j == 2) {
            // w_0 = y, w_1 = y + m1 f_0: w_2 = y + (mu m1 + gamma~ h) f_0 + mu~ h f_1
            const double a = fma(mu, coef(s, 1)[2] * hh, gt);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                w2[r] = w1[r];
                w1[r] = fma(mt, fx[r], fma(a, f0[r], y[r]));
            }
            return;
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            double wn;
            if constexpr (sizeof(R) == 8)
                wn = fma(gt, f0[r], fma(mt, fx[r], fma(nu, w2[r], fma(mu, w1[r], __dmul_rn(c0, y[r])))));
            else
                wn = c0 * y[r] + mu * w1[r] + nu * w2[r] + mt * fx[r] + gt * f0[r];
            w2[r] = w1[r];
            w1[r] = wn;
        }
    }

    // Sum of the squared weighted error components of the step that ends in w1.
    __device__ __forceinline__ double error_sum(double hh)
    {
        double acc = 0.0;
        if constexpr (sizeof(R) == 8) {
            double q[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const double d = fma(0.8, y[r] - w1[r], __dmul_rn(0.4 * hh, f0[r] + fx[r]));
                const double sc = fma(rtol, max_abs(y[r], w1[r]), atol);
                q[r] = valid(r) ? __dmul_rn(d, rcp_newton(sc)) : 0.0;
            }
            acc = grp.sum_sq(q);
        } else {
#pragma unroll
            for (int r = 0; r < NR; ++r)
                if (valid(r)) {
                    const double d = 0.8 * (y[r] - w1[r]) + 0.4 * hh * (f0[r] + fx[r]);
                    const double sc = atol + rtol * fmax(fabs(y[r]), fabs(w1[r]));
                    const double q = d * rcp_newton(sc);
                    acc += q * q;
                }
            acc = group_sum<G>(acc, mask);
        }
        return acc;
    }

    // Integration state of a cell.
    struct Cell {
        double dt, sig, h;                  // flow step, spectral radius, next step size
        double t, hprev, cprev, hh;
        int attempts, since, nacc, nrej;
        int s, j;                           // stages of the step, stage whose f comes next (j > s: f(w_s))
        bool last, sigma_here, last_rej, have_prev;
        // a spectral-radius estimate in progress (groups of less than a warp)
        bool estimating, wait;
        int k;
        double dyn, prev, eps;

        __device__ void start(double dt_, double sig_, double h_)
        {
            dt = dt_;
            sig = sig_;
            h = h_;
            t = hprev = cprev = 0.0;
            attempts = since = nacc = nrej = 0;
            sigma_here = true;
            last_rej = have_prev = estimating = false;
        }
        __device__ bool stale() const { return since >= 25 || (last_rej && !sigma_here); }
    };

    // The next step's size and stages, and w_1.
    __device__ __forceinline__ void begin_step(Cell& U)
    {
        double hh = U.h;
        bool last = false;
        if (hh >= U.dt - U.t) {
            hh = U.dt - U.t;
            last = true;
        }
        int s = stages(hh, U.sig);
        if (s > SMAX) {
            s = SMAX;
            hh = ddiv((SMAX - 1.0) * (SMAX - 1.0) - 1.0, 1.54 * U.sig);
            last = false;
        }
        U.hh = hh;
        U.last = last;
        U.s = s;
        U.j = 2;
        first_stage(s, hh);
    }

    // Error test and step control after f(w_s). Returns a final status, or -1.
    __device__ __forceinline__ int end_step(Cell& U, double invN)
    {
        const double hh = U.hh;
        U.attempts++;
        // x = ||Delta||^2; z = x^(-1/6) = err^(-1/3) (see the lane kernel)
        // (one evaluation of the power serves both branches)
        const double xe = error_sum(hh) * invN;
        // (the mixed-precision path keeps the FP32 power, within 4 ulp: a
        // step-size factor, with the FP32 rates' precision)
        double z = 0.0;
        const bool pos = bits(xe) - 1ull < 0x7fefffffffffffffull;  // 0 < xe < inf (xe is not negative)
        if (pos) {
            if constexpr (sizeof(R) == 4)
                z = f32_normal(xe) ? (double)powf((float)xe, -1.0f / 6.0f) : dpow(xe, -1.0 / 6.0);
            else
                z = rpow6_newton(xe);
        }
        if (bits(xe) <= bits(1.0)) {
            U.nacc++;
            double fac, c3 = 0.0;
            if (xe == 0.0) {
                fac = 10.0;
            } else {
                const double z2 = z * z;
                c3 = xe * (z2 * z2 * z);
                if (U.have_prev && !U.last_rej && U.cprev > 0.0)
                    fac = 0.8 * hh * U.cprev * z2 * rcp_newton(U.hprev);
                else fac = 0.8 * z;
            }
            fac = fmin(10.0, fmax(0.1, fac));
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                y[r] = w1[r];
                f0[r] = fx[r];
            }
            if (U.last) return KIN_CELL_OK;
            U.t += hh;
            U.have_prev = true;
            U.hprev = hh;
            U.cprev = c3;
            U.last_rej = false;
            U.sigma_here = false;
            U.since++;
            U.h = fac * hh;
        } else {
            U.nrej++;
            double fac = pos ? 0.8 * z : 0.1;
            if (fac < 0.1) fac = 0.1;
            U.last_rej = true;
            U.h = fac * hh;
            if (U.h < 1e-20 * U.dt) return KIN_CELL_HMIN;
        }
        return -1;
    }

    // RKC integration of a started cell (y, f0 and ev from the pre-pass).
    // Returns the cell status.
    __device__ int run(Cell& U)
    {
        const double invN = ddiv(1.0, (double)nV);
        for (;;) {
            if (U.attempts >= L.max_steps) return KIN_CELL_MAXSTEPS;
            if (U.stale()) {
                U.sig = sigma(false);
                nsig++;
                U.since = 0;
                U.sigma_here = true;
                if (!isfinite(U.sig)) return KIN_CELL_NONFINITE;
            }
            begin_step(U);
            for (;; ++U.j) {
                f(w1, fx);  // f(w_{j-1}); after the last stage, f(w_s)
                if (U.j > U.s) break;
                stage(U.s, U.j, U.hh);
            }
            const int code = end_step(U, invN);
            if (code >= 0) return code;
        }
    }

    // ---- several cells per warp (FP64): one evaluation of f at a time ----
    // Each call of run's loop would let the warp's groups drift apart, and a
    // group in an estimate would keep the others waiting for its evaluations.
    // Here every pass of the kernel's loop evaluates f once for each group, at
    // the point its cell needs next (w1), and then does that cell's own
    // bookkeeping.

    // The point to evaluate in pass `pass`, once a step or an estimate has ended.
    // Steps start in even passes (nearly all have two evaluations), so that the
    // groups of a warp are in the same part of their steps and run its control
    // together. Returns a final status, or -1.
    __device__ __forceinline__ int next_point(Cell& U, unsigned pass)
    {
        if (U.attempts >= L.max_steps) return KIN_CELL_MAXSTEPS;
        U.wait = false;
        if (!U.stale()) {
            U.estimating = false;
            U.wait = pass & 1u;
            begin_step(U);
            return -1;
        }
        U.estimating = true;
        U.k = 0;
        U.prev = 0.0;
        if (L.sigma_method == KIN_SIGMA_POWER) U.dyn = power_setup();
#pragma unroll
        for (int r = 0; r < NR; ++r) w2[r] = 0.0;  // Gershgorin row sums
        sigma_point(U);
        return -1;
    }

    __device__ __forceinline__ void sigma_point(Cell& U)
    {
        if (L.sigma_method == KIN_SIGMA_POWER) {
#pragma unroll
            for (int r = 0; r < NR; ++r) w1[r] = y[r] + ev[r];
            return;
        }
        const int kr = U.k / G, kl = U.k % G;
        const double yk = grp.from(reg_get(y, kr), kl);
        U.eps = SIG_SQRT_U * fmax(fabs(yk), atol);
#pragma unroll
        for (int r = 0; r < NR; ++r) w1[r] = (r == kr && lane == kl) ? yk + U.eps : y[r];
    }

    // fx = f(w1) of an estimate; true when it has ended (U.sig).
    __device__ __forceinline__ bool sigma_post(Cell& U)
    {
        if (L.sigma_method == KIN_SIGMA_POWER) {
#pragma unroll
            for (int r = 0; r < NR; ++r) fx[r] = fx[r] - f0[r];
            const double wn = dsqrt(grp.sum_sq(fx)), sg = ddiv(wn, U.dyn);
            U.sig = 1.2 * sg;
            if (!(wn > 0.0) || !isfinite(wn)) return true;
            const double sc = ddiv(U.dyn, wn);
#pragma unroll
            for (int r = 0; r < NR; ++r) ev[r] = mul(fx[r], sc);
            if (U.k >= 1 && fabs(sg - U.prev) <= 0.01 * sg) return true;
            U.prev = sg;
            if (++U.k >= 20) return true;
        } else {
            const double ie = rcp_newton(U.eps);
#pragma unroll
            for (int r = 0; r < NR; ++r)
                if (valid(r)) w2[r] += fabs(__dmul_rn(fx[r] - f0[r], ie));
            if (++U.k >= nV) {
                double m = 0.0;
#pragma unroll
                for (int r = 0; r < NR; ++r) m = fmax(m, w2[r]);
                U.sig = grp.max(m);
                return true;
            }
        }
        sigma_point(U);
        return false;
    }

    // What follows f(w1) = fx. Returns a final status, or -1.
    __device__ __forceinline__ int advance(Cell& U, double invN, unsigned pass)
    {
        bool ended = false;
        if (U.estimating) {
            nfs++;
            ended = sigma_post(U);
            if (ended) {
                nsig++;
                U.since = 0;
                U.sigma_here = true;
                if (!isfinite(U.sig)) return KIN_CELL_NONFINITE;
            }
        } else if (U.j <= U.s) {
            stage(U.s, U.j, U.hh);
            U.j++;
        } else {
            const int code = end_step(U, invN);
            if (code >= 0) return code;
            ended = true;
        }
        return ended ? next_point(U, pass + 1) : -1;
    }
};

// Register budget at 256 threads per block. OCC 0: 128 registers (no spills
// for up to 4 vector slots; 16 resident warps per SM); OCC 1, for 2 or fewer
// slots: 48 registers (40 warps per SM, about the most that the shared words
// of a 53-species / 634-reaction cell leave room for; some values spill to
// local memory), or 80 (24 warps) with the energy equation, whose f holds
// more live values; 128 for 4 and 8 slots. The isothermal f evaluation of
// these mechanisms waits on L1 and shared-memory round trips, and more
// resident warps hide more of that latency: on 53 species / 634 reactions,
// mixed precision, 198 K cells/s at 32 warps per SM (64 registers), 217 K at
// 36 (56) and 237 K at 40 (48), against 178 K at 24 (80), before four rounds'
// loads were in flight together; with them 65,536 cells take 199 ms at 40
// warps and 202 ms at 16 (128), 1,024 cells 18.9 and 8.5. With the energy
// equation 74.1 K at 80 registers against 72.1 K at 64.
template <int NR, int OCC, bool EN>
struct WarpBounds {
    static constexpr int min_blocks = NR == 8 ? (OCC ? 2 : 1) : (OCC && NR <= 2 ? (EN ? 3 : 5) : 2);
};

// Pre-pass, one group of G lanes per cell (grid-stride over cells): the cell's rate
// constants (stored cell-major for the main kernel), f(y0), sigma and the
// initial step h1 (Section 2.3).
template <typename R, int NR, int OCC, bool EN, int G>
__global__ void __launch_bounds__(256, WarpBounds<NR, OCC, EN>::min_blocks) warp_init_kernel(const __grid_constant__ Launch L)
{
    WarpRKC<R, NR, EN, G> W(L);
    const MechDev& M = L.M;
    const int lane = W.lane, nK = M.nR + M.nFO, nS = M.nS, nV = L.nV;
    const int64_t ngroups = L.nslots / G;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G; g < L.total; g += ngroups) {
        const int ii = find_inst(L, g);
        const InstDev& I = L.inst[ii];
        const int64_t c = g - L.start[ii];
        const double T = I.T[c], p = I.p[c];
        W.Ctot = ddiv(p * 1e-6, EN && sizeof(R) == 8 ? R_GAS : R_GAS * T);
        W.invCtot = ddiv(1.0, W.Ctot);
        W.CtotR = (R)W.Ctot;
        W.invCtotR = (R)W.invCtot;
        W.atol = I.atol;
        W.rtol = I.rtol;
        W.p = p;
        W.nfe = 0;
        W.nfs = 0;
        if constexpr (!EN) {
            // rate constants (Eq. (E:rxn-const)) in permutation order; with the
            // energy equation they follow T and are formed inside f instead
            // (for the main kernel in the workspace, and for this kernel's own
            // evaluations in the staged copy when there is one)
            R* kc = reinterpret_cast<R*>(L.cell_k) + g * nK;
            R* ks = W.Ks ? W.Ks : kc;
            const double lnT = log(T), invT = ddiv(1.0, T);
            bool kfin = true;
            for (int q = lane; q < M.nR; q += G) {
                const int j = M.rxn_perm[q];
                const double a = M.lnA[j] + M.beta[j] * lnT - M.EaR[j] * invT;
                const R k = Tab<R>::ex(a);
                kc[q] = k;
                ks[q] = k;
                if (sizeof(R) == 8) kfin &= im_finite_k(k);
                const int fo = M.rxnp[q].fo;
                if (fo >= 0) {
                    const double a0 = M.lnA0[j] + M.beta0[j] * lnT - M.Ea0R[j] * invT;
                    const R k0 = Tab<R>::ex(a0 - a);
                    kc[M.nR + fo] = k0;
                    ks[M.nR + fo] = k0;
                    if (sizeof(R) == 8) kfin &= im_finite_k(k0);
                }
            }
            W.grp.sync();
            W.Kc = ks;
            if (sizeof(R) == 8) W.kfin = W.grp.all(kfin);
        }
        W.scale = EN ? -1 : 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int i = lane + G * r;
            W.y[r] = i < nS ? I.Y[(int64_t)i * I.ldY + c] : (i == nS && EN ? T : 0.0);
        }
        W.f(W.y, W.f0);
        bool fin = true;
#pragma unroll
        for (int r = 0; r < NR; ++r) fin &= isfinite(W.f0[r]);
        fin = W.grp.all(fin);
        uint8_t st = fin ? 0 : KIN_CELL_NONFINITE;
        double sig = 0.0, h = I.dt;
        if (fin) {
            sig = W.sigma(true);
            if (!isfinite(sig)) {
                st = KIN_CELL_NONFINITE;
            } else {
                double h0 = sig > 0.0 ? ddiv(1.0, sig) : I.dt;
                if (h0 > I.dt) h0 = I.dt;
#pragma unroll
                for (int r = 0; r < NR; ++r) W.x[r] = W.mul_add(h0, W.f0[r], W.y[r]);
                W.f(W.x, W.fx);
#pragma unroll
                for (int r = 0; r < NR; ++r) W.x[r] = h0 * (W.fx[r] - W.f0[r]);  // Delta_0
                const double e0 = W.rms(W.x, W.y, W.y);
                if (!isfinite(e0)) h = 0.1 * h0;
                else h = e0 > 0.0 ? ddiv(0.1 * h0, dsqrt(e0)) : I.dt;
                if (h > I.dt) h = I.dt;
                if (h < 1e-20 * I.dt) st = KIN_CELL_HMIN;
            }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (W.valid(r)) {
                L.cell_f0[g * nV + lane + G * r] = W.f0[r];
                if (L.cell_ev) L.cell_ev[g * nV + lane + G * r] = W.ev[r];
            }
        if (lane == 0) {
            L.cell_sig[g] = sig;
            L.cell_h[g] = h;
            L.cell_nfe[g] = W.nfe;
            L.cell_nfs[g] = W.nfs;
            L.cell_st[g] = st;
        }
    }
}

// Take cell g into W: its constants, state and pre-pass results. Returns the
// status that the pre-pass decided, or 0.
template <typename R, int NR, bool EN, int G>
__device__ __forceinline__ uint8_t warp_load_cell(WarpRKC<R, NR, EN, G>& W, const InstDev& I, int64_t g, int64_t c)
{
    const Launch& L = W.L;
    const MechDev& M = W.M;
    const int lane = W.lane, nK = M.nR + M.nFO, nS = M.nS, nV = L.nV;
    W.nfe = L.cell_nfe[g];
    W.nfs = L.cell_nfs[g];
    W.nsig = 1;
    const uint8_t pre = L.cell_st[g];
    if (pre != 0) return pre;  // Y stays as given
    const double T = I.T[c], p = I.p[c];
    W.Ctot = ddiv(p * 1e-6, EN && sizeof(R) == 8 ? R_GAS : R_GAS * T);
    W.invCtot = ddiv(1.0, W.Ctot);
    W.CtotR = (R)W.Ctot;
    W.invCtotR = (R)W.invCtot;
    W.atol = I.atol;
    W.rtol = I.rtol;
    W.p = p;
    W.scale = EN ? -1 : 0;
    if constexpr (EN) {
        W.Kc = nullptr;
    } else {
        const R* kg = reinterpret_cast<const R*>(L.cell_k) + g * nK;
        bool kfin = true;
        if (W.Ks || sizeof(R) == 8)
            for (int q = lane; q < nK; q += G) {
                const R k = kg[q];
                if (sizeof(R) == 8) kfin &= im_finite_k(k);
                if (W.Ks) W.Ks[q] = k;  // staged (the last f of the previous cell ended in a sync)
            }
        if (sizeof(R) == 8) W.kfin = W.grp.all(kfin);
        if (W.Ks) W.grp.sync();
        W.Kc = W.Ks ? W.Ks : kg;
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        const bool v = i < nV;
        W.y[r] = i < nS ? I.Y[(int64_t)i * I.ldY + c] : (v ? T : 0.0);
        W.f0[r] = v ? L.cell_f0[g * nV + i] : 0.0;
        W.ev[r] = (v && L.cell_ev) ? L.cell_ev[g * nV + i] : 0.0;
    }
    return 0;
}

// Cell c's result: its state unless the pre-pass decided its status, the
// status and the statistics.
template <typename R, int NR, bool EN, int G>
__device__ __forceinline__ void warp_store_cell(const WarpRKC<R, NR, EN, G>& W, const InstDev& I, int64_t c, bool state,
                                                int code, int nacc, int nrej)
{
    const int lane = W.lane, nS = W.M.nS;
    if (state) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int i = lane + G * r;
            if (i < nS) I.Y[(int64_t)i * I.ldY + c] = W.y[r];
            else if (i == nS && EN) I.T[c] = W.y[r];
        }
    }
    if (lane == 0) {
        if (I.status) I.status[c] = (uint8_t)code;
        if (I.stats) {
            int32_t* st = I.stats + KIN_NSTATS * c;
            st[0] = W.nfe;
            st[1] = nacc;
            st[2] = nrej;
            st[3] = W.nsig;
            st[4] = W.nfs;
        }
    }
}

// Persistent main kernel: each group takes cells from the queue in the
// longest-first order and integrates them one after another.
template <typename R, int NR, int OCC, bool EN, int G>
__global__ void __launch_bounds__(256, WarpBounds<NR, OCC, EN>::min_blocks) warp_integrate_kernel(const __grid_constant__ Launch L)
{
    using Warp = WarpRKC<R, NR, EN, G>;
    Warp W(L);
    typename Warp::Cell U;
    if constexpr (G >= 32) {
        for (;;) {
            unsigned long long q = 0;
            if (W.lane == 0) q = atomicAdd(L.queue, 1ull);
            q = W.grp.from(q, 0);
            if (q >= (unsigned long long)L.total) return;
            const int64_t g = L.order[q];
            const int ii = find_inst(L, g);
            const InstDev& I = L.inst[ii];
            const int64_t c = g - L.start[ii];
            int code = warp_load_cell(W, I, g, c);
            const bool pre = code != 0;  // decided by the pre-pass
            U.nacc = U.nrej = 0;
            if (!pre) {
                U.start(I.dt, L.cell_sig[g], L.cell_h[g]);
                code = W.run(U);
            }
            warp_store_cell(W, I, c, !pre, code, U.nacc, U.nrej);
        }
    } else {
        // the warp's groups together: one evaluation of f per pass (a group
        // without a cell waits)
        const double invN = ddiv(1.0, (double)W.nV);
        bool have = false, more = true;
        int ii = 0;
        int64_t c = 0;
        for (unsigned pass = 0;; ++pass) {
            while (!have && more) {
                unsigned long long q = 0;
                if (W.lane == 0) q = atomicAdd(L.queue, 1ull);
                q = W.grp.from(q, 0);
                more = q < (unsigned long long)L.total;
                if (!more) break;
                const int64_t g = L.order[q];
                ii = find_inst(L, g);
                c = g - L.start[ii];
                int code = warp_load_cell(W, L.inst[ii], g, c);
                const bool pre = code != 0;
                U.start(L.inst[ii].dt, L.cell_sig[g], L.cell_h[g]);
                if (!pre) code = W.next_point(U, pass);
                have = !pre && code < 0;
                if (!have) warp_store_cell(W, L.inst[ii], c, !pre, code, 0, 0);
            }
            if (__all_sync(0xffffffffu, !have)) return;
            const bool go = have && !U.wait;
            U.wait = false;
            if (go) W.f(W.w1, W.fx);
            __syncwarp();
            if (go) {
                const int code = W.advance(U, invN, pass);
                if (code >= 0) {
                    warp_store_cell(W, L.inst[ii], c, true, code, U.nacc, U.nrej);
                    have = false;
                }
            }
        }
    }
}

// ---------------------------------------------------- RKCK, warp per cell --
// Cash-Karp 5(4) with the step rule of Section 2.2 (Table 1, Eq. (E:hnew)),
// one group of G lanes per cell (G = 32, a warp; or G = 16, two cells per
// warp, for states of at most 16 components, where a whole warp would leave
// most of its FP64 lanes idle), in one persistent kernel: RKCK needs no
// spectral radius or initial-step estimate, so there is no pre-pass and no
// cost ordering. A group takes the next cell, forms its rate constants
// (cell-major in the workspace, unless they follow T with the energy
// equation) and integrates it with straight-line control flow; the decisions
// are those of the lane-per-cell kernel. Every collective of a group names
// only the group's lanes.
template <typename R, int NR, bool EN, int G>
struct WarpRKCK {
    const Launch& L;
    const MechDev& M;
    R* C;
    R* OM;
    R* Ks;  // the group's staged rate constants, or null
    const R* Kc;
    double* base;   // the group's shared words
    int lane, nV;
    Group<G> grp;
    unsigned mask;  // the group's lanes
    int scale;      // of the integer FP64 f, kept from one evaluation of a cell to the next
    bool kfin;      // the cell's rate constants are finite
    double Ctot, invCtot, atol, rtol, p;
    R CtotR, invCtotR;  // the same in the rate type
    int nfe;
    double y[NR], x[NR], kx[NR], k[6][NR];

    __device__ explicit WarpRKCK(const Launch& l)
        : L(l), M(l.M), Kc(nullptr), lane(threadIdx.x & (G - 1)), nV(l.nV),
          grp(nullptr, group_set_words<NR, G>()), mask(group_mask<G>()), scale(0), kfin(true)
    {
        base = reinterpret_cast<double*>(kin_smem) + (size_t)(threadIdx.x / G) * warp_group_words<R, NR, EN, G>(M);
        C = reinterpret_cast<R*>(base);
        OM = C + M.nS;
        Ks = warp_k_words<R, EN>(M) ? reinterpret_cast<R*>(base + warp_f_words<R, EN, G>(M)) : nullptr;
    }

    __device__ __forceinline__ bool valid(int r) const { return lane + G * r < nV; }

    __device__ __forceinline__ void f(const double (&in)[NR], double (&o)[NR])
    {
        if constexpr (sizeof(R) == 4) {
            if constexpr (EN) warp_feval_energy<R, NR, G>(M, p, C, OM, in, o, lane, mask);
            else warp_feval<R, R, NR, G>(M, Kc, C, OM, CtotR, invCtotR, in, o, lane, mask);
        } else {
            const IntDev& I = int_tab<G>(M);
            const IntSmem S(M, I, base);
            if constexpr (EN) warp_feval_int_energy<NR, G>(M, I, S, Ctot, invCtot, scale, in, o, lane, grp);
            else
                warp_feval_int<NR, G, false>(M, I, S, RateSource{reinterpret_cast<const double*>(Kc), 0.0, 0.0}, kfin,
                                             Ctot, invCtot, scale, in, o, lane, grp);
        }
        nfe++;
    }

    // Integration state of a cell.
    struct Cell {
        double dt, t, h, hh;
        int attempts, nacc, nrej;
        bool last, due;  // the flow step's last step; f(y) comes next

        __device__ void start(double dt_)
        {
            dt = h = dt_;  // first trial step: the whole flow step
            t = 0.0;
            attempts = nacc = nrej = 0;
            due = true;
        }
    };

    __device__ __forceinline__ bool finite(const double (&v)[NR]) const
    {
        bool fin = true;
#pragma unroll
        for (int r = 0; r < NR; ++r) fin &= isfinite(v[r]);
        return __all_sync(mask, fin);
    }

    // The next step's size.
    __device__ __forceinline__ void begin_step(Cell& U)
    {
        U.hh = U.h;
        U.last = false;
        if (U.hh >= U.dt - U.t) {
            U.hh = U.dt - U.t;
            U.last = true;
        }
    }

    // Stage point y + hh sum_l b_{st,l} k_l in x (stage indices are resolved
    // with unrolled selects, so k stays in registers).
    __device__ __forceinline__ void stage_point(int st, double hh)
    {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            double acc = 0.0;
#pragma unroll
            for (int l = 0; l < 5; ++l)
                if (l < st) acc += CK_B[st][l] * k[l][r];
            x[r] = y[r] + hh * acc;
        }
    }

    // Error test and step control after the six evaluations. Returns a final
    // status, or -1.
    __device__ __forceinline__ int end_step(Cell& U)
    {
        const double hh = U.hh;
        double errmax = 0.0;
        bool blown = false;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            double s5 = 0.0, e = 0.0;
#pragma unroll
            for (int l = 0; l < 6; ++l) {
                s5 += CK_C[l] * k[l][r];
                e += CK_E[l] * k[l][r];
            }
            x[r] = y[r] + hh * s5;
            if (valid(r)) {
                const double tol = rtol * (fabs(y[r]) + fabs(hh * k[0][r])) + atol;
                const double q = fabs(hh * e) * rcp_newton(tol);
                blown |= isnan(q);
                if (q > errmax) errmax = q;
            }
        }
        // group maximum; a NaN component makes the estimate non-finite
        errmax = group_max<G>(errmax, mask);
        if (__any_sync(mask, blown)) errmax = __longlong_as_double(0x7ff8000000000000ll);
        U.attempts++;
        if (errmax <= 1.0) {
            U.nacc++;
#pragma unroll
            for (int r = 0; r < NR; ++r) y[r] = x[r];
            if (U.last) return KIN_CELL_OK;
            U.t += hh;
            const double hn = errmax == 0.0 ? 5.0 * hh : 0.9 * hh * rpow5_newton(errmax);
            U.h = fmin(hn, 5.0 * hh);
            U.due = true;
        } else {
            U.nrej++;
            const double hn = isfinite(errmax) ? 0.9 * hh * rpow4_newton(errmax) : 0.1 * hh;
            U.h = fmax(hn, 0.1 * hh);
            if (U.h < 1e-20 * U.dt) return KIN_CELL_HMIN;
        }
        return -1;
    }
};

// Take cell g into W: its constants and state.
template <typename R, int NR, bool EN, int G>
__device__ __forceinline__ void warp_rkck_load(WarpRKCK<R, NR, EN, G>& W, const InstDev& I, int64_t g, int64_t c)
{
    const Launch& L = W.L;
    const MechDev& M = W.M;
    const int lane = W.lane, nK = M.nR + M.nFO, nS = M.nS;
    const double T = I.T[c], p = I.p[c];
    W.Ctot = ddiv(p * 1e-6, EN && sizeof(R) == 8 ? R_GAS : R_GAS * T);
    W.invCtot = ddiv(1.0, W.Ctot);
    W.CtotR = (R)W.Ctot;
    W.invCtotR = (R)W.invCtot;
    W.atol = I.atol;
    W.rtol = I.rtol;
    W.p = p;
    W.nfe = 0;
    if constexpr (!EN) {
        // formed straight into the staged copy when there is one (the
        // previous cell's last f ended in a sync of the group)
        R* kc = W.Ks ? W.Ks : reinterpret_cast<R*>(L.cell_k) + g * nK;
        const double lnT = log(T), invT = ddiv(1.0, T);
        bool kfin = true;
        for (int qq = lane; qq < M.nR; qq += G) {
            const int j = M.rxn_perm[qq];
            const double a = M.lnA[j] + M.beta[j] * lnT - M.EaR[j] * invT;
            const R k = Tab<R>::ex(a);
            kc[qq] = k;
            if (sizeof(R) == 8) kfin &= im_finite_k(k);
            const int fo = M.rxnp[qq].fo;
            if (fo >= 0) {
                const double a0 = M.lnA0[j] + M.beta0[j] * lnT - M.Ea0R[j] * invT;
                const R k0 = Tab<R>::ex(a0 - a);
                kc[M.nR + fo] = k0;
                if (sizeof(R) == 8) kfin &= im_finite_k(k0);
            }
        }
        __syncwarp(W.mask);
        W.Kc = kc;
        if (sizeof(R) == 8) W.kfin = __all_sync(W.mask, kfin);
    }
    W.scale = EN ? -1 : 0;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        W.y[r] = i < nS ? I.Y[(int64_t)i * I.ldY + c] : (i == nS && EN ? T : 0.0);
    }
}

// The cell's result: its state unless f(y) at the start was not finite, the
// status and the statistics.
template <typename R, int NR, bool EN, int G>
__device__ __forceinline__ void warp_rkck_store(const WarpRKCK<R, NR, EN, G>& W, const InstDev& I, int64_t c, bool state,
                                                int code, int nacc, int nrej)
{
    const int lane = W.lane, nS = W.M.nS;
    if (state) {
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int i = lane + G * r;
            if (i < nS) I.Y[(int64_t)i * I.ldY + c] = W.y[r];
            else if (i == nS && EN) I.T[c] = W.y[r];
        }
    }
    if (lane == 0) {
        if (I.status) I.status[c] = (uint8_t)code;
        if (I.stats) {
            int32_t* st = I.stats + KIN_NSTATS * c;
            st[0] = W.nfe;
            st[1] = nacc;
            st[2] = nrej;
            st[3] = 0;
            st[4] = 0;
        }
    }
}

// Two half-warp groups stay together step by step and evaluation by evaluation
// (a group that has no evaluation due, or no cell, waits): where they only met by
// the compiler's choice, one build ran the 16-species kernel at a third of its
// speed.
template <typename R, int NR, bool EN, int G>
__global__ void __launch_bounds__(256, NR == 8 ? 1 : 2) warp_rkck_kernel(const __grid_constant__ Launch L)
{
    using Warp = WarpRKCK<R, NR, EN, G>;
    Warp W(L);
    typename Warp::Cell U;
    bool have = false, more = true;
    int ii = 0;
    int64_t c = 0;
    for (;;) {
        if (!have && more) {
            unsigned long long q = 0;
            if (W.lane == 0) q = atomicAdd(L.queue, 1ull);
            q = __shfl_sync(W.mask, q, 0, G);
            more = q < (unsigned long long)L.total;
            if (more) {
                ii = find_inst(L, (int64_t)q);
                c = (int64_t)q - L.start[ii];
                warp_rkck_load(W, L.inst[ii], (int64_t)q, c);
                U.start(L.inst[ii].dt);
                have = true;
            }
        }
        if (__all_sync(0xffffffffu, !have)) return;
        if (have && U.due) {
            W.f(W.y, W.k[0]);
            U.due = false;
            if (!W.finite(W.k[0])) {
                warp_rkck_store(W, L.inst[ii], c, U.nacc > 0, KIN_CELL_NONFINITE, U.nacc, U.nrej);
                have = false;
            } else if (U.attempts >= L.max_steps) {
                warp_rkck_store(W, L.inst[ii], c, true, KIN_CELL_MAXSTEPS, U.nacc, U.nrej);
                have = false;
            }
        }
        __syncwarp();
        if (have) W.begin_step(U);
        for (int st = 1; st < 6; ++st) {
            if (have) {
                W.stage_point(st, U.hh);
                W.f(W.x, W.kx);
#pragma unroll
                for (int l = 1; l < 6; ++l)
                    if (l == st)
#pragma unroll
                        for (int r = 0; r < NR; ++r) W.k[l][r] = W.kx[r];
            }
            __syncwarp();
        }
        if (have) {
            int code = W.end_step(U);
            if (code < 0 && !U.due && U.attempts >= L.max_steps) code = KIN_CELL_MAXSTEPS;
            if (code >= 0) {
                warp_rkck_store(W, L.inst[ii], c, true, code, U.nacc, U.nrej);
                have = false;
            }
        }
    }
}

template <typename R, int NR, bool EN, int G>
inline size_t group_smem_bytes(const MechDev& M, int threads)
{
    return (size_t)warp_group_words<R, NR, EN, G>(M) * (threads / G) * 8;
}

template <typename R, int NR, bool EN, int G>
inline cudaError_t warp_rkck_launch_nr(Launch& L, int blocks, int threads, cudaStream_t st)
{
    const size_t sm = group_smem_bytes<R, NR, EN, G>(L.M, threads);
    cudaError_t e = cudaFuncSetAttribute(warp_rkck_kernel<R, NR, EN, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    warp_rkck_kernel<R, NR, EN, G><<<blocks, threads, sm, st>>>(L);
    return cudaGetLastError();
}

template <typename R, int NR, bool EN, int G>
inline cudaError_t warp_rkck_occ_nr(const MechDev& M, int threads, int* bps)
{
    const size_t sm = group_smem_bytes<R, NR, EN, G>(M, threads);
    cudaError_t e = cudaFuncSetAttribute(warp_rkck_kernel<R, NR, EN, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, warp_rkck_kernel<R, NR, EN, G>, threads, sm);
}

template <typename R, int NR, int OCC, bool EN, int G>
inline cudaError_t warp_launch_nr(Launch& L, int blocks, int threads, cudaStream_t st)
{
    const size_t sm = group_smem_bytes<R, NR, EN, G>(L.M, threads);
    cudaError_t e = cudaFuncSetAttribute(warp_init_kernel<R, NR, OCC, EN, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(warp_integrate_kernel<R, NR, OCC, EN, G>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    warp_init_kernel<R, NR, OCC, EN, G><<<blocks, threads, sm, st>>>(L);
    e = launch_sort(L, st);
    if (e != cudaSuccess) return e;
    warp_integrate_kernel<R, NR, OCC, EN, G><<<blocks, threads, sm, st>>>(L);
    return cudaGetLastError();
}

template <typename R, int NR, int OCC, bool EN, int G>
inline cudaError_t warp_occ_nr(const MechDev& M, int precision, int threads, int* bps)
{
    const size_t sm = group_smem_bytes<R, NR, EN, G>(M, threads);
    cudaError_t e = cudaFuncSetAttribute(warp_integrate_kernel<R, NR, OCC, EN, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, warp_integrate_kernel<R, NR, OCC, EN, G>,
                                                         threads, sm);
}

// Register-vector width of a state of n components on groups of G lanes
// (component l + G r, r < NR).
__host__ __device__ inline int warp_nr(int n, int G)
{
    const int r = (n + G - 1) / G;
    return r <= 2 ? r : r <= 4 ? 4 : 8;
}

// The instantiation for groups of `lanes` lanes: FN<NR, G>.
#define KIN_WARP_DISPATCH(FN, n, lanes)                                     \
    if constexpr (sizeof(R) == 8) {                                         \
        if constexpr (OCC == 0) {                                           \
            if (lanes == 8) return FN(2, 8);                                \
        }                                                                   \
        if (lanes == 16) return FN(1, 16);                                  \
        if constexpr (OCC == 0) {                                           \
            if (lanes == 64) return FN(1, 64);                              \
            if (lanes == 128) return warp_nr(n, 128) == 1 ? FN(1, 128) : FN(2, 128); \
        }                                                                   \
    }                                                                       \
    switch (warp_nr(n, 32)) {                                               \
    case 1: return FN(1, 32);                                               \
    case 2: return FN(2, 32);                                               \
    case 4: return FN(4, 32);                                               \
    default: return FN(8, 32);                                              \
    }

template <typename R, int OCC, bool EN>
inline cudaError_t warp_launch(Launch& L, int blocks, int threads, cudaStream_t st)
{
#define KIN_FN(NR, G) warp_launch_nr<R, NR, OCC, EN, G>(L, blocks, threads, st)
    KIN_WARP_DISPATCH(KIN_FN, L.nV, L.lanes)
#undef KIN_FN
}

template <typename R, int OCC, bool EN>
inline cudaError_t warp_occ(const MechDev& M, int nV, int lanes, int precision, int threads, int* bps)
{
#define KIN_FN(NR, G) warp_occ_nr<R, NR, OCC, EN, G>(M, precision, threads, bps)
    KIN_WARP_DISPATCH(KIN_FN, nV, lanes)
#undef KIN_FN
}

template <typename R, bool EN>
inline cudaError_t warp_rkck_launch(Launch& L, int blocks, int threads, cudaStream_t st)
{
    if (L.lanes == 16) return warp_rkck_launch_nr<R, 1, EN, 16>(L, blocks, threads, st);
    switch (warp_nr(L.nV, 32)) {
    case 1: return warp_rkck_launch_nr<R, 1, EN, 32>(L, blocks, threads, st);
    case 2: return warp_rkck_launch_nr<R, 2, EN, 32>(L, blocks, threads, st);
    case 4: return warp_rkck_launch_nr<R, 4, EN, 32>(L, blocks, threads, st);
    default: return warp_rkck_launch_nr<R, 8, EN, 32>(L, blocks, threads, st);
    }
}

template <typename R, bool EN>
inline cudaError_t warp_rkck_occ(const MechDev& M, int nV, int lanes, int precision, int threads, int* bps)
{
    (void)precision;
    if (lanes == 16) return warp_rkck_occ_nr<R, 1, EN, 16>(M, threads, bps);
    switch (warp_nr(nV, 32)) {
    case 1: return warp_rkck_occ_nr<R, 1, EN, 32>(M, threads, bps);
    case 2: return warp_rkck_occ_nr<R, 2, EN, 32>(M, threads, bps);
    case 4: return warp_rkck_occ_nr<R, 4, EN, 32>(M, threads, bps);
    default: return warp_rkck_occ_nr<R, 8, EN, 32>(M, threads, bps);
    }
}

}  // namespace kin
