// lane_int.cuh -- the lane layout's isothermal FP64 f on the integer pipes
// (intf.cuh has the arithmetic), driven by the mechanism's tables.
//
// Each lane keeps its cell's c_k / rho as mantissas and exponents and its
// species' 128-bit sums of rates in shared memory ([element][lane], so a
// warp's words are one contiguous span). One loop over the reactions, the same
// for every lane, forms a rate of progress in registers and adds it to its two
// products' sums and subtracts it from its two reactants'. Third-body factors
// come first, while the sums' words hold the fractions they are made of.
//
// Bound by the latency of a lane's serial chain (shared and L2 loads) at the 16
// warps per SM that its registers and shared words leave: 17 K instructions of a
// full warp per evaluation at 0.44 per cycle and scheduler. The plain FP64 code
// that it replaces kept the FP64 pipe 85 % busy, 64 cycles per instruction.
// GB300, 13 species / 54 reactions RKC: 262,144 cells 122 -> 100 ms (97 without the
// test of the sums' length and the wider limbs), 131,072 64.3 -> 50; 9 / 38 RKCK,
// 60,000 cells 4.7 -> 3.2. Loops over the state's
// vectors unrolled (104 ms) or their loads batched (102 to 139, spills) are
// slower, tables in constant memory no faster (96).
#pragma once
#include "intf.cuh"
#include "kernels.cuh"

namespace kin {

// A reaction of the loop (16 bytes): x = reactants a | b << 8 | products p0 <<
// 16 | p1 << 24; y = consumed species n0 | n1 << 8 | coefficient-of-2 flags <<
// 16 (p0, p1, n0, n1) | (power of rho + 2) << 20 | falloff << 23; z = rate
// constant; w = falloff ordinal. Reactants: nS is an empty slot (a
// concentration of 1). p and n: net coefficients, nS for none.
constexpr uint32_t LI_P0X2 = 1u << 16, LI_P1X2 = 1u << 17, LI_N0X2 = 1u << 18, LI_N1X2 = 1u << 19;
constexpr uint32_t LI_X2 = 15u << 16, LI_FALLOFF = 1u << 23;

// f in plain FP64 for states outside the integer forms' range.
static __device__ __noinline__ void lane_int_general(const MechDev& M, double Ctot, double invCtot, Lane<double> K,
                                                     Lane<double> KR, Lane<double> C, Lane<double> OM, Lane<double> x,
                                                     Lane<double> out)
{
    feval<double, double>(M, Ctot, invCtot, K, KR, C, OM, x, out);
}

// The lane's words in shared memory ([element][lane]): sums, mantissas and exponents
// of c_k / rho (bit 15 the sign, 64 above the double's exponent, so that 1 / W
// never takes it below 0) and of the third-body factors.
struct LaneIntSmem {
    ulonglong2* acc;
    im_u64 *sm, *tm;
    uint16_t *se, *te;

    __device__ __forceinline__ explicit LaneIntSmem(const MechDev& M)
    {
        const int nS = M.nS, T = blockDim.x, nTB = M.li_tb;
        acc = reinterpret_cast<ulonglong2*>(kin_smem) + threadIdx.x;
        sm = reinterpret_cast<im_u64*>(kin_smem) + 2 * (nS + 1) * T + threadIdx.x;
        tm = sm + (nS + 1) * T;
        se = reinterpret_cast<uint16_t*>(reinterpret_cast<im_u64*>(kin_smem) + (3 * (nS + 1) + nTB) * T) + threadIdx.x;
        te = se + (nS + 1) * T;
    }
};

// Mantissas and exponents of rho and 1 / rho.
struct LaneIntRho {
    im_u64 mr, mi;
    uint32_t er, ei;
};

// The species' sums of the reactions' words placed by the exponent sc; returns the
// largest rate's exponent. LOWER: a unit far below the largest rate (lane_int_lower);
// cut: a rate has bits below the unit; live: species that a rate other than zero
// changes.
template <bool LOWER>
__device__ __forceinline__ int lane_int_pass(const MechDev& M, const LaneIntSmem& W, const LaneIntRho& mix, Lane<double> K,
                                             int sc, bool& cut, uint32_t& live)
{
    ulonglong2* const acc = W.acc;
    const im_u64 *const sm = W.sm, *const tm = W.tm;
    const uint16_t *const se = W.se, *const te = W.te;
    const int nS = M.nS, T = blockDim.x, nTB = M.li_tb, up = M.imUp - sc, n = M.li_n;
    int emax = 0;
#pragma unroll 4
    for (int k = 0; k < nS; ++k) acc[k * T] = make_ulonglong2(0ull, 0ull);
    // the next reaction's record and rate constant are on their way
    // while this one is formed (the last record repeats)
    uint4 dn = M.li_rx[0];
    double kn = n ? K[dn.z] : 0.0;
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
        const uint4 d = dn;
        im_u64 Q;
        uint32_t e;
        im_split_k(kn, Q, e);
        if (LOWER && e == 0u) Q = 0ull;
        dn = M.li_rx[j + 1];
        kn = K[dn.z];
        const int a = (d.x & 0xffu) * T, b = ((d.x >> 8) & 0xffu) * T;
        Q = im_mul(im_mul(sm[a], sm[b]), Q);
        const uint32_t ea = se[a], eb = se[b];
        e += (ea & 0x7fffu) + (eb & 0x7fffu);
        if (j < nTB) {
            Q = im_mul(Q << 1, tm[j * T]);
            e += te[j * T] - (uint32_t)(IM_BIAS - 63);
        }
        if ((d.y & (7u << 20)) != (2u << 20)) {  // not rho^2 as for a plain reaction of two
            for (int p = (int)((d.y >> 20) & 7u) - 2; p != 0; p += p > 0 ? -1 : 1) {
                Q = im_mul(Q, p > 0 ? mix.mr : mix.mi);
                e += (p > 0 ? mix.er : mix.ei) - (uint32_t)(IM_BIAS - 64);
            }
        }
        const int L = (int)e + up;
        emax = max(emax, (int)e);
        im_u128 v = im_place(Q, L);
        if constexpr (LOWER) {
            v.hi |= im_shl(Q, (uint32_t)(L - 64));
            if (Q) {
                cut = cut || L < 0;
                live |= 1u << (d.x >> 16 & 0xffu) | 1u << (d.x >> 24) | 1u << (d.y & 0xffu) | 1u << (d.y >> 8 & 0xffu);
            }
        }
        if ((ea ^ eb) & 0x8000u) {
            im_u128 u{0ull, 0ull};
            im_sub(u, v.lo, v.hi);
            v = u;
        }
        ulonglong2* const p0 = acc + (d.x >> 16 & 0xffu) * T;
        ulonglong2* const p1 = acc + (d.x >> 24) * T;
        ulonglong2* const n0 = acc + (d.y & 0xffu) * T;
        ulonglong2* const n1 = acc + (d.y >> 8 & 0xffu) * T;
        const ulonglong2 A = *p0, B = *p1, D = *n0, E = *n1;
        im_u128 wa{A.x, A.y}, wb{B.x, B.y}, wd{D.x, D.y}, we{E.x, E.y};
        im_add(wa, v.lo, v.hi);
        im_add(wb, v.lo, v.hi);
        im_sub(wd, v.lo, v.hi);
        im_sub(we, v.lo, v.hi);
        if (d.y & LI_X2) {
            if (d.y & LI_P0X2) im_add(wa, v.lo, v.hi);
            if (d.y & LI_P1X2) im_add(wb, v.lo, v.hi);
            if (d.y & LI_N0X2) im_sub(wd, v.lo, v.hi);
            if (d.y & LI_N1X2) im_sub(we, v.lo, v.hi);
        }
        *p0 = make_ulonglong2(wa.lo, wa.hi);
        *p1 = make_ulonglong2(wb.lo, wb.hi);
        *n0 = make_ulonglong2(wd.lo, wd.hi);
        *n1 = make_ulonglong2(we.lo, we.hi);
    }
    return emax;
}

// The sums of the species in `left`, which were too short at the scale sc
// (intf.cuh): species without a rate are zero, the others take passes with
// lower units.
static __device__ __noinline__ void lane_int_lower(const MechDev& M, LaneIntRho mix, Lane<double> K, int sc, uint32_t left,
                                                   Lane<double> out)
{
    const LaneIntSmem W(M);
#pragma unroll 1
    while (left) {
        sc -= IM_STEP;
        bool cut = false;
        uint32_t live = 0u;
        lane_int_pass<true>(M, W, mix, K, sc, cut, live);
        uint32_t still = 0u;
        for (int i = 0; i < M.nS; ++i) {
            if (!(left >> i & 1u)) continue;
            const ulonglong2 w = W.acc[i * blockDim.x];
            if (cut && (live >> i & 1u) && im_short(im_u128{w.x, w.y}, M.imShort)) still |= 1u << i;
            else
                out[i] = im_scaled(im_u128{w.x, w.y}, sc - M.imUp - 3 * IM_BIAS, M.imW[i].y, M.imWe[i].y, mix.mr, (int)mix.er);
        }
        left = still;
    }
}

struct IntF {
    // The cell's first scale: 0, or -1 where a rate constant is not finite.
    __device__ static int scale0(const MechDev& M, Lane<double> K, Lane<double> KR)
    {
        bool fin = true;
#pragma unroll 4
        for (int j = 0; j < M.nR; ++j) fin &= im_finite_k(K[j]);
        for (int j = 0; j < M.nFO; ++j) fin &= im_finite_k(KR[j]);
        return fin ? 0 : -1;
    }

    template <typename R, typename KT>
    __device__ __forceinline__ static void eval(const MechDev& M, double Ctot, double invCtot, Lane<KT> K, Lane<KT> KR,
                                                Lane<R> C, Lane<R> OM, Lane<double> x, Lane<double> out, int& scale)
    {
        static_assert(sizeof(R) == 8 && sizeof(KT) == 8, "FP64");
        const int nS = M.nS, T = blockDim.x, nTB = M.li_tb;
        const LaneIntSmem S(M);
        ulonglong2* const acc = S.acc;
        im_u64 *const sm = S.sm, *const tm = S.tm;
        uint16_t *const se = S.se, *const te = S.te;
        // c_k / rho: Y_k / W_k
        double S0 = 0.0, S1 = 0.0;
        bool in = scale >= 0;
        int neg = -100000;
        auto load = [&](int i, double& S) {
            const double v = x[i];
            S = fma(v, M.invW[i], S);
            im_u64 m;
            uint32_t e;
            im_split(v, m, e);
            in = in && (e & 0x7ffu) != 0x7ffu;
            const int z = (int)(e & 0x7ffu) + M.imWe[i].x - 1022 + 64;
            if ((int)e < 0 && m) neg = max(neg, z);
            sm[i * T] = im_mul(m, M.imW[i].x) << 1;
            se[i * T] = (uint16_t)((uint32_t)z | (e >> 31 << 15));
        };
        int i0 = 0;
#pragma unroll 2
        for (; i0 + 1 < nS; i0 += 2) {
            load(i0, S0);
            load(i0 + 1, S1);
        }
        if (i0 < nS) load(i0, S0);
        sm[nS * T] = 1ull << 62;
        se[nS * T] = 1023 + 64;
        const double Sum = S0 + S1;
        const uint32_t top = (uint32_t)__double2hiint(Sum);
        const int eS = (int)(top >> 20);
        // finite, and no species below -2^-9 of the total
        if (!(in && top - 0x00100000u < 0x7fe00000u && neg + 9 <= eS + 64)) {
            lane_int_general(M, Ctot, invCtot, K, KR, C, OM, x, out);
            return;
        }
        const double rho = Ctot * Tab<double>::inv(Sum);
        LaneIntRho mix;
        im_split_k(rho, mix.mr, mix.er);
        im_split_k(Sum * invCtot, mix.mi, mix.ei);
        int bad = 0;
        if (nTB) {
            // fractions of the total in 30 + 29 bits, in the lane's own sums' words
            int2* const F = reinterpret_cast<int2*>(acc);
#pragma unroll 2
            for (int k = 0; k < nS; ++k) {
                const uint32_t e = se[k * T];
                long long f = (long long)((im_shr(sm[k * T], (uint32_t)(eS - (int)(e & 0x7fffu) + 67)) + 1ull) >> 1);
                if (e & 0x8000u) f = -f;
                const int hi = (int)((f + (1 << 28)) >> 29);
                F[2 * k * T] = make_int2(hi, (int)(f - (long long)hi * (1 << 29)));
            }
#pragma unroll 1
            for (int r = 0; r < nTB; ++r) {
                const int2* __restrict__ E = M.li_eff + r * nS;
                long long hi = 0, mid = 0;
#pragma unroll 4
                for (int k = 0; k < nS; ++k) {
                    const int2 u = E[k], f = F[2 * k * T];
                    hi += (long long)u.x * f.x;
                    mid += (long long)u.x * f.y;
                    mid += (long long)u.y * f.x;
                }
                const long long U = hi + (mid >> 29);
                if (U < (1ll << 53)) bad = IM_OUT;  // small beside its terms: the fractions are too coarse
                const int z = max(1, __clzll(U | 1ll));
                im_u64 mm = (im_u64)U << (z - 1);
                uint32_t em = (uint32_t)(eS + M.li_effx[r] + 5 - z);
                const uint4 d = M.li_rx[r];
                if (d.y & LI_FALLOFF) {
                    im_u64 km;
                    uint32_t ke;
                    im_split_k(KR[d.w], km, ke);
                    const double Pr = im_round(im_mul(im_mul(km, mm) << 1, mix.mr), (int)(ke + em + mix.er) - 3 * IM_BIAS + 127, false);
                    im_split(quot(Pr, 1.0 + Pr), mm, em);
                    if (em >= 0x7ffu) bad = IM_OUT;
                }
                tm[r * T] = mm;
                te[r * T] = (uint16_t)em;
            }
        }
        int s0;
#pragma unroll 1
        for (;;) {
            s0 = scale;
            bool cut = false;
            uint32_t live = 0u;
            const int emax = max(bad, lane_int_pass<false>(M, S, mix, K, s0, cut, live));
            if (emax >= IM_OUT) {
                lane_int_general(M, Ctot, invCtot, K, KR, C, OM, x, out);
                return;
            }
            scale = emax;
            if (emax <= s0 + IM_GUARD && emax >= s0 - IM_SLACK) break;
        }
        uint32_t left = 0u;
#pragma unroll 2
        for (int i = 0; i < nS; ++i) {
            // a word's unit at e = s0: 2^(128 + s0 - 2 * 64 - 3 IM_BIAS - imUp)
            const ulonglong2 w = acc[i * T];
            const im_u64 mW = M.imW[i].y;  // 0: no reaction changes the species
            if (mW && im_short(im_u128{w.x, w.y}, M.imShort)) left |= 1u << i;
            out[i] = im_scaled(im_u128{w.x, w.y}, s0 - M.imUp - 3 * IM_BIAS, mW, M.imWe[i].y, mix.mr, (int)mix.er);
        }
        if (left) lane_int_lower(M, mix, K, s0, left, out);
    }

    template <typename R>
    __device__ static void eval_energy(const MechDev&, double, Lane<R>, Lane<R>, Lane<double>, Lane<double>)
    {
    }
};

template <>
struct IntegerF<IntF> {
    static constexpr bool value = true;
};

}  // namespace kin
