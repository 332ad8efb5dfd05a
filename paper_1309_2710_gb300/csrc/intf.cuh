// intf.cuh -- FP64 arithmetic of the source term on the integer pipes.
//
// GB300 runs one FP64 warp instruction per SM sub-partition every 64 cycles
// (DFMA, DADD, DMUL and 64-bit conversions alike; 628 G FMA/s on the chip),
// against 2 cycles for a 32 x 32 + 64 bit multiply-add (IMAD.WIDE) and for a
// 32-bit shift or add. The rates of progress and their sums, nine tenths of
// an FP64 evaluation of f, therefore run faster as integers than on the FP64
// pipe, and that pipe is left to the state vectors and the step control,
// which run beside them:
//  * a factor (rate constant, concentration) is a 63-bit left-aligned
//    mantissa and an exponent, exact for every normal double; a product
//    keeps the top 62 bits of the mantissas' product (three IMAD.WIDE, 6
//    cycles for a DMUL's 64);
//  * a rate of progress is placed into a 128-bit fixed-point word whose unit is
//    far below the largest rate of the evaluation, so every sum of rates is
//    exact (four 32-bit adds) but for the words' own last bits; sums that these
//    bits could matter to are formed again with a lower unit (IM_STEP below);
//  * a third-body sum multiplies 59-bit integer efficiencies by the
//    concentrations as 59-bit fractions of the total. Sums below 2^-7 to 2^-5 of
//    the row's largest efficiency times the total are taken in FP64, where the
//    fractions would be too coarse.
// A product of two loses up to 2^-58, one of five (a third body, the density) up to
// 2^-53, and a sum of rates nothing to the order of its terms. Error of a
// species' rate over the sum of its |terms|, in units of 2^-53, on mixtures of 13,
// 53 and 111 species with given rate constants (tests/test_int_f_species.py): rms
// 1.2 to 2.0, and 1.8 to 2.2 for the plain FP64 form of the same rates. States
// outside the range of the fixed-point forms (not finite, or a concentration
// below -2^-9 of the total) take a plain FP64 evaluation instead.
#pragma once
#ifndef __CUDACC_RTC__
#include <cstdint>
#endif

namespace kin {

typedef unsigned long long im_u64;

// Exponent words: bit 31 the sign, the rest the exponent biased by 1023 as in
// the double; the value is mantissa * 2^(e - IM_BIAS).
constexpr int IM_BIAS = 1023 + 62;

// Top 64 of the 128 bits of a * b, less at most 3 units; a, b < 2^63.
__device__ __forceinline__ im_u64 im_mul(im_u64 a, im_u64 b)
{
    const uint32_t a1 = (uint32_t)(a >> 32), a0 = (uint32_t)a, b1 = (uint32_t)(b >> 32), b0 = (uint32_t)b;
    im_u64 t = (im_u64)a1 * b0;
    t = (im_u64)a0 * b1 + t;
    return (im_u64)a1 * b1 + (t >> 32);
}

// Mantissa and exponent word of a double (a denormal becomes zero).
__device__ __forceinline__ void im_split(double v, im_u64& m, uint32_t& e)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const uint32_t x = (hi >> 20) & 0x7ffu;
    e = x | (hi & 0x80000000u);
    const im_u64 n = ((im_u64)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    m = x ? n << 10 : 0ull;
}

// The same of a positive double; zero and denormals read as about 2^-1023
// (im_normal_k tells).
__device__ __forceinline__ void im_split_k(double v, im_u64& m, uint32_t& e)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    e = hi >> 20;
    m = (((im_u64)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 10;
}

__device__ __forceinline__ bool im_normal_k(double v) { return ((uint32_t)__double2hiint(v) >> 20) != 0u; }
__device__ __forceinline__ bool im_finite_k(double v) { return ((uint32_t)__double2hiint(v) >> 20) < 0x7ffu; }
__device__ __forceinline__ bool im_finite_k(float v) { return (__float_as_uint(v) >> 23) < 0xffu; }

struct im_u128 {
    im_u64 lo, hi;
};

// 64-bit shifts by any unsigned amount (64 and more give zero), and 128-bit
// sums (the plain forms are for host compilers).
#ifdef __CUDACC__
__device__ __forceinline__ im_u64 im_shl(im_u64 v, uint32_t n)
{
    im_u64 r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}
__device__ __forceinline__ im_u64 im_shr(im_u64 v, uint32_t n)
{
    im_u64 r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}
__device__ __forceinline__ void im_add(im_u128& a, im_u64 lo, im_u64 hi)
{
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(a.lo), "+l"(a.hi) : "l"(lo), "l"(hi));
}
__device__ __forceinline__ void im_sub(im_u128& a, im_u64 lo, im_u64 hi)
{
    asm("sub.cc.u64 %0, %0, %2;\n\tsubc.u64 %1, %1, %3;" : "+l"(a.lo), "+l"(a.hi) : "l"(lo), "l"(hi));
}
#else
inline im_u64 im_shl(im_u64 v, uint32_t n) { return n < 64 ? v << n : 0; }
inline im_u64 im_shr(im_u64 v, uint32_t n) { return n < 64 ? v >> n : 0; }
inline void im_add(im_u128& a, im_u64 lo, im_u64 hi)
{
    const im_u64 l = a.lo + lo;
    a.hi += hi + (l < lo);
    a.lo = l;
}
inline void im_sub(im_u128& a, im_u64 lo, im_u64 hi)
{
    a.hi -= hi + (a.lo < lo);
    a.lo -= lo;
}
#endif

// Q * 2^L as a 128-bit word, Q < 2^61, L <= 63 (any L gives some word); bits
// below the unit drop.
__device__ __forceinline__ im_u128 im_place(im_u64 Q, int L)
{
    im_u128 r;
    r.lo = im_shl(Q, (uint32_t)L) | im_shr(Q, (uint32_t)-L);
    r.hi = im_shr(Q, (uint32_t)(64 - L));
    return r;
}

// r * 2^x rounded to a double, 2^52 < r < 2^63 (0 gives 0), negated if neg.
__device__ __forceinline__ double im_round(im_u64 r, int x, bool neg)
{
    if (r == 0ull) return 0.0;
    const int z = __clzll((long long)r);
    const im_u64 m = ((r << (z - 1)) + 512ull) >> 10;  // [2^52, 2^53]
    const int n = 1075 + x + 11 - z;
    im_u64 b = m + ((im_u64)(uint32_t)(n - 1) << 52);  // a carry into 2^53 raises the exponent
    if (n <= 0) b = 0ull;
    if (n >= 0x7ff) b = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(neg ? b | 0x8000000000000000ull : b));
}

// a * 2^-d of a signed 128-bit word, d >= 0.
__device__ __forceinline__ void im_sar(im_u128& a, int d)
{
    for (int k = 0; k < 2 && d >= 64; ++k, d -= 64) {
        a.lo = a.hi;
        a.hi = (im_u64)((long long)a.hi >> 63);
    }
    if (d == 0 || d >= 64) return;
    a.lo = a.lo >> d | a.hi << (64 - d);
    a.hi = (im_u64)((long long)a.hi >> d);
}

// Whether a signed 128-bit word has at most t bits.
__device__ __forceinline__ bool im_short(im_u128 a, int t)
{
    const im_u64 s = (im_u64)((long long)a.hi >> 63);
    const im_u64 hi = a.hi ^ s, lo = a.lo ^ s;
    return t < 64 ? (hi | im_shr(lo, (uint32_t)t)) == 0ull : im_shr(hi, (uint32_t)(t - 64)) == 0ull;
}

// (a 2^x) (u 2^(eu - IM_BIAS)) (v 2^(ev - IM_BIAS)) of a signed 128-bit word and
// two 63-bit mantissas, as a double.
__device__ __forceinline__ double im_scaled(im_u128 a, int x, im_u64 u, int eu, im_u64 v, int ev)
{
    const bool neg = (long long)a.hi < 0;
    if (neg) {
        im_u128 z{0ull, 0ull};
        im_sub(z, a.lo, a.hi);
        a = z;
    }
    if (a.hi == 0ull) {  // far below the largest rate: 64 bits up
        a.hi = a.lo;
        a.lo = 0ull;
        x -= 64;
        if (a.hi == 0ull) return 0.0;
    }
    const int z = __clzll((long long)a.hi);
    im_u64 t = a.hi;
    if (z) t = (t << z) | (a.lo >> (64 - z));
    t = im_mul(t >> 1, u) << 1;
    return im_round(im_mul(t, v), x + 64 - z + 1 + eu + ev - 2 * IM_BIAS + 127, neg);
}

// The tables of im_exp and im_log (int_tables.h), 64 entries: 2^(i / 64) in units
// of 2^-62; c_i just above 64 / (64 + i) in units of 2^-62 and -ln c_i in 2^-59.

// exp(a) as a 63-bit mantissa and exponent, false where a is not a number or
// exp overflows. 2^y, y = a log2(e) in 52 fractional bits: an entry of the table
// for the first six, a polynomial for the rest (degree 5, interpolating 2^(t/64)
// at the Chebyshev nodes of [0, 1]; 2^-59.6). Relative error 2^-52, against
// 2^-47 that an FP64 argument of 50 brings along; 75 integer instructions
// against some 20 on the FP64 pipe.
__device__ __forceinline__ bool im_exp(const im_u64* __restrict__ tab, double a, im_u64& m, uint32_t& e)
{
    im_u64 v;
    uint32_t w;
    im_split(a, v, w);
    const int x = (int)(w & 0x7ffu);
    m = 0ull;
    e = 0u;
    if (x >= 1023 + 10) return x < 0x7ff ? (int)w < 0 : (int)w < 0 && a < 0.0;  // |a| >= 1024
    const im_u64 p = im_mul(v, 6653256548922161246ull);  // |a| log2(e) = p 2^(x - 1083)
    const int s = 1031 - x;
    long long y = (long long)(s > 0 ? (im_shr(p, (uint32_t)(s - 1)) + 1ull) >> 1 : p << -s);
    if ((int)w < 0) y = -y;
    const int n = (int)(y >> 52) + 1023;
    const im_u64 r = (im_u64)y & 0xfffffffffffffull;
    const im_u64 t = (r & 0x3fffffffffffull) << 17;  // of the entry's interval, in 2^-63
    const uint32_t th = (uint32_t)(t >> 31);
    const uint32_t c4 = 2643776176u + (uint32_t)((5757821ull * th) >> 32);
    im_u64 q = 976438624029ull + (((im_u64)c4 * th) >> 32);
    q = 270471001802121ull + (im_mul(q, t) << 1);
    q = 49946518145323239ull + (im_mul(q, t) << 1);
    q = 4611686018427387899ull + (im_mul(q, t) << 1);
    if (n >= 0x7ff) return false;
    if (n <= 0) return true;  // below the smallest normal double
    m = im_mul(tab[r >> 46], q) << 2;
    e = (uint32_t)n;
    return true;
}

// ln T for T in [1, 2^16), as a double (0.5 ulp and 2^-57): T = 2^E m, m c_i = 1 +
// t / 64 for the entry i of m's first six bits, and the series of ln(1 + t / 64)
// to the eighth power.
__device__ __forceinline__ double im_log(const ulonglong2* __restrict__ tab, double T)
{
    im_u64 m;
    uint32_t e;
    im_split_k(T, m, e);
    const ulonglong2 c = tab[(m >> 56) & 63ull];
    const im_u64 t = (im_mul(m, c.x) - (1ull << 60)) << 9;  // in 2^-63
    const uint32_t th = (uint32_t)(t >> 31);
    uint32_t a = 149797u - (uint32_t)((2048ull * th) >> 32);
    a = 11184811u - (uint32_t)(((im_u64)a * th) >> 32);
    a = 858993459u - (uint32_t)(((im_u64)a * th) >> 32);
    im_u64 q = (1ull << 36) - (((im_u64)a * th) >> 32);
    q = 5864062014805ull - (im_mul(q, t) << 1);
    q = (1ull << 49) - (im_mul(q, t) << 1);
    q = (1ull << 56) - (im_mul(q, t) << 1);
    q = im_mul(q, t) << 1;
    const uint32_t n = e - 1023u;
    const im_u64 l = (im_u64)n * 399572145162582989ull + (((im_u64)n * 1582243228u) >> 32);  // n ln 2 in 2^-59
    return im_round(l + c.y + (q >> 3), -59, false);
}

// A word of the largest rate (e = the evaluation's scale) is shifted up by
// MechDev::imUp bits (int_word_bits of int_tables.h): Q < 2^61, so it stays below
// 2^(61 + imUp + 8) where the scale is IM_GUARD octaves too low, which leaves
// room for the entries of the mechanism's longest row and the sign. The words'
// unit is 2^-105 of the largest rate for rows of up to 127 entries (Q >= 2^54),
// 2^-97 where the scale is IM_SLACK octaves too high.
//
// A row's sum of fewer than MechDev::imShort = 53 + log2(entries) bits could
// miss an ulp in the bits below the unit: a species whose rates are all far
// below the cell's largest, or whose rates cancel. Such rows are summed again: with
// the unit of their own largest rate (int_short), or in the lane layout, all of
// them together, with the unit IM_STEP octaves lower, modulo 2^128 (the sum itself
// fits, the words that do not wrap around), and so on until each has its bits or no
// rate has bits below the unit, when the sums are exact (lane_int_lower). The
// workloads' cells have no net rate below 2^-36 of their largest, and a net rate
// of 2^-37 has its bits, so that they pay for the test alone, 2 to 5 % of a call.
// Inside the common code the further sums' registers and branches would cost 5 to
// 38 %.
constexpr int IM_GUARD = 8, IM_SLACK = 8, IM_STEP = 56;

// Exponent that stands for a rate that is not finite.
constexpr int IM_OUT = 1 << 20;

}  // namespace kin
