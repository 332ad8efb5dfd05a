// warp_int.cuh -- the warp layout's FP64 f on the integer pipes, isothermal, with
// the energy equation and alone
// (intf.cuh has the arithmetic, int_tables.h the tables).
//
// One group of G lanes evaluates f for one cell. Concentrations live in
// shared memory as mantissas and exponents; the lanes split the reactions of
// a chunk, leave each rate of progress as a 128-bit word in shared memory,
// and gather the words of the chunk into partial sums per species, G equal
// runs of the chunk's entries. Chunks keep the words of a large mechanism from
// taking the shared memory that resident groups and L1 need.
//
// An evaluation is bound by the latency of its phases, not by a pipe (cycles
// of one evaluation of 53 species / 634 reactions, two warps, 8 cells per
// SM: mixture 2165, products and third-body sums 8390, gather 8391, the rest
// 1780; the FP64 f it replaced took 43 K with one warp, 354 FP64 instructions
// of 64 cycles among them). So a lane's next reaction words, the gather's next
// entries and eight efficiencies of a third-body sum are fetched ahead.
// (Cycles from a build without the test of the sums' length and the wider limbs,
// which add 2 to 5 %.)
// Whole calls on GB300, plain FP64 f and this one: 53 / 634 RKC, 4,096 cells 77.0 and
// 40.0 ms; 111 / 1566 RKC, 16 instances of 2,000 cells in all 1061 and 231 ms;
// 13 / 54 RKC, 1,000 cells 3.75 and 3.08 ms, 30,011 cells 38.4 and 15.9; 9 / 38 RKCK,
// 4,096 cells 0.716 and 0.489 ms; energy equation, 13 / 54, 20,000 cells 66.8 and
// 14.1 (54.6 to 69 from state to state before); f alone, 53 / 634, 50,000 cells 2.80
// and 0.755 ms. Error of whole results against 64 bits: that of plain FP64 (1e-13
// and below, the finite differences of the spectral radius).
#pragma once
#include "intf.cuh"
#include "kernels.cuh"

namespace kin {

// The lanes of this thread's group within its warp.
template <int G>
__device__ __forceinline__ unsigned group_mask()
{
    return G >= 32 ? 0xffffffffu : (((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1)));
}

// Butterfly sum over a group of G lanes (a whole warp, or a 16-lane half
// that owns one cell); mask names the group's lanes.
template <int G, typename T>
__device__ __forceinline__ T group_sum(T v, unsigned mask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
}

template <int G>
__device__ __forceinline__ double group_max(double v, unsigned mask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(mask, v, o));
    return v;
}

// A group of G lanes that evaluates one cell: a half warp, a warp, or several
// warps of a block. Reductions leave every lane with the same bits, and the
// sums do not depend on G: component l + 32 r is added at lane l in the order
// of r, then the 32 (16, 8) lanes in butterfly order (the first step of 16
// lanes adds the components that 8 lanes hold in two slots). Across warps the components
// go through shared words and the group's named barrier; the words alternate
// between two sets, so that one barrier per reduction is enough (a set is
// written again only after the barrier of the reduction in between).
template <int G>
struct Group {
    static constexpr int WARPS = G / 32;
    unsigned mask;
    double* red;  // [2][set_words]
    int set, set_words;

    __device__ explicit Group(double* r, int words) : mask(group_mask<G>()), red(r), set(0), set_words(words) {}

    __device__ __forceinline__ void sync() const
    {
        if constexpr (G <= 32) __syncwarp(mask);
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / G), "n"(G) : "memory");
    }
    // sync, and whether v holds for any of the group's lanes
    __device__ __forceinline__ bool sync_any(bool v) const
    {
        if constexpr (G <= 32) {
            const bool a = __any_sync(mask, v);
            __syncwarp(mask);
            return a;
        } else {
            int a;
            asm volatile(
                "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, %3, p;\n\t"
                "selp.s32 %0, 1, 0, q;\n\t}"
                : "=r"(a)
                : "r"((int)v), "r"(1 + (int)threadIdx.x / G), "n"(G)
                : "memory");
            return a != 0;
        }
    }
    __device__ __forceinline__ double* next_set()
    {
        double* b = red + set * set_words;
        set ^= 1;
        return b;
    }
    // One value per warp, seen by all.
    template <typename T>
    __device__ __forceinline__ const T* exchange(T v)
    {
        static_assert(sizeof(T) <= 8, "one shared word per warp");
        T* t = reinterpret_cast<T*>(next_set());
        if ((threadIdx.x & 31) == 0) t[(threadIdx.x % G) >> 5] = v;
        sync();
        return t;
    }
    // Sum of v, or of its squares, over the components (lane + G r). (__dadd_rn:
    // no product in v is fused into the sum, which only some G could.)
    template <bool SQ, int NR>
    __device__ __forceinline__ double sum_of(const double (&v)[NR])
    {
        double s = 0.0;
        if constexpr (G <= 32) {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                if constexpr (SQ && G == 32) s = fma(v[r], v[r], s);
                else s = __dadd_rn(s, SQ ? __dmul_rn(v[r], v[r]) : v[r]);
            }
        } else {
            double* b = next_set();
#pragma unroll
            for (int r = 0; r < NR; ++r) b[threadIdx.x % G + G * r] = v[r];
            sync();
#pragma unroll
            for (int r = 0; r < NR * WARPS; ++r) {
                const double u = b[(threadIdx.x & 31) + 32 * r];
                s = SQ ? fma(u, u, s) : __dadd_rn(s, u);
            }
        }
        return group_sum<(G < 32 ? G : 32)>(s, mask);
    }
    template <int NR>
    __device__ __forceinline__ double sum(const double (&v)[NR])
    {
        return sum_of<false>(v);
    }
    template <int NR>
    __device__ __forceinline__ double sum_sq(const double (&v)[NR])
    {
        return sum_of<true>(v);
    }
    __device__ __forceinline__ double max(double v)
    {
        v = group_max<(G < 32 ? G : 32)>(v, mask);
        if constexpr (G > 32) {
            const double* b = exchange(v);
            v = b[0];
#pragma unroll
            for (int w = 1; w < WARPS; ++w) v = fmax(v, b[w]);
        }
        return v;
    }
    __device__ __forceinline__ int imax(int v)
    {
        v = __reduce_max_sync(mask, v);
        if constexpr (G > 32) {
            const int* b = exchange(v);
            v = b[0];
#pragma unroll
            for (int w = 1; w < WARPS; ++w) v = ::max(v, b[w]);
        }
        return v;
    }
    __device__ __forceinline__ bool all(bool v)
    {
        if constexpr (G <= 32) return __all_sync(mask, v);
        else return imax(!v) == 0;
    }
    // v of the group's lane k
    template <typename T>
    __device__ __forceinline__ T from(T v, int k)
    {
        if constexpr (G <= 32) return __shfl_sync(mask, v, k, G);
        else {
            double* b = next_set();
            if ((int)(threadIdx.x % G) == k) *reinterpret_cast<T*>(b) = v;
            sync();
            return *reinterpret_cast<const T*>(b);
        }
    }
};
// Shared words of one set of a group's reductions, NR components per lane.
template <int NR, int G>
__host__ __device__ constexpr int group_set_words() { return G > 32 ? NR * G : 0; }

// Where f's rate constants come from: stored (isothermal), or exp(ln A + beta ln T
// - (E / R) / T) at this temperature (K null).
struct RateSource {
    const double* K;
    double lnT, invT;
};

// The cell's mixture, with mantissas and exponents of rho and 1 / rho.
struct IntMix {
    double rho;
    im_u64 mr, mi;
    uint32_t er, ei;
    int eT;  // exponent of the sum of Y_k / W_k
};

// What int_row_sum reads of the cell beside its concentrations.
struct IntCell {
    IntMix mix;
    RateSource rk;
};

// The group's shared arrays.
struct IntSmem {
    ulonglong2* OM;  // [chunk + 1] rates of progress of a chunk, and a zero word
    ulonglong2* P;   // [nslots] partial sums
    int2* CF;        // [nS, even] concentrations as 59-bit fractions: 30 high, 29 low bits
    IntCell* cell;
    im_u64* CM;      // [nS + 1] mantissas, after the constant 1 that empty slots read
    uint32_t* CE;    // [nS + 1] exponent words

    __device__ IntSmem(const MechDev& M, const IntDev& I, double* base)
    {
        OM = reinterpret_cast<ulonglong2*>(base);
        P = OM + I.chunk + 1;
        species(M, reinterpret_cast<int2*>(P + I.nslots));
    }
    // (without OM and P, from the first of the species' arrays)
    __device__ IntSmem(const MechDev& M, int2* f) : OM(nullptr), P(nullptr) { species(M, f); }
    __device__ void species(const MechDev& M, int2* f)
    {
        CF = f;
        cell = reinterpret_cast<IntCell*>(CF + ((M.nS + 1) & ~1));
        CM = reinterpret_cast<im_u64*>(cell + 1);
        CE = reinterpret_cast<uint32_t*>(CM + M.nS + 1);
    }
};

static_assert(sizeof(IntCell) == 8 * INT_CELL_WORDS, "int_group_words counts it");

// Shared FP64 words of a group, a multiple of 4.
__host__ __device__ __forceinline__ int int_smem_words(const MechDev& M, const IntDev& I)
{
    return int_group_words(M.nS, I.chunk, I.nslots);
}

// A c_k / rho back from its mantissa.
__device__ __forceinline__ double int_conc(const IntSmem& S, int k)
{
    const uint32_t e = S.CE[k];
    return im_round(S.CM[k], (int)(e & 0x7fffffffu) - 64 - IM_BIAS, (int)e < 0);
}

// [M] of an efficiency row in FP64, from concentrations c[k + 1] given by get, in
// two interleaved partial sums.
template <typename Get>
__device__ double int_row_dot(const MechDev& M, int row, Get get)
{
    const double2* __restrict__ a = reinterpret_cast<const double2*>(M.effV64) + row;
    double m0 = 0.0, m1 = 0.0;
#pragma unroll 1
    for (int k = 0; k < M.nS; ++k) {
        const double2 e = a[(int64_t)(k >> 1) * M.nM];
        const double m = m1 + ((k & 1) ? e.y : e.x) * get(k + 1);
        m1 = m0;
        m0 = m;
    }
    return m0 + m1;
}

static __device__ __noinline__ double int_row_dot_slow(const MechDev& M, int row, int2* CF)
{
    const IntSmem S(M, CF);
    return int_row_dot(M, row, [&](int k) { return int_conc(S, k); });
}

// The exponents of reaction position q and falloff ordinal fo.
__device__ __forceinline__ double rate_exponent(const MechDev& M, int q, const RateSource& k)
{
    return fma(-M.arr[2 * M.nR + q], k.invT, fma(M.arr[M.nR + q], k.lnT, M.arr[q]));
}
__device__ __forceinline__ double low_exponent(const MechDev& M, int fo, const RateSource& k)
{
    return fma(-M.arr0[2 * M.nFO + fo], k.invT, fma(M.arr0[M.nFO + fo], k.lnT, M.arr0[fo]));
}

// A state outside the integer forms' range (a trial point that blew up, as a Cash-Karp
// step far beyond the stability limit makes them) takes plain FP64, chunk by chunk:
// the lanes' rates of progress from the concentrations c[k + 1] (c[0] = 1), then
// each species' sum over its row, whose entries are in order of position, so that
// the bits depend neither on the lanes nor on the chunks. Out of line; about the
// time of the plain FP64 f that the integer one replaced (with every row forming
// its own rates instead, 111 species / 1566 reactions, 500 cells in RKCK took
// 43.8 ms instead of 17.4; 23.2 in plain FP64 throughout).
template <bool AT_T>
static __device__ __noinline__ void int_general_rates(const MechDev& M, int2* CF, double* om, int q0, int q1, int lane, int lanes)
{
    const IntSmem S(M, CF);
    const RateSource k = S.cell->rk;
    const double* c = reinterpret_cast<const double*>(S.CM);
    const int nP = M.nR - M.nM, nF = M.nR - M.nFO;
#pragma unroll 1
    for (int q = q0 + lane; q < q1; q += lanes) {
        const uint32_t w = M.rxw[q];
        const double a = AT_T ? rate_exponent(M, q, k) : 0.0;
        double v = (AT_T ? exp(a) : k.K[q]) * c[w & 0xffffu] * c[w >> 16];
        if (q >= nP) {
            const double Mc = int_row_dot(M, q - nP, [&](int i) { return c[i]; });
            if (q < nF) {
                v *= Mc;
            } else {
                const double Pr = (AT_T ? exp(low_exponent(M, q - nF, k) - a) : k.K[M.nR + (q - nF)]) * Mc;
                v *= ddiv(Pr, 1.0 + Pr);
            }
        }
        om[q - q0] = v;
    }
}

// w and the rest of species i's row from entry e on, up to position q1.
struct IntRow {
    double w;
    int e;
};
static __device__ __noinline__ IntRow int_general_row(const MechDev& M, const double* om, int i, int q0, int q1, IntRow a)
{
    const int end = M.csr_ptr[i + 1];
#pragma unroll 1
    for (; a.e < end; ++a.e) {
        const int q = M.csrq[a.e] >> 3;
        if (q >= q1) break;
        a.w += M.csrq_nu[a.e] * om[q - q0];
    }
    return a;
}

// f of such a state, from its c_k / rho (the group's lanes together).
template <int NR, int G, bool AT_T>
__device__ __forceinline__ void int_general(const MechDev& M, const IntDev& I, const IntSmem& S, const double (&c)[NR],
                                            double rho, double invrho, double (&out)[NR], int lane, const Group<G>& grp)
{
    double* cs = reinterpret_cast<double*>(S.CM);
    double* om = reinterpret_cast<double*>(S.OM);
    if (lane == 0) cs[0] = 1.0;
    IntRow row[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        row[r] = IntRow{0.0, i < M.nS ? M.csr_ptr[i] : 0};
        if (i < M.nS) cs[i + 1] = c[r] * rho;
    }
    grp.sync();
#pragma unroll 1
    for (int q0 = 0; q0 < M.nR; q0 += I.chunk) {
        const int q1 = min(M.nR, q0 + I.chunk);
        int_general_rates<AT_T>(M, S.CF, om, q0, q1, lane, G);
        grp.sync();
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (lane + G * r < M.nS) row[r] = int_general_row(M, om, lane + G * r, q0, q1, row[r]);
        grp.sync();
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        out[r] = i < M.nS ? __dmul_rn(row[r].w, M.W[i] * invrho) : 0.0;
    }
}

// The rate of progress of the reaction at position q (over a common power of rho) as
// Q < 2^61 and exponent word, from its reactants' word and its rate constant
// (kq), or ln A, beta and E / R (AT_T). False where it is not finite. AHEAD: eight
// efficiencies in flight.
template <bool AT_T, bool AHEAD>
__device__ __forceinline__ bool int_rate(const MechDev& M, const IntSmem& S, const RateSource& rk, const IntMix& mix,
                                         int q, uint32_t w, double kq, double bq, double eq, im_u64& Q, uint32_t& e)
{
    const int nS = M.nS, nR = M.nR, nM = M.nM, nP = nR - nM, nF = nR - M.nFO;
    bool in = true;
    double a = 0.0;
    if constexpr (AT_T) {
        a = fma(-eq, rk.invT, fma(bq, rk.lnT, kq));
        if (!im_exp(M.ex2, a, Q, e)) in = false;
    } else {
        im_split_k(kq, Q, e);
    }
    const uint32_t ra = w & 0xffffu, rb = w >> 16;
    Q = im_mul(im_mul(S.CM[ra], S.CM[rb]), Q);
    e += S.CE[ra] + S.CE[rb];
    if (q >= nP) {
        const int row = q - nP;
        const int4* __restrict__ E = M.effI + row;
        const int4* F = reinterpret_cast<const int4*>(S.CF);
        long long hi = 0, mid = 0;
        auto term = [&](const int4& u, const int4& f) {
            hi += (long long)u.x * f.x;
            mid += (long long)u.x * f.y;
            mid += (long long)u.y * f.x;
            hi += (long long)u.z * f.z;
            mid += (long long)u.z * f.w;
            mid += (long long)u.w * f.z;
        };
        // (sixteen species' products keep mid below 2^63)
        auto carry = [&]() {
            hi += mid >> 29;
            mid &= (1 << 29) - 1;
        };
        const int n2 = (nS + 1) >> 1;
        int k = 0;
#pragma unroll 1
        for (; AHEAD && k + 7 < n2; k += 8) {
            int4 u[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) u[j] = E[(int64_t)(k + j) * nM];
#pragma unroll
            for (int j = 0; j < 8; ++j) term(u[j], F[k + j]);
            carry();
        }
        if constexpr (AHEAD) {
#pragma unroll 4
            for (; k < n2; ++k) term(E[(int64_t)k * nM], F[k]);
        } else {
#pragma unroll 1
            for (; k < n2; ++k) {
                term(E[(int64_t)k * nM], F[k]);
                carry();
            }
        }
        carry();
        const long long U = hi;
        im_u64 mm;
        uint32_t em;
        if (U < (1ll << 53)) {  // small beside its terms: the fractions are too coarse
            im_split(int_row_dot_slow(M, row, S.CF), mm, em);
        } else {
            const int z = __clzll(U);
            mm = (im_u64)U << (z - 1);
            em = (uint32_t)(M.effX[row] + mix.eT + 5 - z);
        }
        if (q >= nF) {
            im_u64 km;
            uint32_t ke;
            if constexpr (AT_T) {
                if (!im_exp(M.ex2, low_exponent(M, q - nF, rk) - a, km, ke)) in = false;
            } else {
                im_split_k(rk.K[nR + (q - nF)], km, ke);
            }
            const double Pr = im_round(im_mul(im_mul(km, mm) << 1, mix.mr),
                                       (int)(ke + (em & 0x7fffffffu) + mix.er) - 3 * IM_BIAS + 127, (int)em < 0);
            im_split(quot(Pr, 1.0 + Pr), mm, em);
            if ((em & 0x7ffu) == 0x7ffu) in = false;
        }
        // (a bit up: four factors cut from a short mantissa would cost half an ulp)
        Q = im_mul(Q << 1, mm);
        e += em - (uint32_t)(IM_BIAS - 63);
    }
    // the rate is rho^2 of what a plain reaction of two gives here
    if (q >= nP || M.imLow) {
        int p = (ra != 0u) + (rb != 0u) + (q >= nP && q < nF) - 2;
        for (; p > 0; --p) {
            Q = im_mul(Q, mix.mr);
            e += mix.er - (uint32_t)(IM_BIAS - 64);
        }
        for (; p < 0; ++p) {
            Q = im_mul(Q, mix.mi);
            e += mix.ei - (uint32_t)(IM_BIAS - 64);
        }
    }
    return in;
}

// Sums that are too short for their last bits (intf.cuh), once more: the lanes'
// rates of a chunk of reactions as mantissas and exponents, then each such species'
// sum over its row (csrq, in order of position), placed by the largest of them so
// far. Rarely taken, so it is out of line with rolled loops, and reads the cell's
// values from shared memory: with more of its registers around, cells without such
// species lose up to 12 % (now 2 to 5 %). A cell with such species takes two to three
// times as long, about the plain FP64 f's time or less: GB300, 53 species / 634
// reactions, unburnt mixtures, 4,096 cells with radicals of zero 2.9 ms (without
// these sums, and wrong, 1.35; plain FP64 2.5), of 1e-22 to 1e-9 7.0 (5.3, 11.5); f
// alone, 50,000 cells 2.1 and 1.4 (0.69, 0.85; 2.8). Row by row with each row's rates
// formed anew it was 12, 11, 10 and 1.9 ms.
// Shift of the largest rate's word there: 61 + 43 bits, the entries of the longest
// row (two for each reaction) and the sign.
constexpr int INT_SHORT_UP = 43;

template <bool AT_T>
static __device__ __noinline__ void int_short_rates(const MechDev& M, int2* CF, ulonglong2* om, int q0, int q1, int lane, int lanes)
{
    const IntSmem S(M, CF);
    const IntMix mix = S.cell->mix;
    const RateSource rk = S.cell->rk;
#pragma unroll 1
    for (int q = q0 + lane; q < q1; q += lanes) {
        const double kq = AT_T ? M.arr[q] : rk.K[q];
        im_u64 Q;
        uint32_t e;
        int_rate<AT_T, false>(M, S, rk, mix, q, M.rxw[q], kq, AT_T ? M.arr[M.nR + q] : 0.0, AT_T ? M.arr[2 * M.nR + q] : 0.0, Q, e);
        if (!AT_T && !im_normal_k(kq)) Q = 0ull;
        om[q - q0] = make_ulonglong2(Q, e);
    }
}

// A species' sum, its scale (-1: no rate so far) and the next entry of its row.
struct IntSum {
    im_u128 w;
    int at, e;
};
// The sum with the row's entries up to position q1.
static __device__ __noinline__ IntSum int_short_row(const MechDev& M, const ulonglong2* om, int q0, int q1, int end, IntSum a)
{
    int next = M.csrq[a.e];  // (the table ends in a word past the last row)
#pragma unroll 1
    for (; a.e < end; ++a.e) {
        const int q = next >> 3, nu = (next & 7) - 4;
        if (q >= q1) break;
        next = M.csrq[a.e + 1];
        const ulonglong2 v = om[q - q0];
        if (v.x == 0ull) continue;
        const int x = (int)(v.y & 0x7fffffffull);
        if (x > a.at) {
            im_sar(a.w, x - max(a.at, 0));
            a.at = x;
        }
        const im_u128 u = im_place(v.x, x - a.at + INT_SHORT_UP);
        const bool neg = (v.y >> 31 != 0ull) != (nu < 0);
        for (int n = abs(nu); n > 0; --n)
            if (neg) im_sub(a.w, u.lo, u.hi);
            else im_add(a.w, u.lo, u.hi);
    }
    return a;
}

// The group's species in `left` (a bit per slot).
template <int NR, int G, bool AT_T>
__device__ __forceinline__ void int_short(const MechDev& M, const IntDev& I, const IntSmem& S, unsigned left,
                                          double (&out)[NR], int lane, const Group<G>& grp)
{
    IntSum a[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) a[r] = IntSum{{0ull, 0ull}, -1, lane + G * r < M.nS ? M.csr_ptr[lane + G * r] : 0};
#pragma unroll 1
    for (int q0 = 0; q0 < M.nR; q0 += I.chunk) {
        const int q1 = min(M.nR, q0 + I.chunk);
        int_short_rates<AT_T>(M, S.CF, S.OM, q0, q1, lane, G);
        grp.sync();
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (left >> r & 1u) a[r] = int_short_row(M, S.OM, q0, q1, M.csr_ptr[lane + G * r + 1], a[r]);
        grp.sync();
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        if (left >> r & 1u)
            out[r] = im_scaled(a[r].w, a[r].at - INT_SHORT_UP - 3 * IM_BIAS, M.imW[i].y, M.imWe[i].y, S.cell->mix.mr,
                               (int)S.cell->mix.er);
    }
}

// v cut to FP32, without the FP64 pipe's conversion (beyond its range: 0, or infinite).
__device__ __forceinline__ float im_f32(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v), s = hi & 0x80000000u;
    const int x = (int)((hi >> 20) & 0x7ffu) - 896;
    if (x <= 0) return 0.0f;
    return __uint_as_float(s | (x >= 255 ? 0x7f800000u : (uint32_t)x << 23 | (hi & 0xfffffu) << 3 | lo >> 29));
}

// About the largest rate's exponent of the lane's reactions, for the first
// evaluation of a cell: a few octaves too high where a third-body sum is small
// beside its largest efficiency, more where a falloff is. A function of the cell
// alone, in FP32 from a table of its own (int_scale_table) and without the third-body
// sums; a whole evaluation to find the scale would double kin_rates.
__device__ __forceinline__ int int_first_scale(const MechDev& M, const IntSmem& S, const RateSource& rk, const IntMix& mix,
                                               int lane, int lanes)
{
    const float lnT = im_f32(rk.lnT), invT = im_f32(rk.invT);
    const int nP = M.nR - M.nM;
    int top = 0;
#pragma unroll 4
    for (int q = lane; q < M.nR; q += lanes) {
        const uint4 d = M.scl[q];
        const float a = fmaf(-__uint_as_float(d.z), invT, fmaf(__uint_as_float(d.y), lnT, __uint_as_float(d.x)));
        int e = (int)floorf(a) + (int)((S.CE[d.w & 0x3ffu] + S.CE[d.w >> 10 & 0x3ffu]) & 0x7fffffffu);
        if (q >= nP || M.imLow) {
            const int p = (int)(d.w >> 20 & 7u) - 2;  // of rho, beyond a plain reaction of two
            if (d.w >> 23) e += mix.eT;
            e += p > 0 ? p * ((int)mix.er - (IM_BIAS - 64)) : -p * ((int)mix.ei - (IM_BIAS - 64));
        }
        top = max(top, e);
    }
    return top;
}

// f for the group's cell. `scale` is the exponent that the fixed-point words are
// placed by, kept by the caller from one evaluation of the cell to the next
// (at the first a value that does not depend on other cells, for the bits of the
// result not to; AT_T: -1, and int_first_scale gives one); an evaluation whose largest rate is more than
// IM_GUARD octaves above it or IM_SLACK below is repeated with that rate's. The
// barriers around the gather carry the two tests, the one at the end whether a
// sum is too short for its last bits (int_short). kfin: the cell's rate constants
// are finite.
template <int NR, int G, bool AT_T>
__device__ __forceinline__ void warp_feval_int(const MechDev& M, const IntDev& I, const IntSmem& S,
                                               const RateSource& rk, bool kfin, double Ctot, double invCtot,
                                               int& scale, const double (&x)[NR], double (&out)[NR], int lane,
                                               Group<G>& grp)
{
    const int nS = M.nS, nR = M.nR;
    // c_k / rho = Y_k / W_k: in FP64 for the mixture sum, and as mantissa and
    // exponent word (64 above the double's, so that 1 / W never takes it below
    // zero) for everything else
    double c[NR];
    im_u64 m[NR];
    uint32_t e[NR];
    int neg = -100000;
    bool in = kfin;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        c[r] = 0.0;
        m[r] = 0ull;
        e[r] = 0u;
        if (i < nS) {
            c[r] = __dmul_rn(x[r], M.invW[i]);
            im_split(x[r], m[r], e[r]);
            in = in && (e[r] & 0x7ffu) != 0x7ffu;
            const int z = (int)(e[r] & 0x7ffu) + M.imWe[i].x - 1022 + 64;
            if ((int)e[r] < 0 && m[r]) neg = max(neg, z);
            m[r] = im_mul(m[r], M.imW[i].x) << 1;
            e[r] = (uint32_t)z | (e[r] & 0x80000000u);
        }
    }
    const double s = grp.sum(c);
    const double rho = Ctot * Tab<double>::inv(s);
    const uint32_t top = (uint32_t)__double2hiint(s);
    const int eT = (int)(top >> 20);
    // finite, and no species below -2^-9 of the total
    in = in && top - 0x00100000u < 0x7fe00000u && neg + 9 <= eT + 64;
    IntMix mix{rho, 0ull, 0ull, 0u, 0u, eT};
    im_split_k(rho, mix.mr, mix.er);
    if (M.imLow) im_split_k(s * invCtot, mix.mi, mix.ei);
    if (lane == 0) {
        S.CM[0] = 1ull << 62;
        S.CE[0] = 1023u + 64u;
        S.OM[I.chunk] = make_ulonglong2(0ull, 0ull);
        *S.cell = IntCell{mix, rk};
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        if (i < nS) {
            S.CM[i + 1] = m[r];
            S.CE[i + 1] = e[r];
            if (M.nM) {
                // 2^59 of twice the total at most: sum |F| < 3 * 2^59
                long long F = (long long)((im_shr(m[r], (uint32_t)(eT - (int)(e[r] & 0xfffu) + 67)) + 1ull) >> 1);
                if ((int)e[r] < 0) F = -F;
                const int hi = (int)((F + (1 << 28)) >> 29);
                S.CF[i] = make_int2(hi, (int)(F - (long long)hi * (1 << 29)));
            }
        } else if (i == nS && (nS & 1)) {
            S.CF[i] = make_int2(0, 0);
        }
    }
    if (grp.sync_any(!in)) {
        int_general<NR, G, AT_T>(M, I, S, c, rho, invCtot * s, out, lane, grp);
        return;
    }
    if constexpr (AT_T) {
        if (scale < 0) scale = grp.imax(int_first_scale(M, S, rk, mix, lane, G));
    }
    im_u128 acc[NR];
    for (;;) {
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] = im_u128{0ull, 0ull};
        int emax = 0;
        bool over = false, under = false;
        auto store = [&](im_u64 Q, uint32_t e, int at) {
            const int x = (int)(e & 0x7fffffffu);
            if (Q) emax = max(emax, x);
            im_u128 v = im_place(Q, x - scale + M.imUp);
            if (e >> 31) {
                im_u128 z{0ull, 0ull};
                im_sub(z, v.lo, v.hi);
                v = z;
            }
            S.OM[at] = make_ulonglong2(v.lo, v.hi);
        };
        // the lane's reactions follow each other through the chunks, so the
        // next one's words are on their way while this one is formed
        uint32_t wn = 0;
        double kn = 0.0, bn = 0.0, en0 = 0.0;
        auto fetch = [&](int q) {
            wn = M.rxw[q];
            if constexpr (AT_T) {
                kn = M.arr[q];
                bn = M.arr[nR + q];
                en0 = M.arr[2 * nR + q];
            } else {
                kn = rk.K[q];
            }
        };
        if (lane < nR) fetch(lane);
#pragma unroll 1
        for (int ch = 0, q0 = 0; ch < I.nchunk; ++ch, q0 += I.chunk) {
            const int q1 = min(nR, q0 + I.chunk);
#pragma unroll 1
            for (int q = q0 + lane; q < q1; q += G) {
                const uint32_t w = wn;
                const double kq = kn, bq = bn, eq = en0;
                if (q + G < nR) fetch(q + G);
                im_u64 Q;
                uint32_t e;
                if (!int_rate<AT_T, true>(M, S, rk, mix, q, w, kq, bq, eq, Q, e)) emax = IM_OUT;
                store(Q, e, q - q0);
            }
            // the run's first entries, fetched ahead of the barrier
            const int k0 = I.step0[ch], K = I.step0[ch + 1] - k0;
            const uint32_t* __restrict__ ent = I.ent + (int64_t)k0 * G + lane;
            ulonglong2* P = S.P + I.slot0[ch * G + lane];
            int part[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) part[r] = lane + G * r < nS ? I.part[ch * nS + lane + G * r] : 0;
            uint32_t en[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) en[j] = j < K ? ent[G * j] : (uint32_t)I.chunk;
            over = grp.sync_any(emax > scale + IM_GUARD);
            im_u128 w{0ull, 0ull};
#pragma unroll 1
            for (int k = 0; k < K; k += 4) {
                uint32_t e[4];
                ulonglong2 v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    e[j] = en[j];
                    v[j] = S.OM[e[j] & INT_POS_MASK];
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) en[j] = k + 4 + j < K ? ent[G * (k + 4 + j)] : (uint32_t)I.chunk;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    im_add(w, v[j].x, v[j].y);
                    if (e[j] & INT_FLUSH) {
                        *P++ = make_ulonglong2(w.lo, w.hi);
                        w = im_u128{0ull, 0ull};
                    }
                }
            }
            under = !grp.sync_any(emax >= scale - IM_SLACK);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const ulonglong2* p = S.P + (part[r] >> 16);
                const int np = (part[r] >> 8) & 0xff, n = np + (part[r] & 0xff);
#pragma unroll 1
                for (int k = 0; k < n; ++k) {
                    const ulonglong2 v = p[k];
                    if (k < np) im_add(acc[r], v.x, v.y);
                    else im_sub(acc[r], v.x, v.y);
                }
            }
        }
        if (!over && !under) {
            unsigned left = 0u;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int i = lane + G * r;
                out[r] = 0.0;
                if (i >= nS) continue;
                const im_u64 w = M.imW[i].y;  // 0: no reaction changes the species
                // a word's unit at e = scale: 2^(128 + scale - 2 * 64 - 3 IM_BIAS - imUp)
                if (w && im_short(acc[r], M.imShort)) left |= 1u << r;
                out[r] = im_scaled(acc[r], scale - M.imUp - 3 * IM_BIAS, w, M.imWe[i].y, mix.mr, (int)mix.er);
            }
            // (the shared words are rewritten after this barrier)
            if (grp.sync_any(left != 0u)) int_short<NR, G, AT_T>(M, I, S, left, out, lane, grp);
            return;
        }
        emax = grp.imax(emax);
        if (emax >= IM_OUT) {  // a falloff factor that is not finite
            int_general<NR, G, AT_T>(M, I, S, c, rho, invCtot * s, out, lane, grp);
            return;
        }
        scale = emax;
    }
}

// Element r of a register vector for a warp-uniform r.
template <int NR>
__device__ __forceinline__ double reg_get(const double (&v)[NR], int r)
{
    double o = v[0];
#pragma unroll
    for (int q = 1; q < NR; ++q)
        if (r == q) o = v[q];
    return o;
}

// Rate constants' source at T.
__device__ __forceinline__ RateSource rates_at(const MechDev& M, double T, double invT)
{
    return RateSource{nullptr, T >= 1.0 && T < 65536.0 ? im_log(M.lnc, T) : log(T), invT};
}

// f with the energy equation (Eqs. (E:mass), (E:energy)) for the group's cell:
// state component nS is T. pR = p / R and its reciprocal in mol K / cm^3. The
// species' enthalpies and heat capacities per mass multiply the species' own
// rates: dT/dt = -(sum_i (Hf_i + cp_i (T - T_REF)) / W_i dY_i/dt) / sum_i Y_i cp_i / W_i.
template <int NR, int G>
__device__ __forceinline__ void warp_feval_int_energy(const MechDev& M, const IntDev& I, const IntSmem& S, double pR,
                                                      double invpR, int& scale, const double (&x)[NR],
                                                      double (&out)[NR], int lane, Group<G>& grp)
{
    const int nS = M.nS;
    const double T = grp.from(reg_get(x, nS / G), nS % G), invT = Tab<double>::inv(T);
    warp_feval_int<NR, G, true>(M, I, S, rates_at(M, T, invT), true, pR * invT, invpR * T, scale, x, out, lane, grp);
    const double dT = T - T_REF;
    double h[NR], c[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int i = lane + G * r;
        h[r] = c[r] = 0.0;
        if (i < nS) {
            const double w = M.cpW[i];
            h[r] = __dmul_rn(fma(w, dT, M.HfW[i]), out[r]);
            c[r] = __dmul_rn(x[r], w);
        }
    }
    const double hw = grp.sum(h), cpm = grp.sum(c);
    const double dTdt = quot(-hw, cpm);
#pragma unroll
    for (int r = 0; r < NR; ++r)
        if (lane + G * r == nS) out[r] = dTdt;
}

}  // namespace kin
