// int_tables.h -- host tables of the warp layout's FP64 f in integer arithmetic
// (plain C++, no CUDA: the library builds them at mechanism upload, and a CPU
// test compiles this header on its own to check them).
//
// Gather (Eq. (E:spec-rate), omega_i = sum_j nu_ij Omega_j): the rates of
// progress are 128-bit fixed-point words in shared memory, CHUNK reactions at
// a time, and omega_i is a sum of such words. Species i has two rows, 2 i for
// its positive and 2 i + 1 for its negative coefficients, so that every entry
// counts once (a coefficient of 2 is two entries) and the inner loop only adds.
// Within a chunk the entries, row by row, are cut into G equal runs of
// K = ceil(n / G), one per lane (G lanes evaluate f for one cell); a lane
// writes one partial sum per row it touches (a "flush") into consecutive
// slots, and the species' owner adds the slots of its positive row and
// subtracts those of its negative one, which follow them. Integer sums are
// exact, so their order does not matter.
//
// An entry is a 32-bit word: the reaction's place in the chunk, and bit 16 set
// where the lane flushes after it. Padding entries name the place after the
// last, which holds zero. The
// entries of a run that belong to one row are ordered so that the eight lanes
// of a 128-byte wavefront read words in distinct 16-byte banks where they can
// (bank = place mod 8).
//
// Third-body sums (Eq. (E:rxn-rate), [M] = sum_k eff_k C_k): a row's
// efficiencies as integers eff_k 2^(58 - x), x the exponent of the row's
// largest, cut into 30 high and 29 low bits (int_eff_limbs).
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

namespace kin {

constexpr uint32_t INT_POS_MASK = 0xffffu;
constexpr uint32_t INT_FLUSH = 0x10000u;

struct IntGather {
    int nchunk = 0, chunk = 0;
    int nslots = 0;                 // partial-sum slots of the fullest chunk
    std::vector<int32_t> step0;     // [nchunk + 1] first step of each chunk
    std::vector<uint32_t> ent;      // [steps][G] entries
    std::vector<int32_t> slot0;     // [nchunk][G] first slot of each lane
    std::vector<int32_t> part;      // [nchunk][nS] first slot << 16 | positive slots << 8 | negative slots
};

// ptr/pos/nu: species-major rows of net coefficients; pos is the reaction's
// permuted position, nu an integer in -2..2.
inline IntGather build_int_gather(int nS, int nR, const int* ptr, const int* pos, const double* nu,
                                  int chunk, int G)
{
    IntGather t;
    t.chunk = chunk;
    t.nchunk = (nR + chunk - 1) / chunk;
    t.step0.assign(1, 0);
    std::vector<std::vector<std::vector<int>>> rows(t.nchunk, std::vector<std::vector<int>>(2 * nS));
    for (int i = 0; i < nS; ++i)
        for (int e = ptr[i]; e < ptr[i + 1]; ++e) {
            const int c = pos[e] / chunk, at = pos[e] % chunk, n = (int)std::abs(nu[e]);
            for (int k = 0; k < n; ++k) rows[c][2 * i + (nu[e] < 0.0)].push_back(at);
        }
    for (int c = 0; c < t.nchunk; ++c) {
        int n = 0;
        for (auto& r : rows[c]) n += (int)r.size();
        const int K = (n + G - 1) / G, base = (int)t.ent.size();
        t.step0.push_back(t.step0.back() + K);
        t.ent.resize(base + (size_t)K * G, (uint32_t)chunk);
        std::vector<int32_t> part(nS, 0), slot0(G, 0);
        struct Seg { std::vector<int> left; };
        std::vector<std::vector<Seg>> lane(G);
        int row = 0, at = 0, slots = 0;
        for (int l = 0; l < G; ++l) {
            slot0[l] = slots;
            for (int room = K; room > 0 && row < 2 * nS;) {
                const int have = (int)rows[c][row].size() - at;
                if (have == 0) { ++row; at = 0; continue; }
                const int take = std::min(room, have);
                if (part[row / 2] == 0) part[row / 2] = slots << 16;
                part[row / 2] += row % 2 ? 1 : 1 << 8;
                ++slots;
                lane[l].push_back(Seg{{rows[c][row].begin() + at, rows[c][row].begin() + at + take}});
                at += take;
                room -= take;
            }
        }
        t.nslots = std::max(t.nslots, slots);
        std::vector<size_t> cur(G, 0);
        for (int k = 0; k < K; ++k) {
            std::vector<int> used(8 * ((G + 7) / 8), 0);
            for (int l = 0; l < G; ++l) {
                if (cur[l] >= lane[l].size()) continue;
                std::vector<int>& L = lane[l][cur[l]].left;
                int* u = &used[8 * (l / 8)];
                size_t best = 0;
                for (size_t q = 1; q < L.size(); ++q)
                    if (u[L[q] % 8] < u[L[best] % 8]) best = q;
                const int p = L[best];
                L.erase(L.begin() + best);
                u[p % 8]++;
                t.ent[base + (size_t)k * G + l] = (uint32_t)p | (L.empty() ? INT_FLUSH : 0u);
                if (L.empty()) ++cur[l];
            }
        }
        t.slot0.insert(t.slot0.end(), slot0.begin(), slot0.end());
        t.part.insert(t.part.end(), part.begin(), part.end());
    }
    return t;
}

// How far up the largest rate's word is shifted, and how many bits a sum needs
// for its last place to be worth an ulp (intf.cuh), for species-major rows whose
// longest counts n entries: n words below 2^(61 + up + 8) stay below 2^127, and n
// units below the sum's 53rd bit. Up to 55 bits, so that a word's shift stays
// below 64.
inline void int_word_bits(int nS, const int* ptr, const double* nu, int* up, int* enough)
{
    int n = 1, bits = 0;
    for (int i = 0; i < nS; ++i) {
        int c = 0;
        for (int e = ptr[i]; e < ptr[i + 1]; ++e) c += (int)std::abs(nu[e]);
        n = std::max(n, c);
    }
    while (n >> bits) ++bits;
    *up = std::min(55, 58 - bits);
    *enough = 53 + bits;
}

// 63-bit left-aligned mantissa of v > 0 and its exponent as in a double.
inline uint64_t int_split(long double v, int* e)
{
    int x = 0;
    const long double f = frexpl(v, &x);  // v = f 2^x, f in [1/2, 1)
    uint64_t m = (uint64_t)llroundl(ldexpl(f, 62)) << 1;
    if (m == 1ull << 63) {
        m >>= 1;
        ++x;
    }
    *e = x - 1 + 1023;
    return m;
}

// The tables of im_exp and im_log (intf.cuh).
inline void int_exp_log_tables(uint64_t* ex2, uint64_t* lnc)
{
    for (int i = 0; i < 64; ++i) {
        ex2[i] = (uint64_t)llroundl(ldexpl(exp2l(i / 64.0L), 61)) << 1;
        // far enough above for m c_i >= 1 after the product's truncation
        const uint64_t c = (uint64_t)ceill(ldexpl(64.0L / (64 + i), 62)) + 16;
        lnc[2 * i] = c;
        lnc[2 * i + 1] = (uint64_t)llroundl(ldexpl(-logl(ldexpl((long double)c, -62)), 59));
    }
}

// A row's efficiencies as 55-bit integers: hi (30 bits, signed) and lo (25
// bits) of round(eff 2^(54 - x)). Returns x.
inline int int_efficiencies(int nS, const double* eff, int32_t* hi, int32_t* lo)
{
    double top = 0.0;
    for (int k = 0; k < nS; ++k) top = std::max(top, std::fabs(eff[k]));
    int x = 0;
    if (top > 0.0) std::frexp(top, &x), --x;
    if (nS > 128) ++x;
    for (int k = 0; k < nS; ++k) {
        const int64_t E = (int64_t)std::nearbyint(std::ldexp(eff[k], 54 - x));
        hi[k] = (int32_t)(E >> 25);
        lo[k] = (int32_t)(E & ((1 << 25) - 1));
    }
    return x;
}

// A reaction's entry of the estimate of a cell's largest rate (int_first_scale of
// warp_int.cuh): three floats, whose sum with weights 1, ln T and -1 / T is the
// rate's exponent word (a double's exponent) without the concentrations' two (and
// the third body's eT), and reactants (0: none) | power of rho + 2 << 20 | third body << 23.
// row: the exponent of its largest efficiency.
inline void int_scale_table(double lnA, double beta, double EaR, const int32_t* reac, int type, int row, uint32_t* out)
{
    const double log2e = 1.4426950408889634;
    const float f[3] = {(float)(lnA * log2e + 1023 + (type == 1 ? row - 1021 : 0)), (float)(beta * log2e),
                        (float)(EaR * log2e)};
    std::memcpy(out, f, sizeof(f));
    const int power = (reac[0] >= 0) + (reac[1] >= 0) + (type == 1) - 2;
    out[3] = (uint32_t)(reac[0] + 1) | (uint32_t)(reac[1] + 1) << 10 | (uint32_t)(power + 2) << 20 | (type == 1 ? 1u << 23 : 0u);
}

// The same in 59 bits, round(eff 2^(58 - x)), as the kernels take them: hi (30
// bits) and lo (29 bits, signed and rounded to nearest, so that the products
// lo lo that they leave out are small and of either sign). Every efficiency down to
// 2^-6 of the row's largest is exact. hi and lo come from int_efficiencies,
// `stride` apart.
inline void int_eff_limbs(int nS, const double* eff, int x, int stride, int32_t* hi, int32_t* lo)
{
    for (int k = 0; k < nS; ++k) {
        const int64_t c = (int64_t)hi[stride * k] * (1 << 25) + lo[stride * k];
        const int64_t E = 16 * c + (int64_t)std::nearbyint(16.0 * (std::ldexp(eff[k], 54 - x) - (double)c));
        hi[stride * k] = (int32_t)((E + (1 << 28)) >> 29);
        lo[stride * k] = (int32_t)(E - (int64_t)hi[stride * k] * (1 << 29));
    }
}

// Tables of the lane layout's f (lane_int.cuh): its reactions in the order
// third bodies first, without those that change nothing.
struct LaneInt {
    int n = 0, tb = 0;
    std::vector<uint32_t> rx;               // [n + 1][4] records
    std::vector<int32_t> eff;               // [tb][nS][2] integer efficiencies
    std::vector<int32_t> effx;              // [tb]
    std::vector<int32_t> row;               // [tb] efficiency rows in reaction order
};

// type: 0 plain, 1 third body, 2 falloff; eff: one row per non-plain reaction,
// in reaction order.
inline LaneInt build_lane_int(int nS, int nR, const int32_t* reac, const int32_t* prod,
                              const int8_t* type, const double* eff)
{
    LaneInt t;
    for (int pass = 0; pass < 2; ++pass) {
        int row = 0, fo = 0;
        for (int j = 0; j < nR; ++j) {
            const int ty = type[j], r = ty ? row++ : -1, f = ty == 2 ? fo++ : 0;
            if ((ty == 0) != (pass == 1)) continue;
            // net coefficients by species
            int sp[4], c[4], m = 0, order = 0;
            for (int k = 0; k < 4; ++k) {
                const int s = k < 2 ? prod[2 * j + k] : reac[2 * j + k - 2];
                if (s < 0) continue;
                order += k >= 2;
                int a = 0;
                while (a < m && sp[a] != s) ++a;
                if (a == m) {
                    sp[m] = s;
                    c[m++] = 0;
                }
                c[a] += k < 2 ? 1 : -1;
            }
            uint32_t slot[4] = {(uint32_t)nS, (uint32_t)nS, (uint32_t)nS, (uint32_t)nS}, flags = 0;  // p0 p1 n0 n1
            int np = 0, nn = 0;
            for (int a = 0; a < m; ++a) {
                if (c[a] == 0) continue;
                const int at = c[a] > 0 ? np++ : 2 + nn++;
                slot[at] = (uint32_t)sp[a];
                if (c[a] == 2 || c[a] == -2) flags |= 1u << (16 + at);
            }
            if (np + nn == 0) continue;
            const uint32_t ra = reac[2 * j] < 0 ? nS : reac[2 * j], rb = reac[2 * j + 1] < 0 ? nS : reac[2 * j + 1];
            const int power = order + (ty == 1) - 2;  // of rho, beyond a plain reaction of two
            t.rx.push_back(ra | rb << 8 | slot[0] << 16 | slot[1] << 24);
            t.rx.push_back(slot[2] | slot[3] << 8 | flags | (uint32_t)(power + 2) << 20 | (ty == 2 ? 1u << 23 : 0u));
            t.rx.push_back((uint32_t)j);
            t.rx.push_back((uint32_t)f);
            ++t.n;
            if (ty) {
                ++t.tb;
                t.row.push_back(r);
                std::vector<int32_t> hi(nS), lo(nS);
                t.effx.push_back(int_efficiencies(nS, eff + (size_t)r * nS, hi.data(), lo.data()));
                for (int k = 0; k < nS; ++k) {
                    t.eff.push_back(hi[k]);
                    t.eff.push_back(lo[k]);
                }
            }
        }
    }
    for (int k = 0; k < 4; ++k) t.rx.push_back(t.n ? t.rx[4 * (t.n - 1) + k] : 0u);
    return t;
}

}  // namespace kin
