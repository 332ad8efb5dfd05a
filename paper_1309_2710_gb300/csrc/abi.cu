// abi.cu -- host side of the C ABI declared in include/kin.h: argument
// validation, mechanism packing and upload, workspace sizing, launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <climits>
#include <cstring>
#include <string>
#include <vector>

#include "codegen.h"
#include "int_tables.h"
#include "kin_dev.cuh"
#include "seg_tables.h"

using namespace kin;

struct kin_mech {
    MechDev dev;  // device pointers into `buf`
    void* buf;
    int device;
    int nS, nR, nM;
    bool thermo;          // cp and Hf given (energy equation available)
    std::string gen_src;  // the generated f (empty when the mechanism is too large for it)
};

namespace {

thread_local char g_err[512] = "";

int fail(int code, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

int cuda_fail(cudaError_t e, const char* what)
{
    return fail(KIN_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

// Device pointer check: the pointer must be device (or managed) memory.
bool is_device_ptr(const void* p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

struct Grid {
    int threads, blocks;  // persistent grid
    int64_t nslots;
    int layout;           // KIN_LAYOUT_LANE or KIN_LAYOUT_WARP (resolved)
    int lanes;            // lanes per cell (1 in the lane layout)
    int occupancy;        // register budget (resolved)
};

// Automatic layout: one warp per cell for large mechanisms (a lane's working
// set would stream from memory) and for calls too small to give every lane of
// the GPU a cell; one lane per cell otherwise. `full`: without the rule below.
int resolve_layout(const kin_mech* m, const kin_opts* o, int64_t cells, int nsm, bool full = true)
{
    if (o->layout != KIN_LAYOUT_AUTO) return o->layout;
    if (m->nR > KIN_WARP_MIN_REACTIONS) return KIN_LAYOUT_WARP;
    if (cells < (int64_t)KIN_WARP_MAX_CELLS_PER_SM * nsm) return KIN_LAYOUT_WARP;
    // FP64 on small mechanisms: the warp layout's integer f beats a lane per cell
    // until the cells fill the GPU's lanes (about 78,000; half of them for RKCK, whose
    // cells take equal times), and at any size where a cell's work fills its
    // group's lanes. Cells per SM up to which it does, from runs at 10,000 to
    // 262,144 cells on GB300, warp against lane in ms:
    //   up to 16 components, by reactions. RKC: 5 / 8, 10,000 cells 0.23 against 0.19,
    //     20,000 0.33 against 0.22;
    //     10 / 12, 40,000 1.44 against 2.15, 71,000 2.4 against 2.3; 13 / 54, 20,000 3.1
    //     against 11, 262,144 35 against 26 (integer f of the lane layout). RKCK: 10 /
    //     12, 20,000 0.24 against 0.20; 14 / 20, 20,000 0.27 against 0.29, 40,000 0.46
    //     against 0.34; 9 / 38, 20,000 0.56 against 0.87, 40,000 1.01 against 0.99.
    //     Energy equation, RKC: 5 / 8, 20,000 0.39 against 0.31; 10 / 12 131,072 6.5
    //     against 6.7, 262,144 12.7 against 9.4; 9 / 38, 262,144 131 against 224.
    //     RKCK: 10 / 12, 20,000 0.32 against 0.30; 14 / 20, 40,000 0.60 against 0.59;
    //     9 / 38, 262,144 9.6 against 10.3.
    //   17 to 32 components, RKC, by reactions + 2 species: 17 / 20, 40,000 16.5
    //     against 19.3, 71,000 29 against 21; 20 / 90, 71,000 36 against 42, 131,072 66
    //     against 56; 28 / 90, 131,072 19.8 against 20.7, 262,144 39 against 36; 32 / 100,
    //     262,144 376 against 387; 24 / 150 578 against 836. Energy equation: 20 / 30,
    //     50,000 7.1 against 9.4, 131,072 18 against 15; 24 / 60, 131,072 16.8 against
    //     17.0; 24 / 100, 262,144 1065 against 1537.
    // A call that names a shape or form of the lane layout keeps it.
    const bool free_shape = o->block_threads == 0 && o->blocks_per_sm == 0 && o->staging == KIN_STAGE_GLOBAL &&
                            o->occupancy == KIN_OCC_DEFAULT && o->feval == KIN_FEVAL_AUTO;
    const int nV = m->nS + o->energy, nR = m->nR, any = INT_MAX;
    if (!full || !free_shape || o->precision != KIN_FP64 || nV > 32) return KIN_LAYOUT_LANE;
    const bool rkc = o->method == KIN_RKC, en = o->energy != 0;
    int most = KIN_WARP_MAX_CELLS_PER_SM;  // cells per SM
    if (nV > 16) {
        const int work = nR + 2 * m->nS;
        if (rkc) most = work < 100 ? 330 : work < 135 ? (en ? 800 : 400) : work < 160 && !en ? 600 : any;
    } else if (nR >= 30) {
        most = en ? any : rkc ? KIN_WARP_RKC_MAX_CELLS_PER_SM : KIN_WARP_RKCK_MAX_CELLS_PER_SM;
    } else if (nR >= 16) {
        most = rkc ? (en ? 860 : KIN_WARP_RKC_MAX_CELLS_PER_SM) : en ? 260 : 150;
    } else if (nR >= 10) {
        most = rkc ? (en ? 860 : KIN_WARP_RKC_MAX_CELLS_PER_SM) : en ? 100 : 70;
    } else if (rkc && !en) {
        most = 100;
    }
    return most == any || cells < (int64_t)most * nsm ? KIN_LAYOUT_WARP : KIN_LAYOUT_LANE;
}

// The mechanism as the small register budget's FP64 kernels see it.
MechDev small_chunks(const MechDev& d)
{
    MechDev s = d;
    if (d.ig[INT_G16S].ent) s.ig[INT_G16] = d.ig[INT_G16S];
    if (d.ig[INT_G32S].ent) s.ig[INT_G32] = d.ig[INT_G32S];
    return s;
}

// Lanes that integrate one cell in the warp layout: half a warp for states of
// at most 16 components (RKCK; RKC in FP64), of which FP64 calls of up to 8
// cells per SM take a whole one (9 species RKCK, 64 cells 0.348 ms with half a
// warp, 0.295 with a whole one; 13 species RKC, 1,000 cells 3.57 and 3.05) and
// FP64 RKC above 64 cells per SM a quarter (13 species, 4,000 cells 4.0 ms with 16 lanes and 5.6 with 8, 16,000
// cells 9.8 and 8.6, 30,000 cells 17.9 and 14.6); else a warp, and in FP64 RKC
// two warps above 32 components and four above 64. An evaluation is a chain of short phases, so more lanes shorten it, and the
// FP64 pipe's vector work per cell stays the same (fewer slots per lane on more
// warps). Measured on GB300, 2 or 4 warps against 1: 53 species, 256 / 4,096 /
// 20,000 cells 10.4 against 18.9, 37.7 against 43.9, 157.9 against 159.4 ms;
// 111 species, 200 / 8,000 cells 42 against 175, 231 against 323 ms. One warp
// where the block size does not hold whole groups, and with the small register
// budget, whose kernels exist for single warps.
int cell_lanes(const kin_opts* o, int occupancy, int nV, int threads, int64_t cells, int nsm)
{
    const bool int_f = o->precision == KIN_FP64, f64 = int_f && o->method == KIN_RKC;
    if (nV <= 16 && int_f && !occupancy && cells <= 8 * (int64_t)nsm) return 32;
    if (nV <= 16 && f64 && !occupancy && cells > (int64_t)KIN_WARP_MAX_CELLS_PER_SM * nsm) return 8;
    if (nV <= 16) return o->method == KIN_RKCK || f64 ? 16 : 32;
    if (!f64 || occupancy || nV <= 32) return 32;
    const int g = nV <= 64 ? 64 : 128;
    return threads % g ? 32 : g;
}

int grid_for(const kin_mech* m, const kin_opts* o, int64_t cells, Grid* g)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev != m->device) return fail(KIN_EINVAL, "mechanism lives on device %d, current device is %d", m->device, dev);
    int nsm = 0;
    e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    int maxsm = 0;
    e = cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    if (o->energy && !m->thermo)
        return fail(KIN_EUNSUPPORTED, "the energy equation needs the mechanism's cp and Hf");
    const int layout = resolve_layout(m, o, cells, nsm);
    int threads = o->block_threads > 0 ? o->block_threads : 128;
    int occ = 0, cap = 0, lanes = 1, budget = o->occupancy;
    if (layout == KIN_LAYOUT_WARP) {
        if (threads % 32 != 0 || threads > 256) return fail(KIN_EINVAL, "block_threads must be a multiple of 32 and <= 256");
        // The small register budget does not serve the FP64 f, which spills at it
        // (GB300, RKC, default against KIN_OCC_HIGH with it: 13 species, 64 / 1,000 /
        // 9,000 cells 2.5 against 4.9, 3.2 against 5.8, 6.2 against 9.3 ms; 24 species,
        // 8,000 cells 20.9 against 22.2; 53 species, 8,000 / 20,000 cells 15.0
        // against 18.7, 90 against 101): it is left to calls that name more blocks per
        // SM than the other holds.
        if (o->precision == KIN_FP64 && o->method == KIN_RKC && budget != KIN_OCC_DEFAULT) {
            kin_opts d = *o;
            d.occupancy = KIN_OCC_DEFAULT;
            d.blocks_per_sm = 0;
            d.layout = KIN_LAYOUT_WARP;
            Grid gd;
            if (grid_for(m, &d, cells, &gd) == KIN_OK && o->blocks_per_sm <= gd.blocks / nsm) budget = KIN_OCC_DEFAULT;
            g_err[0] = 0;
        }
        lanes = cell_lanes(o, budget, m->nS + o->energy, threads, cells, nsm);
        // the layout's limit on a mechanism: C and Omega of a block's cells in
        // shared memory, at half a warp or a warp per cell (the FP64 f's own words
        // need no more: a group's chunk of a large mechanism takes 2 to 5 KB)
        const size_t sm = (size_t)((m->nS + m->nR + 3) & ~3) * 8 * (threads / (o->method == KIN_RKCK && lanes < 32 ? 16 : 32));
        if (sm > (size_t)maxsm)
            return fail(KIN_EUNSUPPORTED, "warp layout needs %zu bytes of shared memory per block (max %d)", sm, maxsm);
        const int nV = m->nS + o->energy;
        if (o->method == KIN_RKCK) {
            e = o->precision == KIN_MIXED ? occ_warp_rkck_f32(m->dev, nV, lanes, o->energy, threads, &occ)
                                          : occ_warp_rkck_f64(m->dev, nV, lanes, o->energy, threads, &occ);
        } else {
            using OccFn = cudaError_t (*)(const MechDev&, int, int, int, int*);
            // [energy][precision][occupancy]
            static const OccFn fns[2][2][2] = {
                {{occ_warp_f64_o0, occ_warp_f64_o1}, {occ_warp_f32_o0, occ_warp_f32_o1}},
                {{occ_warp_f64_en_o0, occ_warp_f64_en_o1}, {occ_warp_f32_en_o0, occ_warp_f32_en_o1}}};
            e = fns[o->energy][o->precision == KIN_MIXED][budget ? 1 : 0](budget ? small_chunks(m->dev) : m->dev, nV, lanes,
                                                                          threads, &occ);
        }
        cap = occ;  // as many as fit
    } else {
        if (threads % 32 != 0 || threads > 128) return fail(KIN_EINVAL, "block_threads must be a multiple of 32 and <= 128");
        const int stg = o->energy ? KIN_STAGE_GLOBAL : o->staging;  // energy: nothing to stage
        if (stg > 0 && smem_bytes(m->dev, o->precision, threads, stg) > (size_t)maxsm)
            return fail(KIN_EUNSUPPORTED, "shared-memory staging needs %zu bytes per block (max %d)",
                        smem_bytes(m->dev, o->precision, threads, stg), maxsm);
        e = integrate_occupancy(m->dev, o->method, o->precision, stg, o->occupancy, o->energy, threads,
                                &occ);
        cap = (o->occupancy ? 768 : 512) / threads;
    }
    if (e != cudaSuccess) return cuda_fail(e, "occupancy query");
    if (occ < 1) return fail(KIN_EUNSUPPORTED, "kernel does not fit on an SM with these options");
    int bps = o->blocks_per_sm;
    if (bps <= 0) bps = std::max(1, std::min(occ, cap));
    if (bps > occ) return fail(KIN_EINVAL, "blocks_per_sm %d exceeds the %d blocks that fit per SM", bps, occ);
    g->threads = threads;
    g->blocks = nsm * bps;
    g->nslots = (int64_t)g->blocks * threads;
    g->layout = layout;
    g->lanes = lanes;
    g->occupancy = budget;
    return KIN_OK;
}

// Blocks of a lane-layout call's persistent grid that run the integer FP64 f,
// or 0 where it does not serve: a layout or f evaluation asked for, mixed
// precision, the energy equation, staged arrays, a mechanism beyond its tables,
// or fewer than LANE_INT_MIN_LANES lanes per SM, asked for or left by its shared
// words. Its lanes wait on their own
// chains, so it needs them: GB300, 13 species RKC, 262,144 cells at 512 and
// 384 lanes per SM 97 and 116 ms, the generated f 122 and 123; 9 species RKCK,
// 400,000 cells at 512 lanes 21.4 against 24.9; 20 species RKCK, 150,000 cells
// at 384 lanes 1.53 against 1.34.
int lane_int_blocks(const kin_mech* m, const kin_opts* o, const Grid& g, int* blocks)
{
    *blocks = 0;
    if (g.layout != KIN_LAYOUT_LANE || o->layout != KIN_LAYOUT_AUTO || o->feval != KIN_FEVAL_AUTO) return KIN_OK;
    if (!m->dev.li_rx || o->precision != KIN_FP64 || o->energy || o->staging != KIN_STAGE_GLOBAL) return KIN_OK;
    int nsm = 0, bps = 0;
    cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    e = occ_lane_int(m->dev, o->method, o->occupancy, g.threads, &bps);
    if (e != cudaSuccess) return cuda_fail(e, "occupancy query");
    bps = std::min(bps, g.blocks / nsm);
    if (bps * g.threads >= LANE_INT_MIN_LANES) *blocks = bps * nsm;
    return KIN_OK;
}

// Workspace bytes; the warp layout keeps no per-lane arrays.
int64_t ws_bytes(const kin_mech* m, const kin_opts* o, const Grid& g, int64_t cells)
{
    const int sig = o->method == KIN_RKC ? o->sigma : KIN_SIGMA_GERSHGORIN;
    return ws_layout(m->dev, o->precision, sig, o->energy, g.layout == KIN_LAYOUT_WARP ? 0 : g.nslots,
                     cells).total;
}

int check_opts(const kin_opts* o)
{
    if (!o) return fail(KIN_EINVAL, "opts is NULL");
    if (o->method != KIN_RKCK && o->method != KIN_RKC) return fail(KIN_EINVAL, "unknown method %d", o->method);
    if (o->precision != KIN_FP64 && o->precision != KIN_MIXED)
        return fail(KIN_EINVAL, "unknown precision %d", o->precision);
    if (o->staging != KIN_STAGE_GLOBAL && o->staging != KIN_STAGE_SHARED &&
        o->staging != KIN_STAGE_SHARED_ALL)
        return fail(KIN_EINVAL, "unknown staging %d", o->staging);
    if (o->occupancy != KIN_OCC_DEFAULT && o->occupancy != KIN_OCC_HIGH)
        return fail(KIN_EINVAL, "unknown occupancy %d", o->occupancy);
    if (o->sigma != KIN_SIGMA_GERSHGORIN && o->sigma != KIN_SIGMA_POWER)
        return fail(KIN_EINVAL, "unknown sigma estimator %d", o->sigma);
    if (o->layout != KIN_LAYOUT_AUTO && o->layout != KIN_LAYOUT_LANE && o->layout != KIN_LAYOUT_WARP)
        return fail(KIN_EINVAL, "unknown layout %d", o->layout);
    if (o->energy != 0 && o->energy != 1) return fail(KIN_EINVAL, "energy must be 0 or 1");
    if (o->feval != KIN_FEVAL_AUTO && o->feval != KIN_FEVAL_TABLE && o->feval != KIN_FEVAL_GENERATED)
        return fail(KIN_EINVAL, "unknown feval %d", o->feval);
    return KIN_OK;
}

bool finite_pos(double x) { return std::isfinite(x) && x > 0.0; }

}  // namespace

int kin::set_last_error(int code, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

int kin::noalloc_opts(const kin_mech* m, const kin_opts* in, int64_t cells, int64_t cap,
                      kin_opts* out)
{
    g_err[0] = 0;
    if (!m) return fail(KIN_EINVAL, "mechanism is NULL");
    if (cells < 0) return fail(KIN_EINVAL, "cells < 0");
    int rc = check_opts(in);
    if (rc) return rc;
    kin_opts o = *in;
    // the layout of kin_integrate's choice; its cells have to fit the array in
    // the lane layout too where only the f evaluation and the launch shape,
    // left to the library, make it the warp layout
    int nsm = 1;
    cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    o.layout = resolve_layout(m, in, cells, nsm);
    const int limit = resolve_layout(m, in, cells, nsm, false);
    // Never compile here: NVRTC and loading the compiled library allocate
    // device memory. The generated f runs only where an earlier call loaded
    // it on this device; otherwise the automatic choice falls back to the
    // tables and a forced one is refused.
    if (o.feval != KIN_FEVAL_TABLE && (m->gen_src.empty() || !gen_loaded(m->device, m->gen_src))) {
        if (o.feval == KIN_FEVAL_GENERATED)
            return fail(KIN_EUNSUPPORTED,
                        "kin_integrate_noalloc: the generated f of this mechanism is not loaded on "
                        "device %d (a kin_integrate call with KIN_FEVAL_GENERATED compiles and loads "
                        "it, which allocates)", m->device);
        o.feval = KIN_FEVAL_TABLE;
    }
    Grid g;
    rc = grid_for(m, &o, cells, &g);  // resolves blocks_per_sm = 0 to "as many as fit"
    if (rc) return rc;
    int64_t need = 0;
    if (limit != o.layout) {
        kin_opts l = o;
        l.layout = limit;
        l.blocks_per_sm = 1;
        Grid gl;
        rc = grid_for(m, &l, cells, &gl);
        if (rc) return rc;
        need = ws_bytes(m, &l, gl, cells);
    }
    for (int bps = need > cap ? 0 : g.blocks / nsm; bps >= 1; --bps) {
        o.blocks_per_sm = bps;
        rc = grid_for(m, &o, cells, &g);
        if (rc) return rc;
        need = ws_bytes(m, &o, g, cells);
        if (need <= cap) {
            // kin_integrate's integer f where it serves, which compiles nothing:
            // a call whose layout is left to the library and that names its
            // blocks takes the lane layout again
            kin_opts a = o;
            a.layout = in->layout;
            a.feval = in->feval;
            int li_blocks = 0;
            rc = lane_int_blocks(m, &a, g, &li_blocks);
            if (rc) return rc;
            *out = li_blocks ? a : o;
            return KIN_OK;
        }
    }
    return fail(KIN_ENOMEM,
                "kin_integrate_noalloc: %lld cells need %lld bytes of working memory even at one "
                "block per SM, more than the %lld-byte fixed array",
                (long long)cells, (long long)need, (long long)cap);
}

extern "C" {

const char* kin_last_error(void) { return g_err; }

const char* kin_version(void) { return "kin 0.3 (sm_103a)"; }

int64_t kin_generated_f_source(const kin_mech_desc* d, char* buf, int64_t cap)
{
    g_err[0] = 0;
    if (!d) return fail(KIN_EINVAL, "desc is NULL");
    if (cap < 0 || (cap > 0 && !buf)) return fail(KIN_EINVAL, "buf is NULL or cap < 0");
    const int nS = d->n_species, nR = d->n_reactions;
    if (nS < 1 || nS > KIN_MAX_SPECIES || nR < 0 || nR > KIN_MAX_REACTIONS)
        return fail(KIN_EINVAL, "n_species %d / n_reactions %d out of range", nS, nR);
    if (!gen_eligible(nS, nR))
        return fail(KIN_EUNSUPPORTED, "the generated f covers at most %d species and %d reactions",
                    KIN_GEN_MAX_SPECIES, KIN_GEN_MAX_REACTIONS);
    if (!d->W || (nR > 0 && (!d->reac || !d->prod || !d->type)))
        return fail(KIN_EINVAL, "W, reac, prod and type must be non-NULL");
    int rows = 0;
    for (int i = 0; i < nS; ++i)
        if (!finite_pos(d->W[i])) return fail(KIN_EINVAL, "W[%d] must be finite and > 0", i);
    for (int j = 0; j < nR; ++j) {
        const int t = d->type[j];
        if (t != KIN_RXN_PLAIN && t != KIN_RXN_THIRD_BODY && t != KIN_RXN_FALLOFF)
            return fail(KIN_EINVAL, "reaction %d: unknown type %d", j, t);
        for (int k = 0; k < 2; ++k)
            if (d->reac[2 * j + k] < -1 || d->reac[2 * j + k] >= nS || d->prod[2 * j + k] < -1 ||
                d->prod[2 * j + k] >= nS)
                return fail(KIN_EINVAL, "reaction %d: species index out of range", j);
        rows += t != KIN_RXN_PLAIN;
    }
    if (rows > 0 && !d->eff) return fail(KIN_EINVAL, "eff is NULL but %d reactions need efficiencies", rows);
    for (int64_t k = 0; k < (int64_t)rows * nS; ++k)
        if (!std::isfinite(d->eff[k])) return fail(KIN_EINVAL, "non-finite efficiency");
    if ((d->cp != nullptr) != (d->Hf != nullptr)) return fail(KIN_EINVAL, "give both cp and Hf, or neither");
    for (int i = 0; d->cp && i < nS; ++i)
        if (!finite_pos(d->cp[i]) || !std::isfinite(d->Hf[i]))
            return fail(KIN_EINVAL, "species %d: cp must be finite and > 0, Hf finite", i);
    if (nR > 0 && (!d->lnA || !d->beta || !d->Ea)) return fail(KIN_EINVAL, "Arrhenius arrays must be non-NULL");
    for (int j = 0; j < nR; ++j)
        if (d->type[j] == KIN_RXN_FALLOFF && (!d->lnA0 || !d->beta0 || !d->Ea0))
            return fail(KIN_EINVAL, "falloff reaction %d needs lnA0, beta0, Ea0", j);
    const std::string src = gen_f_source(d);
    if (cap > 0) {
        const int64_t n = std::min<int64_t>(cap - 1, (int64_t)src.size());
        memcpy(buf, src.data(), (size_t)n);
        buf[n] = 0;
    }
    return (int64_t)src.size();
}

int kin_create_mechanism(const kin_mech_desc* d, kin_mech** out)
{
    g_err[0] = 0;
    if (!d || !out) return fail(KIN_EINVAL, "desc and out must be non-NULL");
    *out = nullptr;
    const int nS = d->n_species, nR = d->n_reactions;
    if (nS < 1 || nS > KIN_MAX_SPECIES) return fail(KIN_EINVAL, "n_species %d out of range", nS);
    if (nR < 0 || nR > KIN_MAX_REACTIONS) return fail(KIN_EINVAL, "n_reactions %d out of range", nR);
    if (!d->W) return fail(KIN_EINVAL, "W is NULL");
    if (nR > 0 && (!d->lnA || !d->beta || !d->Ea || !d->reac || !d->prod || !d->type))
        return fail(KIN_EINVAL, "reaction arrays must be non-NULL");
    for (int i = 0; i < nS; ++i)
        if (!finite_pos(d->W[i])) return fail(KIN_EINVAL, "W[%d] must be finite and > 0", i);

    std::vector<Rxn> rxn(nR);
    std::vector<double> EaR(nR), lnA0(nR, 0.0), beta0(nR, 0.0), Ea0R(nR, 0.0);
    std::vector<std::vector<std::pair<int, double>>> bySp(nS);
    int nM = 0, nFO = 0;
    for (int j = 0; j < nR; ++j) {
        const int t = d->type[j];
        if (t != KIN_RXN_PLAIN && t != KIN_RXN_THIRD_BODY && t != KIN_RXN_FALLOFF)
            return fail(KIN_EINVAL, "reaction %d: unknown type %d", j, t);
        if (!std::isfinite(d->lnA[j]) || !std::isfinite(d->beta[j]) || !std::isfinite(d->Ea[j]))
            return fail(KIN_EINVAL, "reaction %d: non-finite Arrhenius parameter", j);
        int r[2] = {d->reac[2 * j], d->reac[2 * j + 1]};
        int q[2] = {d->prod[2 * j], d->prod[2 * j + 1]};
        for (int k = 0; k < 2; ++k) {
            if (r[k] < -1 || r[k] >= nS) return fail(KIN_EINVAL, "reaction %d: reactant index %d", j, r[k]);
            if (q[k] < -1 || q[k] >= nS) return fail(KIN_EINVAL, "reaction %d: product index %d", j, q[k]);
        }
        rxn[j] = Rxn{(int16_t)r[0], (int16_t)r[1], (int16_t)t, 0, t != KIN_RXN_PLAIN ? nM : -1,
                     t == KIN_RXN_FALLOFF ? nFO : -1};
        if (t != KIN_RXN_PLAIN) ++nM;
        if (t == KIN_RXN_FALLOFF) ++nFO;
        EaR[j] = d->Ea[j] / R_GAS;
        if (t == KIN_RXN_FALLOFF) {
            if (!d->lnA0 || !d->beta0 || !d->Ea0)
                return fail(KIN_EINVAL, "falloff reaction %d needs lnA0, beta0, Ea0", j);
            if (!std::isfinite(d->lnA0[j]) || !std::isfinite(d->beta0[j]) || !std::isfinite(d->Ea0[j]))
                return fail(KIN_EINVAL, "reaction %d: non-finite low-pressure parameter", j);
            lnA0[j] = d->lnA0[j];
            beta0[j] = d->beta0[j];
            Ea0R[j] = d->Ea0[j] / R_GAS;
        }
        // net coefficients nu'' - nu' per species of this reaction
        int sp[4] = {q[0], q[1], r[0], r[1]};
        double c[4] = {1, 1, -1, -1};
        for (int a = 0; a < 4; ++a) {
            if (sp[a] < 0) continue;
            auto& v = bySp[sp[a]];
            if (!v.empty() && v.back().first == j) v.back().second += c[a];
            else v.push_back({j, c[a]});
        }
    }
    if (nM > 0 && !d->eff) return fail(KIN_EINVAL, "eff is NULL but %d reactions need efficiencies", nM);
    for (int64_t k = 0; k < (int64_t)nM * nS; ++k)
        if (!std::isfinite(d->eff[k])) return fail(KIN_EINVAL, "non-finite efficiency");
    std::vector<int> ptr(nS + 1, 0), crx;
    std::vector<double> cnu;
    for (int i = 0; i < nS; ++i) {
        for (auto& pr : bySp[i])
            if (pr.second != 0.0) {  // a species on both sides with equal count cancels
                crx.push_back(pr.first);
                cnu.push_back(pr.second);
            }
        ptr[i + 1] = (int)crx.size();
    }
    const int nnz = (int)crx.size();

    // one device buffer, 256-byte aligned sub-arrays
    std::vector<char> host;
    auto put = [&](const void* src, size_t bytes) {
        size_t off = (host.size() + 255) / 256 * 256;
        host.resize(off + bytes);
        if (bytes) memcpy(host.data() + off, src, bytes);
        return off;
    };
    std::vector<double> invW(nS);
    std::vector<float> invW32(nS), W32(nS), nu32(cnu.begin(), cnu.end());
    for (int i = 0; i < nS; ++i) {
        invW[i] = 1.0 / d->W[i];
        invW32[i] = (float)invW[i];
        W32[i] = (float)d->W[i];
    }
    std::vector<float> eff32((size_t)nM * nS);
    for (size_t k = 0; k < eff32.size(); ++k) eff32[k] = (float)d->eff[k];
    const size_t oW = put(d->W, 8 * nS), oIW = put(invW.data(), 8 * nS), oIW32 = put(invW32.data(), 4 * nS);
    const size_t oW32 = put(W32.data(), 4 * nS);
    const size_t oLA = put(d->lnA, 8 * nR), oB = put(d->beta, 8 * nR), oE = put(EaR.data(), 8 * nR);
    const size_t oLA0 = put(lnA0.data(), 8 * nR), oB0 = put(beta0.data(), 8 * nR), oE0 = put(Ea0R.data(), 8 * nR);
    const size_t oRx = put(rxn.data(), sizeof(Rxn) * nR);
    // warp layout: reactions permuted plain, third-body, falloff (each in
    // reaction order, so falloff ordinals keep their order); efficiency rows
    // transposed to [species][non-plain reaction in permutation order]
    std::vector<int> perm, pos(nR);
    for (int t = KIN_RXN_PLAIN; t <= KIN_RXN_FALLOFF; ++t)
        for (int j = 0; j < nR; ++j)
            if (rxn[j].type == t) perm.push_back(j);
    std::vector<Rxn> rxnp(nR);
    const int nPlain = nR - nM;
    for (int q = 0; q < nR; ++q) {
        pos[perm[q]] = q;
        rxnp[q] = rxn[perm[q]];
        rxnp[q].row = rxnp[q].type != KIN_RXN_PLAIN ? q - nPlain : -1;
    }
    std::vector<int> crxp(nnz);
    for (int e2 = 0; e2 < nnz; ++e2) crxp[e2] = pos[crx[e2]];
    std::vector<double> effV64((size_t)(nS + 1) / 2 * nM * 2, 0.0);
    std::vector<float> effV32((size_t)(nS + 3) / 4 * nM * 4, 0.0f);
    for (int q = nPlain; q < nR; ++q)
        for (int k = 0; k < nS; ++k) {
            const double a = d->eff[(size_t)rxn[perm[q]].row * nS + k];
            const int row = q - nPlain;
            effV64[((size_t)(k / 2) * nM + row) * 2 + k % 2] = a;
            effV32[((size_t)(k / 4) * nM + row) * 4 + k % 4] = (float)a;
        }
    // the warp f derives a reaction's efficiency row and falloff ordinal from
    // its permutation position
    std::vector<uint32_t> rxw(nR);
    for (int q = 0; q < nR; ++q) {
        const Rxn& x = rxnp[q];
        if ((x.type != KIN_RXN_PLAIN) != (q >= nPlain) || (x.type != KIN_RXN_PLAIN && x.row != q - nPlain) ||
            (x.type == KIN_RXN_FALLOFF) != (q >= nR - nFO) || (x.type == KIN_RXN_FALLOFF && x.fo != q - (nR - nFO)))
            return fail(KIN_EUNSUPPORTED, "reaction permutation out of order at %d", q);
        rxw[q] = (uint32_t)(x.r0 + 1) | ((uint32_t)(x.r1 + 1) << 16);
    }
    const size_t oPerm = put(perm.data(), 4 * nR), oRxp = put(rxnp.data(), sizeof(Rxn) * nR);
    const size_t oRxw = put(rxw.data(), 4 * nR);
    const size_t oCrxp = put(crxp.data(), 4 * nnz);
    // the rows once more in order of position
    std::vector<int> crxq(nnz + 1, 0), byPos;
    std::vector<double> cnuq(nnz);
    for (int i = 0; i < nS; ++i) {
        byPos.clear();
        for (int e2 = ptr[i]; e2 < ptr[i + 1]; ++e2) byPos.push_back(e2);
        std::sort(byPos.begin(), byPos.end(), [&](int a, int b) { return crxp[a] < crxp[b]; });
        for (size_t k = 0; k < byPos.size(); ++k) {
            crxq[ptr[i] + k] = crxp[byPos[k]] << 3 | ((int)cnu[byPos[k]] + 4);
            cnuq[ptr[i] + k] = cnu[byPos[k]];
        }
    }
    const size_t oEffV64 = put(effV64.data(), 8 * effV64.size()), oEffV32 = put(effV32.data(), 4 * effV32.size());
    const size_t oPtr = put(ptr.data(), 4 * (nS + 1)), oCrx = put(crx.data(), 4 * nnz);
    const size_t oNu = put(cnu.data(), 8 * nnz), oNu32 = put(nu32.data(), 4 * nnz);
    // the species' molar mass folded into its row (a common factor of the row)
    std::vector<double> cnuW(nnz);
    std::vector<float> nuW32(nnz);
    for (int i = 0; i < nS; ++i)
        for (int e2 = ptr[i]; e2 < ptr[i + 1]; ++e2) {
            cnuW[e2] = cnu[e2] * d->W[i];
            nuW32[e2] = (float)cnuW[e2];
        }
    const size_t oNuW = put(cnuW.data(), 8 * nnz), oNuW32 = put(nuW32.data(), 4 * nnz);
    // ELL copies of the gather entries for the warp layout's 32 lanes
    int ell_base[ELL_SLOTS] = {0};
    int ell_n = 0;
    for (int r = 0; r * 32 < nS; ++r) {
        int len = 0;
        for (int i = 32 * r; i < std::min(nS, 32 * r + 32); ++i) len = std::max(len, ptr[i + 1] - ptr[i]);
        ell_base[r] = ell_n;
        ell_n += 32 * len;
    }
    // Each species' entries are ordered step by step so that the lanes of a
    // step read Omega words in distinct shared-memory banks where they can:
    // for FP32 words the bank is the position mod 32 across the warp; for
    // FP64 words, read by half-warps, the position mod 16 within each half.
    // A greedy pass gives each lane, in turn, its remaining entry in the
    // least used bank of the step. Only the summation order of a row
    // follows from this; its entries do not change.
    std::vector<int> ord32(nnz), ord64(nnz);
    auto order_rows = [&](std::vector<int>& ord, int banks, int group) {
        for (int r = 0; r * 32 < nS; ++r) {
            std::vector<std::vector<int>> left(32);
            int len = 0;
            for (int l = 0; l < 32 && 32 * r + l < nS; ++l) {
                const int i = 32 * r + l;
                for (int e2 = ptr[i]; e2 < ptr[i + 1]; ++e2) left[l].push_back(e2);
                len = std::max(len, ptr[i + 1] - ptr[i]);
            }
            for (int k = 0; k < len; ++k) {
                std::vector<int> used(2 * banks, 0);
                for (int l = 0; l < 32; ++l) {
                    if (left[l].empty()) continue;
                    const int gbase = (l / group) * banks;
                    size_t best = 0;
                    for (size_t c = 1; c < left[l].size(); ++c)
                        if (used[gbase + crxp[left[l][c]] % banks] < used[gbase + crxp[left[l][best]] % banks])
                            best = c;
                    const int e2 = left[l][best];
                    left[l].erase(left[l].begin() + best);
                    used[gbase + crxp[e2] % banks]++;
                    ord[ptr[32 * r + l] + k] = e2;
                }
            }
        }
    };
    order_rows(ord32, 32, 32);
    order_rows(ord64, 16, 16);
    std::vector<CsrW32> ell32(ell_n, CsrW32{0.0f, 0});
    std::vector<CsrW64> ell64(ell_n, CsrW64{0.0, 0, 0});
    for (int i = 0; i < nS; ++i)
        for (int k = 0; k < ptr[i + 1] - ptr[i]; ++k) {
            const int at = ell_base[i / 32] + 32 * k + i % 32;
            const int a = ord32[ptr[i] + k], b = ord64[ptr[i] + k];
            ell32[at] = CsrW32{nuW32[a], crxp[a]};
            ell64[at] = CsrW64{cnuW[b], crxp[b], 0};
        }
    const size_t oEll32 = put(ell32.data(), sizeof(CsrW32) * ell_n);
    const size_t oEll64 = put(ell64.data(), sizeof(CsrW64) * ell_n);
    // the integer FP64 f (int_tables.h), for each group size that the mechanism
    // can take; eight rounds of reactions a chunk, so that the words of a
    // 53-species / 634-reaction cell (7.4 KB for a warp) leave room for 16 warps
    // per SM beside the tables in L1, and sixteen across warps, whose barriers
    // cost more than the shared memory
    IntGather ig[INT_NTAB];
    size_t oIg[INT_NTAB][4];
    const int ig_lanes[INT_NTAB] = {8, 16, 32, 64, 128, 16, 32, 4};
    const bool ig_use[INT_NTAB] = {nS <= 32, nS <= 16, true, nS >= 32 && nS <= 64, nS >= 64,
                                  nS <= 16, nS <= 64, nS <= 16};
    auto put_ig = [&](int v) {
        oIg[v][0] = put(ig[v].step0.data(), 4 * ig[v].step0.size());
        oIg[v][1] = put(ig[v].ent.data(), 4 * ig[v].ent.size());
        oIg[v][2] = put(ig[v].slot0.data(), 4 * ig[v].slot0.size());
        oIg[v][3] = put(ig[v].part.data(), 4 * ig[v].part.size());
    };
    for (int v = 0; v < INT_NTAB; ++v) {
        if (!ig_use[v]) continue;
        int chunk = std::max(32, std::min((nR + 31) / 32 * 32, std::max(64, (ig_lanes[v] > 32 ? 16 : 8) * ig_lanes[v])));
        if (v == INT_G16S || v == INT_G32S) {
            // (with the rate constants that may be staged beside them)
            const int words = INT_SMALL_WARP_WORDS * ig_lanes[v] / 32 - (nS + 2 * nR <= 256 ? nR + nFO : 0);
            while (chunk > 32 && int_group_words(nS, chunk, 2 * nS + ig_lanes[v]) > words) chunk -= 32;
        }
        ig[v] = build_int_gather(nS, nR, ptr.data(), crxp.data(), cnu.data(), chunk, ig_lanes[v]);
        if (v < INT_G16S) put_ig(v);
    }
    std::vector<int32_t> effI((size_t)(nS + 1) / 2 * nM * 4, 0), effX(nM);
    for (int row = 0; row < nM; ++row) {
        std::vector<int32_t> hi(nS), lo(nS);
        const double* e = d->eff + (size_t)rxn[perm[nPlain + row]].row * nS;
        effX[row] = int_efficiencies(nS, e, hi.data(), lo.data());
        int_eff_limbs(nS, e, effX[row], 1, hi.data(), lo.data());
        for (int k = 0; k < nS; ++k) {
            effI[((size_t)(k / 2) * nM + row) * 4 + 2 * (k % 2)] = hi[k];
            effI[((size_t)(k / 2) * nM + row) * 4 + 2 * (k % 2) + 1] = lo[k];
        }
    }
    std::vector<uint64_t> imW(2 * nS);
    std::vector<int32_t> imWe(2 * nS);
    for (int i = 0; i < nS; ++i) {
        imW[2 * i] = int_split(1.0L / d->W[i], &imWe[2 * i]);
        imW[2 * i + 1] = int_split(d->W[i], &imWe[2 * i + 1]);
        if (ptr[i + 1] == ptr[i]) imW[2 * i + 1] = 0;  // no reaction changes it
    }
    int imLow = 0;
    for (int j = 0; j < nR; ++j)
        if ((d->reac[2 * j] >= 0) + (d->reac[2 * j + 1] >= 0) + (rxn[j].type == KIN_RXN_THIRD_BODY) < 2) imLow = 1;
    std::vector<double> arr(3 * nR), arr0(3 * nFO);
    for (int q = 0; q < nR; ++q) {
        const int j = perm[q], fo = rxnp[q].fo;
        arr[q] = d->lnA[j];
        arr[nR + q] = d->beta[j];
        arr[2 * nR + q] = EaR[j];
        if (fo < 0) continue;
        arr0[fo] = lnA0[j];
        arr0[nFO + fo] = beta0[j];
        arr0[2 * nFO + fo] = Ea0R[j];
    }
    std::vector<uint32_t> scl(4 * nR);
    for (int q = 0; q < nR; ++q) {
        const int j = perm[q];
        int_scale_table(d->lnA[j], d->beta[j], EaR[j], d->reac + 2 * j, d->type[j], q >= nPlain ? effX[q - nPlain] : 0, &scl[4 * q]);
    }
    uint64_t ex2[64], lnc[128];
    int_exp_log_tables(ex2, lnc);
    const size_t oArr = put(arr.data(), 8 * arr.size()), oArr0 = put(arr0.data(), 8 * arr0.size());
    const size_t oEx2 = put(ex2, sizeof(ex2)), oLnc = put(lnc, sizeof(lnc));
    const size_t oImW = put(imW.data(), 8 * imW.size()), oImWe = put(imWe.data(), 4 * imWe.size());
    const size_t oEffI = put(effI.data(), 4 * effI.size()), oEffX = put(effX.data(), 4 * effX.size());
    // the lane layout's integer FP64 f, for mechanisms whose shared words leave
    // room for enough lanes
    const bool use_li = lane_int_bytes(nS, nM) <= LANE_INT_MAX_BYTES;
    LaneInt li;
    if (use_li) li = build_lane_int(nS, nR, d->reac, d->prod, d->type, d->eff);
    for (int r = 0; r < li.tb; ++r)
        int_eff_limbs(nS, d->eff + (size_t)li.row[r] * nS, li.effx[r], 2, &li.eff[2 * (size_t)r * nS],
                      &li.eff[2 * (size_t)r * nS + 1]);
    const size_t oLiRx = put(li.rx.data(), 4 * li.rx.size());
    const size_t oLiE = put(li.eff.data(), 4 * li.eff.size()), oLiEx = put(li.effx.data(), 4 * li.effx.size());
    // the segmented FP32 gather of the 32-lane isothermal f, where the packed
    // entries apply and its partial sums fit in the FP32 half of the warp's
    // shared words, past C and Omega
    SegTables seg;
    const int group_floats = 2 * ((nS + nR + 3) & ~3);
    const bool use_seg = build_seg_tables(nS, nR, ptr.data(), crxp.data(), cnu.data(), seg) &&
                         nS + nR + seg.nslots <= group_floats;
    // four steps of a lane side by side; steps past the last have no flush
    const int segK4 = (seg.K + 3) / 4;
    std::vector<uint32_t> segE((size_t)segK4 * 128, 0u);
    for (size_t k = 0; k < seg.ent.size(); ++k) segE[(k / 128 * 32 + k % 32) * 4 + k / 32 % 4] = seg.ent[k];
    const size_t oSegE = use_seg ? put(segE.data(), 4 * segE.size()) : 0;
    const size_t oSegF = use_seg ? put(seg.slot0.data(), 4 * seg.slot0.size()) : 0;
    const size_t oSegP = use_seg ? put(seg.part.data(), 4 * seg.part.size()) : 0;
    const size_t oEff = put(d->eff, 8 * (size_t)nM * nS), oEff32 = put(eff32.data(), 4 * (size_t)nM * nS);
    // thermochemistry for the energy equation: cp, cp/W, Hf
    const bool thermo = d->cp && d->Hf;
    if ((d->cp != nullptr) != (d->Hf != nullptr)) return fail(KIN_EINVAL, "give both cp and Hf, or neither");
    std::vector<double> cpW(thermo ? nS : 0), HfW(thermo ? nS : 0);
    for (int i = 0; thermo && i < nS; ++i) {
        if (!finite_pos(d->cp[i])) return fail(KIN_EINVAL, "cp[%d] must be finite and > 0", i);
        if (!std::isfinite(d->Hf[i])) return fail(KIN_EINVAL, "Hf[%d] must be finite", i);
        cpW[i] = d->cp[i] / d->W[i];
        HfW[i] = d->Hf[i] / d->W[i];
    }
    const size_t oCp = thermo ? put(d->cp, 8 * nS) : 0, oCpW = thermo ? put(cpW.data(), 8 * nS) : 0;
    const size_t oHf = thermo ? put(d->Hf, 8 * nS) : 0, oHfW = thermo ? put(HfW.data(), 8 * nS) : 0;
    // the tables that few calls read come last: between the others they cost the
    // mixed path 2 % (53 / 634, 1,024 cells 8.40 -> 8.56 ms)
    for (int v = INT_G16S; v < INT_NTAB; ++v)
        if (ig_use[v]) put_ig(v);
    const size_t oCrxq = put(crxq.data(), 4 * (nnz + 1)), oCnuq = put(cnuq.data(), 8 * nnz);
    const size_t oScl = put(scl.data(), 4 * scl.size());
    const size_t oTab = put(nullptr, 0);
    const size_t tabBytes = sizeof(double) * RKC_TAB_S * RKC_TAB_S * RKC_TAB_W;
    host.resize(oTab + tabBytes, 0);

    kin_mech* m = new (std::nothrow) kin_mech();
    if (!m) return fail(KIN_ENOMEM, "host allocation failed");
    cudaError_t e = cudaGetDevice(&m->device);
    if (e != cudaSuccess) { delete m; return cuda_fail(e, "cudaGetDevice"); }
    e = cudaMalloc(&m->buf, host.size());
    if (e != cudaSuccess) { delete m; cudaGetLastError(); return fail(KIN_ENOMEM, "cudaMalloc(%zu): %s", host.size(), cudaGetErrorString(e)); }
    e = cudaMemcpy(m->buf, host.data(), host.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) { cudaFree(m->buf); delete m; return cuda_fail(e, "cudaMemcpy"); }
    char* b = (char*)m->buf;
    MechDev& M = m->dev;
    M.nS = nS; M.nR = nR; M.nM = nM; M.nFO = nFO; M.nnz = nnz;
    M.W = (const double*)(b + oW); M.invW = (const double*)(b + oIW); M.invW32 = (const float*)(b + oIW32);
    M.W32 = (const float*)(b + oW32);
    M.lnA = (const double*)(b + oLA); M.beta = (const double*)(b + oB); M.EaR = (const double*)(b + oE);
    M.lnA0 = (const double*)(b + oLA0); M.beta0 = (const double*)(b + oB0); M.Ea0R = (const double*)(b + oE0);
    M.rxn = (const Rxn*)(b + oRx);
    M.rxn_perm = (const int*)(b + oPerm);
    M.rxnp = (const Rxn*)(b + oRxp);
    M.csrp_rxn = (const int*)(b + oCrxp);
    M.csrq = (const int*)(b + oCrxq);
    M.csrq_nu = (const double*)(b + oCnuq);
    M.ell32 = (const CsrW32*)(b + oEll32);
    M.ell64 = (const CsrW64*)(b + oEll64);
    for (int r = 0; r < ELL_SLOTS; ++r) M.ell_base[r] = ell_base[r];
    M.seg_ent = use_seg ? (const uint4*)(b + oSegE) : nullptr;
    M.seg_slot0 = use_seg ? (const int32_t*)(b + oSegF) : nullptr;
    M.seg_part = use_seg ? (const int32_t*)(b + oSegP) : nullptr;
    M.seg_K4 = use_seg ? segK4 : 0;
    for (int v = 0; v < INT_NTAB; ++v) {
        M.ig[v] = IntDev{};
        if (!ig_use[v]) continue;
        M.ig[v] = IntDev{ig[v].nchunk, ig[v].chunk, ig[v].nslots, (const int32_t*)(b + oIg[v][0]),
                         (const uint32_t*)(b + oIg[v][1]), (const int32_t*)(b + oIg[v][2]),
                         (const int32_t*)(b + oIg[v][3])};
    }
    M.effI = (const int4*)(b + oEffI);
    M.effX = (const int32_t*)(b + oEffX);
    M.arr = (const double*)(b + oArr);
    M.arr0 = (const double*)(b + oArr0);
    M.scl = (const uint4*)(b + oScl);
    M.ex2 = (const unsigned long long*)(b + oEx2);
    M.lnc = (const ulonglong2*)(b + oLnc);
    M.imW = (const ulonglong2*)(b + oImW);
    M.imWe = (const int2*)(b + oImWe);
    M.imLow = imLow;
    int_word_bits(nS, ptr.data(), cnu.data(), &M.imUp, &M.imShort);
    M.li_n = li.n;
    M.li_tb = li.tb;
    M.li_rx = use_li ? (const uint4*)(b + oLiRx) : nullptr;
    M.li_eff = (const int2*)(b + oLiE);
    M.li_effx = (const int32_t*)(b + oLiEx);
    M.effV64 = (const double*)(b + oEffV64);
    M.effV32 = (const float*)(b + oEffV32);
    M.rxw = (const uint32_t*)(b + oRxw);
    M.csr_ptr = (const int*)(b + oPtr); M.csr_rxn = (const int*)(b + oCrx);
    M.csr_nu = (const double*)(b + oNu); M.csr_nu32 = (const float*)(b + oNu32);
    M.csr_nuW = (const double*)(b + oNuW); M.csr_nuW32 = (const float*)(b + oNuW32);
    M.eff = (const double*)(b + oEff); M.eff32 = (const float*)(b + oEff32);
    M.rkc = (const double*)(b + oTab);
    M.cp = thermo ? (const double*)(b + oCp) : nullptr;
    M.cpW = thermo ? (const double*)(b + oCpW) : nullptr;
    M.Hf = thermo ? (const double*)(b + oHf) : nullptr;
    M.HfW = thermo ? (const double*)(b + oHfW) : nullptr;
    m->nS = nS; m->nR = nR; m->nM = nM;
    m->thermo = thermo;
    if (gen_eligible(nS, nR)) m->gen_src = gen_f_source(d);
    e = launch_rkc_table((double*)(b + oTab), 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) { cudaFree(m->buf); delete m; return cuda_fail(e, "RKC table"); }
    *out = m;
    return KIN_OK;
}

int kin_destroy(kin_mech* m)
{
    g_err[0] = 0;
    if (!m) return KIN_OK;
    cudaError_t e = cudaFree(m->buf);
    delete m;
    return e == cudaSuccess ? KIN_OK : cuda_fail(e, "cudaFree");
}

// The largest workspace of a call with these options: the automatic layout
// depends on the f evaluation, which a caller may set after sizing the
// workspace.
static int max_ws_bytes(const kin_mech* m, const kin_opts* o, int64_t cells, int64_t* bytes)
{
    Grid g;
    int rc = grid_for(m, o, cells, &g);
    if (rc) return rc;
    *bytes = ws_bytes(m, o, g, cells);
    int nsm = 0;
    const cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    kin_opts lane = *o;
    lane.layout = resolve_layout(m, o, cells, nsm, false);
    if (lane.layout == g.layout) return KIN_OK;
    rc = grid_for(m, &lane, cells, &g);
    if (rc) return rc;
    *bytes = std::max(*bytes, ws_bytes(m, &lane, g, cells));
    return KIN_OK;
}

int64_t kin_workspace_bytes(const kin_mech* m, const kin_opts* o, int64_t cells)
{
    g_err[0] = 0;
    if (!m) return fail(KIN_EINVAL, "mechanism is NULL");
    if (cells < 0) return fail(KIN_EINVAL, "cells < 0");
    int rc = check_opts(o);
    if (rc) return rc;
    int64_t bytes = 0;
    rc = max_ws_bytes(m, o, cells, &bytes);
    return rc ? rc : bytes;
}

int kin_integrate_batch(const kin_mech* m, int32_t n, const kin_instance* inst, const kin_opts* o,
                        void* ws, int64_t ws_size)
{
    g_err[0] = 0;
    if (!m) return fail(KIN_EINVAL, "mechanism is NULL");
    int rc = check_opts(o);
    if (rc) return rc;
    if (n < 1 || n > KIN_MAX_INSTANCES) return fail(KIN_EINVAL, "n_instances %d out of range [1, %d]", n, KIN_MAX_INSTANCES);
    if (!inst) return fail(KIN_EINVAL, "instances is NULL");
    // ~10 KB of launch parameters: built on the heap, copied by the launch
    Launch* Lp = new (std::nothrow) Launch();
    if (!Lp) return fail(KIN_ENOMEM, "host allocation failed");
    struct Free { Launch* p; ~Free() { delete p; } } fr{Lp};
    Launch& P = *Lp;
    int64_t total = 0;
    for (int i = 0; i < n; ++i) {
        const kin_instance& I = inst[i];
        if (I.cells < 0) return fail(KIN_EINVAL, "instance %d: cells < 0", i);
        if (!finite_pos(I.dt)) return fail(KIN_EINVAL, "instance %d: dt must be finite and > 0", i);
        if (!finite_pos(I.rtol)) return fail(KIN_EINVAL, "instance %d: rtol must be finite and > 0", i);
        if (!std::isfinite(I.atol) || I.atol < 0) return fail(KIN_EINVAL, "instance %d: atol must be finite and >= 0", i);
        if (I.cells > 0) {
            if (!I.T || !I.p || !I.Y) return fail(KIN_EINVAL, "instance %d: T, p and Y must be non-NULL", i);
            if (I.ldY < I.cells) return fail(KIN_EINVAL, "instance %d: ldY < cells", i);
            if (I.ldY > INT32_MAX) return fail(KIN_EINVAL, "instance %d: ldY >= 2^31", i);
            if (!is_device_ptr(I.T) || !is_device_ptr(I.p) || !is_device_ptr(I.Y) ||
                (I.status && !is_device_ptr(I.status)) || (I.stats && !is_device_ptr(I.stats)))
                return fail(KIN_EINVAL, "instance %d: T, p, Y, status and stats must be device memory", i);
        }
        P.start[i] = total;
        P.inst[i] = InstDev{I.T, I.p, I.Y, I.ldY, I.dt, I.rtol, I.atol, I.status, I.stats};
        total += I.cells;
    }
    P.start[n] = total;
    if (total == 0) return KIN_OK;
    Grid g;
    rc = grid_for(m, o, total, &g);
    if (rc) return rc;
    const int64_t need = ws_bytes(m, o, g, total);
    if (!ws) return fail(KIN_EINVAL, "workspace is NULL");
    if (((uintptr_t)ws) % 256) return fail(KIN_EINVAL, "workspace must be 256-byte aligned");
    if (ws_size < need) return fail(KIN_ENOMEM, "workspace has %lld bytes, needs %lld", (long long)ws_size, (long long)need);
    if (!is_device_ptr(ws)) return fail(KIN_EINVAL, "workspace must be device memory");
    // never more lanes (warps in the warp layout) than cells
    int blocks = g.blocks;
    const int per_block = g.threads / g.lanes;
    const int64_t want = (total + per_block - 1) / per_block;
    if (want < blocks) blocks = (int)want;
    const int64_t nslots = (int64_t)blocks * g.threads;
    P.M = m->dev;
    P.method = o->method;
    P.precision = o->precision;
    P.max_steps = o->max_steps > 0 ? o->max_steps : 100000;
    P.n_inst = n;
    P.nslots = nslots;
    P.total = total;
    char* base = (char*)ws;
    const int sig = o->method == KIN_RKC ? o->sigma : KIN_SIGMA_GERSHGORIN;
    const WsLayout w = ws_layout(m->dev, o->precision, sig, o->energy,
                                 g.layout == KIN_LAYOUT_WARP ? 0 : nslots, total);
    P.energy = o->energy;
    P.nV = m->nS + o->energy;
    P.lanes = g.lanes;
    P.sigma_method = sig;
    P.cell_ev = sig == KIN_SIGMA_POWER ? (double*)(base + w.ev) : nullptr;
    P.queue = (unsigned long long*)(base + w.header);
    P.hist = (unsigned*)(base + w.header + 256);
    P.vec = (double*)(base + w.vec);
    P.lane_r = base + w.lane_r;
    P.lane_sig = (double*)(base + w.lane_sig);
    P.cell_k = base + w.cell_k;
    P.cell_f0 = (double*)(base + w.f0);
    P.cell_sig = (double*)(base + w.sig);
    P.cell_h = (double*)(base + w.h);
    P.cell_nfe = (int32_t*)(base + w.nfe);
    P.cell_nfs = (int32_t*)(base + w.nfs);
    P.cell_st = (uint8_t*)(base + w.st);
    P.order = (int32_t*)(base + w.order);
    if (total > INT32_MAX) return fail(KIN_EINVAL, "more than 2^31-1 cells in one call");
    // f: integer arithmetic where it serves, tables, or the mechanism's
    // generated code (lane layout, FP64, isothermal)
    int li_blocks = 0;
    rc = lane_int_blocks(m, o, g, &li_blocks);
    if (rc) return rc;
    bool gen = false;
    GenKernels gk{};
    // (the automatic choice leaves the energy equation on the tables: with a
    // per-reaction exp inlined, the generated form measured slower)
    if (o->feval == KIN_FEVAL_GENERATED ||
        (o->feval == KIN_FEVAL_AUTO && total >= KIN_GEN_MIN_CELLS && !o->energy && !li_blocks)) {
        // (the energy equation comes generated too: the mechanism has cp and
        // Hf, checked above, so its source carries that form of f)
        const bool serves = g.layout == KIN_LAYOUT_LANE && o->precision == KIN_FP64 &&
                            o->staging == KIN_STAGE_GLOBAL && !m->gen_src.empty();
        if (serves) {
            std::string log;
            const int grc = gen_kernels(m->device, m->gen_src, &gk, &log);
            if (grc == KIN_OK && (!o->energy || gk.energy)) gen = true;
            else if (o->feval == KIN_FEVAL_GENERATED)
                return fail(grc != KIN_OK ? grc : KIN_EUNSUPPORTED, "generated f: %.400s", log.c_str());
        } else if (o->feval == KIN_FEVAL_GENERATED) {
            return fail(KIN_EUNSUPPORTED, "the generated f serves the lane layout, KIN_FP64, "
                                          "KIN_STAGE_GLOBAL and at most %d species / %d reactions",
                        KIN_GEN_MAX_SPECIES, KIN_GEN_MAX_REACTIONS);
        }
    }
    cudaStream_t st = (cudaStream_t)o->stream;
    cudaError_t e = cudaMemsetAsync(base + w.header, 0, 512, st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
    if (g.layout == KIN_LAYOUT_WARP && o->method == KIN_RKCK) {
        e = o->precision == KIN_MIXED ? launch_warp_rkck_f32(P, blocks, g.threads, st)
                                      : launch_warp_rkck_f64(P, blocks, g.threads, st);
    } else if (g.layout == KIN_LAYOUT_WARP) {
        using LaunchFn = cudaError_t (*)(Launch&, int, int, cudaStream_t);
        if (g.occupancy) P.M = small_chunks(m->dev);
        // [energy][precision][occupancy]
        static const LaunchFn fns[2][2][2] = {
            {{launch_warp_f64_o0, launch_warp_f64_o1}, {launch_warp_f32_o0, launch_warp_f32_o1}},
            {{launch_warp_f64_en_o0, launch_warp_f64_en_o1}, {launch_warp_f32_en_o0, launch_warp_f32_en_o1}}};
        e = fns[o->energy][o->precision == KIN_MIXED][g.occupancy ? 1 : 0](P, blocks, g.threads, st);
    }
    else if (li_blocks) {
        blocks = std::min(blocks, li_blocks);
        P.nslots = (int64_t)blocks * g.threads;
        e = launch_lane_int(P, o->occupancy, blocks, g.threads, st);
    } else if (gen)
        e = gen_launch(gk, P, o->occupancy, blocks, g.threads, st);
    else
        e = launch_integrate(P, o->energy ? KIN_STAGE_GLOBAL : o->staging, o->occupancy, blocks,
                             g.threads, st);
    if (e != cudaSuccess) return cuda_fail(e, "integrate launch");
    return KIN_OK;
}

int kin_integrate(const kin_mech* m, int64_t cells, double* T, const double* p, double* Y,
                  int64_t ldY, double dt, double rtol, double atol, const kin_opts* o,
                  uint8_t* status, int32_t* stats, void* ws, int64_t ws_size)
{
    kin_instance I{cells, T, p, Y, ldY, dt, rtol, atol, status, stats};
    return kin_integrate_batch(m, 1, &I, o, ws, ws_size);
}

static int64_t al256(int64_t x) { return (x + 255) / 256 * 256; }

int64_t kin_host_buffer_bytes(const kin_mech* m, const kin_opts* o, int64_t cells)
{
    g_err[0] = 0;
    if (cells < 0) return fail(KIN_EINVAL, "cells < 0");
    int64_t ws = kin_workspace_bytes(m, o, cells);
    if (ws < 0) return ws;
    return al256(ws) + 2 * al256(8 * cells) + al256(8 * cells * m->nS) + al256(cells) + al256(4 * KIN_NSTATS * cells);
}

int kin_integrate_host(const kin_mech* m, int64_t cells, double* T, const double* p, double* Y,
                       int64_t ldY, double dt, double rtol, double atol, const kin_opts* o,
                       uint8_t* status, int32_t* stats, void* buf, int64_t bytes)
{
    g_err[0] = 0;
    const int64_t need = kin_host_buffer_bytes(m, o, cells);
    if (need < 0) return (int)need;
    if (cells == 0) return KIN_OK;
    if (!T || !p || !Y) return fail(KIN_EINVAL, "T, p and Y must be non-NULL");
    if (ldY < cells) return fail(KIN_EINVAL, "ldY < cells");
    if (!buf || ((uintptr_t)buf) % 256) return fail(KIN_EINVAL, "device_buffer must be non-NULL and 256-byte aligned");
    if (bytes < need) return fail(KIN_ENOMEM, "device_buffer has %lld bytes, needs %lld", (long long)bytes, (long long)need);
    if (!is_device_ptr(buf)) return fail(KIN_EINVAL, "device_buffer must be device memory");
    const int64_t ws = kin_workspace_bytes(m, o, cells);
    char* b = (char*)buf;
    int64_t off = al256(ws);
    double* Td = (double*)(b + off); off += al256(8 * cells);
    double* pd = (double*)(b + off); off += al256(8 * cells);
    double* Yd = (double*)(b + off); off += al256(8 * cells * m->nS);
    uint8_t* sd = (uint8_t*)(b + off); off += al256(cells);
    int32_t* xd = (int32_t*)(b + off);
    cudaStream_t st = (cudaStream_t)o->stream;
    cudaError_t e = cudaMemcpyAsync(Td, T, 8 * cells, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(pd, p, 8 * cells, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpy2DAsync(Yd, 8 * cells, Y, 8 * ldY, 8 * cells, m->nS, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_fail(e, "host-to-device copy");
    int rc = kin_integrate(m, cells, Td, pd, Yd, cells, dt, rtol, atol, o, sd, stats ? xd : nullptr, buf, ws);
    if (rc) return rc;
    e = cudaMemcpy2DAsync(Y, 8 * ldY, Yd, 8 * cells, 8 * cells, m->nS, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && o->energy) e = cudaMemcpyAsync(T, Td, 8 * cells, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && status) e = cudaMemcpyAsync(status, sd, cells, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && stats) e = cudaMemcpyAsync(stats, xd, 4 * KIN_NSTATS * cells, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return cuda_fail(e, "device-to-host copy");
    return KIN_OK;
}

int kin_rates(const kin_mech* m, int64_t cells, const double* T, const double* p, const double* Y,
              int64_t ldY, double* dYdt, int32_t precision, void* stream, void* ws, int64_t ws_size)
{
    g_err[0] = 0;
    if (!m) return fail(KIN_EINVAL, "mechanism is NULL");
    if (precision != KIN_FP64 && precision != KIN_MIXED) return fail(KIN_EINVAL, "unknown precision %d", precision);
    if (cells < 0) return fail(KIN_EINVAL, "cells < 0");
    if (cells == 0) return KIN_OK;
    if (!T || !p || !Y || !dYdt) return fail(KIN_EINVAL, "T, p, Y and dYdt must be non-NULL");
    if (ldY < cells) return fail(KIN_EINVAL, "ldY < cells");
    if (ldY > INT32_MAX) return fail(KIN_EINVAL, "ldY >= 2^31");
    if (!is_device_ptr(T) || !is_device_ptr(p) || !is_device_ptr(Y) || !is_device_ptr(dYdt))
        return fail(KIN_EINVAL, "T, p, Y and dYdt must be device memory");
    kin_opts o{KIN_RKC, precision, 0, 0, 0, KIN_STAGE_GLOBAL, KIN_OCC_DEFAULT, 0, KIN_LAYOUT_LANE, 0,
               KIN_FEVAL_TABLE, stream};
    Grid g;
    int rc = grid_for(m, &o, cells, &g);
    if (rc) return rc;
    const int64_t need = ws_bytes(m, &o, g, cells);
    if (!ws || ((uintptr_t)ws) % 256) return fail(KIN_EINVAL, "workspace must be non-NULL and 256-byte aligned");
    if (ws_size < need) return fail(KIN_ENOMEM, "workspace has %lld bytes, needs %lld", (long long)ws_size, (long long)need);
    if (!is_device_ptr(ws)) return fail(KIN_EINVAL, "workspace must be device memory");
    int nsm = 0;
    cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, m->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    e = precision == KIN_MIXED ? launch_rates_f32(m->dev, cells, T, p, Y, ldY, dYdt, ws, g.nslots, g.blocks, g.threads,
                                                  (cudaStream_t)stream)
                               : launch_rates_f64(m->dev, cells, T, p, Y, ldY, dYdt, nsm, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "rates launch");
    return KIN_OK;
}

}  // extern "C"
