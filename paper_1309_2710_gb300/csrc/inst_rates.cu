// inst_rates.cu -- f alone in FP64 (kin_rates): one group of lanes per cell, with
// the integer f and exponential of the warp layout (warp_int.cuh).
//
// A cell of 53 species / 634 reactions takes 659 exponentials and 8,160 other
// operations; on the FP64 pipe the exponentials alone (some 20 instructions
// each) take 1.1 ms for 50,000 cells, and the lane-per-cell form streamed its
// rate constants and rates of progress through L2 besides: 2.80 ms, 0.755 now.
// Each cell's scale comes from the cell itself (int_first_scale), so its bits do
// not depend on the call's other cells.
#include "warp.cuh"

namespace kin {

template <int NR, int G>
__global__ void __launch_bounds__(128, 4)
    warp_rates_kernel(const __grid_constant__ MechDev M, int64_t cells, const double* __restrict__ T,
                      const double* __restrict__ p, const double* Y, int64_t ldY, double* dYdt)
{
    const IntDev& I = int_tab<G>(M);
    double* base = reinterpret_cast<double*>(kin_smem) + (size_t)(threadIdx.x / G) * int_smem_words(M, I);
    const IntSmem S(M, I, base);
    Group<G> grp(nullptr, 0);
    const int lane = threadIdx.x & (G - 1);
    const int64_t ngroups = (int64_t)gridDim.x * (blockDim.x / G);
    const int64_t first = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    // every group of a warp takes part in every pass; those past the end repeat
    // the last cell and leave its result alone
    for (int64_t c0 = first; c0 - (threadIdx.x & 31) / G < cells; c0 += ngroups) {
        const int64_t c = c0 < cells ? c0 : cells - 1;
        const double t = T[c], pR = p[c] * (1e-6 / R_GAS), invT = Tab<double>::inv(t);
        double x[NR], out[NR];
        int scale = -1;
#pragma unroll
        for (int r = 0; r < NR; ++r) x[r] = lane + G * r < M.nS ? Y[(int64_t)(lane + G * r) * ldY + c] : 0.0;
        warp_feval_int<NR, G, true>(M, I, S, rates_at(M, t, invT), true, pR * invT, quot(t, pR), scale, x,
                                    out, lane, grp);
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (lane + G * r < M.nS && c0 < cells) dYdt[(int64_t)(lane + G * r) * ldY + c] = out[r];
    }
}

template <int NR, int G>
static cudaError_t launch_nr(const MechDev& M, int64_t cells, const double* T, const double* p, const double* Y,
                             int64_t ldY, double* dYdt, int nsm, cudaStream_t st)
{
    const int threads = 128, per = threads / G;
    const size_t sm = (size_t)int_smem_words(M, int_tab<G>(M)) * per * 8;
    cudaError_t e = cudaFuncSetAttribute(warp_rates_kernel<NR, G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    int bps = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, warp_rates_kernel<NR, G>, threads, sm);
    if (e != cudaSuccess) return e;
    const int64_t want = (cells + per - 1) / per, fit = (int64_t)nsm * (bps > 0 ? bps : 1);
    warp_rates_kernel<NR, G><<<(int)(want < fit ? want : fit), threads, sm, st>>>(M, cells, T, p, Y, ldY, dYdt);
    return cudaGetLastError();
}

cudaError_t launch_rates_f64(const MechDev& M, int64_t cells, const double* T, const double* p, const double* Y,
                             int64_t ldY, double* dYdt, int nsm, cudaStream_t st)
{
    // Lanes per cell by the mechanism alone, so that a cell's bits do not depend on
    // the call. With few reactions more lanes would only wait; GB300, 400,000 cells,
    // plain FP64 with a lane per cell / more lanes / these: 5 species / 8 reactions
    // 0.223 / 0.291 / 0.189 ms, 10 / 12 0.321 / 0.360 / 0.243, 14 / 20 0.491 / 0.409 /
    // 0.344, 17 / 20 0.515 / 0.941 / 0.455, 20 / 30 0.722 / 0.968 / 0.525; more lanes
    // for 9 / 38 (0.423; 2,000 cells 0.026 against 0.031) and 32 / 80 (1.59; 2,000 cells
    // 0.031 against 0.039).
    if (M.nS <= 8 && M.nR < 24) return launch_nr<2, 4>(M, cells, T, p, Y, ldY, dYdt, nsm, st);
    if (M.nS <= 16 && M.nR < 24) return launch_nr<4, 4>(M, cells, T, p, Y, ldY, dYdt, nsm, st);
    if (M.nS <= 16) return launch_nr<2, 8>(M, cells, T, p, Y, ldY, dYdt, nsm, st);
    if (M.nS <= 32 && M.nR < 40) return launch_nr<4, 8>(M, cells, T, p, Y, ldY, dYdt, nsm, st);
    switch (warp_nr(M.nS, 32)) {
    case 1: return launch_nr<1, 32>(M, cells, T, p, Y, ldY, dYdt, nsm, st);
    case 2: return launch_nr<2, 32>(M, cells, T, p, Y, ldY, dYdt, nsm, st);
    case 4: return launch_nr<4, 32>(M, cells, T, p, Y, ldY, dYdt, nsm, st);
    default: return launch_nr<8, 32>(M, cells, T, p, Y, ldY, dYdt, nsm, st);
    }
}

}  // namespace kin
