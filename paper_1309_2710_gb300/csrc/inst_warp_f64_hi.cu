// inst_warp_f64_hi.cu -- the warp-per-cell RKC kernels with double rate arithmetic and
// the high-occupancy register budget (own translation unit so the build runs in
// parallel).
#include "warp.cuh"

namespace kin {

cudaError_t launch_warp_f64_o1(Launch& L, int blocks, int threads, cudaStream_t st)
{
    return warp_launch<double, 1, false>(L, blocks, threads, st);
}

cudaError_t occ_warp_f64_o1(const MechDev& M, int nV, int lanes, int threads, int* bps)
{
    return warp_occ<double, 1, false>(M, nV, lanes, KIN_FP64, threads, bps);
}

}  // namespace kin
