// inst_warp_energy_f64.cu -- the warp-per-cell RKC kernels with the
// energy equation (Eq. (E:energy)), double rate arithmetic and the default
// register budget (own translation unit so the build runs in parallel).
#include "warp.cuh"

namespace kin {

cudaError_t launch_warp_f64_en_o0(Launch& L, int blocks, int threads, cudaStream_t st)
{
    return warp_launch<double, 0, true>(L, blocks, threads, st);
}

cudaError_t occ_warp_f64_en_o0(const MechDev& M, int nV, int lanes, int threads, int* bps)
{
    return warp_occ<double, 0, true>(M, nV, lanes, KIN_FP64, threads, bps);
}

}  // namespace kin
