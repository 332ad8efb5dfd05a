// inst_lane_int.cu -- the lane kernels with the integer FP64 f, both methods
// and register budgets (own translation unit so the build runs in parallel).
#include "lane_int.cuh"

namespace kin {

static size_t lane_int_smem(const MechDev& M, int threads)
{
    return (size_t)threads * lane_int_bytes(M.nS, M.li_tb);
}

template <int METHOD>
static cudaError_t launch_m(Launch& L, int occ, int blocks, int threads, cudaStream_t st)
{
    const size_t sm = lane_int_smem(L.M, threads);
    return occ ? launch_all<METHOD, double, 0, 1, false, IntF>(L, blocks, threads, st, sm)
               : launch_all<METHOD, double, 0, 0, false, IntF>(L, blocks, threads, st, sm);
}

cudaError_t launch_lane_int(Launch& L, int occ, int blocks, int threads, cudaStream_t st)
{
    return L.method == KIN_RKCK ? launch_m<KIN_RKCK>(L, occ, blocks, threads, st)
                                : launch_m<KIN_RKC>(L, occ, blocks, threads, st);
}

cudaError_t occ_lane_int(const MechDev& M, int method, int occ, int threads, int* bps)
{
    const size_t sm = lane_int_smem(M, threads);
    if (method == KIN_RKCK)
        return occ ? occ_one<KIN_RKCK, double, 0, 1, false, IntF>(threads, sm, bps)
                   : occ_one<KIN_RKCK, double, 0, 0, false, IntF>(threads, sm, bps);
    return occ ? occ_one<KIN_RKC, double, 0, 1, false, IntF>(threads, sm, bps)
               : occ_one<KIN_RKC, double, 0, 0, false, IntF>(threads, sm, bps);
}

}  // namespace kin
