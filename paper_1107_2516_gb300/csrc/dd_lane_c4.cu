// Kernel 3 instantiation of kLaneSmall, the shape of launches with few blocks.
#include "dd_lane_impl.cuh"

namespace dd {

cudaError_t lane_launch_small(dd_dtype t, const LaneLaunch &a, bool fours, cudaStream_t s)
{
    return fours ? lane_launch_cfg<kLaneSmall.ti, kLaneSmall.dr, kLaneSmall.nw, kLaneSmall.minb, true>(t, a, s)
                 : lane_launch_cfg<kLaneSmall.ti, kLaneSmall.dr, kLaneSmall.nw, kLaneSmall.minb>(t, a, s);
}

cudaError_t lane_prepare_small(size_t optin)
{
    const cudaError_t e = lane_prepare_one<kLaneSmall.ti, kLaneSmall.dr, kLaneSmall.nw, kLaneSmall.minb>(optin);
    return e != cudaSuccess ? e : lane_prepare_one<kLaneSmall.ti, kLaneSmall.dr, kLaneSmall.nw, kLaneSmall.minb, true>(optin);
}

}  // namespace dd
