// Kernel 3 instantiations for rows that start anywhere: kLaneCfg[kLaneAny] and kLaneSmall.
#include "dd_lane_impl.cuh"

namespace dd {

constexpr LaneShape kA = kLaneCfg[kLaneAny], kS = kLaneSmall;

cudaError_t lane_launch_any(dd_dtype t, const LaneLaunch &a, bool small, bool fours, cudaStream_t s)
{
    if (small && fours) return lane_launch_cfg<kS.ti, kS.dr, kS.nw, kS.minb, true, true>(t, a, s);
    return small ? lane_launch_cfg<kS.ti, kS.dr, kS.nw, kS.minb, false, true>(t, a, s)
                 : lane_launch_cfg<kA.ti, kA.dr, kA.nw, kA.minb, false, true>(t, a, s);
}

cudaError_t lane_prepare_any(size_t optin)
{
    cudaError_t e = lane_prepare_one<kS.ti, kS.dr, kS.nw, kS.minb, false, true>(optin);
    if (e == cudaSuccess) e = lane_prepare_one<kS.ti, kS.dr, kS.nw, kS.minb, true, true>(optin);
    return e != cudaSuccess ? e : lane_prepare_one<kA.ti, kA.dr, kA.nw, kA.minb, false, true>(optin);
}

}  // namespace dd
