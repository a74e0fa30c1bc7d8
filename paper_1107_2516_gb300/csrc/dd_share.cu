// Kernel 5 instantiations (its compiled shapes, three input types).
#include "dd_share_impl.cuh"

namespace dd {

template <int TI, int DR, int NW, int MINB, int NS>
static cudaError_t share_launch_cfg(dd_dtype t, const ShareLaunch &a, cudaStream_t s)
{
    const unsigned grid = (unsigned)(a.ntile * a.nblk);
    switch (t) {
    case DD_F32: share_kernel<float, false, TI, DR, NW, kShCS, kShNP, NS, MINB><<<grid, NW * 32, a.smem, s>>>(a); break;
    case DD_F16: share_kernel<__half, false, TI, DR, NW, kShCS, kShNP, NS, MINB><<<grid, NW * 32, a.smem, s>>>(a); break;
    case DD_U8: share_kernel<uint8_t, true, TI, DR, NW, kShCS, kShNP, NS, MINB><<<grid, NW * 32, a.smem, s>>>(a); break;
    }
    return cudaGetLastError();
}

template <int TI, int DR, int NW, int MINB, int NS>
static cudaError_t share_prepare_cfg(size_t optin)
{
    cudaError_t e = allow_max_dynamic_smem((const void *)share_kernel<float, false, TI, DR, NW, kShCS, kShNP, NS, MINB>, optin);
    if (e == cudaSuccess)
        e = allow_max_dynamic_smem((const void *)share_kernel<__half, false, TI, DR, NW, kShCS, kShNP, NS, MINB>, optin);
    if (e == cudaSuccess)
        e = allow_max_dynamic_smem((const void *)share_kernel<uint8_t, true, TI, DR, NW, kShCS, kShNP, NS, MINB>, optin);
    return e;
}

// The warp-specialised shape: PW stage-1 warps + NW stage-2 warps per block,
// subbands of 4 or 8 channels, rows on 16-byte boundaries or anywhere.
using ShareWsFn = void (*)(ShareLaunch);

template <int TI, int DR, int NW, int PW, int PB, int CS, bool kAny>
static ShareWsFn share_ws_fn(dd_dtype t)
{
    switch (t) {
    case DD_F32: return share_ws_kernel<float, false, TI, DR, NW, PW, CS, kShNP, PB, kAny>;
    case DD_F16: return share_ws_kernel<__half, false, TI, DR, NW, PW, CS, kShNP, PB, kAny>;
    default: return share_ws_kernel<uint8_t, true, TI, DR, NW, PW, CS, kShNP, PB, kAny>;
    }
}

template <int TI, int DR, int NW, int PW, int PB>
static ShareWsFn share_ws_fn(dd_dtype t, int cs, bool any)
{
    if (cs == 8) return any ? share_ws_fn<TI, DR, NW, PW, PB, 8, true>(t) : share_ws_fn<TI, DR, NW, PW, PB, 8, false>(t);
    return any ? share_ws_fn<TI, DR, NW, PW, PB, 4, true>(t) : share_ws_fn<TI, DR, NW, PW, PB, 4, false>(t);
}

template <int TI, int DR, int NW, int PW, int PB>
static cudaError_t share_ws_launch_cfg(dd_dtype t, const ShareLaunch &a, cudaStream_t s)
{
    share_ws_fn<TI, DR, NW, PW, PB>(t, a.cs, a.shifted)<<<(unsigned)(a.ntile * a.nblk), (NW + PW + kWsStage) * 32, a.smem, s>>>(a);
    return cudaGetLastError();
}

template <int TI, int DR, int NW, int PW, int PB>
static cudaError_t share_ws_prepare_cfg(size_t optin)
{
    cudaError_t e = cudaSuccess;
    for (dd_dtype t : {DD_F32, DD_F16, DD_U8})
        for (int form = 0; form < 4; ++form)
            if (e == cudaSuccess)
                e = allow_max_dynamic_smem((const void *)share_ws_fn<TI, DR, NW, PW, PB>(t, form & 1 ? 8 : 4, form & 2), optin);
    return e;
}

template <int TI, int DR, int NW, int PW, int PB>
static bool share_ws_regs_ok_cfg(dd_dtype t)
{
    using Regs = WsRegs<NW, PW>;
    for (int form = 0; form < 4; ++form) {
        cudaFuncAttributes at{};
        if (cudaFuncGetAttributes(&at, (const void *)share_ws_fn<TI, DR, NW, PW, PB>(t, form & 1 ? 8 : 4, form & 2)) != cudaSuccess ||
            at.numRegs < Regs::kNeed)
            return false;
    }
    return true;
}

#define DD_SHARE_CFG(k) kShareCfg[k].ti, kShareCfg[k].dr, kShareCfg[k].nw, kShareCfg[k].minb, kShareCfg[k].ns
#define DD_SHARE_WS_CFG(k) kShareCfg[k].ti, kShareCfg[k].dr, kShareCfg[k].nw, kShareCfg[k].pw, kShareCfg[k].pb
static_assert(kNumShareCfg == 4, "one case per compiled shape");
static_assert(kShareCfg[0].pw == 0 && kShareCfg[1].pw == 0 && kShareCfg[2].pw == 0 && kShareCfg[3].pw > 0,
              "shapes 0-2 are the one-barrier kernel, shape 3 the warp-specialised one");

cudaError_t share_launch(int k, dd_dtype t, const ShareLaunch &a, cudaStream_t s)
{
    switch (k) {
    case 0: return share_launch_cfg<DD_SHARE_CFG(0)>(t, a, s);
    case 1: return share_launch_cfg<DD_SHARE_CFG(1)>(t, a, s);
    case 2: return share_launch_cfg<DD_SHARE_CFG(2)>(t, a, s);
    default: return share_ws_launch_cfg<DD_SHARE_WS_CFG(3)>(t, a, s);
    }
}

cudaError_t share_prepare(int k, size_t optin)
{
    switch (k) {
    case 0: return share_prepare_cfg<DD_SHARE_CFG(0)>(optin);
    case 1: return share_prepare_cfg<DD_SHARE_CFG(1)>(optin);
    case 2: return share_prepare_cfg<DD_SHARE_CFG(2)>(optin);
    default: return share_ws_prepare_cfg<DD_SHARE_WS_CFG(3)>(optin);
    }
}

bool share_regs_ok(int k, dd_dtype t)
{
    switch (k) {
    case 3: return share_ws_regs_ok_cfg<DD_SHARE_WS_CFG(3)>(t);
    default: return true;
    }
}

// Mixed persistent batch: kernel 5 shape 0 with kernel 3 shape 2.
constexpr ShareShape kMS = kShareCfg[kMixedShare];
constexpr LaneShape kML = kLaneCfg[kMixedLane];
static_assert(kMS.ti == kML.ti && kMS.dr == kML.dr && kMS.nw == kML.nw && kMS.minb == kML.minb,
              "the mixed batch's kernel 3 and kernel 5 shapes must share the block geometry");

cudaError_t mixed_batch_launch(const LaneBatchLaunch &b, int sms, size_t smem, cudaStream_t s)
{
    mixed_batch_kernel<kMS.ti, kMS.dr, kMS.nw, kShCS, kShNP, kMS.ns, kMS.minb><<<sms * kMS.minb, kMS.nw * 32, smem, s>>>(b);
    return cudaGetLastError();
}

int mixed_batch_occupancy(size_t smem)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, mixed_batch_kernel<kMS.ti, kMS.dr, kMS.nw, kShCS, kShNP, kMS.ns, kMS.minb>, kMS.nw * 32, smem) !=
        cudaSuccess)
        return 0;
    return n;
}

cudaError_t mixed_batch_prepare(size_t optin)
{
    return allow_max_dynamic_smem((const void *)mixed_batch_kernel<kMS.ti, kMS.dr, kMS.nw, kShCS, kShNP, kMS.ns, kMS.minb>,
                                  optin);
}

}  // namespace dd
