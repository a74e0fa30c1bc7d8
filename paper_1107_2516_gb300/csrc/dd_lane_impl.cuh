// Kernel 3: lane-interleaved brute-force de-dispersion (Section 3.1),
//   out[dm][t] = sum_c in[c][t + d(c,dm)].
//
// Block = NW warps sharing one time tile of 32*TI samples; lane l owns
// samples t0 + l + 32*i (i < TI) and each warp owns DR DM trials, so a thread
// accumulates DR x TI outputs.  Per channel the block stages (one TMA bulk
// copy) the input span of all its DM trials; for each DM trial a warp adds
// row[o + l + 32 i] with o the trial's warp-uniform offset: 32 consecutive
// words per load, conflict-free at any alignment, no branches.  Every add
// costs one shared-memory word, so the kernel is bounded by shared-memory
// bandwidth (32 words/clk/SM = 1/4 of the FP32 add rate); it trades kernel
// 2's register reuse for straight-line code and high occupancy.
#pragma once

#include "dd_fast_impl.cuh"

#include <type_traits>

namespace dd {

struct LaneLaunch {
    const void *in;
    int64_t pitch, nsamp_in_al;
    int nchans, ndm;
    int64_t nout;
    const int32_t *offs;   // [nblk][nchans][NW*DR] element offsets within the staged row
    const int32_t *base;   // [nblk][nchans] row start relative to the tile start (aligned)
    int rs, ch, bar_off, nblk;
    int64_t ntile;
    int dgroup;
    void *out, *partials;
    int *err;
    size_t smem;
    int dtype;             // dd_dtype of `in` (batched launches)
    int64_t t_base;        // lane_kernel: first output sample of the launch's tile range
    int kind;              // mixed batch: 0 = this kernel 3 launch, 1 = the beam's kernel 5 launch
    int in_res;            // rows that start anywhere: element of its 16-byte unit that `in` points at
};

template <typename Tin> __device__ __forceinline__ float lane_ld(const Tin *p);
template <> __device__ __forceinline__ float lane_ld<float>(const float *p) { return *p; }
template <> __device__ __forceinline__ float lane_ld<__half>(const __half *p) { return __half2float(*p); }
template <> __device__ __forceinline__ float lane_ld<uint8_t>(const uint8_t *p) { return (float)*p; }

// Swaps a bit of v's index with a bit of the lane's number.  Lanes that hold
// four consecutive samples each (4 l + e) would store words 4 apart, and every
// store of the warp would touch the sectors of four; afterwards each covers 32
// consecutive samples, wherever the row starts (4 channels uint8, 200 trials x
// 30 000 samples: 12.4 us with one sample a lane, 16.5 us with the words apart,
// 12.4 us now).
template <int kReg, int kLane, int N>
__device__ __forceinline__ void swap_with_lane_bit(uint32_t (&v)[N], int lane)
{
    const bool up = lane & kLane;
#pragma unroll
    for (int k = 0; k < N; ++k)
        if (!(k & kReg)) {
            const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? v[k] : v[k | kReg], kLane);
            if (up) v[k] = got;
            else v[k | kReg] = got;
        }
}
// Sample (of 32) in a lane's registers after bits 0 and 1 were swapped with the lane's bits 3 and 4.
__device__ __forceinline__ int quad_sample(int lane) { return 4 * (lane & 7) + (lane >> 3); }

// Sums of bytes, four consecutive samples a step: lane l owns samples 4 l + 128
// i + e (i < TI / 4, e < 4).  A trial's four bytes start anywhere in a word:
// two word loads and a funnel shift, then their even and odd bytes are added
// as pairs of 16 bits over up to four channels, and each pair into two 32-bit
// sums: the word (low + 2^16 high, modulo 2^32) and its high half.  Seven
// instructions for four adds and half the shared-memory words of a byte load
// per add, which also takes a conversion to float (a quarter-rate
// instruction).  Whole numbers: the same results.  A persistent batch of 8
// small beams, 4 of them uint8: 0.97 -> 0.51 ms.
template <int TI, int DR>
struct ByteSums {
    static_assert(TI % 4 == 0 && DR % 4 == 0, "quads of samples, offsets four at a time");
    uint32_t a[DR][TI / 4][2], h[DR][TI / 4][2];   // [..][0]: samples e = 0, 2, [..][1]: e = 1, 3

    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int j = 0; j < DR; ++j)
#pragma unroll
            for (int i = 0; i < TI / 4; ++i)
#pragma unroll
                for (int e = 0; e < 2; ++e) { a[j][i][e] = 0u; h[j][i][e] = 0u; }
    }

    // M channels: their staged rows from `rows` on, rs apart; this warp's
    // trials' offsets from `so` on, os apart, plus xo(c).
    template <int M, typename X>
    __device__ __forceinline__ void add(const uint8_t *rows, int rs, const int32_t *so, int os, int lane, X xo)
    {
        constexpr uint32_t kEven = 0x00ff00ffu;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(rows) + lane;
        const int rw = rs >> 2;
#pragma unroll
        for (int q = 0; q < DR; q += 4) {
            int o[M][4];
#pragma unroll
            for (int c = 0; c < M; ++c) {
                const int4 v = *reinterpret_cast<const int4 *>(so + c * os + q);
                const int x = xo(c);
                o[c][0] = v.x + x; o[c][1] = v.y + x; o[c][2] = v.z + x; o[c][3] = v.w + x;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < TI / 4; ++i) {
                    uint32_t ev = 0, od = 0;
#pragma unroll
                    for (int c = 0; c < M; ++c) {
                        const uint32_t *p = w + c * rw + (o[c][j] >> 2) + 32 * i;
                        const uint32_t x = __funnelshift_r(p[0], p[1], (uint32_t)o[c][j] << 3);
                        ev += x & kEven;
                        od += __byte_perm(x, 0u, 0x4341);
                    }
                    a[q + j][i][0] += ev;
                    a[q + j][i][1] += od;
                    h[q + j][i][0] = __dp2a_lo(ev, 0x0100u, h[q + j][i][0]);   // + the high half
                    h[q + j][i][1] = __dp2a_lo(od, 0x0100u, h[q + j][i][1]);
                }
        }
    }

    template <typename X>
    __device__ __forceinline__ void add_stage(const uint8_t *rows, int rs, const int32_t *so, int os, int cn, int lane, X xo)
    {
        int c = 0;
        for (; c + 4 <= cn; c += 4) add<4>(rows + (size_t)c * rs, rs, so + c * os, os, lane, [&](int k) { return xo(c + k); });
        for (; c < cn; ++c) add<1>(rows + (size_t)c * rs, rs, so + c * os, os, lane, [&](int k) { return xo(c + k); });
    }

    // The sums of trial j's samples 128 i on: v[k] that of sample 128 i + 32 k + quad_sample(lane).
    __device__ __forceinline__ void at(int j, int i, int lane, uint32_t (&v)[4]) const
    {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = e >= 2 ? h[j][i][e & 1] : a[j][i][e] - (h[j][i][e] << 16);
        swap_with_lane_bit<1, 8>(v, lane);
        swap_with_lane_bit<2, 16>(v, lane);
    }
};

// DM block / time tile of linear block index `lin` (DM blocks in groups, time
// tiles slowest within a group, as kernel 2).
template <int TI>
__device__ __forceinline__ void lane_raster(const LaneLaunch &a, int64_t lin, int &blk, int64_t &t0)
{
    const int64_t per_group = (int64_t)a.dgroup * a.ntile;
    const int64_t grp = lin / per_group;
    const int64_t rr = lin - grp * per_group;
    const int gsize = min(a.dgroup, a.nblk - (int)grp * a.dgroup);
    blk = (int)grp * a.dgroup + (int)(rr % gsize);
    t0 = (rr / gsize) * (32 * TI);
}

// One work item: DM block `blk` x the time tile at t0 of the plan in `a`;
// partials record `lin`.  `gstage` is the block's running stage count (the
// mbarrier ring persists across the items of a persistent block: stage s
// of this item uses buffer (gstage+s) % kStages, parity (gstage+s) / kStages).
// Returns false if a bounded wait gave up.
// The tile addresses the block's dynamic shared memory through the extern
// symbol (not a pointer argument), so that its loads and stores stay
// shared-space instructions in the out-of-line copies the persistent kernels
// call.
// kFours (ch a multiple of 4, nchans too): four channels are summed before
// they are added, kernel 5's order with subbands of 4 and so its float sums to
// the bit.  kAny: rows that start anywhere, staged as in share_ws_kernel: whole
// 16-byte units around a row's samples, in rows one unit longer.
template <typename Tin, bool kInt, int TI, int DR, int NW, bool kFours = false, bool kAny = false>
__device__ __forceinline__ bool lane_tile(const LaneLaunch &a, int blk, int64_t t0, int64_t lin,
                                          uint64_t *bar, uint32_t &gstage)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int kDmBlk = DR * NW;
    const Tin *__restrict__ in = static_cast<const Tin *>(a.in);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nchans = a.nchans, rs = a.rs, ch = a.ch;
    const int dm0 = blk * kDmBlk;

    // layout: [kStages][ch][rs] Tin rows | [kStages][ch][kDmBlk] int32 offsets | mbar at bar_off
    const size_t stage_elems = (size_t)ch * rs;
    Tin *rows = reinterpret_cast<Tin *>(smem);
    int32_t *soffs = reinterpret_cast<int32_t *>(smem + kStages * stage_elems * sizeof(Tin));
    const int32_t *boffs = a.offs + (size_t)blk * nchans * kDmBlk;
    const int32_t *bbase = a.base + (size_t)blk * nchans;
    const int nst = (nchans + ch - 1) / ch;
    const uint32_t g0 = gstage;

    // Stage s's copies: lane l of warp w issues row w + NW l, the last warp the
    // offsets too.  A bulk copy holds the thread that issues it some 270 cycles,
    // so the block's copies are spread over its warps (one thread used to issue
    // all of them, and every warp waited for its warp at the stage's barrier:
    // the subband kernel, which has the same body, took 12.06 and 10.03 ms for
    // its stages of the LOFAR-like plan and takes 10.87 and 8.17).  The row's
    // start is loaded one stage early.
    constexpr int kAl = 16 / (int)sizeof(Tin);
    const int pitch_res = (int)(a.pitch & (kAl - 1));
    auto res = [&](int c) { return kAny ? (a.in_res + c * pitch_res) & (kAl - 1) : 0; };
    const int mine = warp + NW * lane;
    int rb = mine < ch ? bbase[min(mine, nchans - 1)] : 0;   // of the next stage to issue
    auto issue = [&](int s) {
        const int buf = (int)((g0 + s) % kStages);
        const int c0 = s * ch;
        const int cn = min(ch, nchans - c0);
        const int most = kAny ? rs - kAl : rs;
        int64_t g = t0 + rb;
        int64_t n = a.nsamp_in_al - g;
        n = n < 0 || mine >= cn ? 0 : (n > most ? most : n);
        if (kAny && n > 0) {
            const int d = res(c0 + mine);
            n = (n + d + kAl - 1) & ~(int64_t)(kAl - 1);
            g -= d;
        }
        const uint32_t nb = (uint32_t)(n * (int64_t)sizeof(Tin)), ob = (uint32_t)(cn * kDmBlk * sizeof(int32_t));
        const uint32_t bytes = __reduce_add_sync(0xffffffffu, nb) + (warp == NW - 1 ? ob : 0u);
        if (lane == 0) {
            mbar_arrive_tx(&bar[buf], bytes);
            if (warp == NW - 1) bulk_g2s(soffs + (size_t)buf * ch * kDmBlk, boffs + (size_t)c0 * kDmBlk, ob, &bar[buf]);
        }
        __syncwarp();
        if (nb)
            bulk_g2s(rows + (size_t)buf * stage_elems + (size_t)mine * rs, in + (size_t)(c0 + mine) * a.pitch + g, nb,
                     &bar[buf]);
        if (mine < ch) rb = bbase[min(c0 + ch + mine, nchans - 1)];
    };

    constexpr bool kBytes = std::is_same<Tin, uint8_t>::value;
    static_assert(kBytes == kInt, "byte input gives integer sums");
    float acc[kBytes ? 1 : DR][kBytes ? 1 : TI];
    ByteSums<kBytes ? TI : 4, kBytes ? DR : 4> bs;
    if constexpr (kBytes) {
        bs.clear();
    } else {
#pragma unroll
        for (int j = 0; j < DR; ++j)
#pragma unroll
            for (int i = 0; i < TI; ++i) acc[j][i] = 0.f;
    }

    for (int s = 0; s < kStages - 1 && s < nst; ++s) issue(s);

    const bool idle = dm0 + warp * DR >= a.ndm;   // none of the warp's trials exist
    bool ok = true;
    for (int s = 0; s < nst; ++s) {
        if (s + kStages - 1 < nst) issue(s + kStages - 1);
        const uint32_t g = g0 + s;
        const int buf = (int)(g % kStages);
        ok = __all_sync(0xffffffffu, mbar_wait(&bar[buf], (g / kStages) & 1u, a.err));
        if (!ok) { sit_out(bar, g0, s, nst, kStages, a.err); break; }
        const int cn = idle ? 0 : min(ch, nchans - s * ch);
        const Tin *srow = rows + (size_t)buf * stage_elems + lane;
        const int32_t *so = soffs + (size_t)buf * ch * kDmBlk + warp * DR;
        const int c0 = s * ch;
        if constexpr (kBytes) bs.add_stage(srow - lane, rs, so, kDmBlk, cn, lane, [&](int c) { return res(c0 + c); });
        else if constexpr (kFours) for (int cc = 0; cc < cn; cc += 4) {
            const Tin *r = srow + (size_t)cc * rs;
#pragma unroll
            for (int j = 0; j < DR; j += 4) {
                int o[4][4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int4 v = *reinterpret_cast<const int4 *>(so + (cc + c) * kDmBlk + j);
                    const int x = res(c0 + cc + c);
                    o[0][c] = v.x + x; o[1][c] = v.y + x; o[2][c] = v.z + x; o[3][c] = v.w + x;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int i = 0; i < TI; ++i) {
                        float v = lane_ld<Tin>(r + o[e][0] + 32 * i);
#pragma unroll
                        for (int c = 1; c < 4; ++c) v += lane_ld<Tin>(r + c * rs + o[e][c] + 32 * i);
                        acc[j + e][i] += v;
                    }
            }
        }
        else for (int cc = 0; cc < cn; ++cc) {
            const Tin *r = srow + (size_t)cc * rs + res(c0 + cc);
            // the warp's DR offsets: uniform 16-byte loads, one shared-memory
            // wavefront per 4 offsets (the data path is the kernel's bound)
            int o[DR];
            static_assert(DR % 4 == 0, "offsets are loaded 4 at a time");
#pragma unroll
            for (int j = 0; j < DR; j += 4) {
                const int4 v = *reinterpret_cast<const int4 *>(so + cc * kDmBlk + j);
                o[j] = v.x; o[j + 1] = v.y; o[j + 2] = v.z; o[j + 3] = v.w;
            }
#pragma unroll
            for (int j = 0; j < DR; ++j) {
                const Tin *p = r + o[j];
#pragma unroll
                for (int i = 0; i < TI; ++i) acc[j][i] += lane_ld<Tin>(p + 32 * i);
            }
        }
        __syncthreads();
    }
    gstage = g0 + nst;
    ok = __syncthreads_and(ok);
    if (!ok) return false;

    // epilogue: lanes hold consecutive samples, so stores are coalesced directly
    const int64_t nout = a.nout;
    if constexpr (kInt) {
        long long n = 0, s = 0;
        unsigned long long q = 0;
        int32_t *out = reinterpret_cast<int32_t *>(a.out);
        const int left = (int)min(nout - t0 - quad_sample(lane), (int64_t)32 * TI);
#pragma unroll
        for (int j = 0; j < DR; ++j) {
            const int dm = dm0 + warp * DR + j;
            int32_t *row = out + (size_t)dm * nout + t0 + quad_sample(lane);
#pragma unroll
            for (int i = 0; i < TI / 4; ++i) {
                uint32_t v[4];
                bs.at(j, i, lane, v);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (dm < a.ndm && 128 * i + 32 * k < left) {
                        row[128 * i + 32 * k] = (int32_t)v[k];
                        n++; s += v[k]; q += (unsigned long long)v[k] * v[k];
                    }
            }
        }
        block_stat_i(n, s, q, reinterpret_cast<StatI *>(a.partials) + lin);
    } else {
        int n = 0;
        float s = 0.f;
        float *out = reinterpret_cast<float *>(a.out);
#pragma unroll
        for (int j = 0; j < DR; ++j) {
            const int dm = dm0 + warp * DR + j;
#pragma unroll
            for (int i = 0; i < TI; ++i) {
                const int64_t t = t0 + lane + 32 * i;
                if (dm < a.ndm && t < nout) {
                    out[(size_t)dm * nout + t] = acc[j][i];
                    n++; s += acc[j][i];
                }
            }
        }
        const float m = n ? s / (float)n : 0.f;
        float q = 0.f;
#pragma unroll
        for (int j = 0; j < DR; ++j) {
            const int dm = dm0 + warp * DR + j;
#pragma unroll
            for (int i = 0; i < TI; ++i) {
                const int64_t t = t0 + lane + 32 * i;
                if (dm < a.ndm && t < nout) { const float d = acc[j][i] - m; q += d * d; }
            }
        }
        block_stat_f32(n, s, q, reinterpret_cast<StatF *>(a.partials) + lin);
    }
    return true;
}

// One plan: one block per work item, grid = nblk * ntile.
template <typename Tin, bool kInt, int TI, int DR, int NW, int MINB, bool kFours = false, bool kAny = false>
__global__ void __launch_bounds__(NW * 32, MINB) lane_kernel(LaneLaunch a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + a.bar_off);
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(&bar[s], NW);
        mbar_fence_init();
    }
    __syncthreads();
    int blk;
    int64_t t0;
    lane_raster<TI>(a, blockIdx.x, blk, t0);
    t0 += a.t_base;
    uint32_t gstage = 0;
    lane_tile<Tin, kInt, TI, DR, NW, kFours, kAny>(a, blk, t0, blockIdx.x, bar, gstage);
}

// lane_tile as an out-of-line function: the persistent kernel calls one per
// input type, each compiled with the full register budget.
template <typename Tin, bool kInt, int TI, int DR, int NW>
__device__ __noinline__ bool lane_tile_call(const LaneLaunch &a, int blk, int64_t t0, int64_t lin,
                                            uint64_t *bar, uint32_t &gstage)
{
    return lane_tile<Tin, kInt, TI, DR, NW>(a, blk, t0, lin, bar, gstage);
}

// Batched plans with kernel 3: a persistent grid (MINB blocks per SM) pulls
// work items (beam, linear tile index) from a device queue, heaviest beams
// first; each beam brings its own tables, buffers and input type.
struct ShareLaunch;

struct LaneBatchLaunch {
    const LaneLaunch *beams;
    const uint2 *items;
    int nitems;
    int bar_off;
    unsigned int *counter;
    const ShareLaunch *sbeams;   // mixed batch: each kind-1 beam's kernel 5 launch
};

template <int TI, int DR, int NW, int MINB>
__global__ void __launch_bounds__(NW * 32, MINB) lane_batch_kernel(LaneBatchLaunch b)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_item;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + b.bar_off);
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(&bar[s], NW);
        mbar_fence_init();
    }
    __syncthreads();
    uint32_t gstage = 0;
    while (true) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(b.counter, 1u);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= b.nitems) break;
        const uint2 w = b.items[it];
        const LaneLaunch &a = b.beams[w.x];
        int blk;
        int64_t t0;
        lane_raster<TI>(a, w.y, blk, t0);
        bool ok;
        switch (a.dtype) {
        case DD_F32: ok = lane_tile_call<float, false, TI, DR, NW>(a, blk, t0, w.y, bar, gstage); break;
        case DD_F16: ok = lane_tile_call<__half, false, TI, DR, NW>(a, blk, t0, w.y, bar, gstage); break;
        default: ok = lane_tile_call<uint8_t, true, TI, DR, NW>(a, blk, t0, w.y, bar, gstage); break;
        }
        if (!ok) break;
        __syncthreads();
        if (threadIdx.x == 0) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
}

template <int TI, int DR, int NW, int MINB, bool kFours = false, bool kAny = false>
cudaError_t lane_launch_cfg(dd_dtype t, const LaneLaunch &a, cudaStream_t s)
{
    const unsigned grid = (unsigned)(a.ntile * a.nblk);
    switch (t) {
    case DD_F32: lane_kernel<float, false, TI, DR, NW, MINB, kFours, kAny><<<grid, NW * 32, a.smem, s>>>(a); break;
    case DD_F16: lane_kernel<__half, false, TI, DR, NW, MINB, kFours, kAny><<<grid, NW * 32, a.smem, s>>>(a); break;
    case DD_U8: lane_kernel<uint8_t, true, TI, DR, NW, MINB, false, kAny><<<grid, NW * 32, a.smem, s>>>(a); break;
    }
    return cudaGetLastError();
}

template <int TI, int DR, int NW, int MINB, bool kFours = false, bool kAny = false>
cudaError_t lane_prepare_one(size_t optin)
{
    cudaError_t e = allow_max_dynamic_smem((const void *)lane_kernel<float, false, TI, DR, NW, MINB, kFours, kAny>, optin);
    if (e == cudaSuccess)
        e = allow_max_dynamic_smem((const void *)lane_kernel<__half, false, TI, DR, NW, MINB, kFours, kAny>, optin);
    if (e == cudaSuccess)
        e = allow_max_dynamic_smem((const void *)lane_kernel<uint8_t, true, TI, DR, NW, MINB, false, kAny>, optin);
    return e;
}

template <int TI, int DR, int NW, int MINB>
cudaError_t lane_prepare_cfg(size_t optin)
{
    cudaError_t e = lane_prepare_one<TI, DR, NW, MINB>(optin);
    if (e == cudaSuccess)
        e = allow_max_dynamic_smem((const void *)lane_batch_kernel<TI, DR, NW, MINB>, optin);
    return e;
}

// Persistent launch: grid = MINB blocks per SM (the occupancy the shared
// memory budget of the configuration allows).
template <int TI, int DR, int NW, int MINB>
cudaError_t lane_batch_launch_cfg(const LaneBatchLaunch &b, int sms, size_t smem, cudaStream_t s)
{
    lane_batch_kernel<TI, DR, NW, MINB><<<sms * MINB, NW * 32, smem, s>>>(b);
    return cudaGetLastError();
}

// Configurations compiled into the library: {samples per lane, DM trials per
// warp, warps per block, resident blocks per SM the register budget targets}.
struct LaneShape { int ti, dr, nw, minb; };
constexpr int kNumLaneCfg = 4;
constexpr LaneShape kLaneCfg[kNumLaneCfg] = {{16, 4, 8, 2}, {16, 8, 8, 1}, {16, 8, 4, 3}, {8, 16, 4, 3}};

// A finer shape for launches whose blocks would not fill the SMs (16 trials x
// 128 samples a block instead of 32 x 512 or kernel 5's 64 x 512): the same
// sums in kernel 3's order or (fours) in kernel 5's.
constexpr LaneShape kLaneSmall = {4, 4, 4, 4};
cudaError_t lane_launch_small(dd_dtype t, const LaneLaunch &a, bool fours, cudaStream_t s);
cudaError_t lane_prepare_small(size_t optin);
// Rows that start anywhere: shape kLaneAny or (small; fours: kFours) kLaneSmall.
constexpr int kLaneAny = 2;
cudaError_t lane_launch_any(dd_dtype t, const LaneLaunch &a, bool small, bool fours, cudaStream_t s);
cudaError_t lane_prepare_any(size_t optin);

cudaError_t lane_launch_c0(dd_dtype t, const LaneLaunch &a, cudaStream_t s);
cudaError_t lane_launch_c1(dd_dtype t, const LaneLaunch &a, cudaStream_t s);
cudaError_t lane_launch_c2(dd_dtype t, const LaneLaunch &a, cudaStream_t s);
cudaError_t lane_launch_c3(dd_dtype t, const LaneLaunch &a, cudaStream_t s);
cudaError_t lane_prepare_c0(size_t optin);
cudaError_t lane_prepare_c1(size_t optin);
cudaError_t lane_prepare_c2(size_t optin);
cudaError_t lane_prepare_c3(size_t optin);
cudaError_t lane_batch_launch_c0(const LaneBatchLaunch &b, int sms, size_t smem, cudaStream_t s);
cudaError_t lane_batch_launch_c1(const LaneBatchLaunch &b, int sms, size_t smem, cudaStream_t s);
cudaError_t lane_batch_launch_c2(const LaneBatchLaunch &b, int sms, size_t smem, cudaStream_t s);
cudaError_t lane_batch_launch_c3(const LaneBatchLaunch &b, int sms, size_t smem, cudaStream_t s);

}  // namespace dd
