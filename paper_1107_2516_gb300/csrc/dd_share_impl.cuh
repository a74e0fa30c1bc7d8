// Kernel 5: the Section 3.1 sum with exactly shared subband partial sums,
//   out[dm][t] = sum_c in[c][t + d(c,dm)]
//              = sum_s P_s,pat(dm)[t + d(ref(s),dm)],
//   P_s,pat[u] = sum_{c in s} in[c][u + r_pat(c)],  r_pat(c) = d(c,dm) - d(ref(s),dm),
// over subbands s of CS consecutive channels, ref(s) the subband's channel
// with the smallest delay.  DM trials of a block whose relative delays
// r(c) within a subband coincide (a "pattern") share one partial sum: the
// result is exactly the brute-force sum (same integer delays; FP32 rounding
// order differs), computed with about #patterns x (CS + 1) + #trials
// shared-memory words per subband and output sample instead of #trials x CS.
//
// Block = NW warps on a tile of 32*TI samples (lanes interleaved as kernel 3)
// and DR*NW DM trials.  Per subband (one TMA stage: its CS input rows and
// its table record):
//   stage 1: the block forms every pattern's partial sum over the samples
//            its trials need (P, double-buffered in shared memory).  The
//            patterns' sums are laid end to end in one index space e < E,
//            cut into rows of 32 (each row inside one pattern), and each warp
//            sums the contiguous run of rows the table assigns it, several
//            rows per step: the pattern's fields are uniform in the warp and
//            reloaded only where a pattern ends, and every warp gets the same
//            number of rows;
//   stage 2: each warp adds, for its trials, P_pat[t + offset] (one
//            conflict-free shared word per add, as kernel 3).
// One-barrier shapes (share_tile): one __syncthreads per subband; stage 1 of
// subband s+1 writes the other P buffer while stage 2 of s reads this one;
// each warp takes its trials' offsets into registers during stage 1 (the
// stage's record may be reused by the next copy before stage 2 ends).  The
// input ring has NS stages: NS - 1 subbands' copies are in flight while one is
// summed.  The tile body serves the one-plan kernel and the persistent batch
// kernel.  Warp-specialised shape: share_ws_kernel below.
#pragma once

#include "dd_lane_impl.cuh"

#include <type_traits>

namespace dd {

// Table record of one (DM block, subband), int32 (16-byte multiple):
//   [0 .. DB) q_j (index into P of trial j's t = t0 term) | [DB] E (the
//   subband's P length) | 3 unused |
//   per pattern p < NPMAX, kPatLen words: {end_p, b_0 .. b_{CS-1}, start_p,
//   rows_p, unused} |
//   stage-1 split: [kWarp + w] (w <= kMaxWarps) first row of warp w (the
//   row count R at w = the block's warp count), [kWarp + kMaxWarps + 1 + w]
//   the pattern holding that row.
// start_p / end_p = the index range of pattern p's sums in P; b_c such that
// the term of channel c in P[e] (e in pattern p) is staged element b_c + e of
// the stage's rows (b_c = c * rs + the row offset of the pattern's first
// sample minus start_p); rows_p = the rows of 32 sums before pattern p (the
// patterns' sums are cut into rows of 32, each row inside one pattern).
// Records of packed sums (uint8 input in the warp-specialised shape) have the
// same layout and count P in quads of four sums: start_p, end_p and rows of 32
// are in quads, staged element b_c + 4 e is channel c's term of quad e's first
// sum, and q_j is the word that holds trial j's first pair (see the kernel).
template <int CS, int NPMAX, int DB>
struct ShareRec {
    static_assert(DB % 4 == 0, "trial offsets are loaded 4 at a time");
    static constexpr int kTrial = 0;
    static constexpr int kE = DB;
    static constexpr int kPat = DB + 4;                 // first pattern field (16-byte aligned)
    static constexpr int kPatLen = (CS + 3 + 3) / 4 * 4;   // end, CS row offsets, start, rows before
    static constexpr int kPatStart = 1 + CS, kPatRows = 2 + CS;
    static constexpr int kMaxWarps = 8;
    static constexpr int kWarp = kPat + NPMAX * kPatLen;
    static constexpr int kLen = kWarp + (2 * kMaxWarps + 1 + 3) / 4 * 4;
};

struct ShareLaunch {
    const void *in;
    int64_t pitch, nsamp_in_al;
    int nchans, ndm, nsub;
    int64_t nout;
    const int32_t *rec;    // [nblk][nsub][kLen]
    const int32_t *base;   // [nblk][nchans] staged row start relative to the tile start (aligned)
    const int32_t *rlen;   // [nblk][nchans] elements of that row the block's trials read (<= rs, aligned)
    int rs, pmax, bar_off, nblk;
    int64_t ntile;         // tiles of this launch, starting at output sample t_base
    int64_t t_base;
    int dgroup;
    void *out, *partials;
    int *err;
    size_t smem;
    int skew;              // 1: DM block b takes the time tiles in a rotated order (share_raster)
    // warp-specialised shape
    int cs;                // channels per subband: 4 or 8
    int ns;                // input stages
    int shifted;           // 1: rows start anywhere (in or pitch not 16-byte aligned)
    int in_res;            // element of its 16-byte unit that `in` points at
};

// DM block / time tile of linear block index `lin`, as lane_raster, and with
// a.skew set (a launch over every time tile of the plan) each DM block's
// tiles rotated back by its own delay offset: block b takes tile (s - k_b)
// mod ntile where lane_raster gives tile s, k_b = the block's row start in
// the middle channel in whole tiles.  Blocks that run at the same time then
// stage nearly the same input columns instead of windows up to the whole
// delay span apart, so the staged input stays in L2 between them.  A
// permutation of each block's tiles: every (block, tile) is still taken once.
template <int TI>
__device__ __forceinline__ void share_raster(const ShareLaunch &a, int64_t lin, int &blk, int64_t &t0)
{
    LaneLaunch r{};
    r.dgroup = a.dgroup; r.ntile = a.ntile; r.nblk = a.nblk;
    lane_raster<TI>(r, lin, blk, t0);
    if (a.skew) {
        constexpr int64_t kTile = 32 * TI;
        const int64_t k = ((int64_t)a.base[(size_t)blk * a.nchans + a.nchans / 2] / kTile) % a.ntile;
        t0 = ((t0 / kTile + a.ntile - k) % a.ntile) * kTile;
    }
}

// Stage 1 of one subband: P[e] for e < E (the patterns' sums end to end).
// Each pattern's sums form rows of 32 consecutive e (the last one partial);
// warp w takes the contiguous rows the record assigns it (the host splits
// the R rows in order, equal shares), so a row's pattern (its fields) is
// uniform in the warp and changes only at pattern ends, and lane l sums
// element row_start + l of each of its rows: whole rows RPS at a time with
// the pattern's offsets set up once (every load of a step issued before its
// stores), then the pattern's leftover rows in predicated steps of LRS rows.
// xo[c] is added to channel c's staged elements (rows that start anywhere).
template <typename Tin, typename R, int CS, int NW, int RPS = 4, int LRS = RPS>
__device__ __forceinline__ void share_stage1(const int32_t *rec, const Tin *srow, float *Pb, int warp, int lane,
                                             const int (&xo)[CS])
{
    static_assert(NW <= R::kMaxWarps, "stage-1 split recorded for at most kMaxWarps warps");
    int r = rec[R::kWarp + warp];
    const int r1 = rec[R::kWarp + warp + 1];
    int p = rec[R::kWarp + R::kMaxWarps + 1 + warp];
    while (r < r1) {
        const int32_t *pr = rec + R::kPat + p * R::kPatLen;
        int b[R::kPatLen];
#pragma unroll
        for (int v = 0; v < R::kPatLen; v += 4) {
            const int4 x = *reinterpret_cast<const int4 *>(pr + v);
            b[v] = x.x; b[v + 1] = x.y; b[v + 2] = x.z; b[v + 3] = x.w;
        }
        const int pend = b[0], pst = b[R::kPatStart], pexcl = b[R::kPatRows];
        const int rend = min(r1, pexcl + ((pend - pst + 31) >> 5));
        const int rfull = min(rend, pexcl + ((pend - pst) >> 5));    // rows wholly inside the pattern
        // row r's element for this lane: e = e0 + 32 r
        const int e0 = pst - (pexcl << 5) + lane;
        int src[CS];                                                   // staged element of channel c at e0
#pragma unroll
        for (int c = 0; c < CS; ++c) src[c] = b[1 + c] + xo[c] + e0;
        for (; r + RPS <= rfull; r += RPS) {
            // all RPS x CS loads before the RPS stores: the staged rows and P
            // are both shared memory, so the compiler may not move a store
            // above a later load
            float x[RPS][CS];
#pragma unroll
            for (int u = 0; u < RPS; ++u)
#pragma unroll
                for (int c = 0; c < CS; ++c) x[u][c] = lane_ld<Tin>(srow + (src[c] + ((r + u) << 5)));
#pragma unroll
            for (int u = 0; u < RPS; ++u) {
                float v = x[u][0];
#pragma unroll
                for (int c = 1; c < CS; ++c) v += x[u][c];
                Pb[e0 + ((r + u) << 5)] = v;
            }
        }
        for (; r < rend; r += LRS) {
            // the pattern's leftover rows (fewer than RPS whole rows and the
            // partial last one), LRS per step; only the rows and lanes inside
            // the pattern load and store
            float x[LRS][CS];
            bool in[LRS];
#pragma unroll
            for (int u = 0; u < LRS; ++u) {
                const int o = (r + u) << 5;
                in[u] = r + u < rend && e0 + o < pend;
#pragma unroll
                for (int c = 0; c < CS; ++c) x[u][c] = in[u] ? lane_ld<Tin>(srow + (src[c] + o)) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < LRS; ++u) {
                float v = x[u][0];
#pragma unroll
                for (int c = 1; c < CS; ++c) v += x[u][c];
                if (in[u]) Pb[e0 + ((r + u) << 5)] = v;
            }
        }
        r = rend;
        ++p;
    }
}

// Stage 1 on bytes: lane l sums the four consecutive sums (a quad) of element
// l of each of its rows of 32 quads.  Channel c's four bytes start anywhere in
// a word: two word loads, one funnel shift, and their even and odd bytes are
// added as pairs of 16-bit sums (whole numbers of at most 8 x 255: exact).  Stage 2 reads pairs of
// sums (u, u + 1) at any u, so P is stored twice, as pairs from even u (Pe)
// and from odd u (Po); the pair that ends in the next quad takes that quad's
// first sum from the bytes behind the four, one permute per two channels.
// Per quad and lane 2 CS + 4 shared words for four sums, against 4 (CS + 1)
// with one byte load (and a conversion to float) per term; stage 2 reads half
// the words.  Bound by instructions, no longer by shared memory (ncu: issue
// 75%, shared-memory wavefronts 65% of their peaks).  LOFAR-like beam of 2^18
// uint8 samples, 2000 trials: 30.0 -> 20.2 ms; 4096 channels x 65536 samples,
// 1500 trials: 24.7 -> 13.5 ms.  Exact step sizes for the rows that are left,
// and the high half added with one dp2a instead of a shift and an add, are
// 1.10x of that.
template <typename R, int CS, int NW>
__device__ __forceinline__ void share_stage1_bytes(const int32_t *rec, const uint8_t *srow, uint32_t *Pe, uint32_t *Po,
                                                   int warp, int lane, const int (&xo)[CS])
{
    static_assert(NW <= R::kMaxWarps, "stage-1 split recorded for at most kMaxWarps warps");
    constexpr uint32_t kEven = 0x00ff00ffu;
    const uint32_t *words = reinterpret_cast<const uint32_t *>(srow);
    int r = rec[R::kWarp + warp];
    const int r1 = rec[R::kWarp + warp + 1];
    int p = rec[R::kWarp + R::kMaxWarps + 1 + warp];
    while (r < r1) {
        const int32_t *pr = rec + R::kPat + p * R::kPatLen;
        int b[R::kPatLen];
#pragma unroll
        for (int v = 0; v < R::kPatLen; v += 4) {
            const int4 x = *reinterpret_cast<const int4 *>(pr + v);
            b[v] = x.x; b[v + 1] = x.y; b[v + 2] = x.z; b[v + 3] = x.w;
        }
        const int pend = b[0], pst = b[R::kPatStart], pexcl = b[R::kPatRows];
        const int rend = min(r1, pexcl + ((pend - pst + 31) >> 5));
        int g = pst + ((r - pexcl) << 5) + lane;               // this lane's quad of row r
        int src[CS];                                            // its first word of each channel, at g = 0
        uint32_t sh[CS], sel[CS / 2];
#pragma unroll
        for (int c = 0; c < CS; ++c) {
            const int e = b[1 + c] + xo[c];
            src[c] = e >> 2;
            sh[c] = (uint32_t)e << 3;                           // funnel shifts take it modulo 32
        }
#pragma unroll
        for (int c = 0; c < CS; c += 2)                         // the bytes behind the four
            sel[c / 2] = ((b[1 + c] + xo[c]) & 3) | (((b[2 + c] + xo[c + 1]) & 3) << 8) | 0x400;
        // kRows rows from row r on, all loads before the first store.  Lanes past
        // the pattern's end load too, at most 132 bytes behind the staged
        // rows: records and slots follow them.
        auto rows = [&](auto n) {
            constexpr int kRows = decltype(n)::value;
            uint32_t lo[kRows][CS], hi[kRows][CS];
#pragma unroll
            for (int u = 0; u < kRows; ++u)
#pragma unroll
                for (int c = 0; c < CS; ++c) {
                    lo[u][c] = words[src[c] + g + 32 * u];
                    hi[u][c] = words[src[c] + g + 32 * u + 1];
                }
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                uint32_t ev = 0, od = 0, nx = 0;
#pragma unroll
                for (int c = 0; c < CS; ++c) {
                    const uint32_t x = __funnelshift_r(lo[u][c], hi[u][c], sh[c]);
                    ev += x & kEven;
                    od += __byte_perm(x, 0u, 0x4341);
                }
#pragma unroll
                for (int c = 0; c < CS; c += 2) nx += __byte_perm(hi[u][c], hi[u][c + 1], sel[c / 2]) & kEven;
                nx += nx >> 16;
                if (u + 1 < kRows || g + 32 * u < pend) {       // only the last row can be partial
                    const int w = 2 * (g + 32 * u);
                    *reinterpret_cast<uint2 *>(Pe + w) = make_uint2(__byte_perm(ev, od, 0x5410), __byte_perm(ev, od, 0x7632));
                    *reinterpret_cast<uint2 *>(Po + w) = make_uint2(__byte_perm(od, ev, 0x7610), __byte_perm(od, nx, 0x5432));
                }
            }
        };
        // 32 loads a step, then the leftover rows (pairs only: 5% longer)
        constexpr int kStep = CS == 4 ? 4 : 2;
        auto step = [&](auto n) {
            rows(n);
            r += decltype(n)::value;
            g += 32 * decltype(n)::value;
        };
        while (r + kStep <= rend) step(std::integral_constant<int, kStep>());
        if (kStep == 4 && r + 2 <= rend) step(std::integral_constant<int, 2>());
        if (r < rend) step(std::integral_constant<int, 1>());
        ++p;
    }
}

// One thread's share of the block's partial statistics.
template <bool kInt> struct ShareStat;
template <> struct ShareStat<true> { long long n = 0, s = 0; unsigned long long q = 0; };
template <> struct ShareStat<false> { int n = 0; float s = 0.f, q = 0.f; };

// Store one warp's DR trials x 32*TI samples and accumulate their statistics.
template <bool kInt, int TI, int DR>
__device__ __forceinline__ void share_store(const ShareLaunch &a, const float (&acc)[DR][TI], int dmw, int64_t t0,
                                            int lane, ShareStat<kInt> &st)
{
    const int64_t nout = a.nout;
    if constexpr (kInt) {
        int32_t *out = reinterpret_cast<int32_t *>(a.out);
#pragma unroll
        for (int j = 0; j < DR; ++j) {
            const int dm = dmw + j;
#pragma unroll
            for (int i = 0; i < TI; ++i) {
                const int64_t t = t0 + lane + 32 * i;
                if (dm < a.ndm && t < nout) {
                    const long long v = __float2int_rn(acc[j][i]);
                    __stcs(&out[(size_t)dm * nout + t], (int32_t)v);
                    st.n++; st.s += v; st.q += (unsigned long long)(v * v);
                }
            }
        }
    } else {
        float *out = reinterpret_cast<float *>(a.out);
#pragma unroll
        for (int j = 0; j < DR; ++j) {
            const int dm = dmw + j;
#pragma unroll
            for (int i = 0; i < TI; ++i) {
                const int64_t t = t0 + lane + 32 * i;
                if (dm < a.ndm && t < nout) {
                    __stcs(&out[(size_t)dm * nout + t], acc[j][i]);   // streamed: read back only by the search
                    st.n++; st.s += acc[j][i];
                }
            }
        }
        const float m = st.n ? st.s / (float)st.n : 0.f;
#pragma unroll
        for (int j = 0; j < DR; ++j) {
            const int dm = dmw + j;
#pragma unroll
            for (int i = 0; i < TI; ++i) {
                const int64_t t = t0 + lane + 32 * i;
                if (dm < a.ndm && t < nout) { const float d = acc[j][i] - m; st.q += d * d; }
            }
        }
    }
}

// The same for sums kept as pairs (packed stage 2): lane l's pair i holds the
// samples t0 + 2 l + 64 i and the next one; a = low + 2^16 high and h = high
// of the pair, modulo 2^32.
template <int TI, int DR>
__device__ __forceinline__ void share_store_pairs(const ShareLaunch &a, const uint32_t (&s)[DR][TI / 2],
                                                  const uint32_t (&h)[DR][TI / 2], int dmw, int64_t t0, int lane,
                                                  ShareStat<true> &st)
{
    int32_t *out = reinterpret_cast<int32_t *>(a.out);
#pragma unroll
    for (int j = 0; j < DR; ++j) {
        const int dm = dmw + j;
        if (dm >= a.ndm) break;
        int32_t *row = out + (size_t)dm * a.nout;
#pragma unroll
        for (int i = 0; i < TI / 2; ++i) {
            const uint32_t v[2] = {s[j][i] - (h[j][i] << 16), h[j][i]};
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t t = t0 + 2 * lane + 64 * i + e;
                if (t < a.nout) {
                    __stcs(row + t, (int32_t)v[e]);
                    st.n++; st.s += v[e]; st.q += (unsigned long long)v[e] * v[e];
                }
            }
        }
    }
}

// The block's partial statistics into record `lin` (every thread of the
// block calls this).
template <bool kInt>
__device__ __forceinline__ void share_stat_flush(const ShareLaunch &a, const ShareStat<kInt> &st, int64_t lin)
{
    if constexpr (kInt)
        block_stat_i(st.n, st.s, st.q, reinterpret_cast<StatI *>(a.partials) + lin);
    else
        block_stat_f32(st.n, st.s, st.q, reinterpret_cast<StatF *>(a.partials) + lin);
}

// One work item: DM block `blk` x the time tile at t0; partial statistics
// record `lin`.  bar[NS] is the block's input ring; `gstage` its running stage
// count (a persistent block keeps the ring across items: subband s of this
// item uses buffer (gstage + s) % NS, parity ((gstage + s) / NS) & 1; each
// warp arrives once per stage).
// Returns false if a bounded wait gave up.
template <typename Tin, bool kInt, int TI, int DR, int NW, int CS, int NPMAX, int NS>
__device__ __forceinline__ bool share_tile(const ShareLaunch &a, int blk, int64_t t0, int64_t lin,
                                           uint64_t *bar, uint32_t &gstage)
{
    extern __shared__ __align__(128) unsigned char smem[];   // as lane_tile: shared-space accesses
    constexpr int kDmBlk = DR * NW, kT = NW * 32;
    using R = ShareRec<CS, NPMAX, kDmBlk>;
    const Tin *__restrict__ in = static_cast<const Tin *>(a.in);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rs = a.rs, nsub = a.nsub;
    const int dm0 = blk * kDmBlk;

    // layout: [NS][CS][rs] Tin rows | [NS][kLen] int32 records | [2][pmax] float P
    const size_t stage_elems = (size_t)CS * rs;
    Tin *rows = reinterpret_cast<Tin *>(smem);
    int32_t *srec = reinterpret_cast<int32_t *>(smem + NS * stage_elems * sizeof(Tin));
    float *P = reinterpret_cast<float *>(srec + NS * R::kLen);
    const int32_t *brec = a.rec + (size_t)blk * nsub * R::kLen;
    const uint32_t g0 = gstage;
    gstage += (uint32_t)nsub;

    // Warp w < CS issues row w of subband s, the last warp the record: a bulk
    // copy holds the thread that issues it some 270 cycles, so they are spread.
    // A row's start and length are loaded one subband early (the global loads'
    // latency stays off the barrier path); the row is the rl elements that
    // the block's DM trials read from column t0 + b on, cut at the input's end.
    static_assert(CS <= NW, "a warp per row");
    int rb = 0, rl = 0;                                // of the next subband to issue
    auto load_rb = [&](int s) {
        const size_t i = (size_t)blk * a.nchans + s * CS + min(warp, CS - 1);
        rb = a.base[i];
        rl = a.rlen[i];
    };
    auto issue = [&](int s) {
        if (lane != 0) return;
        const int buf = (int)((g0 + s) % NS);
        const int64_t g = t0 + rb;
        int64_t n = a.nsamp_in_al - g;
        n = n < 0 || warp >= CS ? 0 : (n > rl ? rl : n);
        const uint32_t nb = (uint32_t)(n * (int64_t)sizeof(Tin)), rec_b = (uint32_t)(R::kLen * sizeof(int32_t));
        mbar_arrive_tx(&bar[buf], nb + (warp == NW - 1 ? rec_b : 0u));
        if (warp == NW - 1) bulk_g2s(srec + (size_t)buf * R::kLen, brec + (size_t)s * R::kLen, rec_b, &bar[buf]);
        if (nb)
            bulk_g2s_hint(rows + (size_t)buf * stage_elems + (size_t)warp * rs, in + (size_t)(s * CS + warp) * a.pitch + g,
                          nb, &bar[buf], l2_evict_last());   // other DM blocks of this tile stage these rows soon
    };

    float acc[DR][TI];
#pragma unroll
    for (int j = 0; j < DR; ++j)
#pragma unroll
        for (int i = 0; i < TI; ++i) acc[j][i] = 0.f;

    for (int s = 0; s < NS - 1 && s < nsub; ++s) { load_rb(s); issue(s); }
    if (NS - 1 < nsub) load_rb(NS - 1);

    bool ok = true;
    int q[DR];
    for (int s = 0; s < nsub; ++s) {
        if (s + NS - 1 < nsub) {
            issue(s + NS - 1);
            if (s + NS < nsub) load_rb(s + NS);
        }
        const int buf = (int)((g0 + s) % NS);
        ok = __all_sync(0xffffffffu, mbar_wait(&bar[buf], (uint32_t)(((g0 + s) / NS) & 1), a.err));
        if (!ok) { sit_out(bar, g0, s, nsub, NS, a.err); break; }
        const int32_t *rec = srec + (size_t)buf * R::kLen;
        const Tin *srow = rows + (size_t)buf * stage_elems;
        float *Pb = P + (size_t)(s & 1) * a.pmax;
        // stage 1: every pattern's partial sum over the samples its trials need
        const int xo[CS] = {};
        share_stage1<Tin, R, CS, NW>(rec, srow, Pb, warp, lane, xo);
        // this warp's trials: index of their t = t0 term in P
#pragma unroll
        for (int j = 0; j < DR; j += 4) {
            const int4 v = *reinterpret_cast<const int4 *>(rec + R::kTrial + warp * DR + j);
            q[j] = v.x; q[j + 1] = v.y; q[j + 2] = v.z; q[j + 3] = v.w;
        }
        __syncthreads();
        // stage 2: one shared word per add
#pragma unroll
        for (int j = 0; j < DR; ++j) {
            const float *pp = Pb + q[j] + lane;
#pragma unroll
            for (int i = 0; i < TI; ++i) acc[j][i] += pp[32 * i];
        }
    }
    ok = __syncthreads_and(ok);
    if (!ok) return false;
    ShareStat<kInt> st;
    share_store<kInt, TI, DR>(a, acc, dm0 + warp * DR, t0, lane, st);
    share_stat_flush<kInt>(a, st, lin);
    return true;
}

// One plan: one block per work item, grid = nblk * ntile.
template <typename Tin, bool kInt, int TI, int DR, int NW, int CS, int NPMAX, int NS, int MINB>
__global__ void __launch_bounds__(NW * 32, MINB) share_kernel(ShareLaunch a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + a.bar_off);
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) mbar_init(&bar[s], NW);
        mbar_fence_init();
    }
    __syncthreads();
    int blk;
    int64_t t0;
    share_raster<TI>(a, blockIdx.x, blk, t0);
    t0 += a.t_base;
    uint32_t gstage = 0;
    share_tile<Tin, kInt, TI, DR, NW, CS, NPMAX, NS>(a, blk, t0, blockIdx.x, bar, gstage);
}

// share_tile as an out-of-line function for the persistent batch kernel.
template <typename Tin, bool kInt, int TI, int DR, int NW, int CS, int NPMAX, int NS>
__device__ __noinline__ bool share_tile_call(const ShareLaunch &a, int blk, int64_t t0, int64_t lin,
                                             uint64_t *bar, uint32_t &gstage)
{
    return share_tile<Tin, kInt, TI, DR, NW, CS, NPMAX, NS>(a, blk, t0, lin, bar, gstage);
}

// Persistent batch of beams, each on kernel 5 (kind 1: its ShareLaunch) or on
// kernel 3 (kind 0: its LaneLaunch) with the same block geometry (DR*NW
// trials x 32*TI samples), so both enumerate the same work items.  Two input
// rings: kernel 3's kStages mbarriers at b.bar_off, kernel 5's NS right after;
// each with its own running stage count.
template <int TI, int DR, int NW, int CS, int NPMAX, int NS, int MINB>
__global__ void __launch_bounds__(NW * 32, MINB) mixed_batch_kernel(LaneBatchLaunch b)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_item;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + b.bar_off), *sbar = bar + kStages;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(&bar[s], NW);
        for (int s = 0; s < NS; ++s) mbar_init(&sbar[s], NW);
        mbar_fence_init();
    }
    __syncthreads();
    uint32_t gl = 0, gs = 0;
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
        if (a.kind == 1) {
            const ShareLaunch &sa = b.sbeams[w.x];
            switch (a.dtype) {
            case DD_F32: ok = share_tile_call<float, false, TI, DR, NW, CS, NPMAX, NS>(sa, blk, t0, w.y, sbar, gs); break;
            case DD_F16: ok = share_tile_call<__half, false, TI, DR, NW, CS, NPMAX, NS>(sa, blk, t0, w.y, sbar, gs); break;
            default: ok = share_tile_call<uint8_t, true, TI, DR, NW, CS, NPMAX, NS>(sa, blk, t0, w.y, sbar, gs); break;
            }
        } else {
            switch (a.dtype) {
            case DD_F32: ok = lane_tile_call<float, false, TI, DR, NW>(a, blk, t0, w.y, bar, gl); break;
            case DD_F16: ok = lane_tile_call<__half, false, TI, DR, NW>(a, blk, t0, w.y, bar, gl); break;
            default: ok = lane_tile_call<uint8_t, true, TI, DR, NW>(a, blk, t0, w.y, bar, gl); break;
            }
        }
        if (!ok) break;
        __syncthreads();
        if (threadIdx.x == 0) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
}

// Arrive on an mbarrier (no transaction bytes); release semantics at CTA scope.
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Partial statistics of warps [gw0, gw0 + ngw) of the block (the accumulator
// warps of the warp-specialised kernel; the others have left): the same
// combination as block_stat_f32 / block_stat_i over those warps only, joined
// by named barrier 1.  Every thread of those warps calls it; the group's
// first thread writes record `lin`.
template <bool kInt>
__device__ __forceinline__ void group_stat_flush(const ShareLaunch &a, const ShareStat<kInt> &st, int64_t lin,
                                                 int gw0, int ngw)
{
    __shared__ double gn[32], gm[32], gq[32];
    __shared__ long long gs[32], gc[32];
    __shared__ unsigned long long gu[32];
    const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) - gw0;
    if constexpr (kInt) {
        long long n = st.n, s = st.s;
        unsigned long long q = st.q;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            n += __shfl_xor_sync(0xffffffffu, n, off);
            s += __shfl_xor_sync(0xffffffffu, s, off);
            q += __shfl_xor_sync(0xffffffffu, q, off);
        }
        if (lane == 0) { gc[w] = n; gs[w] = s; gu[w] = q; }
    } else {
        int nw = st.n;
        float sw = st.s;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            nw += __shfl_xor_sync(0xffffffffu, nw, off);
            sw += __shfl_xor_sync(0xffffffffu, sw, off);
        }
        const float mw = nw ? sw / (float)nw : 0.f;
        const float mt = st.n ? st.s / (float)st.n : 0.f;
        const float d = mt - mw;
        float qw = st.q + (float)st.n * d * d;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) qw += __shfl_xor_sync(0xffffffffu, qw, off);
        if (lane == 0) { gn[w] = nw; gm[w] = mw; gq[w] = qw; }
    }
    asm volatile("bar.sync 1, %0;" ::"r"(ngw * 32) : "memory");
    if (w == 0 && lane == 0) {
        if constexpr (kInt) {
            long long N = 0, S = 0;
            unsigned long long Q = 0;
            for (int v = 0; v < ngw; ++v) { N += gc[v]; S += gs[v]; Q += gu[v]; }
            StatI *dst = reinterpret_cast<StatI *>(a.partials) + lin;
            dst->n = N; dst->sum = S; dst->sumsq = Q;
        } else {
            double N = 0, S = 0;
            for (int v = 0; v < ngw; ++v) { N += gn[v]; S += gn[v] * (double)gm[v]; }
            const double M = N > 0 ? S / N : 0.0;
            double Q = 0;
            for (int v = 0; v < ngw; ++v) {
                const double e = (double)gm[v] - M;
                Q += (double)gq[v] + gn[v] * e * e;
            }
            StatF *dst = reinterpret_cast<StatF *>(a.partials) + lin;
            dst->n = N; dst->mean = M; dst->m2 = Q;
        }
    }
}

// Registers of the warp-specialised block: a launch of T threads gets at
// most 65536 / T per thread (a multiple of 8).  When that is below what the
// stage-2 warps need (their DR x TI accumulators: kWsAccRegs), the stage-1
// warps give registers back with setmaxnreg.dec and the stage-2 warps take
// them with setmaxnreg.inc; the two shares together stay within the block's
// launch allocation (checked on the host against the compiled register count
// before the shape is used: an increase the block cannot cover would wait
// forever).
// Stage-2 warps hold 128 accumulators: 144 registers keep enough loads in
// flight beside them, and what they leave lets a stage-1 warp (80) issue 40
// loads before the first use.  With 160 and 64 (32 loads) the LOFAR-like beam
// took 6% longer; with 136 the accumulators spill (1.5 times).
constexpr int kWsAccRegs = 144;
constexpr int kWsStageRegs = 32;     // staging warps
constexpr int kWsStage = 4;          // staging warps: a warpgroup
template <int NW, int PW>
struct WsRegs {
    static constexpr int kWarps = NW + PW + kWsStage;
    static constexpr int kLaunch = (65536 / (kWarps * 32)) / 8 * 8;
    static constexpr int kProd = (kWarps * kLaunch - NW * kWsAccRegs - kWsStage * kWsStageRegs) / PW / 8 * 8;
    static_assert(kLaunch < kWsAccRegs && kProd >= 24 && kProd <= kLaunch, "the stage-2 warps take registers from the others");
    static_assert(PW % 4 == 0 && NW % 4 == 0 && kWsStage % 4 == 0, "setmaxnreg acts on whole warpgroups");
    // the compiled register count per thread the split needs
    static constexpr int kNeed = (kWsStage * kWsStageRegs + PW * kProd + NW * kWsAccRegs + kWarps - 1) / kWarps;
    static_assert(kNeed <= kLaunch, "the shares stay within the launch's registers");
};

// Whether the phase has completed, without waiting.
__device__ __forceinline__ bool mbar_done(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Kernel 5, warp-specialised: the same two stages on separate warps.  Warps
// [0, PW) form subband s's partial sums (stage 1) into P slot s % PB and copy
// the block's trial offsets next to them; warps [PW, PW + NW) add slot s into
// their trials' accumulators (stage 2); the last four stage the input.
// Hand-offs are mbarriers, not a block barrier per subband:
//   full[i]   input stage i has landed,
//   empty[i]  every stage-1 warp is done with input stage i,
//   pfull[b]  every stage-1 warp has written slot b,
//   pempty[b] every stage-2 warp has read slot b,
// so stage 1 runs up to PB - 1 subbands ahead of stage 2, the staging up to ns
// ahead of stage 1, and the two stages keep the shared-memory pipe busy together.
//
// A thread that issues a bulk copy is held 250 to 300 cycles, whatever the
// copy's size (clock64 around the issue).  When lane 0 of a stage-1 warp issued
// the 5 copies of a subband it took 1277 of the subband's 2546 cycles on the
// LOFAR-like plan, and everything waited for that warp's rows.  Four warps of
// their own issue 1 to 3 copies each and are never waited for (626 of 2361
// cycles; 888 of 2895 with 8 rows; 133.1 -> 127.7 ms for the whole plan's call).  Measured against it: 16-byte cp.async by
// the stage-2 threads (731 cycles a subband on the critical side) or by the
// staging warps (1102; the copies then also take the loads' path into shared
// memory: 31.9 against 30.5 ms on a quarter of the LOFAR-like plan).
// One block per SM: NW * DR trials x 32 * TI samples of accumulators take
// most of the register file, the stage-1 warps the rest.
// Every wait is bounded; a warp whose wait gives up stops, the others then
// give up on theirs, and the staging warps wait (bounded) for their copies still
// in flight before they return.
//
// kAny: rows that start anywhere (in or pitch not 16-byte aligned).  Channel
// c's copy starts res(c) elements early, at the 16-byte unit that holds its
// first element, and ends with the unit of its last one, in a staged row one
// unit longer; stage 1 reads res(c) elements on.
template <typename Tin, bool kInt, int TI, int DR, int NW, int PW, int CS, int NPMAX, int PB, bool kAny>
__global__ void __launch_bounds__((NW + PW + kWsStage) * 32, 1) share_ws_kernel(ShareLaunch a)
{
    using Regs = WsRegs<NW, PW>;
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int kDmBlk = DR * NW;
    using R = ShareRec<CS, NPMAX, kDmBlk>;
    static_assert(PB >= 2, "the slot ring needs two entries");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rs = a.rs, nsub = a.nsub, ns = a.ns;

    // layout: [ns][CS][rs] Tin rows | [ns][kLen] int32 records |
    //         [PB] slots {int32 q[kDmBlk], float P[pmax]} | mbarriers at bar_off
    const size_t stage_elems = (size_t)CS * rs;
    Tin *rows = reinterpret_cast<Tin *>(smem);
    int32_t *srec = reinterpret_cast<int32_t *>(smem + ns * stage_elems * sizeof(Tin));
    int32_t *slots = srec + ns * R::kLen;
    const size_t slot_len = (size_t)kDmBlk + a.pmax;      // packed sums: two halves of pmax / 2 words
    uint64_t *pfull = reinterpret_cast<uint64_t *>(smem + a.bar_off);
    uint64_t *pempty = pfull + PB, *full = pfull + 2 * PB, *empty = full + ns;
    if (tid == 0) {
        for (int i = 0; i < ns; ++i) { mbar_init(&full[i], kWsStage); mbar_init(&empty[i], PW); }
        for (int b = 0; b < PB; ++b) { mbar_init(&pfull[b], PW); mbar_init(&pempty[b], NW); }
        mbar_fence_init();
    }
    __syncthreads();
    int blk;
    int64_t t0;
    share_raster<TI>(a, blockIdx.x, blk, t0);
    t0 += a.t_base;
    constexpr int kAl = 16 / (int)sizeof(Tin);
    const int pitch_res = (int)(a.pitch & (kAl - 1));
    auto res = [&](int c) { return (a.in_res + c * pitch_res) & (kAl - 1); };

    if (warp < PW) {
        // ---- stage 1
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Regs::kProd));
        int ib = 0, pb = 0;                      // input stage, slot
        uint32_t fpar = 0, epar = 1;             // their phases' parities (a fresh slot counts as read)
        for (int s = 0; s < nsub; ++s) {
            const bool e = mbar_done(&pempty[pb], epar), f = mbar_done(&full[ib], fpar);
            bool ok = e && f;
            if (!ok) ok = mbar_wait(&pempty[pb], epar, a.err) && mbar_wait(&full[ib], fpar, a.err);
            if (!__all_sync(0xffffffffu, ok)) break;
            const int32_t *rec = srec + (size_t)ib * R::kLen;
            const Tin *srow = rows + (size_t)ib * stage_elems;
            int32_t *slot = slots + (size_t)pb * slot_len;
            int xo[CS] = {};
            if constexpr (kAny) {
#pragma unroll
                for (int cc = 0; cc < CS; ++cc) xo[cc] = cc * kAl + res(s * CS + cc);   // the records' rows are one unit shorter
            }
            if constexpr (kInt) {
                uint32_t *P = reinterpret_cast<uint32_t *>(slot + kDmBlk);
                share_stage1_bytes<R, CS, PW>(rec, srow, P, P + a.pmax / 2, warp, lane, xo);
            } else {
                // 40 loads a step (no accumulators here): 10 or 5 whole rows;
                // leftover rows 3 or 2 a step
                constexpr int kRows = 40 / CS;
                share_stage1<Tin, R, CS, PW, kRows, (kRows + 3) / 4>(rec, srow, reinterpret_cast<float *>(slot + kDmBlk), warp,
                                                               lane, xo);
            }
            if (warp == PW - 1)
                for (int j = lane; j < kDmBlk; j += 32) slot[j] = rec[R::kTrial + j];
            __syncwarp();
            if (lane == 0) { mbar_arrive(&pfull[pb]); mbar_arrive(&empty[ib]); }
            if (++pb == PB) { pb = 0; epar ^= 1u; }
            if (++ib == ns) { ib = 0; fpar ^= 1u; }
        }
        return;
    }

    if (warp >= PW + NW) {
        // ---- staging: warp w stages rows w, w + 4, .. of the subband, the last
        // one its record too.  A row's start and length are loaded one
        // subband early, by lane i for the warp's i-th row.
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kWsStageRegs));
        constexpr int kRows = CS / kWsStage;       // rows per warp
        const int w = warp - PW - NW, mine = w + kWsStage * min(lane, kRows - 1);
        const Tin *in = static_cast<const Tin *>(a.in) + t0;
        const int32_t *rb_p = a.base + (size_t)blk * a.nchans + mine, *rl_p = a.rlen + (size_t)blk * a.nchans + mine;
        const int32_t *rec_p = a.rec + (size_t)blk * nsub * R::kLen;
        const bool with_rec = w == kWsStage - 1;
        const uint64_t pol = l2_evict_last();      // other DM blocks of this tile stage these rows soon
        int rb = rb_p[0], rl = rl_p[0], ib = 0, s = 0;
        uint32_t par = 1;                          // a fresh stage counts as done with
        for (; s < nsub; ++s) {
            if (!__all_sync(0xffffffffu, mbar_wait(&empty[ib], par, a.err))) break;
            // lane i: its row's first element and 16-byte units
            int64_t g = (int64_t)(s * CS + mine) * a.pitch + rb, n = a.nsamp_in_al - (t0 + rb);
            n = n < 0 ? 0 : (n > rl ? rl : n);
            if constexpr (kAny) {
                const int d = res(s * CS + mine);
                g -= d;
                if (n > 0) n += d;
            }
            const int units = lane < kRows ? (int)((n + kAl - 1) / kAl) : 0;
            if (s + 1 < nsub) { rb = rb_p[(s + 1) * CS]; rl = rl_p[(s + 1) * CS]; }
            Tin *dst = rows + (size_t)ib * stage_elems + (size_t)w * rs;
            int32_t *rdst = srec + (size_t)ib * R::kLen;
            const int32_t *rsrc = rec_p + (size_t)s * R::kLen;
            const int all = __reduce_add_sync(0xffffffffu, units);
            if (lane == 0) mbar_arrive_tx(&full[ib], (uint32_t)(all * 16 + (with_rec ? R::kLen * 4 : 0)));
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                const int64_t gi = __shfl_sync(0xffffffffu, g, i);
                const int ui = __shfl_sync(0xffffffffu, units, i);
                if (lane == 0 && ui)
                    bulk_g2s_hint(dst + (size_t)(i * kWsStage) * rs, in + gi, (uint32_t)ui * 16, &full[ib], pol);
            }
            if (lane == 0 && with_rec) bulk_g2s(rdst, rsrc, R::kLen * 4, &full[ib]);
            if (++ib == ns) { ib = 0; par ^= 1u; }
        }
        // after a wait gave up: let the copies still in flight land before leaving
        if (lane == 0)
            for (int u = max(0, s - ns); u < s; ++u) mbar_wait(&full[u % ns], (uint32_t)((u / ns) & 1), a.err);
        return;
    }

    // ---- stage 2: one shared word per add
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kWsAccRegs));
    // Packed sums: a word holds the sums of two consecutive samples, and is
    // added whole (low + 2^16 high, modulo 2^32) and by its high half: the two
    // sums follow exactly from the two accumulators, with one word per two adds.
    const int cw = warp - PW;
    float acc[kInt ? 1 : DR][kInt ? 1 : TI];
    uint32_t pa[kInt ? DR : 1][kInt ? TI / 2 : 1], ph[kInt ? DR : 1][kInt ? TI / 2 : 1];
    if constexpr (kInt) {
#pragma unroll
        for (int j = 0; j < DR; ++j)
#pragma unroll
            for (int i = 0; i < TI / 2; ++i) { pa[j][i] = 0u; ph[j][i] = 0u; }
    } else {
#pragma unroll
        for (int j = 0; j < DR; ++j)
#pragma unroll
            for (int i = 0; i < TI; ++i) acc[j][i] = 0.f;
    }

    bool ok = true;
    int pb = 0;
    uint32_t ppar = 0;
    for (int s = 0; s < nsub; ++s) {
        ok = mbar_done(&pfull[pb], ppar) || mbar_wait(&pfull[pb], ppar, a.err);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const int32_t *slot = slots + (size_t)pb * slot_len;
        const float *Pb = reinterpret_cast<const float *>(slot + kDmBlk);
        int q[DR];
#pragma unroll
        for (int j = 0; j < DR; j += 4) {
            const int4 v = *reinterpret_cast<const int4 *>(slot + cw * DR + j);
            q[j] = v.x; q[j + 1] = v.y; q[j + 2] = v.z; q[j + 3] = v.w;
        }
#pragma unroll
        for (int j = 0; j < DR; ++j) {
            if constexpr (kInt) {
                const uint32_t *pp = reinterpret_cast<const uint32_t *>(Pb) + q[j] + lane;
#pragma unroll
                for (int i = 0; i < TI / 2; ++i) {
                    const uint32_t v = pp[32 * i];
                    pa[j][i] += v;
                    ph[j][i] = __dp2a_lo(v, 0x0100u, ph[j][i]);   // + its high half
                }
            } else {
                const float *pp = Pb + q[j] + lane;
#pragma unroll
                for (int i = 0; i < TI; ++i) acc[j][i] += pp[32 * i];
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&pempty[pb]);
        if (++pb == PB) { pb = 0; ppar ^= 1u; }
    }
    ShareStat<kInt> st;
    if (ok) {
        if constexpr (kInt) share_store_pairs<TI, DR>(a, pa, ph, blk * kDmBlk + cw * DR, t0, lane, st);
        else share_store<kInt, TI, DR>(a, acc, blk * kDmBlk + cw * DR, t0, lane, st);
    }
    group_stat_flush<kInt>(a, st, blockIdx.x, PW, NW);
}

// Compiled shapes: subbands of 4 channels (the warp-specialised shape also 8),
// at most 16 patterns per (block, subband); {samples per lane, DM trials per
// warp, warps (stage-2 warps in the warp-specialised form), resident blocks
// per SM the register budget targets, input stages (at most, in the
// warp-specialised form), stage-1 warps (0: the one-barrier-per-subband
// kernel, whose warps do both stages), partial-sum slots}.
constexpr int kShCS = 4, kShNP = 16;
struct ShareShape { int ti, dr, nw, minb, ns, pw, pb; };
constexpr int kNumShareCfg = 4;
constexpr int kShareWs = 3;          // the warp-specialised shape
constexpr ShareShape kShareCfg[kNumShareCfg] = {
    {16, 8, 4, 3, 2, 0, 2}, {8, 8, 4, 5, 2, 0, 2}, {16, 8, 6, 2, 2, 0, 2}, {16, 8, 8, 1, 6, 8, 3}};
template <int DB>
using ShareRecDB = ShareRec<kShCS, kShNP, DB>;

cudaError_t share_launch(int k, dd_dtype t, const ShareLaunch &a, cudaStream_t s);
cudaError_t share_prepare(int k, size_t optin);
// false if shape k's kernels for this input type were compiled with fewer
// registers than their register split needs (they are then not used)
bool share_regs_ok(int k, dd_dtype t);
// Mixed persistent batch of kernel 5 shape 0 and kernel 3 shape 2 (the same
// block geometry): grid = sms * that shape's resident blocks per SM.
cudaError_t mixed_batch_launch(const LaneBatchLaunch &b, int sms, size_t smem, cudaStream_t s);
cudaError_t mixed_batch_prepare(size_t optin);
int mixed_batch_occupancy(size_t smem);   // resident blocks per SM with `smem` dynamic bytes
constexpr int kMixedLane = 2, kMixedShare = 0;

}  // namespace dd
