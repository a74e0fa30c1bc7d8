// Generic de-dispersion kernel (kernel 1), statistics and the boxcar
// threshold search.
//
// Section 3.1 (brute force): out[dm][t] = sum_c in[c][t + d(c,dm)].
// Section 3 (output stage): mean and standard deviation over the whole
// processed buffer, an n-sigma threshold, every point above it reported.
#include "dd_internal.h"
#include "dd_device.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace dd {

// ---------------------------------------------------------------------------
// Kernel 1: generic shared-memory de-dispersion.
//
// Block = kGenDms DM trials x kGenTile samples.  For each stage of `chunk`
// channels the block copies, per channel, the input span covering all its
// DM trials ([t0 + base, t0 + base + kGenTile + span)) into shared memory,
// converting to float; each thread then adds, for each of its samples and
// DM trials, the element at its delay offset.  One shared load per add.
// With chunk == 0 (span too large for shared memory) it reads global memory
// directly.
// ---------------------------------------------------------------------------
template <typename Tin, bool kInt>
__global__ void __launch_bounds__(kGenThreads)
generic_kernel(const Tin *__restrict__ in, int64_t pitch, int64_t nsamp_in, int nchans,
               const int32_t *__restrict__ goffs,   // [dmblk][nchans][kGenDms]
               const int32_t *__restrict__ gbase,   // [dmblk][nchans]
               const int32_t *__restrict__ gspan,   // [dmblk][nchans]
               int ndm, int64_t nout, void *__restrict__ out_, void *__restrict__ partials,
               int chunk, int stride)
{
    extern __shared__ float smem[];
    const int tid = threadIdx.x;
    const int64_t t0 = (int64_t)blockIdx.x * kGenTile;
    const int blk = blockIdx.y;
    const int dm0 = blk * kGenDms;
    const int ndb = min(kGenDms, ndm - dm0);
    const int32_t *boffs = goffs + (size_t)blk * nchans * kGenDms;
    const int32_t *bbase = gbase + (size_t)blk * nchans;
    const int32_t *bspan = gspan + (size_t)blk * nchans;

    float acc[kGenDms][kGenTimes];
#pragma unroll
    for (int j = 0; j < kGenDms; ++j)
#pragma unroll
        for (int k = 0; k < kGenTimes; ++k) acc[j][k] = 0.f;

    if (chunk > 0) {
        float *rows = smem;
        int *offs = reinterpret_cast<int *>(smem + (size_t)chunk * stride);
        for (int c0 = 0; c0 < nchans; c0 += chunk) {
            const int cn = min(chunk, nchans - c0);
            __syncthreads();
            for (int i = tid; i < cn * kGenDms; i += kGenThreads)
                offs[i] = boffs[(size_t)c0 * kGenDms + i];
            for (int c = 0; c < cn; ++c) {
                const int64_t s0 = t0 + bbase[c0 + c];
                const int len = kGenTile + bspan[c0 + c];
                const Tin *src = in + (size_t)(c0 + c) * pitch;
                float *dst = rows + (size_t)c * stride;
                for (int i = tid; i < len; i += kGenThreads) {
                    const int64_t s = s0 + i;
                    dst[i] = (s < nsamp_in) ? to_f(src[s]) : 0.f;
                }
            }
            __syncthreads();
            for (int c = 0; c < cn; ++c) {
                const float *r = rows + (size_t)c * stride + tid;
                const int *o = offs + c * kGenDms;
#pragma unroll
                for (int j = 0; j < kGenDms; ++j) {
                    const int oj = o[j];
#pragma unroll
                    for (int k = 0; k < kGenTimes; ++k) acc[j][k] += r[oj + k * kGenThreads];
                }
            }
        }
    } else {
        for (int c = 0; c < nchans; ++c) {
            const Tin *src = in + (size_t)c * pitch + bbase[c];
            const int32_t *o = boffs + (size_t)c * kGenDms;
#pragma unroll
            for (int j = 0; j < kGenDms; ++j) {
                const int oj = o[j];
#pragma unroll
                for (int k = 0; k < kGenTimes; ++k) {
                    const int64_t s = t0 + tid + k * kGenThreads + oj;
                    if (s + bbase[c] < nsamp_in) acc[j][k] += to_f(src[s]);
                }
            }
        }
    }

    // Epilogue: store, then per-block partial statistics.
    const int64_t pidx = (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
    if constexpr (kInt) {
        int32_t *out = reinterpret_cast<int32_t *>(out_);
        long long n = 0, s = 0;
        unsigned long long q = 0;
#pragma unroll
        for (int j = 0; j < kGenDms; ++j)
#pragma unroll
            for (int k = 0; k < kGenTimes; ++k) {
                const int64_t t = t0 + tid + k * kGenThreads;
                if (j < ndb && t < nout) {
                    const int v = __float2int_rn(acc[j][k]);
                    out[(size_t)(dm0 + j) * nout + t] = v;
                    n += 1; s += v; q += (unsigned long long)((long long)v * v);
                }
            }
        block_stat_i(n, s, q, reinterpret_cast<StatI *>(partials) + pidx);
    } else {
        float *out = reinterpret_cast<float *>(out_);
        int n = 0;
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < kGenDms; ++j)
#pragma unroll
            for (int k = 0; k < kGenTimes; ++k) {
                const int64_t t = t0 + tid + k * kGenThreads;
                if (j < ndb && t < nout) {
                    out[(size_t)(dm0 + j) * nout + t] = acc[j][k];
                    n += 1; s += acc[j][k];
                }
            }
        const float m = n ? s / (float)n : 0.f;
        float q = 0.f;
#pragma unroll
        for (int j = 0; j < kGenDms; ++j)
#pragma unroll
            for (int k = 0; k < kGenTimes; ++k) {
                const int64_t t = t0 + tid + k * kGenThreads;
                if (j < ndb && t < nout) { const float d = acc[j][k] - m; q += d * d; }
            }
        block_stat_f32(n, s, q, reinterpret_cast<StatF *>(partials) + pidx);
    }
}

// ---------------------------------------------------------------------------
// Statistics straight from an `out` buffer (used when dd_search is given a
// buffer other than the one the last dd_execute produced).
// ---------------------------------------------------------------------------
constexpr int kStatThreads = 256;
constexpr int kStatPer = 16;   // elements per thread

template <bool kInt>
__global__ void __launch_bounds__(kStatThreads)
stats_kernel(const void *__restrict__ out_, int64_t total, void *__restrict__ partials)
{
    const int64_t base = (int64_t)blockIdx.x * kStatThreads * kStatPer;
    if constexpr (kInt) {
        const int32_t *x = reinterpret_cast<const int32_t *>(out_);
        long long n = 0, s = 0;
        unsigned long long q = 0;
        for (int k = 0; k < kStatPer; ++k) {
            const int64_t i = base + (int64_t)k * kStatThreads + threadIdx.x;
            if (i < total) { const long long v = x[i]; n++; s += v; q += (unsigned long long)(v * v); }
        }
        block_stat_i(n, s, q, reinterpret_cast<StatI *>(partials) + blockIdx.x);
    } else {
        const float *x = reinterpret_cast<const float *>(out_);
        float v[kStatPer];
        int n = 0;
        float s = 0.f;
        for (int k = 0; k < kStatPer; ++k) {
            const int64_t i = base + (int64_t)k * kStatThreads + threadIdx.x;
            v[k] = i < total ? x[i] : 0.f;
            if (i < total) { n++; s += v[k]; }
        }
        const float m = n ? s / (float)n : 0.f;
        float q = 0.f;
        for (int k = 0; k < kStatPer; ++k) {
            const int64_t i = base + (int64_t)k * kStatThreads + threadIdx.x;
            if (i < total) { const float d = v[k] - m; q += d * d; }
        }
        block_stat_f32(n, s, q, reinterpret_cast<StatF *>(partials) + blockIdx.x);
    }
}

// ---------------------------------------------------------------------------
// Finalise: merge the per-block partials into mu and sigma (population, over
// the whole buffer) and form the per-width thresholds
//   T_w = w*mu + k*sigma*sqrt(w)
// in double (Section 3's n-sigma test applied to boxcar sums).  Each
// threshold is stored as the largest float <= T_w and as floor(T_w), so the
// kernels' FP32 / integer comparisons decide B_w > T_w exactly as a double
// comparison of the same B_w would.  It also clears the hit count that the
// search adds to.
//
// The LOFAR-like plan leaves 64 288 partials (1.5 MB).  One block of 1024
// threads took 122 us for them: two passes of dependent loads by one SM, and
// FP64 at two lanes a clock.  Here each block merges its own run of about
// kFinRun partials and the last block to finish (a ticket in the plan's
// scratch) merges the blocks' records with the same code, so the loads and
// the FP64 work spread over the SMs: 122 -> 10 us there, 291 -> 16 us for
// the 168 756 partials of the subband plan.  The runs depend on the number
// of partials alone: the result is the same from call to call.
// ---------------------------------------------------------------------------
constexpr int kFinThreads = 128;
constexpr int kFinRun = 512;        // partials per block (at least; kFinBlocks blocks at most)
static_assert(kFinThreads >= kMaxWidths, "one thread per width forms the thresholds");

template <typename T>
__device__ __forceinline__ T fin_block_sum(T v, T *sh)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    T r = sh[0];
#pragma unroll
    for (int w = 1; w < kFinThreads / 32; ++w) r += sh[w];
    return r;
}

// Records [lo, hi) merged, in every thread of the block: two passes, no
// division per record, mean = sum n_b*mean_b / N, M2 = sum [M2_b + n_b*(mean_b - mean)^2].
__device__ __forceinline__ StatF fin_merge(const StatF *p, int64_t lo, int64_t hi)
{
    __shared__ double sh[kFinThreads / 32];
    double n = 0, s = 0, q = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += kFinThreads) { n += p[i].n; s += p[i].n * p[i].mean; }
    StatF r;
    r.n = fin_block_sum(n, sh);
    s = fin_block_sum(s, sh);
    r.mean = r.n > 0 ? s / r.n : 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += kFinThreads) {
        const double e = p[i].mean - r.mean;
        q += p[i].m2 + p[i].n * e * e;
    }
    r.m2 = fin_block_sum(q, sh);
    return r;
}

// The same for integer records: exact sums, the squares in 128 bits.
__device__ __forceinline__ FinI fin_merge(const StatI *p, const FinI *f, int64_t lo, int64_t hi)
{
    __shared__ long long sh[kFinThreads / 32];
    __shared__ unsigned long long shu[kFinThreads / 32];
    long long n = 0, s = 0;
    unsigned long long q0 = 0, q1 = 0, q2 = 0;   // 32-bit limbs: sums of up to 2^32 records stay exact
    for (int64_t i = lo + threadIdx.x; i < hi; i += kFinThreads) {
        const unsigned long long l = p ? p[i].sumsq : f[i].q_lo, h = p ? 0ull : f[i].q_hi;
        n += p ? p[i].n : f[i].n;
        s += p ? p[i].sum : f[i].sum;
        q0 += l & 0xffffffffull; q1 += l >> 32; q2 += h;
    }
    FinI r;
    r.n = fin_block_sum(n, sh);
    r.sum = fin_block_sum(s, sh);
    q0 = fin_block_sum(q0, shu);
    q1 = fin_block_sum(q1, shu);
    q2 = fin_block_sum(q2, shu);
    const unsigned __int128 q = (unsigned __int128)q0 + ((unsigned __int128)q1 << 32) + ((unsigned __int128)q2 << 64);
    r.q_lo = (unsigned long long)q;
    r.q_hi = (unsigned long long)(q >> 64);
    return r;
}

template <bool kInt>
__global__ void __launch_bounds__(kFinThreads)
finalize_kernel(const void *__restrict__ partials, int64_t np, const int32_t *__restrict__ widths,
                int nw, double k, SearchParams *__restrict__ prm, unsigned long long *__restrict__ count,
                FinScratch *__restrict__ scr)
{
    using Rec = typename std::conditional<kInt, FinI, StatF>::type;
    __shared__ bool last_s;
    const int64_t lo = np * blockIdx.x / gridDim.x, hi = np * (blockIdx.x + 1) / gridDim.x;
    Rec r;
    if constexpr (kInt) r = fin_merge(static_cast<const StatI *>(partials), nullptr, lo, hi);
    else r = fin_merge(static_cast<const StatF *>(partials), lo, hi);
    if (gridDim.x > 1) {
        Rec *rec;
        if constexpr (kInt) rec = scr->i; else rec = scr->f;
        if (threadIdx.x == 0) {
            rec[blockIdx.x] = r;
            __threadfence();
            last_s = atomicAdd(&scr->ticket, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last_s) return;
        __threadfence();
        if constexpr (kInt) r = fin_merge(nullptr, rec, 0, gridDim.x);
        else r = fin_merge(rec, 0, gridDim.x);
        if (threadIdx.x == 0) scr->ticket = 0;      // for the next launch
    }
    double mu, sg;
    if constexpr (kInt) {
        const unsigned __int128 Q = ((unsigned __int128)r.q_hi << 64) | r.q_lo;
        // N*Q - S^2 >= 0 exactly (Cauchy-Schwarz), then one rounding each.
        const __int128 num = (__int128)((unsigned __int128)r.n * Q) - (__int128)r.sum * (__int128)r.sum;
        const double dn = (double)r.n;
        mu = (double)r.sum / dn;
        sg = sqrt((double)num / (dn * dn));
    } else {
        mu = r.mean;
        sg = sqrt(r.m2 / r.n);
    }
    if (threadIdx.x == 0) { prm->mu = mu; prm->sigma = sg; prm->nw = nw; *count = 0; }
    if (threadIdx.x < nw) {
        const double w = (double)widths[threadIdx.x];
        const double T = w * mu + k * sg * sqrt(w);
        prm->thr_f[threadIdx.x] = __double2float_rd(T);
        double f = floor(T);
        f = fmin(fmax(f, -4.0e18), 4.0e18);
        prm->thr_i[threadIdx.x] = (long long)f;
    }
}

// ---------------------------------------------------------------------------
// Per-DM-row statistics (search option): one block per row reads the row once.
// Float rows: each thread sums x - K and (x - K)^2 in FP32 with K its first
// value (a shift near the mean keeps the second moment free of cancellation),
// the block merges (n, mean, M2) in FP64.  Integer rows: exact int64 sums,
// 128-bit merge.  Then mu_row, sigma_row (population) and the row's
// thresholds T_w = w*mu_row + k*sigma_row*sqrt(w) in the exact float/integer
// forms of finalize_kernel.
// ---------------------------------------------------------------------------
constexpr int kRowThreads = 512;

template <bool kInt>
__global__ void __launch_bounds__(kRowThreads)
row_stats_kernel(const void *__restrict__ out_, int64_t nout, const int32_t *__restrict__ widths, int nw,
                 double k, RowParams *__restrict__ rp)
{
    __shared__ double sa[kRowThreads], sb[kRowThreads], sc[kRowThreads];
    __shared__ double mu_s, sg_s;
    const int row = blockIdx.x;
    const int tid = threadIdx.x;
    if constexpr (kInt) {
        const int32_t *x = reinterpret_cast<const int32_t *>(out_) + (size_t)row * nout;
        long long n = 0, s = 0, q = 0;
        int64_t t = tid;
        for (; t + 7 * kRowThreads < nout; t += 8 * kRowThreads) {     // 8 loads in flight
            int32_t v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = x[t + u * kRowThreads];
#pragma unroll
            for (int u = 0; u < 8; ++u) { s += v[u]; q += (long long)v[u] * v[u]; }
            n += 8;
        }
        for (; t < nout; t += kRowThreads) {
            const long long v = x[t];
            n++; s += v; q += v * v;
        }
        __shared__ long long sn[kRowThreads], ss[kRowThreads];
        __shared__ unsigned long long ql[kRowThreads], qh[kRowThreads];
        sn[tid] = n; ss[tid] = s; ql[tid] = (unsigned long long)q; qh[tid] = 0;
        __syncthreads();
        for (int h = kRowThreads / 2; h > 0; h >>= 1) {
            if (tid < h) {
                sn[tid] += sn[tid + h];
                ss[tid] += ss[tid + h];
                unsigned __int128 a = ((unsigned __int128)qh[tid] << 64) | ql[tid];
                const unsigned __int128 b = ((unsigned __int128)qh[tid + h] << 64) | ql[tid + h];
                a += b;
                ql[tid] = (unsigned long long)a;
                qh[tid] = (unsigned long long)(a >> 64);
            }
            __syncthreads();
        }
        if (tid == 0) {
            const long long N = sn[0], S = ss[0];
            const unsigned __int128 Q = ((unsigned __int128)qh[0] << 64) | ql[0];
            const __int128 num = (__int128)((unsigned __int128)N * Q) - (__int128)S * (__int128)S;
            const double dn = (double)N;
            mu_s = (double)S / dn;
            sg_s = sqrt((double)num / (dn * dn));
        }
    } else {
        const float *x = reinterpret_cast<const float *>(out_) + (size_t)row * nout;
        const float K = tid < nout ? x[tid] : 0.f;
        float s = 0.f, q = 0.f;
        int n = 0;
        int64_t t = tid;
        for (; t + 7 * kRowThreads < nout; t += 8 * kRowThreads) {     // 8 loads in flight
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = x[t + u * kRowThreads];
#pragma unroll
            for (int u = 0; u < 8; ++u) { const float d = v[u] - K; s += d; q += d * d; }
            n += 8;
        }
        for (; t < nout; t += kRowThreads) {
            const float d = x[t] - K;
            s += d; q += d * d; n++;
        }
        // thread (n, mean, M2) in double: mean = K + s/n, M2 = q - s^2/n
        const double dn = (double)n;
        const double m = n ? (double)K + (double)s / dn : 0.0;
        const double m2 = n ? fmax((double)q - (double)s * (double)s / dn, 0.0) : 0.0;
        sa[tid] = dn; sb[tid] = dn * m;
        __syncthreads();
        for (int h = kRowThreads / 2; h > 0; h >>= 1) {
            if (tid < h) { sa[tid] += sa[tid + h]; sb[tid] += sb[tid + h]; }
            __syncthreads();
        }
        const double N = sa[0], M = N > 0 ? sb[0] / N : 0.0;
        __syncthreads();
        const double e = m - M;
        sc[tid] = m2 + dn * e * e;
        __syncthreads();
        for (int h = kRowThreads / 2; h > 0; h >>= 1) {
            if (tid < h) sc[tid] += sc[tid + h];
            __syncthreads();
        }
        if (tid == 0) { mu_s = M; sg_s = sqrt(sc[0] / N); }
    }
    __syncthreads();
    if (tid == 0) { rp[row].mu = mu_s; rp[row].sigma = sg_s; }
    if (tid < nw) {
        const double w = (double)widths[tid];
        const double T = w * mu_s + k * sg_s * sqrt(w);
        rp[row].thr_f[tid] = __double2float_rd(T);
        double f = floor(T);
        f = fmin(fmax(f, -4.0e18), 4.0e18);
        rp[row].thr_i[tid] = (long long)f;
    }
}

// ---------------------------------------------------------------------------
// Boxcar threshold search.  Block = one DM row x a tile of samples.  Both
// kernels test a whole run of samples per thread by its largest boxcar sum
// (one max per sample and width, one comparison per run and width); only runs
// whose largest sum is a hit are gone through again sample by sample.  Their
// hits go to a list in shared memory, so that a pulse's hits, which lie in one
// or two threads' runs, are finished by all threads of the block: the S/N, (B_w
// - w*mu) / (sigma*sqrt(w)) in double (slow units here), and the record.
// ---------------------------------------------------------------------------
// S/N and record of one hit into slot pos.
__device__ __forceinline__ void put_candidate(dd_candidate *cands, int64_t cap, unsigned long long pos, int row, int w,
                                              int width_idx, int64_t t, double value, const SearchParams *prm,
                                              const RowParams *rp)
{
    if ((int64_t)pos >= cap) return;
    const double dw = (double)w;
    const double mu = rp ? rp[row].mu : prm->mu, sg = rp ? rp[row].sigma : prm->sigma;
    dd_candidate c;
    c.dm_idx = row; c.width_idx = width_idx; c.t = t;
    c.snr = (float)((value - dw * mu) / (sg * sqrt(dw)));
    c.reserved = 0.f; c.value = value;
    cands[pos] = c;
}

// Any widths: thread = kPer consecutive samples.  For the widths in ascending
// order it extends B_w at its first sample from the previous width's sum, then
// slides it along its samples (B_w(t+1) = B_w(t) + x[t+w] - x[t]); its own
// samples x[t] stay in registers.  31 samples a thread (25 integers): an odd
// stride, so that the threads' words fall in distinct banks without padding
// and every shared address is the thread's base plus a constant or the width
// (with 16 samples and a pad word after each 16, index arithmetic was most of
// the kernel's instructions, and each sample and width was compared).
//
// Every slide of a floating-point sum rounds, and a sample that swamps the sum
// (or an infinity) spoils the windows behind it until the next sum formed
// afresh.  So a run of 31 has two: 15 slides at most, as in runs of 16.  (One
// per 25 samples: r.m.s. error on noise 1.05 to 1.24 times that of runs of 16;
// now 0.98 of it.)  Integers slide through the whole run.
//
// A width more than kSearchGap above the previous one starts from the sums of
// the half runs it covers (16 and 15 samples, formed once) with at most 15
// single samples behind them: 3000 samples take 208 adds, and round less than
// one by one.
//
// 600 rows x 253 443 float32 samples without hits: widths 1, 3, 7, 20, 50 0.67 ms
// with runs of 16, 0.21 with one fresh sum per 25 samples, 0.22 now; 1, 30, 300,
// 3000 4.70, 2.03, 0.97 ms; 1 to 64 6.85, 1.39, 1.37 ms.
//
// The block takes a width's hits together: every run with one marks its hits in
// a mask and copies their sums to the list, which the block's threads finish when
// it is full.  (Each thread by itself, sample by sample with one shared atomic
// per hit and FP64 S/N once the list was full: 64 rows x 6600 samples with 85 000
// hits of 64 widths 1.10 ms, one global atomic per hit 0.51 ms, now 0.14 ms.)
constexpr int kSearchThreads = 128;
constexpr int kSearchGap = 64;
template <bool kInt>
struct SearchShape {
    static constexpr int kRun = kInt ? 13 : 16;        // samples of a first half run
    static constexpr int kPer = 2 * kRun - 1;          // samples per thread
    static constexpr int kTile = kSearchThreads * kPer;
    // half runs of the staged samples (a tile and wmax - 1 more)
    static __host__ __device__ constexpr int halves(int wmax) { return 2 * ((kTile + wmax - 1 + kPer - 1) / kPer); }
    // staged samples and, for wide gaps, the half runs' sums
    static constexpr size_t smem(int wmax, bool wide) { return (size_t)(kTile + wmax - 1 + (wide ? halves(wmax) : 0)) * 4; }
};
// with the kernel's own 10 or 14.4 KB within what any launch may have
static_assert(SearchShape<false>::smem(4096, true) + 10 * 1024 <= 48 * 1024 &&
              SearchShape<true>::smem(4096, true) + 15 * 1024 <= 48 * 1024, "no attribute to set on each call");
constexpr int kHitList = 1024;      // hits a block finishes per round
static_assert(kMaxWidths <= 64, "a hit's code holds its width in 6 bits");

template <bool kInt>
__global__ void __launch_bounds__(kSearchThreads, kInt ? 5 : 6)
search_kernel(const void *__restrict__ out_, int64_t nout,
              const int32_t *__restrict__ wsorted, int nw, int wmax, int wide,
              const SearchParams *__restrict__ prm, const RowParams *__restrict__ rp,
              dd_candidate *__restrict__ cands, int64_t cap, unsigned long long *__restrict__ count)
{
    using T = typename std::conditional<kInt, int32_t, float>::type;
    using Acc = typename std::conditional<kInt, long long, float>::type;
    extern __shared__ __align__(16) unsigned char sraw[];
    __shared__ int sw[kMaxWidths], sidx[kMaxWidths];
    __shared__ Acc sthr[kMaxWidths];
    __shared__ Acc hval[kHitList];                  // the block's hits: their sums and
    __shared__ int hcode[kHitList];                 // sample << 6 | sorted width
    __shared__ double wmu[kMaxWidths], wsg[kMaxWidths];    // w mu, sigma sqrt(w)
    __shared__ int nlist;
    __shared__ unsigned long long first;
    using S = SearchShape<kInt>;
    constexpr int kSearchPer = S::kPer, kSearchRun = S::kRun, kSearchTile = S::kTile;
    T *x = reinterpret_cast<T *>(sraw);
    const int row = blockIdx.y;
    const int64_t t0 = (int64_t)blockIdx.x * kSearchTile;
    if (threadIdx.x == 0) nlist = 0;
    const int len = kSearchTile + wmax - 1;
    if (threadIdx.x < nw) {
        const int o = wsorted[nw + threadIdx.x];
        sw[threadIdx.x] = wsorted[threadIdx.x];
        sidx[threadIdx.x] = o;
        if constexpr (kInt) sthr[threadIdx.x] = rp ? rp[row].thr_i[o] : prm->thr_i[o];
        else sthr[threadIdx.x] = rp ? rp[row].thr_f[o] : prm->thr_f[o];
    }
    const T *src = reinterpret_cast<const T *>(out_) + (size_t)row * nout + t0;
    const int64_t avail = nout - t0;
    {
        T r[kSearchPer];
        if (avail >= kSearchTile) {
#pragma unroll
            for (int q = 0; q < kSearchPer; ++q) r[q] = __ldcs(src + q * kSearchThreads + threadIdx.x);
        } else {
#pragma unroll
            for (int q = 0; q < kSearchPer; ++q) {
                const int i = q * kSearchThreads + threadIdx.x;
                r[q] = i < avail ? __ldcs(src + i) : (T)0;
            }
        }
#pragma unroll
        for (int q = 0; q < kSearchPer; ++q) x[q * kSearchThreads + threadIdx.x] = r[q];
    }
    for (int i = kSearchTile + threadIdx.x; i < len; i += kSearchThreads) x[i] = i < avail ? src[i] : (T)0;
    __syncthreads();
    const int base = threadIdx.x * kSearchPer;
    const T *xb = x + base;
    T own[kSearchPer];
#pragma unroll
    for (int i = 0; i < kSearchPer; ++i) own[i] = xb[i];
    T *half = x + len;   // the sums of the half runs: 2 u at sample kPer u, 2 u + 1 kRun samples behind it
    if (wide) {
        T a = own[0], b = own[kSearchRun];
#pragma unroll
        for (int i = 1; i < kSearchRun; ++i) a += own[i];
#pragma unroll
        for (int i = kSearchRun + 1; i < kSearchPer; ++i) b += own[i];
        half[2 * threadIdx.x] = a;
        half[2 * threadIdx.x + 1] = b;
        for (int h = 2 * kSearchThreads + threadIdx.x; h < S::halves(wmax); h += kSearchThreads) {
            const int s = (h >> 1) * kSearchPer + (h & 1) * kSearchRun;
            const int e = min(s + kSearchRun - (h & 1), len);
            T v = 0;
            for (int j = s; j < e; ++j) v += x[j];
            half[h] = v;
        }
        __syncthreads();
    }
    // B_w at sample c * kRun of the thread's run from its whole half runs
    auto cover = [&](int c, int w) {
        Acc v = 0;
        int h = 2 * threadIdx.x + c, n = 0;
        for (int l; n + (l = kSearchRun - (h & 1)) <= w; n += l, ++h) v += (Acc)half[h];
        for (; n < w; ++n) v += (Acc)xb[c * kSearchRun + n];
        return v;
    };
    // the list's records by all threads; the terms that depend on the width alone once
    bool terms = false;
    auto finish = [&]() {
        const int n = min(nlist, kHitList);
        if (threadIdx.x == 0) first = atomicAdd(count, (unsigned long long)n);
        if (!terms && (int)threadIdx.x < nw) {
            const double dw = (double)sw[threadIdx.x];
            wmu[threadIdx.x] = dw * (rp ? rp[row].mu : prm->mu);
            wsg[threadIdx.x] = (rp ? rp[row].sigma : prm->sigma) * sqrt(dw);
        }
        terms = true;
        __syncthreads();
        for (int q = threadIdx.x; q < n; q += kSearchThreads) {
            const int p = hcode[q] & 63;
            const unsigned long long pos = first + q;
            if ((int64_t)pos >= cap) continue;
            dd_candidate c;
            c.dm_idx = row; c.width_idx = sidx[p]; c.t = t0 + (hcode[q] >> 6);
            c.value = (double)hval[q];
            c.snr = (float)((c.value - wmu[p]) / wsg[p]);
            c.reserved = 0.f;
            cands[pos] = c;
        }
        __syncthreads();
        if (threadIdx.x == 0) nlist = 0;
        __syncthreads();
    };
    Acc b0 = 0, b1 = 0;  // B_w at the thread's first sample and (floating point) at sample kRun
    int wprev = 0;
    for (int p = 0; p < nw; ++p) {
        const int w = sw[p];
        if (w - wprev > kSearchGap) {
            b0 = cover(0, w);
            if constexpr (!kInt) b1 = cover(1, w);
        } else {
#pragma unroll 4
            for (int j = wprev; j < w; ++j) {
                b0 += (Acc)xb[j];
                if constexpr (!kInt) b1 += (Acc)xb[kSearchRun + j];
            }
        }
        wprev = w;
        const Acc thr = sthr[p];
        const T *xw = xb + (w - 1);              // xw[i] = x[base + i - 1 + w], the sample that enters at i
        Acc b = b0, m = b0;
#pragma unroll
        for (int i = 1; i < kSearchPer; ++i) {
            if (!kInt && i == kSearchRun) b = b1;
            else b += (Acc)xw[i] - (Acc)own[i - 1];
            if constexpr (kInt) m = b > m ? b : m;
            else m = fmaxf(m, b);
        }
        const bool hit = m > thr;
        if (!__syncthreads_or(hit)) continue;
        // runs with a hit: their samples one by one (the same sums again)
        unsigned mask = 0;
        if (hit) {
            b = b0;
#pragma unroll
            for (int i = 0; i < kSearchPer; ++i) {
                if (!kInt && i == kSearchRun) b = b1;
                else if (i > 0) b += (Acc)xw[i] - (Acc)own[i - 1];
                mask |= (unsigned)(b > thr) << i;
            }
            const int64_t lim = avail - base - w + 1;        // tests with t + w <= nout
            if (lim < kSearchPer) mask &= lim > 0 ? (1u << lim) - 1u : 0u;
        }
        while (__syncthreads_or(mask != 0u)) {
            int at = mask ? atomicAdd(&nlist, __popc(mask)) : kHitList;
            if (at < kHitList) {
                b = b0;
#pragma unroll
                for (int i = 0; i < kSearchPer; ++i) {
                    if (!kInt && i == kSearchRun) b = b1;
                    else if (i > 0) b += (Acc)xw[i] - (Acc)own[i - 1];
                    if ((mask >> i & 1u) && at < kHitList) {
                        hval[at] = b;
                        hcode[at++] = (base + i) << 6 | p;
                        mask &= ~(1u << i);
                    }
                }
            }
            __syncthreads();
            if (nlist >= kHitList) finish();
        }
    }
    if (nlist > 0) finish();
}

// The same search for the common width set {1, 2, 4, ..., 2^(K-1)}: each
// thread takes kPow2Per consecutive samples and the 2^(K-1) - 1 that follow
// into registers and forms the boxcars as a doubling tree, B_2w(i) = B_w(i) +
// B_w(i + w): one add per sample and width, two at a time from w = 4 on
// (add.f32x2).  Integer data stay in int32 (at most 65536 channels x 255 x 64
// < 2^31).
//
// The bound is the one read of the buffer.  What kept an earlier form at 38% of
// that was its instructions, 27 a sample: 16 samples a thread (so that the
// overlap of 2^(K-1) - 1 samples cost as much as the samples themselves) and a
// comparison and a mask bit per sample and width.  32 samples a thread and the
// largest sum of each width (three-input max) take about 9 a sample: 3.25 ->
// 1.46 ms for 8.22 GB (5.6 TB/s), and 1.05 -> 0.38 ms for 1.93 GB of integers.
// A pulse's hits used to be written by the one or two threads that own its
// samples (38 of the 47 us of a search of 13 MB with 7000 hits); through the
// list all threads of the block share them: 8 us.  The staged tile is padded by 4 words after every 32: the
// threads' 16-byte window loads then touch all banks evenly.
constexpr int kPow2Threads = 128;
constexpr int kPow2Per = 32;
constexpr int kPow2Tile = kPow2Threads * kPow2Per;

__host__ __device__ __forceinline__ int spad32(int i) { return i + ((i >> 5) << 2); }

__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ int32_t max3(int32_t a, int32_t b, int32_t c) { return __vimax3_s32(a, b, c); }

// (a0, a1) + (b0, b1), each correctly rounded
__device__ __forceinline__ void add2(float &a0, float &a1, float b0, float b1)
{
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\tadd.rn.f32x2 a, a, b;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "+f"(a0), "+f"(a1) : "f"(b0), "f"(b1));
}
__device__ __forceinline__ void add2(int32_t &a0, int32_t &a1, int32_t b0, int32_t b1) { a0 += b0; a1 += b1; }

// B_w at xs[0 .. w) of the padded tile, w = 2^p, by the tree of the search.
template <typename T, int P>
__device__ __forceinline__ T tree_sum(const T *x, int i)
{
    if constexpr (P == 0) return x[spad32(i)];
    else return tree_sum<T, P - 1>(x, i) + tree_sum<T, P - 1>(x, i + (1 << (P - 1)));
}

template <typename T, int K>
__device__ __forceinline__ T tree_sum_p(const T *x, int i, int p)
{
    if constexpr (K == 1) return tree_sum<T, 0>(x, i);
    else return p == K - 1 ? tree_sum<T, K - 1>(x, i) : tree_sum_p<T, K - 1>(x, i, p);
}

template <bool kInt, int K>
__global__ void __launch_bounds__(kPow2Threads)
search_pow2_kernel(const void *__restrict__ out_, int64_t nout, const int32_t *__restrict__ wsorted,
                   const SearchParams *__restrict__ prm, const RowParams *__restrict__ rp,
                   dd_candidate *__restrict__ cands, int64_t cap, unsigned long long *__restrict__ count)
{
    using T = typename std::conditional<kInt, int32_t, float>::type;
    constexpr int W = 1 << (K - 1);                 // widest boxcar
    constexpr int kWin = (kPow2Per + W + 3) / 4 * 4;   // samples of a window, and some that no test uses
    extern __shared__ __align__(16) unsigned char sraw[];
    __shared__ int sidx[K];
    __shared__ float thf[K];
    __shared__ long long thi[K];
    __shared__ unsigned short list[kHitList];       // thread << 8 | sorted width << 5 | sample
    __shared__ int nlist;
    __shared__ unsigned long long first;
    T *x = reinterpret_cast<T *>(sraw);
    const int row = blockIdx.y;
    const int64_t t0 = (int64_t)blockIdx.x * kPow2Tile;
    if (threadIdx.x < K) {
        const int o = wsorted[K + threadIdx.x];     // original index of sorted width 2^threadIdx.x
        sidx[threadIdx.x] = o;
        thf[threadIdx.x] = rp ? rp[row].thr_f[o] : prm->thr_f[o];
        thi[threadIdx.x] = rp ? rp[row].thr_i[o] : prm->thr_i[o];
    }
    if (threadIdx.x == 0) nlist = 0;
    const T *src = reinterpret_cast<const T *>(out_) + (size_t)row * nout + t0;
    const int64_t avail = nout - t0;                // > 0
    {
        T r[kPow2Per];
        if (avail >= kPow2Tile) {
#pragma unroll
            for (int q = 0; q < kPow2Per; ++q) r[q] = __ldcs(src + q * kPow2Threads + threadIdx.x);
        } else {
#pragma unroll
            for (int q = 0; q < kPow2Per; ++q) {
                const int i = q * kPow2Threads + threadIdx.x;
                r[q] = i < avail ? __ldcs(src + i) : (T)0;
            }
        }
        const int i = kPow2Tile + threadIdx.x;
        if ((int)threadIdx.x < W) x[spad32(i)] = i < avail ? src[i] : (T)0;
#pragma unroll
        for (int q = 0; q < kPow2Per; ++q) x[spad32(q * kPow2Threads + threadIdx.x)] = r[q];
    }
    __syncthreads();
    const int base = threadIdx.x * kPow2Per;
    const T *xb = x + spad32(base);
    bool hit = false;
    {
        T b[kWin];
#pragma unroll
        for (int k = 0; k < kWin; k += 4) {
            const int4 v = *reinterpret_cast<const int4 *>(xb + spad32(k));
            if constexpr (kInt) { b[k] = v.x; b[k + 1] = v.y; b[k + 2] = v.z; b[k + 3] = v.w; }
            else {
                b[k] = __int_as_float(v.x); b[k + 1] = __int_as_float(v.y);
                b[k + 2] = __int_as_float(v.z); b[k + 3] = __int_as_float(v.w);
            }
        }
#pragma unroll
        for (int p = 0; p < K; ++p) {
            const int w = 1 << p;
            // b[k] = B_{w/2}(k) -> B_w(k); ascending k reads b[k + w/2] before it changes
            if (p == 1) {
#pragma unroll
                for (int k = 0; k + w <= kWin; ++k) b[k] = b[k] + b[k + 1];
            } else if (p > 1) {
#pragma unroll
                for (int k = 0; k + w < kWin; k += 2) add2(b[k], b[k + 1], b[k + w / 2], b[k + 1 + w / 2]);
            }
            T m0 = b[0], m1 = b[1];
#pragma unroll
            for (int i = 2; i < kPow2Per - 2; i += 4) {
                m0 = max3(m0, b[i], b[i + 1]);
                m1 = max3(m1, b[i + 2], b[i + 3]);
            }
            m0 = max3(m0, m1, b[kPow2Per - 2]);
            m1 = b[kPow2Per - 1];
            if constexpr (kInt) hit |= (long long)m0 > thi[p] || (long long)m1 > thi[p];
            else hit |= m0 > thf[p] || m1 > thf[p];
        }
    }
    if (!__syncthreads_or(hit)) return;

    // Runs with a hit again, sample by sample; their hits through the list.
    unsigned hits[K];
#pragma unroll
    for (int p = 0; p < K; ++p) hits[p] = 0u;
    if (hit) {
        const int64_t rem = avail - base;           // samples from this thread's first one on
        T b[kWin];
#pragma unroll
        for (int k = 0; k < kWin; ++k) b[k] = xb[spad32(k)];
#pragma unroll
        for (int p = 0; p < K; ++p) {
            const int w = 1 << p;
            if (p > 0) {
#pragma unroll
                for (int k = 0; k + w <= kWin; ++k) b[k] = b[k] + b[k + w / 2];
            }
            unsigned m = 0;
#pragma unroll
            for (int i = 0; i < kPow2Per; ++i) {
                bool h;
                if constexpr (kInt) h = (long long)b[i] > thi[p];
                else h = b[i] > thf[p];
                m |= (unsigned)h << i;
            }
            const int64_t lim = rem - w + 1;        // tests with t + w <= nout
            if (lim < kPow2Per) m &= lim > 0 ? (1u << lim) - 1u : 0u;
            hits[p] = m;
        }
    }
    for (;;) {
        int mine = 0;
#pragma unroll
        for (int p = 0; p < K; ++p) mine += __popc(hits[p]);
        int at = mine ? atomicAdd(&nlist, mine) : 0;
#pragma unroll
        for (int p = 0; p < K; ++p)
            while (hits[p] && at < kHitList) {
                list[at++] = (unsigned short)(threadIdx.x << 8 | p << 5 | (__ffs((int)hits[p]) - 1));
                hits[p] &= hits[p] - 1;
                --mine;
            }
        __syncthreads();
        const int n = min(nlist, kHitList);
        if (threadIdx.x == 0) first = atomicAdd(count, (unsigned long long)n);
        __syncthreads();
        for (int q = threadIdx.x; q < n; q += kPow2Threads) {
            const int code = list[q], p = code >> 5 & 7, i = (code >> 8) * kPow2Per + (code & 31);
            const T v = tree_sum_p<T, K>(x, i, p);   // B_w(i) again, by the same tree (the same value)
            put_candidate(cands, cap, first + q, row, 1 << p, sidx[p], t0 + i, (double)v, prm, rp);
        }
        if (threadIdx.x == 0) nlist = 0;
        if (!__syncthreads_or(mine > 0)) return;
    }
}

template <bool kInt, int K>
static void launch_search_pow2(dim3 grid, cudaStream_t s, const void *out, const dd_plan *p)
{
    const size_t smem = (size_t)spad32(kPow2Tile + kPow2Per + (1 << (K - 1)) + 4) * 4;
    search_pow2_kernel<kInt, K><<<grid, kPow2Threads, smem, s>>>(out, p->nsamp_out, p->d_wsorted, p->d_params,
                                                                    p->row_stats ? p->d_rowprm : nullptr,
                                                                    p->d_cands, p->cand_cap, p->d_count);
}

// K if the plan's widths are exactly {1, 2, ..., 2^(K-1)} with K <= 7, else 0.
static int pow2_widths(const dd_plan *p)
{
    std::vector<int> w(p->widths.begin(), p->widths.end());
    std::sort(w.begin(), w.end());
    if (w.size() > 7) return 0;
    for (size_t i = 0; i < w.size(); ++i)
        if (w[i] != (1 << i)) return 0;
    return (int)w.size();
}

template <bool kInt>
static void launch_search_pow2_k(int K, dim3 grid, cudaStream_t s, const void *out, const dd_plan *p)
{
    switch (K) {
    case 1: launch_search_pow2<kInt, 1>(grid, s, out, p); break;
    case 2: launch_search_pow2<kInt, 2>(grid, s, out, p); break;
    case 3: launch_search_pow2<kInt, 3>(grid, s, out, p); break;
    case 4: launch_search_pow2<kInt, 4>(grid, s, out, p); break;
    case 5: launch_search_pow2<kInt, 5>(grid, s, out, p); break;
    case 6: launch_search_pow2<kInt, 6>(grid, s, out, p); break;
    default: launch_search_pow2<kInt, 7>(grid, s, out, p); break;
    }
}

// Boxcars that cross a chunk boundary (streaming search variant): per DM row,
// x = [the previous chunk's last L outputs | this chunk's first L outputs],
// L = wmax - 1; every window of width w starting at i in [L - w + 1, L) (it
// starts in the previous chunk and ends in this one) is tested against this
// chunk's thresholds.  Hits get t = i - L < 0: the window starts |t| samples
// before this chunk's first output.  S/N is formed on the host.
template <bool kInt>
__global__ void __launch_bounds__(128)
boundary_search_kernel(const void *__restrict__ tail_, const void *__restrict__ out_, int64_t nout, int L,
                       const int32_t *__restrict__ widths, int nw, const SearchParams *__restrict__ prm,
                       const RowParams *__restrict__ rp, dd_candidate *__restrict__ cands, int64_t cap,
                       unsigned long long *__restrict__ count)
{
    using T = typename std::conditional<kInt, int32_t, float>::type;
    using Acc = typename std::conditional<kInt, long long, float>::type;
    extern __shared__ __align__(16) unsigned char sraw[];
    T *x = reinterpret_cast<T *>(sraw);
    const int row = blockIdx.x;
    const T *tail = reinterpret_cast<const T *>(tail_) + (size_t)row * L;
    const T *head = reinterpret_cast<const T *>(out_) + (size_t)row * nout;
    for (int i = threadIdx.x; i < L; i += blockDim.x) { x[i] = tail[i]; x[L + i] = head[i]; }
    __syncthreads();
    for (int q = threadIdx.x; q < nw * L; q += blockDim.x) {
        const int p = q / L, i = q - p * L, w = widths[p];
        if (i < L - w + 1) continue;                 // window ends before this chunk
        Acc b = 0;
        for (int j = 0; j < w; ++j) b += (Acc)x[i + j];
        bool hit;
        if constexpr (kInt) hit = (long long)b > (rp ? rp[row].thr_i[p] : prm->thr_i[p]);
        else hit = b > (rp ? rp[row].thr_f[p] : prm->thr_f[p]);
        if (hit) {
            const unsigned long long pos = atomicAdd(count, 1ull);
            if ((int64_t)pos < cap) {
                dd_candidate c;
                c.dm_idx = row; c.width_idx = p; c.t = (int64_t)i - L;
                c.snr = 0.f; c.reserved = 0.f; c.value = (double)b;
                cands[pos] = c;
            }
        }
    }
}

int boundary_search_launch(dd_plan *p, const void *tail, const void *out, int L, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(p->d_count, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return cuda_fail(e, "memset count");
    const int32_t *w_orig = p->d_wsorted + 2 * p->nwidths;
    const RowParams *rp = p->row_stats ? p->d_rowprm : nullptr;
    const size_t smem = (size_t)2 * L * 4;
    if (p->dtype == DD_U8)
        boundary_search_kernel<true><<<(unsigned)p->ndm, 128, smem, s>>>(tail, out, p->nsamp_out, L, w_orig, p->nwidths,
                                                                        p->d_params, rp, p->d_cands, p->cand_cap,
                                                                        p->d_count);
    else
        boundary_search_kernel<false><<<(unsigned)p->ndm, 128, smem, s>>>(tail, out, p->nsamp_out, L, w_orig,
                                                                         p->nwidths, p->d_params, rp, p->d_cands,
                                                                         p->cand_cap, p->d_count);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "launch boundary_search_kernel");
    return DD_OK;
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
static size_t stat_size(const dd_plan *p)
{
    return p->dtype == DD_U8 ? sizeof(StatI) : sizeof(StatF);
}

// The dynamic shared-memory limit is a per-kernel (not per-plan) attribute:
// set it once to everything the device allows so that plans of different
// geometry never lower it under one another.
cudaError_t allow_max_dynamic_smem(const void *fn, size_t optin)
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, fn);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(optin - a.sharedSizeBytes));
}

int ensure_partials_public(dd_plan *p, int64_t n)
{
    if (n <= p->n_partials_cap) return DD_OK;
    // An outgrown buffer stays until the plan goes: a graph captured before (a
    // batch's, or a caller's own) holds its address, and its kernels write and
    // read their partials there.  Shapes differ in their number of blocks (the
    // finer shape of a launch of few blocks has 8 times the others'), so a plan
    // outgrows its buffer at most once per shape.
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, (size_t)n * stat_size(p));
    if (e != cudaSuccess) return set_error(DD_ERR_NOMEM, "cudaMalloc(partials, %lld): %s",
                                           (long long)n, cudaGetErrorString(e));
    if (p->d_partials) p->old_partials.push_back(p->d_partials);
    p->d_partials = q;
    p->n_partials_cap = n;
    return DD_OK;
}

int generic_configure(dd_plan *p)
{
    const int nblk = (p->ndm + kGenDms - 1) / kGenDms;
    const int C = p->nchans;
    std::vector<int32_t> offs((size_t)nblk * C * kGenDms), base((size_t)nblk * C), span((size_t)nblk * C);
    int maxspan = 0;
    for (int b = 0; b < nblk; ++b) {
        const int dm0 = b * kGenDms, ndb = std::min(kGenDms, p->ndm - dm0);
        for (int c = 0; c < C; ++c) {
            int lo = INT32_MAX, hi = INT32_MIN;
            for (int j = 0; j < ndb; ++j) {
                const int d = p->delays[(size_t)(dm0 + j) * C + c];
                lo = std::min(lo, d); hi = std::max(hi, d);
            }
            base[(size_t)b * C + c] = lo;
            span[(size_t)b * C + c] = hi - lo;
            maxspan = std::max(maxspan, hi - lo);
            for (int j = 0; j < kGenDms; ++j) {
                const int jj = std::min(j, ndb - 1);
                offs[((size_t)b * C + c) * kGenDms + j] = p->delays[(size_t)(dm0 + jj) * C + c] - lo;
            }
        }
    }
    // Shared-memory geometry: rows of kGenTile + maxspan floats (rounded to 4).
    const int stride = ((kGenTile + maxspan + 3) / 4) * 4;
    const size_t budget = std::min<size_t>(p->smem_optin, 100 * 1024);
    const size_t per_chan = (size_t)stride * sizeof(float) + kGenDms * sizeof(int);
    int chunk = (int)std::min<size_t>(16, budget / per_chan);
    if (chunk < 1) chunk = 0;
    p->gen_stride = stride;
    p->gen_chunk = chunk;
    p->gen_smem = chunk ? (size_t)chunk * per_chan : 0;

    // Device copies, packed as [offs | base | span] in one allocation.
    void *dptr = nullptr;
    const size_t bytes = (offs.size() + base.size() + span.size()) * sizeof(int32_t);
    cudaError_t e = cudaMalloc(&dptr, bytes);
    if (e != cudaSuccess) return set_error(DD_ERR_NOMEM, "cudaMalloc(generic tables): %s", cudaGetErrorString(e));
    int32_t *d = static_cast<int32_t *>(dptr);
    e = cudaMemcpy(d, offs.data(), offs.size() * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d + offs.size(), base.data(), base.size() * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d + offs.size() + base.size(), span.data(), span.size() * 4, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) { cudaFree(dptr); return cuda_fail(e, "upload generic tables"); }
    p->d_gen = d;
    if (chunk) {
        auto set = [&](const void *fn) {
            return allow_max_dynamic_smem(fn, p->smem_optin);
        };
        cudaError_t a = cudaSuccess;
        a = set((const void *)generic_kernel<float, false>);
        if (a == cudaSuccess) a = set((const void *)generic_kernel<__half, false>);
        if (a == cudaSuccess) a = set((const void *)generic_kernel<uint8_t, true>);
        if (a != cudaSuccess) return cuda_fail(a, "cudaFuncSetAttribute(generic)");
    }
    return DD_OK;
}

int generic_execute(dd_plan *p, const void *in, int64_t pitch, void *out, cudaStream_t s)
{
    const int nblk = (p->ndm + kGenDms - 1) / kGenDms;
    const int64_t ntile = (p->nsamp_out + kGenTile - 1) / kGenTile;
    if (ntile > INT32_MAX || nblk > 65535) return set_error(DD_ERR_ARG, "problem too large for kernel 1 grid");
    const int64_t np = ntile * nblk;
    int rc = ensure_partials_public(p, np);
    if (rc) return rc;
    const size_t noffs = (size_t)nblk * p->nchans * kGenDms;
    const int32_t *goffs = p->d_gen;
    const int32_t *gbase = goffs + noffs;
    const int32_t *gspan = gbase + (size_t)nblk * p->nchans;
    dim3 grid((unsigned)ntile, (unsigned)nblk);
    switch (p->dtype) {
    case DD_F32:
        generic_kernel<float, false><<<grid, kGenThreads, p->gen_smem, s>>>(
            (const float *)in, pitch, p->nsamp_in, p->nchans, goffs, gbase, gspan, p->ndm,
            p->nsamp_out, out, p->d_partials, p->gen_chunk, p->gen_stride);
        break;
    case DD_F16:
        generic_kernel<__half, false><<<grid, kGenThreads, p->gen_smem, s>>>(
            (const __half *)in, pitch, p->nsamp_in, p->nchans, goffs, gbase, gspan, p->ndm,
            p->nsamp_out, out, p->d_partials, p->gen_chunk, p->gen_stride);
        break;
    case DD_U8:
        generic_kernel<uint8_t, true><<<grid, kGenThreads, p->gen_smem, s>>>(
            (const uint8_t *)in, pitch, p->nsamp_in, p->nchans, goffs, gbase, gspan, p->ndm,
            p->nsamp_out, out, p->d_partials, p->gen_chunk, p->gen_stride);
        break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "launch generic_kernel");
    p->n_partials = np;
    p->stats_out = out;
    return DD_OK;
}

int stats_from_out(dd_plan *p, const void *out, cudaStream_t s)
{
    const int64_t total = (int64_t)p->ndm * p->nsamp_out;
    const int64_t per = (int64_t)kStatThreads * kStatPer;
    const int64_t nb = (total + per - 1) / per;
    if (nb > INT32_MAX) return set_error(DD_ERR_ARG, "buffer too large for the stats kernel");
    int rc = ensure_partials_public(p, nb);
    if (rc) return rc;
    if (p->dtype == DD_U8)
        stats_kernel<true><<<(unsigned)nb, kStatThreads, 0, s>>>(out, total, p->d_partials);
    else
        stats_kernel<false><<<(unsigned)nb, kStatThreads, 0, s>>>(out, total, p->d_partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "launch stats_kernel");
    p->n_partials = nb;
    p->stats_out = out;
    return DD_OK;
}

int search_launch(dd_plan *p, const void *out, cudaStream_t s)
{
    const bool isint = p->dtype == DD_U8;
    // widths are stored original-order in [0,nw) of d_wsorted's tail region
    const int32_t *w_orig = p->d_wsorted + 2 * p->nwidths;
    const unsigned nfin = (unsigned)std::max<int64_t>(1, std::min<int64_t>(kFinBlocks, (p->n_partials + kFinRun - 1) / kFinRun));
    if (isint)
        finalize_kernel<true><<<nfin, kFinThreads, 0, s>>>(p->d_partials, p->n_partials, w_orig, p->nwidths,
                                                           p->sigma_k, p->d_params, p->d_count, p->d_fin);
    else
        finalize_kernel<false><<<nfin, kFinThreads, 0, s>>>(p->d_partials, p->n_partials, w_orig, p->nwidths,
                                                            p->sigma_k, p->d_params, p->d_count, p->d_fin);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "launch finalize_kernel");
    const RowParams *rp = nullptr;
    if (p->row_stats && p->d_rowprm) {
        if (isint)
            row_stats_kernel<true><<<(unsigned)p->ndm, kRowThreads, 0, s>>>(out, p->nsamp_out, w_orig, p->nwidths,
                                                                           p->sigma_k, p->d_rowprm);
        else
            row_stats_kernel<false><<<(unsigned)p->ndm, kRowThreads, 0, s>>>(out, p->nsamp_out, w_orig, p->nwidths,
                                                                            p->sigma_k, p->d_rowprm);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "launch row_stats_kernel");
        rp = p->d_rowprm;
    }
    int wmax = 0;
    for (int w : p->widths) wmax = std::max(wmax, w);
    const int K = pow2_widths(p);
    const int tile = K ? kPow2Tile : isint ? SearchShape<true>::kTile : SearchShape<false>::kTile;
    const dim3 grid((unsigned)((p->nsamp_out + tile - 1) / tile), (unsigned)p->ndm);
    int ws[kMaxWidths];
    std::copy(p->widths.begin(), p->widths.end(), ws);
    std::sort(ws, ws + p->nwidths);
    bool wide = false;
    for (int i = 0; i < p->nwidths; ++i) wide |= ws[i] - (i ? ws[i - 1] : 0) > kSearchGap;
    const size_t smem = isint ? SearchShape<true>::smem(wmax, wide) : SearchShape<false>::smem(wmax, wide);
    if (K) {
        if (isint) launch_search_pow2_k<true>(K, grid, s, out, p);
        else launch_search_pow2_k<false>(K, grid, s, out, p);
    } else if (isint)
        search_kernel<true><<<grid, kSearchThreads, smem, s>>>(out, p->nsamp_out, p->d_wsorted, p->nwidths,
                                                               wmax, wide, p->d_params, rp, p->d_cands, p->cand_cap,
                                                               p->d_count);
    else
        search_kernel<false><<<grid, kSearchThreads, smem, s>>>(out, p->nsamp_out, p->d_wsorted, p->nwidths,
                                                                wmax, wide, p->d_params, rp, p->d_cands, p->cand_cap,
                                                                p->d_count);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "launch search_kernel");
    return DD_OK;
}

}  // namespace dd
