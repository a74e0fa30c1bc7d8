// Front end of the real-time pipeline (Section 5, Tables 5-6): the
// channeliser (an nfft-point FFT of each block of a subband's complex
// voltages), the intensity |X|^2 summed over polarisations, and the corner
// turn to channel-major order, fused into one pass over the voltages.
//
// Thread = one block b of one subband s: it loads nfft complex samples per
// polarisation with 16-byte loads (consecutive threads read consecutive
// blocks: coalesced), transforms them in registers (radix-2, decimation in
// time), and writes the nfft intensities to rows s*nfft + j of the output at
// column b.  Consecutive threads write consecutive columns of each row, so
// the corner turn needs no shared-memory transpose.  Every voltage is read
// once (8 bytes per sample and polarisation) and every intensity written once
// (4 bytes per nfft samples): the kernel is HBM-bound.
#include "dd_internal.h"

#include <algorithm>

namespace dd {

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// cos and sin of 2 pi m / 32, m < 16, rounded once: the twiddles of every
// transform length, as constants of the unrolled butterflies (sincospif of
// constant arguments was computed at run time, 31 of them per 32-point
// transform).  From the Taylor series in double, |x| <= pi.
struct Twiddles {
    float c[16], s[16];
    constexpr Twiddles() : c(), s()
    {
        for (int m = 0; m < 16; ++m) {
            const double x = 2.0 * 3.14159265358979323846 * m / 32.0;
            double term = 1.0, cs = 0.0, sn = 0.0;
            for (int k = 0; k < 40; k += 4) {
                cs += term; term *= x / (k + 1);
                sn += term; term *= x / (k + 2);
                cs -= term; term *= x / (k + 3);
                sn -= term; term *= x / (k + 4);
            }
            c[m] = m == 8 ? 0.f : (float)cs;
            s[m] = (float)sn;
        }
    }
};

// In-place radix-2 DIT FFT of F points (F a power of two), forward sign.
template <int F>
__device__ __forceinline__ void fft_inplace(float2 (&x)[F])
{
    constexpr Twiddles tw;
    // bit-reversal permutation
#pragma unroll
    for (int i = 0; i < F; ++i) {
        int r = 0;
#pragma unroll
        for (int b = 1, v = i; b < F; b <<= 1, v >>= 1) r = (r << 1) | (v & 1);
        if (r > i) { const float2 t = x[i]; x[i] = x[r]; x[r] = t; }
    }
#pragma unroll
    for (int len = 2; len <= F; len <<= 1) {
#pragma unroll
        for (int m = 0; m < len / 2; ++m) {
            const float2 w = make_float2(tw.c[m * (32 / len)], -tw.s[m * (32 / len)]);     // W_len^m
#pragma unroll
            for (int i = 0; i < F; i += len) {
                const float2 u = x[i + m], v = m == 0 ? x[i + m + len / 2] : cmul(w, x[i + m + len / 2]);
                x[i + m] = make_float2(u.x + v.x, u.y + v.y);
                x[i + m + len / 2] = make_float2(u.x - v.x, u.y - v.y);
            }
        }
    }
}

template <int F, int NPOL>
__global__ void __launch_bounds__(256) channelise_kernel(const float2 *__restrict__ volt, int nsub,
                                                         int64_t nsamp, int64_t nblk,
                                                         float *__restrict__ out, int64_t out_pitch)
{
    const int s = blockIdx.y;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nblk;
         b += (int64_t)gridDim.x * blockDim.x) {
        float pw[F];
#pragma unroll
        for (int k = 0; k < F; ++k) pw[k] = 0.f;
#pragma unroll
        for (int p = 0; p < NPOL; ++p) {
            const float4 *src = reinterpret_cast<const float4 *>(volt + ((size_t)p * nsub + s) * nsamp + b * F);
            float2 x[F];
#pragma unroll
            for (int q = 0; q < F / 2; ++q) {
                const float4 v = __ldg(src + q);
                x[2 * q] = make_float2(v.x, v.y);
                x[2 * q + 1] = make_float2(v.z, v.w);
            }
            fft_inplace<F>(x);
#pragma unroll
            for (int k = 0; k < F; ++k) pw[k] += x[k].x * x[k].x + x[k].y * x[k].y;
        }
        // channel j of the subband: bin (F/2 - 1 - j) mod F (descending frequency)
#pragma unroll
        for (int j = 0; j < F; ++j)
            out[((size_t)s * F + j) * out_pitch + b] = pw[(F / 2 - 1 - j + F) % F];
    }
}

// The same for long transforms: a thread's block of F samples is 8 F
// consecutive bytes, so that with 16-byte loads straight from memory a warp's
// loads of F = 32 lie 256 bytes apart.  Here the block's threads fetch their
// blocks together, consecutive threads consecutive 16 bytes (cp.async, every
// polarisation at once), into shared rows padded by 16 bytes, from which each
// thread reads its own without bank conflicts: 2 polarisations x 64 subbands x
// 2^19 samples, 32 points, 141 -> 98 us (6.9 TB/s).
template <int F, int NPOL>
constexpr int staged_threads() { return F * NPOL >= 64 ? 64 : 128; }    // rows within 48 KB

template <int F, int NPOL>
__global__ void __launch_bounds__(staged_threads<F, NPOL>()) channelise_staged_kernel(const float2 *__restrict__ volt, int nsub, int64_t nsamp,
                                                                int64_t nblk, float *__restrict__ out, int64_t out_pitch)
{
    constexpr int kT = staged_threads<F, NPOL>(), kUnits = F / 2;              // 16-byte units per block of samples
    extern __shared__ __align__(16) float4 tile[];        // [NPOL][kT][kUnits + 1]
    const int s = blockIdx.y, tid = threadIdx.x;
    const int64_t b0 = (int64_t)blockIdx.x * kT;
    const int nb = (int)min((int64_t)kT, nblk - b0);
#pragma unroll
    for (int p = 0; p < NPOL; ++p) {
        const float4 *src = reinterpret_cast<const float4 *>(volt + ((size_t)p * nsub + s) * nsamp + b0 * F);
        float4 *dst = tile + p * kT * (kUnits + 1);
        for (int k = tid; k < nb * kUnits; k += kT) {
            const unsigned d = (unsigned)__cvta_generic_to_shared(dst + k + k / kUnits);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src + k) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    float pw[F];
#pragma unroll
    for (int k = 0; k < F; ++k) pw[k] = 0.f;
#pragma unroll
    for (int p = 0; p < NPOL; ++p) {
        if (p + 1 < NPOL) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (tid < nb) {
            const float4 *src = tile + (p * kT + tid) * (kUnits + 1);
            float2 x[F];
#pragma unroll
            for (int q = 0; q < kUnits; ++q) {
                const float4 v = src[q];
                x[2 * q] = make_float2(v.x, v.y);
                x[2 * q + 1] = make_float2(v.z, v.w);
            }
            fft_inplace<F>(x);
#pragma unroll
            for (int k = 0; k < F; ++k) pw[k] += x[k].x * x[k].x + x[k].y * x[k].y;
        }
    }
    if (tid < nb)
#pragma unroll
        for (int j = 0; j < F; ++j)
            out[((size_t)s * F + j) * out_pitch + b0 + tid] = pw[(F / 2 - 1 - j + F) % F];
}

template <int F, int NPOL>
static cudaError_t channelise_staged_launch(const float2 *v, int nsub, int64_t nsamp, float *out, int64_t out_pitch,
                                            cudaStream_t s)
{
    const int64_t nblk = nsamp / F;
    constexpr int kT = staged_threads<F, NPOL>();
    constexpr size_t kSmem = (size_t)NPOL * kT * (F / 2 + 1) * 16;
    static_assert(kSmem <= 48 * 1024, "no attribute to set on each call");
    channelise_staged_kernel<F, NPOL><<<dim3((unsigned)((nblk + kT - 1) / kT), (unsigned)nsub), kT, kSmem, s>>>(
        v, nsub, nsamp, nblk, out, out_pitch);
    return cudaGetLastError();
}

template <int F>
static cudaError_t channelise_launch(const float2 *v, int npol, int nsub, int64_t nsamp, float *out,
                                     int64_t out_pitch, cudaStream_t s)
{
    if constexpr (F >= 16) {
        // blocks of samples of 128 bytes and more (nsamp even keeps every row on 16 bytes)
        return npol == 1 ? channelise_staged_launch<F, 1>(v, nsub, nsamp, out, out_pitch, s)
                         : channelise_staged_launch<F, 2>(v, nsub, nsamp, out, out_pitch, s);
    } else {
        const int64_t nblk = nsamp / F;
        const dim3 grid((unsigned)std::min<int64_t>((nblk + 255) / 256, 65535), (unsigned)nsub);
        if (npol == 1)
            channelise_kernel<F, 1><<<grid, 256, 0, s>>>(v, nsub, nsamp, nblk, out, out_pitch);
        else
            channelise_kernel<F, 2><<<grid, 256, 0, s>>>(v, nsub, nsamp, nblk, out, out_pitch);
        return cudaGetLastError();
    }
}

}  // namespace dd

using namespace dd;

extern "C" int dd_channelise(const void *volt_dev, int32_t npol, int32_t nsub, int64_t nsamp, int32_t nfft,
                             float *out_dev, int64_t out_pitch, void *stream)
{
    if (!volt_dev || !out_dev) return set_error(DD_ERR_ARG, "NULL buffer");
    if (npol < 1 || npol > 2) return set_error(DD_ERR_ARG, "npol must be 1 or 2");
    if (nsub < 1 || nsub > 65535) return set_error(DD_ERR_ARG, "nsub must be in 1..65535");
    if (nfft != 2 && nfft != 4 && nfft != 8 && nfft != 16 && nfft != 32)
        return set_error(DD_ERR_ARG, "nfft must be 2, 4, 8, 16 or 32");
    if (nsamp < nfft || nsamp % 2) return set_error(DD_ERR_ARG, "nsamp must be even and >= nfft");
    if ((uintptr_t)volt_dev & 15u) return set_error(DD_ERR_ARG, "voltages must be 16-byte aligned");
    if (out_pitch < nsamp / nfft) return set_error(DD_ERR_ARG, "out_pitch < nsamp / nfft");
    const float2 *v = static_cast<const float2 *>(volt_dev);
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    switch (nfft) {
    case 2: e = channelise_launch<2>(v, npol, nsub, nsamp, out_dev, out_pitch, s); break;
    case 4: e = channelise_launch<4>(v, npol, nsub, nsamp, out_dev, out_pitch, s); break;
    case 8: e = channelise_launch<8>(v, npol, nsub, nsamp, out_dev, out_pitch, s); break;
    case 16: e = channelise_launch<16>(v, npol, nsub, nsamp, out_dev, out_pitch, s); break;
    default: e = channelise_launch<32>(v, npol, nsub, nsamp, out_dev, out_pitch, s); break;
    }
    if (e != cudaSuccess) return cuda_fail(e, "launch channelise_kernel");
    return DD_OK;
}
