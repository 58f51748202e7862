// isr_linefit.cu -- plasma-line frequency by spectral peak fit on integrated spectra.
//
// The plasma line's frequency carries the electron density (Eq. 1 of the paper: f_r^2 =
// f_p^2 + thermal and magnetic terms, f_p ~ sqrt(n_e)), so the product of an integration is
// the line position per gate.  Per gate: the largest bin of the band, refined by a
// three-point parabola through the logarithm of the power (exact for a Gaussian-shaped
// peak), in double precision; plus the ratio of the peak to the band's mean power.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>

#include "isr.h"
#include "isr_ff.cuh"
#include "isr_kernels.cuh"

namespace {

constexpr int kFitThreads = 256;

// One CTA per gate.  4 bytes per bin bound it; the band's sum runs in float-float on the FP32 pipe
// (an FP64 conversion and addition per bin bound it before: 34.7 us for 1000 gates x 4608 bins), and
// the three logarithms and the two quotients run side by side in lanes of one warp, each FP64
// instruction of which occupies the narrow pipe as long for one lane as for all.  A band whose
// float-float sum is not finite (an infinity, a NaN, or an FP32 overflow) is summed again in FP64.
__global__ void __launch_bounds__(kFitThreads) peak_fit_kernel(const float* __restrict__ spectra, int nfft,
                                                               int band_lo, int band_hi, double* __restrict__ freq_bin,
                                                               float* __restrict__ snr)
{
    constexpr int W = kFitThreads / 32, U = 8;
    const int r = blockIdx.x;
    const float* P = spectra + (size_t)r * nfft;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    float best = -INFINITY;
    int best_i = band_lo;
    isr::ff sum{0.f, 0.f};
    auto take = [&](int i, float v) {
        if (v > best) {  // strided scan in increasing i keeps the lowest index on ties
            best = v;
            best_i = i;
        }
        isr::ff_acc(sum, v);
    };
    int i = band_lo + threadIdx.x;
    for (; i + (U - 1) * kFitThreads < band_hi; i += U * kFitThreads) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = P[i + u * kFitThreads];
#pragma unroll
        for (int u = 0; u < U; ++u) take(i + u * kFitThreads, v[u]);
    }
    for (; i < band_hi; i += kFitThreads) take(i, P[i]);
    // block reduction: max value, lowest index among equal maxima; sum
    __shared__ float s_best[W];
    __shared__ int s_idx[W];
    __shared__ isr::ff s_sum[W];
    auto merge = [&](float ob, int oi) {
        if (ob > best || (ob == best && oi < best_i)) {
            best = ob;
            best_i = oi;
        }
    };
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, best_i, o);
        merge(ob, oi);
    }
    sum = isr::ff_warp_sum(isr::ff_norm(sum.h, sum.l));
    if (l == 0) {
        s_best[w] = best;
        s_idx[w] = best_i;
        s_sum[w] = sum;
    }
    __syncthreads();
    if (w != 0) return;
    best = s_best[0];
    best_i = s_idx[0];
    for (int k = 1; k < W; ++k) merge(s_best[k], s_idx[k]);
    sum = isr::ff_warp_sum(l < W ? s_sum[l] : isr::ff{0.f, 0.f});
    double total = isr::ff_to_double(sum);
    if (!isfinite(sum.h) || !isfinite(sum.l)) {
        total = 0.0;
        for (int j = band_lo + l; j < band_hi; j += 32) total += (double)P[j];
        for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    }
    // lanes 0, 1, 2: the bins before, at and after the peak
    const int at = l == 0 ? (best_i - 1 + nfft) % nfft : l == 2 ? (best_i + 1) % nfft : best_i;
    const double v = l == 1 ? (double)best : (double)P[at];
    const bool positive = (__ballot_sync(0xffffffffu, v > 0.0) & 7u) == 7u;
    const double y = positive ? log(v) : 0.0;
    const double ym = __shfl_sync(0xffffffffu, y, 0), y0 = __shfl_sync(0xffffffffu, y, 1),
                 yp = __shfl_sync(0xffffffffu, y, 2);
    const double d = ym - 2.0 * y0 + yp;
    // lane 0: the parabola's offset; lane 1: peak over mean, as best / (total / n)
    const double mean = total / (double)(band_hi - band_lo);
    const double quot = (l == 0 ? 0.5 * (ym - yp) : (double)best) / (l == 0 ? d : mean);
    if (l == 0) {
        double delta = positive && d < 0.0 ? quot : 0.0;
        if (positive) delta = fmin(0.5, fmax(-0.5, delta));
        freq_bin[r] = (double)best_i + delta;
    } else if (l == 1) {
        snr[r] = mean > 0.0 ? (float)quot : 0.f;
    }
}

}  // namespace

extern "C" isr_status isr_peak_fit(const float* spectra, int32_t n_ranges, int32_t nfft, int32_t band_lo,
                                   int32_t band_hi, double* freq_bin, float* snr, void* stream)
{
    isr::clear_error();
    if (!spectra || !freq_bin || !snr) return isr::fail(ISR_ERR_INVALID_ARG, "isr_peak_fit: NULL pointer");
    if (n_ranges < 1 || nfft < 8 || band_lo < 0 || band_hi > nfft || band_hi - band_lo < 1)
        return isr::fail(ISR_ERR_INVALID_ARG, "isr_peak_fit: need n_ranges >= 1, nfft >= 8, 0 <= band_lo < band_hi <= nfft");
    peak_fit_kernel<<<n_ranges, kFitThreads, 0, static_cast<cudaStream_t>(stream)>>>(spectra, nfft, band_lo, band_hi,
                                                                                   freq_bin, snr);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return isr::fail(ISR_ERR_CUDA, "isr_peak_fit: %s", cudaGetErrorString(e));
    return ISR_OK;
}
