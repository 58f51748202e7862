// isr_estimator.cu -- learned plasma-line estimator: forward, backward and Adam kernels.
//
// The plasma line's frequency carries the electron density (Eq. 1 of the paper).  A small
// network reads one gate's integrated spectrum (standardised log power over a band) and
// returns the line position and a presence probability:
//   4 x [conv1d 9 taps, 32 channels, zero padding, ReLU] -> location logits z (1x1 conv)
//   and presence logit q from an MLP on [max over bins, mean over bins] of the last layer.
// Loss: BCE(q, present) + present * cross-entropy(softmax(z), Gaussian target of width
// 1 bin at the true position).  Parameters are kept in FP32 (master copy, Adam moments);
// activations and working weights are stored in the plan's precision (FP32 or BF16) and
// every product is accumulated in FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <new>
#include <type_traits>

#include "isr.h"
#include "isr_ff.cuh"
#include "isr_kernels.cuh"

namespace {

constexpr int CH = 32;      // channels
constexpr int KT = 9;       // taps
constexpr int HALF = KT / 2;
constexpr int WIN = 3;      // soft-argmax half window
constexpr float SIGMA_T = 1.0f;

// flat parameter layout (matches the documented order)
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + CH * 1 * KT;
constexpr int OFF_W2 = OFF_B1 + CH, OFF_B2 = OFF_W2 + CH * CH * KT;
constexpr int OFF_W3 = OFF_B2 + CH, OFF_B3 = OFF_W3 + CH * CH * KT;
constexpr int OFF_W4 = OFF_B3 + CH, OFF_B4 = OFF_W4 + CH * CH * KT;
constexpr int OFF_W5 = OFF_B4 + CH, OFF_B5 = OFF_W5 + CH;
constexpr int OFF_WA = OFF_B5 + 1, OFF_BA = OFF_WA + CH * 2 * CH;
constexpr int OFF_WB = OFF_BA + CH, OFF_BB = OFF_WB + CH;
constexpr int NPARAM = OFF_BB + 1;
static_assert(NPARAM == ISR_EST_N_PARAMS, "parameter count");

__host__ __device__ constexpr int w_off(int l) { return l == 1 ? OFF_W1 : l == 2 ? OFF_W2 : l == 3 ? OFF_W3 : OFF_W4; }
__host__ __device__ constexpr int b_off(int l) { return l == 1 ? OFF_B1 : l == 2 ? OFF_B2 : l == 3 ? OFF_B3 : OFF_B4; }

template <class T> __device__ __forceinline__ float ld(const T* p, size_t i);
template <> __device__ __forceinline__ float ld<float>(const float* p, size_t i) { return p[i]; }
template <> __device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16* p, size_t i)
{
    return __bfloat162float(p[i]);
}
template <class T> __device__ __forceinline__ T cvt(float v);
template <> __device__ __forceinline__ float cvt<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 cvt<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
// ---------------------------------------------------------------- features
// x[i] = (ln max(P[lo+i], 1e-30) - mean) / (std + 1e-6) over the band; one CTA per gate.
// Bytes bound it (4 in, 4 out per bin), so the logarithm and both moments run in float-float on the
// FP32 pipe instead of FP64, of which the part has about two operations per SM and clock: 1000 gates
// x 4608 bins took 618 us with two FP64 logarithms per bin, 32 us now.  The moments are taken about the first
// bin's logarithm, so the variance loses nothing to cancellation.  A thread keeps the logarithms of
// up to FT_KEEP bins in registers; bands beyond FT_THREADS x FT_KEEP bins form the rest again in the
// second pass.  A band with an infinite bin goes through the FP64 form, whose infinities and NaN are
// the defined result.
constexpr int FT_THREADS = 512;
constexpr int FT_KEEP = 10;

__device__ const isr::LnTable g_ln_table{};

__global__ void __launch_bounds__(FT_THREADS) features_kernel(const float* __restrict__ spectra, int nfft, int lo, int L,
                                                              float* __restrict__ x)
{
    const float* P = spectra + (size_t)blockIdx.x * nfft + lo;
    float* xo = x + (size_t)blockIdx.x * L;
    __shared__ isr::LnTable tab;
    __shared__ isr::ff r1[FT_THREADS / 32], r2[FT_THREADS / 32];
    __shared__ isr::ff mean_s, inv_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    float p[FT_KEEP];
#pragma unroll
    for (int k = 0; k < FT_KEEP; ++k) {
        const int i = tid + k * FT_THREADS;
        p[k] = i < L ? P[i] : 0.f;
    }
    const float pivot_p = P[0];
    for (int i = tid; i < (int)(sizeof(isr::LnTable) / 4); i += FT_THREADS)
        reinterpret_cast<float*>(&tab)[i] = reinterpret_cast<const float*>(&g_ln_table)[i];
    bool inf = false;
#pragma unroll
    for (int k = 0; k < FT_KEEP; ++k) inf |= p[k] == INFINITY;
    for (int i = tid + FT_KEEP * FT_THREADS; i < L; i += FT_THREADS) inf |= P[i] == INFINITY;
    if (__syncthreads_or(inf)) {
        double s = 0, s2 = 0;
        for (int i = tid; i < L; i += FT_THREADS) {
            const double y = log(fmax((double)P[i], 1e-30));
            s += y;
            s2 += y * y;
        }
        __shared__ double d1[FT_THREADS / 32], d2[FT_THREADS / 32];
        for (int o = 16; o; o >>= 1) {
            s += __shfl_down_sync(0xffffffffu, s, o);
            s2 += __shfl_down_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) {
            d1[warp] = s;
            d2[warp] = s2;
        }
        __syncthreads();
        double a = 0, b = 0;
        for (int w = 0; w < FT_THREADS / 32; ++w) {
            a += d1[w];
            b += d2[w];
        }
        const double m = a / L, inv = 1.0 / (sqrt(fmax(b / L - m * m, 0.0)) + 1e-6);
        for (int i = tid; i < L; i += FT_THREADS) xo[i] = (float)((log(fmax((double)P[i], 1e-30)) - m) * inv);
        return;
    }

    // ln max(v, 1e-30) less the pivot; NaN counts as 1e-30 (1e-30f is the first float above 1e-30)
    constexpr double kLnFloor = -30.0 * isr::LnTable::ln(1.25) - 90.0 * isr::LnTable::ln(2.0);   // ln 1e-30
    constexpr float fh = (float)kLnFloor, fl = (float)(kLnFloor - (double)fh);
    auto ln_of = [&](float v) { return v >= 1e-30f ? isr::ff_log(v, tab) : isr::ff{fh, fl}; };
    const float pivot = ln_of(pivot_p).h;
    auto dev = [&](float v) {
        const isr::ff y = ln_of(v);
        float s, e;
        isr::two_sum(y.h, -pivot, s, e);
        return isr::ff_norm(s, e + y.l);
    };
    isr::ff s1{0.f, 0.f}, s2{0.f, 0.f};
    auto add = [&](isr::ff d) {
        isr::ff_acc(s1, d.h);
        s1.l += d.l;
        const float sq = __fmul_rn(d.h, d.h);
        isr::ff_acc(s2, sq);
        s2.l += fmaf(2.f * d.h, d.l, fmaf(d.h, d.h, -sq));
    };
    isr::ff d[FT_KEEP];
#pragma unroll
    for (int k = 0; k < FT_KEEP; ++k) {
        const int i = tid + k * FT_THREADS;
        if (i < L) {
            d[k] = dev(p[k]);
            add(d[k]);
        }
    }
    for (int i = tid + FT_KEEP * FT_THREADS; i < L; i += FT_THREADS) add(dev(P[i]));
    s1 = isr::ff_warp_sum(isr::ff_norm(s1.h, s1.l));
    s2 = isr::ff_warp_sum(isr::ff_norm(s2.h, s2.l));
    if (lane == 0) {
        r1[warp] = s1;
        r2[warp] = s2;
    }
    __syncthreads();
    if (warp == 0) {
        static_assert(FT_THREADS / 32 <= 32, "one lane per warp");
        const bool in = lane < FT_THREADS / 32;
        const isr::ff a = isr::ff_warp_sum(in ? r1[lane] : isr::ff{0.f, 0.f});
        const isr::ff b = isr::ff_warp_sum(in ? r2[lane] : isr::ff{0.f, 0.f});
        if (lane == 0) {
            const double rl = 1.0 / L, m = isr::ff_to_double(a) * rl;
            const double var = fmax(isr::ff_to_double(b) * rl - m * m, 0.0);
            mean_s = isr::ff_of(m);
            inv_s = isr::ff_of(1.0 / (sqrt(var) + 1e-6));
        }
    }
    __syncthreads();
    const isr::ff mean = mean_s, inv = inv_s;
    auto out = [&](isr::ff v) {
        const isr::ff r = isr::ff_mul(isr::ff_add(v, isr::ff{-mean.h, -mean.l}), inv);
        return r.h;
    };
#pragma unroll
    for (int k = 0; k < FT_KEEP; ++k) {
        const int i = tid + k * FT_THREADS;
        if (i < L) xo[i] = out(d[k]);
    }
    for (int i = tid + FT_KEEP * FT_THREADS; i < L; i += FT_THREADS) xo[i] = out(dev(P[i]));
}

template <class T>
__global__ void cast_kernel(const float* __restrict__ in, size_t n, T* __restrict__ out)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = cvt<T>(in[i]);
}

// working conv weights: forward layout [ci][k][co] and the backward-data layout of the
// flipped transpose, [co][k'][ci] = W[co][ci][8 - k'] (both in the storage type); with
// tf and tb (tensor-core path, layers 2-4) also the GEMM rows [co][k][ci] of the forward
// weights and [ci][k'][co] of the flipped transpose
template <class T>
__global__ void relayout_kernel(const float* __restrict__ theta, T* __restrict__ wf, T* __restrict__ wb,
                                T* __restrict__ tf, T* __restrict__ tb)
{
    // layers 1..4 packed back to back: layer 1 has Cin = 1
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int n1 = CH * KT, n = CH * CH * KT;
    if (i >= n1 + 3 * n) return;
    int l, e, cin;
    if (i < n1) {
        l = 1; e = i; cin = 1;
    } else {
        l = 2 + (i - n1) / n; e = (i - n1) % n; cin = CH;
    }
    // e indexes [co][ci][k]
    int co = e / (cin * KT), rem = e % (cin * KT), ci = rem / KT, k = rem % KT;
    float w = theta[w_off(l) + e];
    size_t base = l == 1 ? 0 : (size_t)n1 + (size_t)(l - 2) * n;
    wf[base + ((size_t)ci * KT + k) * CH + co] = cvt<T>(w);
    if (l > 1) wb[(size_t)(l - 2) * n + ((size_t)co * KT + (KT - 1 - k)) * CH + ci] = cvt<T>(w);
    if (l > 1 && tf) {
        tf[(size_t)(l - 2) * n + ((size_t)co * KT + k) * CH + ci] = cvt<T>(w);
        tb[(size_t)(l - 2) * n + ((size_t)ci * KT + (KT - 1 - k)) * CH + co] = cvt<T>(w);
    }
}

// ---------------------------------------------------------------- convolution
// out[b][co][i] = sum_{ci,k} w[ci][k][co] in[b][ci][i + k - 4]  (+ bias, ReLU) or, for the
// backward-data use, times the ReLU mask of `mask` (the layer below's activations).  FP32 storage.
// CTA: 8 P positions of one row; warp = P positions, lane = output channel.  Bound by FMAs while enough
// CTAs share an SM: the launch takes the P for which the fullest SM has least to do (conv_positions; 37
// rows of 1101 positions at P = 16 gave some SMs three CTAs and most two).  The outputs go through
// shared memory, since a store of one position of 32 channels touches 32 lines.  That launch, P = 16 and
// direct stores: 29 us forward, 31 backward-data; now 21 and 25.
constexpr size_t conv_smem_bytes(int p) { return sizeof(float) * (size_t)CH * ((8 * p + KT - 1) + KT * CH); }

template <bool FWD, int P>
__global__ void __launch_bounds__(256) conv_kernel(const float* __restrict__ in, const float* __restrict__ w,
                                                   const float* __restrict__ bias, const float* __restrict__ mask,
                                                   int L, float* __restrict__ out)
{
    constexpr int CT = 8 * P, XW = CT + KT - 1;
    static_assert(P % 4 == 0 && CH * (CT + 1) <= CH * XW + CH * KT * CH, "16-byte rows; the outputs fit");
    extern __shared__ __align__(16) float conv_smem[];
    float* xs = conv_smem;                // [CH][XW]
    float* ws = conv_smem + CH * XW;      // [CH][KT][CH]
    const int b = blockIdx.y;
    const int i0 = blockIdx.x * CT;
    const float* inb = in + (size_t)b * CH * L;
    // staging, every load of the thread in flight before its first store (with a few at a time the
    // 54 KB took half of the kernel)
    constexpr int XPER = (CH * XW + 255) / 256, WPER = CH * KT * CH / 4 / 256;
    static_assert(CH * KT * CH == WPER * 4 * 256, "whole 16-byte pieces per thread");
    float xq[XPER];
#pragma unroll
    for (int u = 0; u < XPER; ++u) {
        const int e = threadIdx.x + u * 256, ci = e / XW, pos = i0 + e % XW - HALF;
        xq[u] = (e < CH * XW && pos >= 0 && pos < L) ? inb[(size_t)ci * L + pos] : 0.f;
    }
    float4 wq[WPER];
#pragma unroll
    for (int u = 0; u < WPER; ++u) wq[u] = reinterpret_cast<const float4*>(w)[threadIdx.x + u * 256];
#pragma unroll
    for (int u = 0; u < WPER; ++u) reinterpret_cast<float4*>(ws)[threadIdx.x + u * 256] = wq[u];
#pragma unroll
    for (int u = 0; u < XPER; ++u) {
        const int e = threadIdx.x + u * 256;
        if (e < CH * XW) xs[e] = xq[u];
    }
    __syncthreads();
    const int co = threadIdx.x & 31;
    const int p0 = (threadIdx.x >> 5) * P;
    float acc[P];
    const float bv = FWD ? bias[co] : 0.f;
#pragma unroll
    for (int p = 0; p < P; ++p) acc[p] = bv;
    for (int ci = 0; ci < CH; ++ci) {
        float xv[P + KT - 1];   // the same for all lanes: 16-byte loads (XW and p0 are multiples of 4)
#pragma unroll
        for (int j = 0; j < P + KT - 1; j += 4)
            *reinterpret_cast<float4*>(xv + j) = *reinterpret_cast<const float4*>(xs + ci * XW + p0 + j);
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            const float wv = ws[(ci * KT + k) * CH + co];
#pragma unroll
            for (int p = 0; p < P; ++p) acc[p] = fmaf(wv, xv[p + k], acc[p]);
        }
    }
    __syncthreads();
    float* os = conv_smem;   // [CH][CT + 1]
#pragma unroll
    for (int p = 0; p < P; ++p) os[co * (CT + 1) + p0 + p] = acc[p];
    __syncthreads();
#pragma unroll 8
    for (int e = threadIdx.x; e < CH * CT; e += 256) {
        const int c = e / CT, j = e % CT, i = i0 + j;
        if (i < L) {
            const size_t o = ((size_t)b * CH + c) * L + i;
            float v = os[c * (CT + 1) + j];
            if (FWD) v = fmaxf(v, 0.f);
            else v = mask[o] > 0.f ? v : 0.f;
            out[o] = v;
        }
    }
}

// Positions per warp: the choice whose fullest SM has least to do, a CTA's staging and stores counted as
// two positions (P = 16 for many rows).
inline int conv_positions(int L, int n, int sms)
{
    int best = 16;
    int64_t best_cost = INT64_MAX;
    for (int p : {16, 12, 8}) {
        const int64_t ctas = (int64_t)n * ((L + 8 * p - 1) / (8 * p)), cost = (ctas + sms - 1) / sms * (p + 2);
        if (cost < best_cost) best = p, best_cost = cost;
    }
    return best;
}

template <bool FWD>
void launch_conv(const float* in, const float* w, const float* bias, const float* mask, int L, int n, int sms, float* out,
                 cudaStream_t s)
{
    const int p = conv_positions(L, n, sms);
    auto* k = p == 16 ? conv_kernel<FWD, 16> : p == 12 ? conv_kernel<FWD, 12> : conv_kernel<FWD, 8>;
    k<<<dim3((L + 8 * p - 1) / (8 * p), n), 256, conv_smem_bytes(p), s>>>(in, w, bias, mask, L, out);
}

// ---------------------------------------------------------------- tensor-core convolution
// Layers 2-4 (32 -> 32 channels) with BF16 storage, as a GEMM on the warp-level tensor-core
// instruction mma.m16n8k16 (BF16 operands, FP32 accumulation):
//   out[co][i] = sum_kk A[co][kk] B[kk][i],   kk = 32 k + ci,   B[kk][i] = in[ci][i + k - 4],
// with A the weights in [co][k][ci] order (K = 288).  B is never formed: the CTA stages its
// input as a position-major tile, one 80-byte row of 32 channels per position (halo included),
// so the 8 x 8 blocks of B at tap k are rows i + k of that tile and ldmatrix reads them as they
// are.  Row pitches of 80 B (tile) and 592 B (weights) put the eight rows an ldmatrix reads on
// 32 distinct banks.  The backward-data convolution is the same GEMM on the flipped transposed
// weights; its FP32 input (the gradient) is split into two BF16 parts, hi + lo, and both are
// multiplied, so the products keep ~16 bits of the gradient and the FP32 accumulation.
// CTA: CF_CT = 512 positions x 32 output channels, 16 warps; warp w: positions [32 w, 32 w + 32),
// all channels (a CTA stages the 18 KB of weights once per 512 positions).
constexpr int CF_CT = 512;                 // positions per convolution CTA
constexpr int CF_THREADS = 16 * 32;
constexpr int CF_XW = CF_CT + KT - 1;      // staged positions, halo included
constexpr int CF_OR = CF_CT + 8;           // output staging row (elements)
constexpr int TC_CT = 256;                 // positions per weight-gradient chunk
constexpr int TC_XW = TC_CT + KT - 1;
constexpr int TC_XR = CH + 8;              // bf16 per staged position (80 B)
constexpr int TC_K = KT * CH;              // GEMM depth
constexpr int TC_WR = TC_K + 8;            // bf16 per staged weight row (592 B)
constexpr size_t tc_smem_bytes(bool fwd)
{
    return (size_t)2 * ((fwd ? 1 : 2) * CF_XW * TC_XR + CH * TC_WR);
}
static_assert(CF_CT == CF_THREADS, "a warp per 32 positions");
static_assert((size_t)CH * CF_OR * 4 <= (size_t)2 * 2 * CF_XW * TC_XR, "FP32 output tile fits the input tiles");
static_assert((size_t)CH * CF_OR * 2 <= (size_t)2 * CF_XW * TC_XR, "BF16 output tile fits the input tile");

// BF16 storage runs the 32 -> 32 channel convolutions on the tensor cores
template <class T> constexpr bool kTensorConv = false;
template <> constexpr bool kTensorConv<__nv_bfloat16> = true;

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// Position-major staging of one row's 32 channels, positions i0 - 4 + j for j < XW (zero
// outside [0, L)): xs[j][c] at a TC_XR-element pitch.  With L a multiple of 8 every channel row
// is read in 16-byte pieces along the positions (lane = channel, so the 2-byte shared stores of
// a warp fill 64 contiguous bytes); otherwise two channels per 32-bit word, element by element.
template <int XW>
__device__ __forceinline__ void stage_act_tile(const unsigned short* __restrict__ rows, int L, int i0,
                                               unsigned short* xs)
{
    static_assert(XW % 8 == 0 && XW * (CH / 2) % 32 == 0, "staging pieces tile the halo'd window");
    if ((L & 7) == 0) {
        // pieces v cover positions i0 - 8 + 8 v .. +7, v < XW / 8 + 1
        for (int e = threadIdx.x; e < CH * (XW / 8 + 1); e += blockDim.x) {
            const int c = e & (CH - 1), v = e / CH;
            const int pos0 = i0 - 8 + 8 * v;
            const unsigned short* src = rows + (size_t)c * L;
            unsigned short t[8];
            if (pos0 >= 0 && pos0 + 8 <= L) {
                const uint4 q = *reinterpret_cast<const uint4*>(src + pos0);
                const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    t[2 * k] = (unsigned short)(w[k] & 0xffffu);
                    t[2 * k + 1] = (unsigned short)(w[k] >> 16);
                }
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) t[k] = (pos0 + k >= 0 && pos0 + k < L) ? src[pos0 + k] : 0;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int j = 8 * v - HALF + k;
                if (j >= 0 && j < XW) xs[j * TC_XR + c] = t[k];
            }
        }
    } else {
        uint32_t* xw = reinterpret_cast<uint32_t*>(xs);
        for (int w = threadIdx.x; w < XW * (CH / 2); w += blockDim.x) {
            const int grp = w >> 5, l = w & 31;
            const int j = (grp >> 2) * 8 + (l & 7), cp = (grp & 3) * 4 + (l >> 3);
            const int pos = i0 - HALF + j;
            const size_t o = (size_t)(2 * cp) * L + pos;
            const bool inside = pos >= 0 && pos < L;
            const uint32_t v0 = inside ? rows[o] : 0u, v1 = inside ? rows[o + L] : 0u;
            xw[j * (TC_XR / 2) + cp] = v0 | (v1 << 16);
        }
    }
}

// The same tile from FP32 rows, split into BF16 hi and lo tiles (with L a multiple of 4, read
// in 16-byte pieces; positions i0 - 4 + 4 v .. +3, v < XW / 4).
template <int XW>
__device__ __forceinline__ void stage_split_tile(const float* __restrict__ rows, int L, int i0, unsigned short* xh,
                                                 unsigned short* xl)
{
    for (int e = threadIdx.x; e < CH * (XW / 4); e += blockDim.x) {
        const int c = e & (CH - 1), v = e / CH;
        const int pos0 = i0 - HALF + 4 * v;
        const float* src = rows + (size_t)c * L;
        float t[4];
        if ((L & 3) == 0 && pos0 >= 0 && pos0 + 4 <= L) {
            const float4 q = *reinterpret_cast<const float4*>(src + pos0);
            t[0] = q.x; t[1] = q.y; t[2] = q.z; t[3] = q.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) t[k] = (pos0 + k >= 0 && pos0 + k < L) ? src[pos0 + k] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
            uint32_t hi, lo;
            isr::split2<true>(t[k], t[k + 1], hi, lo);
            const int j = 4 * v + k;
            xh[j * TC_XR + c] = (unsigned short)(hi & 0xffffu);
            xh[(j + 1) * TC_XR + c] = (unsigned short)(hi >> 16);
            xl[j * TC_XR + c] = (unsigned short)(lo & 0xffffu);
            xl[(j + 1) * TC_XR + c] = (unsigned short)(lo >> 16);
        }
    }
}


// FWD: in = BF16 activations [B][32][L], out = BF16 relu(conv + bias).
// !FWD: in = FP32 gradient [B][32][L], out = FP32 conv masked by mask > 0 (BF16 activations
// of the layer below), no bias.
template <bool FWD>
__global__ void __launch_bounds__(CF_THREADS) conv_tc_kernel(const void* __restrict__ in, const __nv_bfloat16* __restrict__ wt,
                                                      const float* __restrict__ bias,
                                                      const __nv_bfloat16* __restrict__ mask, int L,
                                                      void* __restrict__ out)
{
    constexpr int NX = FWD ? 1 : 2;                    // staged input parts
    constexpr int XWORDS = CF_XW * TC_XR / 2;          // 32-bit words per staged part
    extern __shared__ __align__(16) unsigned char tc_smem[];
    uint32_t* xs = reinterpret_cast<uint32_t*>(tc_smem);
    uint4* ws = reinterpret_cast<uint4*>(tc_smem + (size_t)4 * NX * XWORDS);
    const int b = blockIdx.y, i0 = blockIdx.x * CF_CT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // weights: [co][288] rows, 16-byte copies into 592-byte rows
    const uint4* w4 = reinterpret_cast<const uint4*>(wt);
    for (int e = tid; e < CH * (TC_K / 8); e += CF_THREADS) {
        const int co = e / (TC_K / 8), q = e - co * (TC_K / 8);
        ws[co * (TC_WR / 8) + q] = w4[e];
    }
    // input: position-major tile of positions i0 - 4 + j (FP32 input: hi and lo tiles)
    if constexpr (FWD)
        stage_act_tile<CF_XW>(static_cast<const unsigned short*>(in) + (size_t)b * CH * L, L, i0,
                              reinterpret_cast<unsigned short*>(xs));
    else
        stage_split_tile<CF_XW>(static_cast<const float*>(in) + (size_t)b * CH * L, L, i0,
                                reinterpret_cast<unsigned short*>(xs), reinterpret_cast<unsigned short*>(xs + XWORDS));
    __syncthreads();

    float acc[2][4][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[mt][nt][q] = 0.f;
    const uint32_t xs_s = isr::smem_u32(xs), ws_s = isr::smem_u32(ws);
    const int r8 = lane & 7, mq = lane >> 3;
    // ldmatrix rows: weights, matrix mq = (rows +8 if mq odd, columns +8 if mq >= 2), giving
    // the A fragment registers in order; tile, matrix mq = (n-tile mq / 2, channels +8 if mq
    // odd), giving (b0, b1) of two n-tiles
    const uint32_t a_row = ws_s + 2u * (uint32_t)(((mq & 1) * 8 + r8) * TC_WR + (mq >> 1) * 8);
    const uint32_t b_row = xs_s + 2u * (uint32_t)((warp * 32 + (mq >> 1) * 8 + r8) * TC_XR + (mq & 1) * 8);
#pragma unroll 2
    for (int s = 0; s < TC_K / 16; ++s) {              // k-step s: tap s / 2, channels 16 (s % 2) ..
        const int tap = s >> 1, ci0 = (s & 1) * 16;
        uint32_t a[2][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) ldsm_x4(a[mt], a_row + 2u * (uint32_t)(mt * 16 * TC_WR + s * 16));
#pragma unroll
        for (int part = 0; part < NX; ++part) {
            uint32_t bq[2][4];
#pragma unroll
            for (int p = 0; p < 2; ++p)
                ldsm_x4(bq[p], b_row + 4u * (uint32_t)(part * XWORDS) + 2u * (uint32_t)((p * 16 + tap) * TC_XR + ci0));
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const uint4 af = make_uint4(a[mt][0], a[mt][1], a[mt][2], a[mt][3]);
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
                    isr::mma16816<true>(acc[mt][nt], af, bq[nt >> 1][(nt & 1) * 2], bq[nt >> 1][(nt & 1) * 2 + 1]);
            }
        }
    }
    __syncthreads();   // every warp is done with the tiles: the output tile reuses them

    // accumulator (mt, nt, q): channel mt 16 + g + 8 (q >= 2), position 32 warp + 8 nt + 2 t + (q & 1)
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int co = mt * 16 + h * 8 + g;
            const float bv = FWD ? __ldg(bias + co) : 0.f;
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                const int pl = warp * 32 + nt * 8 + 2 * t4;
                const float v0 = acc[mt][nt][2 * h] + bv, v1 = acc[mt][nt][2 * h + 1] + bv;
                if constexpr (FWD)
                    reinterpret_cast<uint32_t*>(tc_smem)[(co * CF_OR + pl) / 2] =
                        isr::pack2<true>(fmaxf(v0, 0.f), fmaxf(v1, 0.f));
                else
                    reinterpret_cast<float2*>(tc_smem)[(co * CF_OR + pl) / 2] = make_float2(v0, v1);
            }
        }
    __syncthreads();
    // coalesced rows: warp w writes channels w and w + 16
    for (int co = warp; co < CH; co += CF_THREADS / 32) {
        const size_t row = ((size_t)b * CH + co) * L;
        for (int q = lane; q < CF_CT; q += 32) {
            const int i = i0 + q;
            if (i >= L) break;
            if constexpr (FWD) {
                static_cast<__nv_bfloat16*>(out)[row + i] = reinterpret_cast<const __nv_bfloat16*>(tc_smem)[co * CF_OR + q];
            } else {
                const float v = reinterpret_cast<const float*>(tc_smem)[co * CF_OR + q];
                static_cast<float*>(out)[row + i] = __bfloat162float(mask[row + i]) > 0.f ? v : 0.f;
            }
        }
    }
}

// ---------------------------------------------------------------- tcgen05 operand staging
// Activations as operand planes of the tcgen05 weight gradient: a tile of 128 TPC positions (halo
// included) position-major in four planes of eight channels, [rows][8 ch] with 16-byte rows, so every
// 8 x 16-byte core matrix of the no-swizzle layout is eight consecutive rows of one plane, and tap k is
// the same tile started k rows later.
template <int TPC> struct C5 {
    static constexpr int CT = 128 * TPC;                   // positions per tile
    static constexpr int XW = CT + KT - 1;                 // staged rows (halo included)
    static constexpr int PLANE = XW * 16 + 16;             // bytes per channel plane (+16: planes 4 banks apart)
    static constexpr int PART = 4 * PLANE;                 // one staged part (32 channels)
    static_assert(PLANE % 16 == 0 && (PLANE / 4) % 32 == 4, "planes 16-byte aligned, four banks apart");
};

// 16-bit index of (row j, channel c) in a staged part of plane size PLANE bytes
template <int PLANE>
__device__ __forceinline__ int c5_idx(int j, int c) { return (c >> 3) * (PLANE / 2) + j * 8 + (c & 7); }

// Staging of one row's 32 channels, positions i0 - 4 + j for j < XW (zero outside [0, L)), into
// planes, in two phases so that a pipelined caller keeps the global loads in flight while it does
// other work: c5_act_load issues every global load of the thread into registers, c5_act_store
// writes them to the planes.  A warp takes pieces of eight positions, four neighbouring ones (lane >> 3)
// of eight channels (lane & 7): 64 bytes of a row at a time, since a load costs the L1 a cycle for every
// line that its lanes touch (one channel per lane: 32 lines).  When L is not a multiple of 8 the 16-byte
// loads do not apply: c5_act_load does nothing and c5_act_store stages word by word.  Called by NT threads.
template <int TPC, int NT> struct C5Act {
    static constexpr int NV = C5<TPC>::XW / 8 + 1;             // pieces of a row
    static constexpr int ROUNDS = CH / 8 * ((NV + 3) / 4);     // warp rounds: channel group fastest
    static constexpr int PER = (ROUNDS + NT / 32 - 1) / (NT / 32);
};

template <int TPC, int NT>
__device__ __forceinline__ void c5_act_load(const unsigned short* __restrict__ rows, int L, int i0,
                                            uint4 (&q)[C5Act<TPC, NT>::PER])
{
    if ((L & 7) != 0) return;
#pragma unroll
    for (int u = 0; u < C5Act<TPC, NT>::PER; ++u) {
        const int e = (threadIdx.x >> 5) + u * (NT / 32), lane = threadIdx.x & 31;
        const int c = 8 * (e & 3) + (lane & 7), v = 4 * (e >> 2) + (lane >> 3);
        const int pos0 = i0 - 8 + 8 * v;   // a multiple of 8 (i0 is): the piece lies inside [0, L) or outside
        q[u] = make_uint4(0u, 0u, 0u, 0u);
        if (v < C5Act<TPC, NT>::NV && pos0 >= 0 && pos0 + 8 <= L)
            q[u] = *reinterpret_cast<const uint4*>(rows + (size_t)c * L + pos0);
    }
}

template <int TPC, int NT>
__device__ __forceinline__ void c5_act_store(const unsigned short* __restrict__ rows, int L, int i0,
                                             const uint4 (&q)[C5Act<TPC, NT>::PER], unsigned short* xs)
{
    using G = C5<TPC>;
    constexpr int XW = G::XW, THREADS = NT, P = G::PLANE;
    static_assert(CH == 32, "four channel groups");
    if ((L & 7) == 0) {
        // lanes c, c ^ 1 swap halves of their 8 positions, so that the even lane holds positions 0-3 and
        // the odd lane positions 4-7 of both channels and writes one 32-bit word (channels c & ~1, c | 1)
        // per position.  Pieces v are 32 banks apart, so lanes of piece v start with position v & 3: the
        // four pieces, two halves and four channel pairs of a store fill 32 banks.
#pragma unroll
        for (int u = 0; u < C5Act<TPC, NT>::PER; ++u) {
            const int e = (threadIdx.x >> 5) + u * (NT / 32), lane = threadIdx.x & 31;
            if (e >= C5Act<TPC, NT>::ROUNDS) break;
            const int c = 8 * (e & 3) + (lane & 7), v = 4 * (e >> 2) + (lane >> 3), odd = c & 1, rot = v & 3;
            const uint32_t r0 = __shfl_xor_sync(0xffffffffu, odd ? q[u].x : q[u].z, 1);
            const uint32_t r1 = __shfl_xor_sync(0xffffffffu, odd ? q[u].y : q[u].w, 1);
            const uint32_t m0 = odd ? q[u].z : q[u].x, m1 = odd ? q[u].w : q[u].y;
            const uint32_t e0 = odd ? r0 : m0, o0 = odd ? m0 : r0;   // even / odd channel, positions 0-1 of the half
            const uint32_t e1 = odd ? r1 : m1, o1 = odd ? m1 : r1;   // positions 2-3
            const uint32_t w[4] = {__byte_perm(e0, o0, 0x5410), __byte_perm(e0, o0, 0x7632),
                                   __byte_perm(e1, o1, 0x5410), __byte_perm(e1, o1, 0x7632)};
            uint32_t x[4], y[4];   // y[k] = w[(k + rot) & 3]
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = rot & 1 ? w[(k + 1) & 3] : w[k];
#pragma unroll
            for (int k = 0; k < 4; ++k) y[k] = rot & 2 ? x[(k + 2) & 3] : x[k];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = 8 * v - HALF + 4 * odd + ((k + rot) & 3);
                if (j >= 0 && j < XW) *reinterpret_cast<uint32_t*>(xs + c5_idx<P>(j, c & ~1)) = y[k];
            }
        }
    } else {
        for (int e = threadIdx.x; e < XW * (CH / 2); e += THREADS) {
            const int j = e / (CH / 2), cp = e - j * (CH / 2);
            const int pos = i0 - HALF + j;
            const size_t o = (size_t)(2 * cp) * L + pos;
            const bool inside = pos >= 0 && pos < L;
            const uint32_t v0 = inside ? rows[o] : 0u, v1 = inside ? rows[o + L] : 0u;
            *reinterpret_cast<uint32_t*>(xs + c5_idx<P>(j, 2 * cp)) = v0 | (v1 << 16);
        }
    }
}

__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

__device__ __forceinline__ void ldsm_x2_trans(uint32_t (&r)[2], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(addr));
}

// Weight gradient of layers 2-4 with BF16 storage on the tensor cores:
//   dW[co][ci][k] = sum_{b,i} da[b][co][i] h[b][ci][i + k - 4],  db[co] = sum_{b,i} da[b][co][i],
// the GEMM D[co][kk] = sum_i A[co][i] B[i][kk] with kk = (k, ci), A = da (FP32, split into BF16
// hi + lo, both multiplied) and B[i][(k, ci)] = h[ci][i + k - 4].  B's 8 x 8 blocks are read
// transposed (ldmatrix.trans) from the position-major activation tile of the forward kernel,
// whose rows i + k start on 16-byte boundaries for every tap k.  CTA: `span` positions of one
// row in chunks of TC_CT; warp w: output channels 16 (w % 2) .., input channels 8 (w / 2) ..
// at all 9 taps; the CTA's partial dW and db are added with one atomic per element.  Four
// CTAs per SM (64 registers, 55 KB of shared memory each) hide the staging loads.
constexpr int WT_DR = TC_CT + 8;   // bf16 per staged gradient row (528 B)
constexpr size_t wgrad_tc_smem_bytes() { return (size_t)2 * (2 * CH * WT_DR + TC_XW * TC_XR); }

// Chunks per CTA for n rows of L positions with `slots` resident CTAs: the shortest span whose
// CTAs fit in one wave (else one CTA per row).  Every CTA ends with an atomic add to each of the
// same 9216 weights, so more, shorter CTAs contend there: at 128 rows x 4608 positions 2, 4 and 5
// chunks per CTA took 235, 195 and 157 us per launch.
int wgrad_span_chunks(int L, int n, int slots)
{
    const int cpr = (L + TC_CT - 1) / TC_CT;
    for (int k = 1; k <= cpr; ++k)
        if ((int64_t)n * ((cpr + k - 1) / k) <= slots) return k;
    return cpr;
}

__global__ void __launch_bounds__(256, 4) wgrad_tc_kernel(const __nv_bfloat16* __restrict__ h, const float* __restrict__ da,
                                                       int L, int span, float* __restrict__ dW,
                                                       float* __restrict__ db)
{
    extern __shared__ __align__(16) unsigned char wt_smem[];
    uint32_t* dah = reinterpret_cast<uint32_t*>(wt_smem);   // [CH][WT_DR / 2] words, hi parts
    uint32_t* dal = dah + CH * WT_DR / 2;                   // lo parts
    uint32_t* xs = dal + CH * WT_DR / 2;                    // [TC_XW][TC_XR / 2] words
    __shared__ float db_s[CH];
    const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < CH) db_s[tid] = 0.f;
    const int mt = warp & 1, ci0 = (warp >> 1) * 8;
    const int r8 = lane & 7, mq = lane >> 3;
    const uint32_t a_hi = isr::smem_u32(dah) + 2u * (uint32_t)((mt * 16 + (mq & 1) * 8 + r8) * WT_DR + (mq >> 1) * 8);
    const uint32_t a_lo = a_hi + 2u * (uint32_t)(CH * WT_DR);
    // transposed B blocks: matrix mq = (positions +8 if mq odd, tap +1 if mq >= 2)
    const uint32_t b_row = isr::smem_u32(xs) + 2u * (uint32_t)(((mq >> 1) + (mq & 1) * 8 + r8) * TC_XR + ci0);
    float acc[KT][4];
#pragma unroll
    for (int k = 0; k < KT; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[k][q] = 0.f;
    const int span_end = min(L, (int)(blockIdx.x + 1) * span);
    for (int p0 = blockIdx.x * span; p0 < span_end; p0 += TC_CT) {
        __syncthreads();   // the previous chunk's tiles are consumed (and db_s is initialised)
        // gradient: word (co, pp) = positions p0 + 2 pp, +1 of channel co (zero past the span);
        // the 32 lanes of a warp share co, so the bias gradient reduces per warp first
        for (int e = tid; e < CH * TC_CT / 2; e += 256) {
            const int co = e / (TC_CT / 2), pp = e - co * (TC_CT / 2);
            const int pos = p0 + 2 * pp;
            const float* src = da + ((size_t)b * CH + co) * L;
            const float v0 = pos < span_end ? src[pos] : 0.f;
            const float v1 = pos + 1 < span_end ? src[pos + 1] : 0.f;
            uint32_t hi, lo;
            isr::split2<true>(v0, v1, hi, lo);
            dah[co * (WT_DR / 2) + pp] = hi;
            dal[co * (WT_DR / 2) + pp] = lo;
            float s = v0 + v1;
            for (int o = 16; o; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) atomicAdd(&db_s[co], s);
        }
        // activations: position-major tile of positions p0 - 4 + j (zero outside the row)
        stage_act_tile<TC_XW>(reinterpret_cast<const unsigned short*>(h) + (size_t)b * CH * L, L, p0,
                              reinterpret_cast<unsigned short*>(xs));
        __syncthreads();
#pragma unroll 2
        for (int s = 0; s < TC_CT / 16; ++s) {   // k-step: positions p0 + 16 s ..
            uint32_t ah[4], al[4];
            ldsm_x4(ah, a_hi + 2u * (uint32_t)(16 * s));
            ldsm_x4(al, a_lo + 2u * (uint32_t)(16 * s));
            const uint4 fh = make_uint4(ah[0], ah[1], ah[2], ah[3]), fl = make_uint4(al[0], al[1], al[2], al[3]);
#pragma unroll
            for (int tp = 0; tp < KT - 1; tp += 2) {
                uint32_t bq[4];
                ldsm_x4_trans(bq, b_row + 2u * (uint32_t)((16 * s + tp) * TC_XR));
                isr::mma16816<true>(acc[tp], fh, bq[0], bq[1]);
                isr::mma16816<true>(acc[tp], fl, bq[0], bq[1]);
                isr::mma16816<true>(acc[tp + 1], fh, bq[2], bq[3]);
                isr::mma16816<true>(acc[tp + 1], fl, bq[2], bq[3]);
            }
            uint32_t b8[2];   // tap 8: matrices 0 and 1 only (lanes 0-15 give the rows)
            ldsm_x2_trans(b8, b_row + 2u * (uint32_t)((16 * s + KT - 1 - (mq >> 1)) * TC_XR));
            isr::mma16816<true>(acc[KT - 1], fh, b8[0], b8[1]);
            isr::mma16816<true>(acc[KT - 1], fl, b8[0], b8[1]);
        }
    }
    // accumulator (k, q): output channel 16 mt + g + 8 (q >= 2), input channel ci0 + 2 t + (q & 1)
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int k = 0; k < KT; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int co = mt * 16 + g + (q >> 1) * 8, ci = ci0 + 2 * t4 + (q & 1);
            atomicAdd(&dW[((size_t)co * CH + ci) * KT + k], acc[k][q]);
        }
    __syncthreads();
    if (tid < CH) atomicAdd(&db[tid], db_s[tid]);
}

// Weight gradient of layers 2-4 on tcgen05 (ISR_EST_BF16):
//   dW[co][ci][k] = sum_p da[co][p] h[ci][p + k - 4]   over the CTA's chunks,
// as D_g[(k, i)][n] = sum_p A_g[(k, i)][p] B[n][p] with K = positions (16 per MMA): A_g = the
// activation planes of channel group g (8 channels per 16-byte row, positions as rows) as an
// MN-major operand whose 8-row M-groups are 16 bytes apart, so M-group k reads channels 8 g + i at
// position p + k, i.e. tap k (groups 9-15 are padding); B = the gradient's BF16 hi parts (rows
// 0-31) and lo parts (rows 32-63; their sum keeps ~16 bits of the FP32 gradient), K-major 8 x 8
// blocks staged from the channel-major rows; N = 64, M = 128, TMEM columns 64 g, 256 a set.  In
// the no-swizzle layouts of both majors the descriptor's leading-byte offset steps along K and its
// stride-byte offset along M or N.  Four 128 x 64 x 16 MMAs per K-step (64 per chunk) read 6 KB of
// shared memory each: 384 KB per chunk, where 32-column MMAs per tap needed 144 MMAs and 720 KB,
// which the tensor pipe could not stream while the CTA staged the next chunk.  Chunks of 256
// positions are double-buffered; 16 warps stage (and run the epilogue), one more issues the MMAs;
// the CTAs are dealt to the three layers in turn and a layer's n_rows x ceil(L / 256) chunks, row after
// row, split into contiguous ranges of equal length (+-1) over its CTAs, so a CTA's range may cross
// from one row into the next: the sum over positions and rows does not care.  One CTA per SM.
// The accumulators drop low bits at every MMA, an error that grows with the MMAs behind a sum, so a sum
// is taken over to shared memory after as many chunks as a launch of one layer on all SMs would give it,
// while the next ones go to the other of two sets of accumulators.
// At 128 rows x 4608 positions the three layers take 132 us in this one launch (46 chunks a CTA); a
// launch per layer over all SMs, with one channel per lane in the loads, took 3 x 51.  The MMAs alone
// would take about 115 us (75 cycles each: A's core matrices start off the 128-byte lines), the staging
// alone 104, the loads alone 71; without drains it is 126.  Loads one chunk further ahead (+4 us:
// registers) and M = 64 with tap 8 as a fifth product, for no padding rows (+19 us: as many cycles per
// MMA), gave nothing.
// one arrival (release semantics at CTA scope) on the barrier's current phase
// Bounded waits of the tcgen05 kernels on their products.  One that runs out ends the work of its threads:
// they note it, wait once more for what is in flight (with the same bound) and give the tensor memory back;
// the host reports it.
struct EstWait {
    unsigned limit;   // polls
    int* status;      // device word
    int* host;        // pinned host word
};
__device__ __forceinline__ void est_timed_out(const EstWait& w)
{
    atomicOr(w.status, 1);
    *static_cast<volatile int*>(w.host) = 1;
    __threadfence_system();
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

constexpr int W5_CHUNK = 256;                    // positions per chunk (16 K-steps)
constexpr int W5_THREADS = 512;                  // staging (and epilogue) threads
constexpr int W5_BLOCK = W5_THREADS + 32;        // + one warp that issues the MMAs
constexpr int W5_ASBO = W5_CHUNK / 8 * 128;      // bytes per 8-row group of the gradient (all its blocks)
constexpr int W5_ABUF = 8 * W5_ASBO;             // one gradient buffer: 8 row groups (hi 0-3, lo 4-7)
constexpr int W5_LAYERS = 3;                     // layers 2-4, one launch
struct W5Args {
    const __nv_bfloat16* h[W5_LAYERS];
    const float* da[W5_LAYERS];
    float *dW[W5_LAYERS], *db[W5_LAYERS];
    int L, n_rows, drain;   // chunks between drains of the accumulators
    EstWait wait;
};
using W5X = C5<2>;                               // activation tile: 256 + 8 rows, 4 planes
static_assert(W5X::CT == W5_CHUNK, "activation tile matches the chunk");
constexpr int W5_ROWS = 8 * KT;                  // real rows of an accumulator
constexpr int W5_SUM = 4 * CH * W5_ROWS * 4;     // bytes of the drained sums, [channel group][co][row]
constexpr size_t w5_smem_bytes() { return (size_t)2 * W5_ABUF + 2 * W5X::PART + 64 + W5_SUM; }
// dynamic shared memory requested at launch: more than half an SM's, so that one CTA has the SM to
// itself (its 544 threads need the register file)
constexpr size_t W5_SMEM_LAUNCH = 144 * 1024;
constexpr int W5_DCOLS = 4 * 2 * CH;             // D_g of the four channel groups
constexpr int W5_TMEM_COLS = 2 * W5_DCOLS;       // two sets of them
static_assert(w5_smem_bytes() <= W5_SMEM_LAUNCH, "launch request covers the layout");
// the padding M-groups (taps 9-15) of the last plane of the second buffer read up to 4336 bytes
// from that plane's start: still inside the launch allocation
static_assert((size_t)2 * W5_ABUF + W5X::PART + 3 * W5X::PLANE + (W5_CHUNK - 16) * 16 + 15 * 16 + 256 <= W5_SMEM_LAUNCH,
              "A's padding rows stay in shared memory");
// ... and the 9 real taps stay inside their plane (rows < XW)
static_assert((W5_CHUNK - 16) + 15 + (KT - 1) < W5X::XW, "real taps read staged rows only");

template <bool DROP>
__global__ void __launch_bounds__(W5_BLOCK, 1) wgrad_tc05_kernel(const __grid_constant__ W5Args args)
{
    // CTAs are dealt to the layers in turn
    const int layer = blockIdx.x % W5_LAYERS, part = blockIdx.x / W5_LAYERS;
    const int parts = (gridDim.x - layer + W5_LAYERS - 1) / W5_LAYERS;
    const __nv_bfloat16* __restrict__ h = args.h[layer];
    const float* __restrict__ da = args.da[layer];
    float* __restrict__ dW = args.dW[layer];
    float* __restrict__ db = args.db[layer];
    const int L = args.L, n_rows = args.n_rows;
    extern __shared__ __align__(128) unsigned char w5_smem[];
    unsigned char* abuf = w5_smem;                                  // [2][8 row groups][W5_ASBO]
    unsigned char* xbuf = w5_smem + 2 * W5_ABUF;                    // [2][W5X::PART]
    // mbar[b]: the MMAs of the chunk in buffer b completed (one commit); full[b]: buffer b staged
    // (one arrival per staging warp)
    uint64_t* mbar = reinterpret_cast<uint64_t*>(w5_smem + 2 * W5_ABUF + 2 * W5X::PART);   // [2]
    uint64_t* full = mbar + 2;                                                              // [2]
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 4);
    uint64_t* drained = mbar + 5;   // everything issued completed, where a wait ran out
    float* sum = reinterpret_cast<float*>(mbar + 8);
    __shared__ float db_s[CH];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cpr = (L + W5_CHUNK - 1) / W5_CHUNK;                 // chunks per row
    const int64_t total = (int64_t)n_rows * cpr;
    const int q_begin = (int)(part * total / parts);
    const int nch = (int)((part + 1) * total / parts) - q_begin;
    if (tid < CH) db_s[tid] = 0.f;
    if (tid == 0) {
        isr::mbar_init(isr::smem_u32(&mbar[0]), 1);
        isr::mbar_init(isr::smem_u32(&mbar[1]), 1);
        isr::mbar_init(isr::smem_u32(drained), 1);
        isr::mbar_init(isr::smem_u32(&full[0]), W5_THREADS / 32);
        isr::mbar_init(isr::smem_u32(&full[1]), W5_THREADS / 32);
    }
    if (warp == 0) isr::tmem_alloc(isr::smem_u32(tslot), W5_TMEM_COLS);

    // stage chunk c into buffer c & 1: da as hi / lo 8 x 8 blocks, the activations as planes; in
    // two phases, all global loads of the chunk (gradient and activations) into registers first,
    // then the shared stores.  A warp's gradient items are four 8-position blocks (lane >> 3) of eight
    // channels (lane & 7): 128 bytes of a row at a time, and the eight lanes of a 16-byte store phase
    // write one 128-byte core matrix.
    constexpr int PER = CH * (W5_CHUNK / 8) / W5_THREADS, KSTEP = W5_THREADS / CH;
    static_assert(CH == 32 && W5_CHUNK / 8 == KSTEP * PER, "warp = channel group and four blocks");
    const int co = 8 * (warp & 3) + (lane & 7), kb0 = 4 * ((warp >> 2) & 3) + (lane >> 3);
    struct Regs {
        float4 q0[PER], q1[PER];
        uint4 qa[C5Act<2, W5_THREADS>::PER];
    };
    float dbacc = 0.f;   // bias gradient of channel co
    auto load = [&](int c, Regs& v) {
        const int q = q_begin + c, b = q / cpr, p0 = (q - b * cpr) * W5_CHUNK;
        const int span_end = min(L, p0 + W5_CHUNK);
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int pos = p0 + 8 * (kb0 + KSTEP * u);
            const float* src = da + ((size_t)b * CH + co) * L + pos;
            if ((L & 3) == 0 && pos + 8 <= span_end) {
                v.q0[u] = *reinterpret_cast<const float4*>(src);
                v.q1[u] = *reinterpret_cast<const float4*>(src + 4);
            } else {
                float t[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) t[k] = pos + k < span_end ? src[k] : 0.f;
                v.q0[u] = make_float4(t[0], t[1], t[2], t[3]);
                v.q1[u] = make_float4(t[4], t[5], t[6], t[7]);
            }
        }
        c5_act_load<2, W5_THREADS>(reinterpret_cast<const unsigned short*>(h) + (size_t)b * CH * L, L, p0, v.qa);
    };
    auto store = [&](int c, const Regs& v) {
        const int q = q_begin + c, b = q / cpr, p0 = (q - b * cpr) * W5_CHUNK;
        unsigned char* a = abuf + (c & 1) * W5_ABUF;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const float t[8] = {v.q0[u].x, v.q0[u].y, v.q0[u].z, v.q0[u].w, v.q1[u].x, v.q1[u].y, v.q1[u].z, v.q1[u].w};
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) isr::split2<true>(t[2 * k], t[2 * k + 1], hi[k], lo[k]);
            const uint32_t o = (uint32_t)((co >> 3) * W5_ASBO + (kb0 + KSTEP * u) * 128 + (co & 7) * 16);
            *reinterpret_cast<uint4*>(a + o) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(a + o + 4 * W5_ASBO) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            dbacc += ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
        }
        c5_act_store<2, W5_THREADS>(reinterpret_cast<const unsigned short*>(h) + (size_t)b * CH * L, L, p0, v.qa,
                                    reinterpret_cast<unsigned short*>(xbuf + (c & 1) * W5X::PART));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    };

    isr::fence_barrier_init();
    isr::tmem_fence_before_sync();
    __syncthreads();
    isr::tmem_fence_after_sync();
    const uint32_t tbase = *tslot;
    bool ok = true;
    // D_g (columns 64 g ..) row 8 t + i (TMEM lane) = tap t, input channel 8 g + i; columns 0-31 the hi and
    // 32-63 the lo part of output channel o.  Warp w reads lane quarter w % 4 (taps 4 (w % 4) ..) of channel
    // group g = w / 4; taps 9-15 are padding.  out(o, value) with the sums drained before if there are any.
    static_assert(W5_THREADS == 512, "sixteen epilogue warps: four lane quarters x four channel groups");
    const int quarter = warp & 3, g4 = warp >> 2, row = 32 * quarter + lane;
    float* sum_row = sum + (size_t)g4 * CH * W5_ROWS + row;
    int seg = 0;   // segments drained
    auto take = [&](auto out) {
        if (quarter == 3) return;
        const bool more = seg > 0;
        const uint32_t d = isr::tmem_warp_lane_base(tbase) + (uint32_t)(W5_DCOLS * (seg & 1) + 2 * CH * g4);
        uint32_t rh[32], rl[32];
        isr::tmem_ld32(d, rh);
        isr::tmem_ld32(d + CH, rl);
        isr::tmem_wait_ld32(rh);
        isr::tmem_wait_ld32(rl);
        if (row < W5_ROWS) {
#pragma unroll
            for (int o = 0; o < CH; ++o) {
                const float x = __uint_as_float(rh[o]) + __uint_as_float(rl[o]);
                out(o, more ? sum_row[o * W5_ROWS] + x : x);
            }
        }
    };
    auto drain = [&]() {
        isr::tmem_fence_after_sync();
        take([&](int o, float d) { sum_row[o * W5_ROWS] = d; });
        isr::tmem_fence_before_sync();
        ++seg;
    };
    if (warp < W5_THREADS / 32) {
        // staging warps: chunk c goes into buffer c & 1 once chunk c - 2's MMAs, which read that buffer,
        // have completed; each warp then arrives on full[c & 1]
        Regs v;
        int left = args.drain + 1;
        for (int c = 0; c < nch; ++c) {
            if (left-- == 0) {   // chunk c - 2 ended a segment: drain it under the next one's MMAs
                ok = isr::mbar_wait(isr::smem_u32(&mbar[c & 1]), (uint32_t)((c - 2) >> 1) & 1u, args.wait.limit);
                if (!ok) break;
                drain();
                left = args.drain - 1;
            }
            load(c, v);
            if (c >= 2 && !isr::mbar_wait(isr::smem_u32(&mbar[c & 1]), (uint32_t)((c - 2) >> 1) & 1u, args.wait.limit)) {
                ok = false;
                break;
            }
            store(c, v);
            __syncwarp();
            if (lane == 0) mbar_arrive(isr::smem_u32(&full[c & 1]));
        }
    } else if (lane == 0) {
        // the issuing warp: a tcgen05.mma issue holds its thread until the tensor pipe takes it,
        // so this thread does nothing else.  A = the activation planes, MN-major (bit 15): LBO =
        // 128 B along K (8 positions), SBO = 16 B along M, so M-group j (rows 8 j ..) is channel
        // group g started j rows later, i.e. tap j; B = the gradient's hi / lo rows, K-major: LBO =
        // 128 B along K, SBO = W5_ASBO along N (8 rows).  N = 64, M = 128 (M-groups 9-15 unused).
        constexpr uint32_t idesc =
            (isr::tc05_idesc<true>() & ~(0x3Fu << 17)) | ((uint32_t)(2 * CH >> 3) << 17) | (1u << 15);
        int left = 0;
        uint32_t set = tbase + W5_DCOLS;
        for (int c = 0; c < nch; ++c, --left) {
            const bool anew = left == 0;
            if (anew) {
                left = args.drain;
                set = tbase + (set == tbase ? W5_DCOLS : 0);
            }
            if (!isr::mbar_wait(isr::smem_u32(&full[c & 1]), (uint32_t)(c >> 1) & 1u, args.wait.limit)) {
                ok = false;
                break;
            }
            if constexpr (DROP) continue;
            isr::tmem_fence_after_sync();
            // descriptors built once per chunk; K-step s adds two blocks of eight positions to the
            // 16-byte-unit start fields (addresses stay below 0x40000 B: the field never carries)
            const uint64_t bd0 = isr::tc05_desc(isr::smem_u32(abuf + (c & 1) * W5_ABUF), 128, W5_ASBO);
            const uint32_t xa = isr::smem_u32(xbuf + (c & 1) * W5X::PART);
            uint64_t ad0[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) ad0[g] = isr::tc05_desc(xa + g * W5X::PLANE, 128, 16);
#pragma unroll 1
            for (int s = 0; s < W5_CHUNK / 16; ++s) {
                const uint32_t acc = !anew || s > 0 ? 1u : 0u;
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    isr::tc05_mma(set + (uint32_t)(2 * CH * g), ad0[g] + 16u * (uint32_t)s, bd0 + 16u * (uint32_t)s,
                                  idesc, acc);
            }
            isr::tc05_commit(isr::smem_u32(&mbar[c & 1]));
        }
        if (!ok) {
            isr::tc05_commit(isr::smem_u32(drained));
            isr::mbar_wait(isr::smem_u32(drained), 0u, args.wait.limit);
        }
    }
    if (warp < W5_THREADS / 32) {   // the four lanes of a channel
        for (int o = 8; o < 32; o <<= 1) dbacc += __shfl_xor_sync(0xffffffffu, dbacc, o);
        if (lane < 8) atomicAdd(&db_s[co], dbacc);
    }
    // the last commit covers every MMA of this CTA; a thread whose wait ran out skips it
    if (nch > 0 && ok) ok = isr::mbar_wait(isr::smem_u32(&mbar[(nch - 1) & 1]), (uint32_t)((nch - 1) >> 1) & 1u, args.wait.limit);
    isr::tmem_fence_before_sync();
    ok = __syncthreads_and(ok) != 0;
    isr::tmem_fence_after_sync();
    if (!ok && tid == 0) est_timed_out(args.wait);
    if (ok && warp < W5_THREADS / 32) {
        while ((seg + 1) * args.drain < nch) drain();   // the segment before the last may end one chunk earlier
        take([&](int o, float d) {
            atomicAdd(&dW[((size_t)o * CH + 8 * g4 + (lane & 7)) * KT + (row >> 3)], d);
        });
    }
    isr::tmem_fence_before_sync();
    __syncthreads();
    isr::tmem_fence_after_sync();
    if (warp == 0) isr::tmem_dealloc(tbase, W5_TMEM_COLS);
    if (tid < CH) atomicAdd(&db[tid], db_s[tid]);
}

// dW[co][ci][k] += sum_i da[b][co][i] h[b][ci][i + k - 4];  db[co] += sum_i da[b][co][i]
// CTA: one row b, positions [i0, i0 + span); lane = co, warp = four input channels.  Bound by shared
// loads and FMAs: the activations are the same for all lanes, so they come 16 bytes at a time (16 loads
// per 144 FMAs instead of 52).  The span shrinks until the launch has about four CTAs per SM: with one of
// 1152 positions per row, 37 rows of 1101 left three quarters of the SMs idle (121 -> 32 us, 26-29 with tiles of 96).  The sums
// go out through shared memory so that the atomics of a warp fall on runs of 18 addresses instead of 32
// sectors.  The CTAs add to WG_COPIES copies of the gradient in turn, which wgrad_sum_kernel adds up: in
// one copy each of the 444 additions rounds at the size of the whole sum, which leaves a layer's gradient a
// relative RMS error of 3e-7 to 4e-7 (one span per row 1e-7 to 2e-7, the copies 3e-8 to 4e-8; the sums of
// such a batch formed in these orders).  The whole gradient is within 1.5e-7 of FP64 (one copy 3.3e-7), and
// the pass no slower (37 rows of 1101: 309 -> 304 us).
constexpr int WG_MAX_SPAN = 1152;
constexpr int WG_COPIES = 16;
constexpr int WG_SIZE = OFF_W5 - OFF_W2;   // floats of a copy: weights and biases of layers 2 to 4

inline int wgrad_span(int L, int n, int sms, int ct)
{
    int span = WG_MAX_SPAN;
    while (span > ct && (int64_t)n * ((L + span - 1) / span) < 4 * (int64_t)sms) span -= ct;
    return span;
}

// Positions of a tile, 128 or 96: the one whose fullest SM has least to do, a CTA's staging and atomics
// counted as 32 positions (37 rows of 1101 positions: 444 CTAs of 96 make three on every SM, 333 of 128
// three on some and two on most: 26-29 us, 32).
inline int wgrad_tile(int L, int n, int sms)
{
    auto cost = [&](int ct) {
        const int span = wgrad_span(L, n, sms, ct);
        return ((int64_t)n * ((L + span - 1) / span) + sms - 1) / sms * (span + 32);
    };
    return cost(96) < cost(128) ? 96 : 128;
}

// dW, db: the layer's gradients in the first copy
template <class TH, int CT>
__global__ void __launch_bounds__(256) wgrad_kernel(const TH* __restrict__ h, const float* __restrict__ da, int L, int span,
                                                    float* __restrict__ dW, float* __restrict__ db)
{
    const size_t copy = (blockIdx.y * gridDim.x + blockIdx.x) % WG_COPIES;
    dW += copy * WG_SIZE;
    db += copy * WG_SIZE;
    constexpr int CPW = CH / 8, HW = CT + KT - 1, RUN = CPW / 2 * KT;
    static_assert(HW % 4 == 0 && WG_MAX_SPAN % CT == 0, "aligned window rows, whole tiles");
    __shared__ __align__(16) float sm[CT * (CH + 1) + CH * HW];
    static_assert(8 * CH * RUN <= CT * (CH + 1) + CH * HW, "output staging");
    float* das = sm;                    // [CT][CH + 1]
    float* hs = sm + CT * (CH + 1);     // [CH][HW]
    static_assert(CT * (CH + 1) % 4 == 0, "16-byte rows");
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float acc[CPW][KT];
#pragma unroll
    for (int c = 0; c < CPW; ++c)
#pragma unroll
        for (int k = 0; k < KT; ++k) acc[c][k] = 0.f;
    float dbacc = 0.f;
    const int span_end = min(L, (int)(blockIdx.x + 1) * span);
    for (int i0 = blockIdx.x * span; i0 < span_end; i0 += CT) {
        __syncthreads();
        for (int e = threadIdx.x; e < CT * CH; e += 256) {
            const int co = e / CT, j = e % CT, pos = i0 + j;
            das[j * (CH + 1) + co] = pos < span_end ? da[((size_t)b * CH + co) * L + pos] : 0.f;
        }
        for (int e = threadIdx.x; e < CH * HW; e += 256) {
            const int ci = e / HW, j = e % HW, pos = i0 + j - HALF;
            hs[e] = (pos >= 0 && pos < L) ? ld<TH>(h, ((size_t)b * CH + ci) * L + pos) : 0.f;
        }
        __syncthreads();
        for (int j = 0; j < CT; j += 4) {
            float d[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) d[q] = das[(j + q) * (CH + 1) + lane];
            if (warp == 0) dbacc += d[0] + d[1] + d[2] + d[3];
#pragma unroll
            for (int c = 0; c < CPW; ++c) {
                const float* hr = hs + (warp * CPW + c) * HW + j;
                float hv[4 + KT - 1];
#pragma unroll
                for (int q = 0; q < 4 + KT - 1; q += 4)
                    *reinterpret_cast<float4*>(hv + q) = *reinterpret_cast<const float4*>(hr + q);
#pragma unroll
                for (int k = 0; k < KT; ++k)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[c][k] = fmaf(d[q], hv[q + k], acc[c][k]);
            }
        }
    }
    if (warp == 0) atomicAdd(&db[lane], dbacc);
    float* st = sm + warp * CH * RUN;   // [co][two channels x 9 taps]
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        if (half == 0) __syncthreads();
        else __syncwarp();
#pragma unroll
        for (int r = 0; r < RUN; ++r) st[lane * RUN + r] = acc[half * (CPW / 2) + r / KT][r % KT];
        __syncwarp();
        for (int e = lane; e < CH * RUN; e += 32)
            atomicAdd(&dW[(size_t)(e / RUN) * CH * KT + (warp * CPW + half * (CPW / 2)) * KT + e % RUN], st[e]);
    }
}

// grad[i] = sum over the copies, in FP64 (under half a million additions)
__global__ void __launch_bounds__(256) wgrad_sum_kernel(const float* __restrict__ copies, float* __restrict__ grad)
{
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= WG_SIZE) return;
    float v[WG_COPIES];
#pragma unroll
    for (int c = 0; c < WG_COPIES; ++c) v[c] = copies[(size_t)c * WG_SIZE + i];
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < WG_COPIES; ++c) s += (double)v[c];
    grad[i] = (float)s;
}

// Weight gradient of the one-channel first layer:
//   dW1[co][k] += sum_i da[b][co][i] x[b][i + k - 4],  db1[co] += sum_i da[b][co][i]
// The n_rows x ceil(L / W1_SPAN) spans, row after row, are split into gridDim.x contiguous ranges
// (two CTAs per SM), and a CTA keeps its sums in registers over its spans.  Lane l is output
// channel l, so a thread holds only that channel's nine tap sums and its bias sum and the
// registers go to loads in flight.  Spans are short (512 positions) so that CTAs get near-equal
// numbers of them.  Within a span [i0, i0 + W1_SPAN) of row b warp w takes the positions
// i0 + 64 w .. i0 + 64 w + 63 in rounds of eight steps of 8 positions: per step a
// lane reads 8 consecutive positions of its channel's gradient row (two 16-byte loads; a round's
// loads are all issued before the first is used) and the 16 inputs x[p - 4 .. p + 11] as four
// 16-byte broadcast reads of the span's input row in shared memory.  At the end the eight warps'
// sums of each channel are added in shared memory and every weight receives one atomic per CTA.
constexpr int W1_SPAN = 512;
constexpr int W1_STEP = 8;                              // positions per lane and step
constexpr int W1_U = 8;                                 // steps per round (their loads in flight)
constexpr int W1_WSPAN = W1_SPAN / 8;                   // positions per warp and span
static_assert(W1_WSPAN % (W1_STEP * W1_U) == 0, "whole rounds per warp and span");

template <class TH>
__global__ void __launch_bounds__(256, 2) wgrad1_kernel(const TH* __restrict__ x, const float* __restrict__ da, int L,
                                                        int n_rows, float* __restrict__ dW, float* __restrict__ db)
{
    __shared__ __align__(16) float xs[W1_SPAN + 16];    // xs[j] = x[b][i0 - 4 + j]
    __shared__ float red[8][CH * (KT + 1)];             // the warps' sums: [warp][channel][tap, bias]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int spr = (L + W1_SPAN - 1) / W1_SPAN;                 // spans per row
    const int64_t total = (int64_t)n_rows * spr;
    const int q_begin = (int)((int64_t)blockIdx.x * total / gridDim.x);
    const int q_end = (int)((int64_t)(blockIdx.x + 1) * total / gridDim.x);
    float acc[KT], dbacc = 0.f;
#pragma unroll
    for (int k = 0; k < KT; ++k) acc[k] = 0.f;
    const bool vec = (L & 3) == 0;   // 16-byte gradient loads (8-position pieces start at multiples of 8)
    for (int q = q_begin; q < q_end; ++q) {
        const int b = q / spr, i0 = (q - b * spr) * W1_SPAN, iend = min(L, i0 + W1_SPAN);
        __syncthreads();   // the previous span's reads of xs are done
        for (int j = threadIdx.x; j < W1_SPAN + 16; j += 256) {
            const int pos = i0 - HALF + j;
            xs[j] = (pos >= 0 && pos < L) ? ld<TH>(x, (size_t)b * L + pos) : 0.f;
        }
        __syncthreads();
        const float* dar = da + ((size_t)b * CH + lane) * L;
#pragma unroll 1
        for (int r = 0; r < W1_WSPAN / (W1_STEP * W1_U); ++r) {
            const int pbase = i0 + warp * W1_WSPAN + r * W1_STEP * W1_U;
            float d[W1_U][W1_STEP];
#pragma unroll
            for (int u = 0; u < W1_U; ++u) {
                const int p = pbase + W1_STEP * u;
                if (vec && p + W1_STEP <= iend) {
                    const float4 a0 = __ldg(reinterpret_cast<const float4*>(dar + p));
                    const float4 a1 = __ldg(reinterpret_cast<const float4*>(dar + p + 4));
                    d[u][0] = a0.x; d[u][1] = a0.y; d[u][2] = a0.z; d[u][3] = a0.w;
                    d[u][4] = a1.x; d[u][5] = a1.y; d[u][6] = a1.z; d[u][7] = a1.w;
                } else {
#pragma unroll
                    for (int t = 0; t < W1_STEP; ++t) d[u][t] = p + t < iend ? __ldg(dar + p + t) : 0.f;
                }
            }
#pragma unroll
            for (int u = 0; u < W1_U; ++u) {
                const int j = pbase + W1_STEP * u - i0;   // zero gradient past iend: no effect
                const float4* x4 = reinterpret_cast<const float4*>(&xs[j]);
                float xw[16];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const float4 t4 = x4[v];
                    xw[4 * v] = t4.x; xw[4 * v + 1] = t4.y; xw[4 * v + 2] = t4.z; xw[4 * v + 3] = t4.w;
                }
#pragma unroll
                for (int t = 0; t < W1_STEP; ++t) {
                    const float dv = d[u][t];
                    dbacc += dv;
#pragma unroll
                    for (int k = 0; k < KT; ++k) acc[k] = fmaf(dv, xw[t + k], acc[k]);
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < KT; ++k) red[warp][lane * (KT + 1) + k] = acc[k];
    red[warp][lane * (KT + 1) + KT] = dbacc;
    __syncthreads();
    for (int e = threadIdx.x; e < CH * (KT + 1); e += 256) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += red[w][e];
        const int co = e / (KT + 1), k = e - co * (KT + 1);
        atomicAdd(k < KT ? &dW[co * KT + k] : &db[co], t);
    }
}

// ---------------------------------------------------------------- first layer (one input channel)
// h1[b][co][i] = relu(b1[co] + sum_k W1[co][k] x[b][i + k - 4]).  A thread takes two adjacent
// positions and loops over the channels, so every channel row is written in coalesced pairs.
constexpr int L1_CT = 512;   // positions per CTA

template <class T> __device__ __forceinline__ void store_pair(T* o, float a, float b);
template <> __device__ __forceinline__ void store_pair<float>(float* o, float a, float b)
{
    *reinterpret_cast<float2*>(o) = make_float2(a, b);
}
template <> __device__ __forceinline__ void store_pair<__nv_bfloat16>(__nv_bfloat16* o, float a, float b)
{
    *reinterpret_cast<__nv_bfloat162*>(o) = __floats2bfloat162_rn(a, b);
}
template <class T>
__global__ void __launch_bounds__(256) conv1_kernel(const T* __restrict__ x, const T* __restrict__ w1,
                                                    const float* __restrict__ b1, int L, T* __restrict__ out)
{
    __shared__ float xs[L1_CT + KT - 1];
    __shared__ __align__(16) float ws[CH][12];   // W1[co][0..8], b1[co], 0, 0
    const int b = blockIdx.y, i0 = blockIdx.x * L1_CT;
    const T* xb = x + (size_t)b * L;
    for (int j = threadIdx.x; j < L1_CT + KT - 1; j += 256) {
        const int pos = i0 - HALF + j;
        xs[j] = (pos >= 0 && pos < L) ? ld<T>(xb, pos) : 0.f;
    }
    for (int e = threadIdx.x; e < CH * 12; e += 256) {
        const int co = e / 12, k = e - co * 12;
        ws[co][k] = k < KT ? ld<T>(w1, (size_t)k * CH + co) : (k == KT ? b1[co] : 0.f);   // w1: [k][co]
    }
    __syncthreads();
    const int p = 2 * threadIdx.x, i = i0 + p;
    if (i >= L) return;
    float xv[KT + 1];
#pragma unroll
    for (int j = 0; j < KT + 1; ++j) xv[j] = xs[p + j];
    const bool pair = i + 1 < L && (L & 1) == 0;   // even row offsets: aligned pair stores
#pragma unroll 4
    for (int co = 0; co < CH; ++co) {
        const float4 wa = *reinterpret_cast<const float4*>(&ws[co][0]);
        const float4 wb = *reinterpret_cast<const float4*>(&ws[co][4]);
        const float4 wc = *reinterpret_cast<const float4*>(&ws[co][8]);
        const float w[KT] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w, wc.x};
        float s0 = wc.y, s1 = wc.y;
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            s0 = fmaf(w[k], xv[k], s0);
            s1 = fmaf(w[k], xv[k + 1], s1);
        }
        s0 = fmaxf(s0, 0.f);
        s1 = fmaxf(s1, 0.f);
        T* o = out + ((size_t)b * CH + co) * L + i;
        if (pair) {
            store_pair<T>(o, s0, s1);
        } else {
            o[0] = cvt<T>(s0);
            if (i + 1 < L) o[1] = cvt<T>(s1);
        }
    }
}

// ---------------------------------------------------------------- head
// Forward head in two kernels.  head_chunk_kernel: CTA (chunk x of HD_CT positions, row b)
// writes z for its positions and, per channel, the chunk's max, first arg-max and sum.
// head_mlp_kernel: per row, the chunk partials -> max / arg-max (first index) / mean per
// channel, then the presence MLP.
constexpr int HD_CT = 512;

template <class T>
__global__ void __launch_bounds__(256) head_chunk_kernel(const T* __restrict__ h4, const float* __restrict__ theta,
                                                         int L, int nx, float* __restrict__ z,
                                                         float* __restrict__ pmax, int* __restrict__ pidx,
                                                         float* __restrict__ psum, float* __restrict__ zmax,
                                                         int* __restrict__ zidx)
{
    const int b = blockIdx.y, xc = blockIdx.x, i0 = xc * HD_CT, iend = min(L, i0 + HD_CT);
    const T* hb = h4 + (size_t)b * CH * L;
    __shared__ float w5[CH];
    if (threadIdx.x < CH) w5[threadIdx.x] = theta[OFF_W5 + threadIdx.x];
    __syncthreads();
    const float b5 = theta[OFF_B5];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float zm = -INFINITY;   // the chunk's largest z and its first position
    int zi = i0;
    // BF16 rows with L a multiple of 8 are read once: warp w loads its channels 4w .. 4w + 3 with
    // 16-byte loads (lane: positions p = i0 + 8 lane + 256 r, all loads issued first), keeps their
    // max / first arg-max / sum and adds their part of z into zp[w]; z = b5 + the eight parts.
    // Other rows: z over all channels per position, then each channel's statistics, scalar loads.
    bool vec = false;
    if constexpr (std::is_same<T, __nv_bfloat16>::value) vec = (L & 7) == 0;
    if constexpr (std::is_same<T, __nv_bfloat16>::value) if (vec) {
        constexpr int HV = 8, HR = HD_CT / (32 * HV);
        __shared__ __align__(16) float zp[8][HD_CT];
        const T* hw = hb + (size_t)warp * 4 * L;
        uint4 hq[HR][4];
#pragma unroll
        for (int r = 0; r < HR; ++r) {
            const int p = i0 + HV * lane + 32 * HV * r;
#pragma unroll
            for (int cc = 0; cc < 4; ++cc)
                hq[r][cc] = p < iend ? *reinterpret_cast<const uint4*>(hw + (size_t)cc * L + p) : make_uint4(0u, 0u, 0u, 0u);
        }
        float mx[4], sum[4];
        int mi[4];
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            mx[cc] = -INFINITY;
            sum[cc] = 0.f;
            mi[cc] = i0;
        }
#pragma unroll
        for (int r = 0; r < HR; ++r) {
            const int p = i0 + HV * lane + 32 * HV * r;
            if (p >= iend) break;
            float zpart[HV];
#pragma unroll
            for (int k = 0; k < HV; ++k) {
                zpart[k] = 0.f;
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    const uint32_t w = (&hq[r][cc].x)[k >> 1];
                    const float v = __uint_as_float((k & 1) ? (w & 0xffff0000u) : (w << 16));   // BF16 -> FP32
                    zpart[k] = fmaf(w5[warp * 4 + cc], v, zpart[k]);
                    if (v > mx[cc]) {
                        mx[cc] = v;
                        mi[cc] = p + k;
                    }
                    sum[cc] += v;
                }
            }
            float4* zq = reinterpret_cast<float4*>(&zp[warp][p - i0]);
            zq[0] = make_float4(zpart[0], zpart[1], zpart[2], zpart[3]);
            zq[1] = make_float4(zpart[4], zpart[5], zpart[6], zpart[7]);
        }
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            for (int o = 16; o; o >>= 1) {
                const float om = __shfl_down_sync(0xffffffffu, mx[cc], o);
                const int oi = __shfl_down_sync(0xffffffffu, mi[cc], o);
                sum[cc] += __shfl_down_sync(0xffffffffu, sum[cc], o);
                if (om > mx[cc] || (om == mx[cc] && oi < mi[cc])) {
                    mx[cc] = om;
                    mi[cc] = oi;
                }
            }
            if (lane == 0) {
                const size_t o = ((size_t)b * nx + xc) * CH + warp * 4 + cc;
                pmax[o] = mx[cc];
                pidx[o] = mi[cc];
                psum[o] = sum[cc];
            }
        }
        __syncthreads();
        for (int i = i0 + threadIdx.x; i < iend; i += 256) {
            float s = b5;
#pragma unroll
            for (int w = 0; w < 8; ++w) s += zp[w][i - i0];
            z[(size_t)b * L + i] = s;
            if (s > zm) {
                zm = s;
                zi = i;
            }
        }
    }
    if (!vec) {
        for (int i = i0 + threadIdx.x; i < iend; i += 256) {
            float s = b5;
#pragma unroll 8
            for (int c = 0; c < CH; ++c) s = fmaf(w5[c], ld<T>(hb, (size_t)c * L + i), s);
            z[(size_t)b * L + i] = s;
            if (s > zm) {
                zm = s;
                zi = i;
            }
        }
    }
    for (int o = 16; o; o >>= 1) {
        const float om = __shfl_down_sync(0xffffffffu, zm, o);
        const int oi = __shfl_down_sync(0xffffffffu, zi, o);
        if (om > zm || (om == zm && oi < zi)) {
            zm = om;
            zi = oi;
        }
    }
    __shared__ float zm_s[8];
    __shared__ int zi_s[8];
    if (lane == 0) {
        zm_s[warp] = zm;
        zi_s[warp] = zi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w)
            if (zm_s[w] > zm_s[0] || (zm_s[w] == zm_s[0] && zi_s[w] < zi_s[0])) {
                zm_s[0] = zm_s[w];
                zi_s[0] = zi_s[w];
            }
        zmax[(size_t)b * nx + xc] = zm_s[0];
        zidx[(size_t)b * nx + xc] = zi_s[0];
    }
    // warp w: channels 4w .. 4w+3 (done above for the vector path)
    if (!vec) for (int cc = 0; cc < 4; ++cc) {
        const int c = warp * 4 + cc;
        float mx = -INFINITY, sum = 0.f;
        int mi = i0;
        for (int i = i0 + lane; i < iend; i += 32) {
            const float v = ld<T>(hb, (size_t)c * L + i);
            if (v > mx) {
                mx = v;
                mi = i;
            }
            sum += v;
        }
        for (int o = 16; o; o >>= 1) {
            const float om = __shfl_down_sync(0xffffffffu, mx, o);
            const int oi = __shfl_down_sync(0xffffffffu, mi, o);
            sum += __shfl_down_sync(0xffffffffu, sum, o);
            if (om > mx || (om == mx && oi < mi)) {
                mx = om;
                mi = oi;
            }
        }
        if (lane == 0) {
            const size_t o = ((size_t)b * nx + xc) * CH + c;
            pmax[o] = mx;
            pidx[o] = mi;
            psum[o] = sum;
        }
    }
}

// Head of one row from its chunk statistics, in HM_THREADS threads: max / first
// arg-max / mean per channel and the presence MLP; with PREDICT also the prediction: position =
// softmax-weighted mean over the 7 bins around the first arg-max of z (+ band_lo), presence =
// sigmoid(q).  Latency bound (a few KB per row): warp w takes the chunks w, w + 8, ... with a lane per
// channel, the first warp the chunks' largest logits with a lane per chunk, and eight threads share
// each hidden unit.
constexpr int HM_THREADS = 256;
struct HeadScratch {
    float mx[HM_THREADS / 32][CH], sum[HM_THREADS / 32][CH];
    float pool[2 * CH], u[CH];
};
struct HeadArgs {
    const float* theta;
    int L, nx, lo;
    const float *pmax, *psum, *z, *zmax;
    const int *pidx, *zidx;
    int* amax;
    float *pooled, *u, *q, *pos, *pres;
};

template <bool PREDICT>
__global__ void __launch_bounds__(HM_THREADS) head_mlp_kernel(const HeadArgs a)
{
    __shared__ HeadScratch sc;
    __shared__ int mi_s[HM_THREADS / 32][CH];
    const int b = blockIdx.x, tid = threadIdx.x;
    constexpr int NW = HM_THREADS / 32;
    const int lane = tid & 31, warp = tid >> 5, nx = a.nx, L = a.L;
    const float* theta = a.theta;
    // hidden unit j's weights for inputs 8 part .. 8 part + 7, on their way meanwhile
    const int j = tid >> 3, part = tid & 7;
    float wa[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) wa[e] = theta[OFF_WA + j * 2 * CH + 8 * part + e];
    {
        float mx = -INFINITY, sum = 0.f;
        int mi = 0;
        for (int xc = warp; xc < nx; xc += NW) {   // ascending: ties keep the first
            const size_t o = ((size_t)b * nx + xc) * CH + lane;
            const float v = a.pmax[o];
            if (v > mx) {
                mx = v;
                if constexpr (!PREDICT) mi = a.pidx[o];   // only the backward pass asks where
            }
            sum += a.psum[o];
        }
        sc.mx[warp][lane] = mx;
        sc.sum[warp][lane] = sum;
        if constexpr (!PREDICT) mi_s[warp][lane] = mi;
    }
    if (PREDICT && warp == 0) {
        float mx = -INFINITY;
        int mi = 0x7fffffff;
        for (int xc = lane; xc < nx; xc += 32) {
            const float v = a.zmax[(size_t)b * nx + xc];
            if (v > mx) {
                mx = v;
                mi = a.zidx[(size_t)b * nx + xc];
            }
        }
        for (int o = 16; o; o >>= 1) {
            const float om = __shfl_xor_sync(0xffffffffu, mx, o);
            const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
            if (om > mx || (om == mx && oi < mi)) {
                mx = om;
                mi = oi;
            }
        }
        if (mi == 0x7fffffff) mi = 0;   // no logit above -infinity
        const int i = mi - WIN + lane;
        double wgt = 0.0;
        if (lane <= 2 * WIN && i >= 0 && i < L) wgt = exp((double)a.z[(size_t)b * L + i] - (double)mx);
        double sw = 0, swi = 0;
        for (int k = 0; k <= 2 * WIN; ++k) {   // ascending positions
            const double wk = __shfl_sync(0xffffffffu, wgt, k);
            const int ik = mi - WIN + k;
            if (ik < 0 || ik >= L) continue;
            sw += wk;
            swi += wk * ik;
        }
        if (lane == 0) a.pos[b] = (float)(a.lo + swi / sw);
    }
    __syncthreads();
    if (tid < CH) {
        float mx = sc.mx[0][tid], sum = sc.sum[0][tid];
        int mi = PREDICT ? 0 : mi_s[0][tid];
        for (int w = 1; w < NW; ++w) {
            const float om = sc.mx[w][tid];
            const int oi = PREDICT ? 0 : mi_s[w][tid];
            if (om > mx || (om == mx && om > -INFINITY && oi < mi)) {
                mx = om;
                mi = oi;
            }
            sum += sc.sum[w][tid];
        }
        sc.pool[tid] = mx;
        sc.pool[CH + tid] = sum / L;
        if constexpr (!PREDICT) a.amax[b * CH + tid] = mi;
    }
    __syncthreads();
    {
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) s = fmaf(wa[e], sc.pool[8 * part + e], s);
        for (int o = 4; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (part == 0) {
            s += theta[OFF_BA + j];
            sc.u[j] = fmaxf(s, 0.f);
            if constexpr (!PREDICT) a.u[b * CH + j] = sc.u[j];
        }
    }
    if constexpr (!PREDICT) {
        if (tid < 2 * CH) a.pooled[b * 2 * CH + tid] = sc.pool[tid];
    }
    __syncthreads();
    if (warp == 0) {
        float s = theta[OFF_WB + lane] * sc.u[lane];
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            s += theta[OFF_BB];
            if constexpr (!PREDICT) a.q[b] = s;
            else a.pres[b] = 1.f / (1.f + expf(-s));
        }
    }
}

// ---------------------------------------------------------------- fused forward pass (BF16, tcgen05)
// The whole network up to the head's chunk statistics in one kernel: a tile's activations never leave the
// SM (in training they are written out for the backward pass, but not read again).  Launched per layer,
// conv1, three convolutions and the head took 16 + 3 x 33 + 14 us for 128 rows x 4608 positions, bound by
// staging channel-major rows into the operand layout; here the epilogue of a layer writes the next
// layer's operand.
//
// A tile is FI_W = 512 positions of one row, of which FI_P = 488 come out of the fourth layer (four
// 9-tap layers use up 8 positions each, the first computes 512 of the 520 the second could read).  It
// goes to the tensor cores as 128 rows of four positions each:
//   D[r][32 p' + co] = sum_{t, ci} X[4 r + t][ci] W[co][ci][t - p],   p' = 3 - p,  t = 0 .. 11,
// M = 128, N = 128 (four positions x 32 channels), K = 12 taps x 32 channels, 24 MMAs of 64 cycles where
// four M = 128, N = 32 tiles are 72 of 46: a quarter of the products are with zeros, but an N = 32 MMA is
// bound by reading its A operand.  The operand B of tap t is the 128 rows starting at tap t of the
// weights laid out [8-channel group][3 zero taps, 9 taps][32 co][8 ci] (the next group's zeros follow), so
// the Toeplitz matrix costs little more room than the weights.  Positions of equal index mod 4 form the
// planes of A ([8-channel group][index mod 4][index / 4][8 ci]), so tap t is plane t mod 4 started t / 4
// rows later.  Each output accumulates the same products in the same order as one 9-tap convolution
// (the added ones are zeros); a zero times an infinity would not be one, so a tile that holds an infinity
// or a NaN issues the products of each p' alone, without the zero taps.
//
// A CTA (one per SM) holds the three layers' weights and SLOTS tiles, each worked on by eight warps with
// 128 TMEM columns of its own: while one tile's MMAs run, the others are in their first layer or
// epilogues.  The activations are overwritten in place once a layer's MMAs have completed.
// Measured, 128 rows x 4608 positions: inference 59 us with the head's 9 (separate kernels 139), training
// 76 us (separate 136).  Two tiles in inference 68 us, a turn for issuing one tile's MMAs after the
// other's 60 us, the row's head in its last tile's warps (one atomic per tile) 70 us.  The tensor pipe is
// active on about 45 % of cycles: the tiles run through their phases nearly together.  Thread
// (warp w, lane) of a tile: row r = 32 (w mod 4) + lane, its four positions, channels 16 (w / 4) .. + 15.
constexpr int FI_W = 512, FI_P = FI_W - 24;      // positions of a tile, positions it finishes
constexpr int FI_ST = 256;                       // threads per tile
constexpr int FI_ROWS = FI_W / 4 + 2;            // rows of a plane (taps reach two rows beyond)
constexpr int FI_PLANE = FI_ROWS * 16;           // bytes; 8 banks past a multiple of 32, so planes interleave
constexpr int FI_BUF = 16 * FI_PLANE;            // one part (32 channels) of a tile
constexpr int FI_WCG = (KT + 3) * CH * 16;       // bytes between 8-channel groups: 3 zero taps and 9 taps
constexpr int FI_WLAYER = 4 * FI_WCG;
constexpr int FI_WBYTES = 3 * FI_WLAYER + 3 * CH * 16;   // the last group's taps are followed by zeros too
constexpr int FI_OFF_BUF = (FI_WBYTES + 127) / 128 * 128;
constexpr int FI_XW = FI_W + KT - 1;
constexpr int HC = CH / 2;                       // channels of a thread
static_assert((FI_PLANE / 4) % 32 == 8 && FI_PLANE % 16 == 0, "plane pitch");

__host__ __device__ constexpr int fi_cols(int slots) { return slots > 2 ? 512 : 128 * slots; }   // a power of two

// two values as stored (BF16), and relu of them: max with 0 after rounding (NaN becomes 0, as fmaxf gives)
__device__ __forceinline__ uint32_t fi_relu2(float a, float b)
{
    const __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(a, b), __floats2bfloat162_rn(0.f, 0.f));
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t fi_max2(uint32_t a, uint32_t b)
{
    const __nv_bfloat162 h = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&h);
}
// whether a word that is the maximum of magnitude bit patterns has an infinity or NaN in either half
__device__ __forceinline__ bool fi_inf2(uint32_t m) { return (m & 0x7fffu) >= 0x7f80u || (m >> 16 & 0x7fffu) >= 0x7f80u; }
__device__ __forceinline__ float fi_half(uint32_t w, int half) { return __uint_as_float(half ? (w & 0xffff0000u) : (w << 16)); }

// v[c] (16 channels) combined over the warp's lanes: lanes 2 c, 2 c + 1 receive channel c's
template <class T, class OP>
__device__ __forceinline__ T fi_scatter(T (&v)[HC], int lane, OP op)
{
#pragma unroll
    for (int o = HC / 2; o; o >>= 1) {
        const bool up = (lane & (2 * o)) != 0;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const T keep = up ? v[k + o] : v[k], give = up ? v[k] : v[k + o];
            v[k] = op(keep, __shfl_xor_sync(0xffffffffu, give, 2 * o));
        }
    }
    return op(v[0], __shfl_xor_sync(0xffffffffu, v[0], 1));
}

// the barrier of a slot's 256 threads, with a vote
__device__ __forceinline__ bool fi_slot_or(int slot, bool pred)
{
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(any)
        : "r"((uint32_t)pred), "r"(1 + slot), "n"(FI_ST)
        : "memory");
    return any != 0;
}

// weights of three layers, rows [co][tap][ci], to [layer][ci / 8][3 zero taps, 9 taps][co][8 ci]
template <int NT>
__device__ __forceinline__ void fi_stage_weights(unsigned char* dst, const __nv_bfloat16* __restrict__ wt, int tid)
{
    constexpr int PER = (FI_WBYTES / 16 + NT - 1) / NT;
    uint4 v[PER];   // all loads first
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = tid + i * NT, co = e % CH, tp = e / CH % (KT + 3), gr = e / (CH * (KT + 3)), l = gr / 4, cg = gr % 4;
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (tp >= 3 && e < FI_WBYTES / 16)
            v[i] = __ldg(reinterpret_cast<const uint4*>(wt + ((size_t)(l * CH + co) * KT + (tp - 3)) * CH + cg * 8));
    }
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (tid + i * NT < FI_WBYTES / 16) *reinterpret_cast<uint4*>(dst + (tid + i * NT) * 16) = v[i];
}

// one thread: the MMAs of a layer on a tile of PARTS operand parts (hi and lo of a split operand), into the
// 128 TMEM columns at d, committed to mbar
template <int PARTS>
__device__ __forceinline__ void fi_issue(uint32_t d, uint32_t mbar, const unsigned char* buf, const unsigned char* w, bool inf)
{
    constexpr uint32_t idesc32 = isr::tc05_idesc<true>();                                  // M 128, N 32
    constexpr uint32_t idesc = (idesc32 & ~(0x3fu << 17)) | ((128u >> 3) << 17);           // N 128
    const uint64_t ad = isr::tc05_desc(isr::smem_u32(buf), 4 * FI_PLANE, 128);
    const uint64_t bd = isr::tc05_desc(isr::smem_u32(w), FI_WCG, 128);
    // descriptors step in 16-byte units of the start field (addresses stay below 0x40000)
    auto a_at = [&](int part, int t, int ks) {
        return ad + (uint32_t)((part * FI_BUF + (2 * ks * 4 + (t & 3)) * FI_PLANE + (t >> 2) * 16) >> 4);
    };
    auto b_at = [&](int tap, int ks) { return bd + (uint32_t)((2 * ks * FI_WCG + tap * CH * 16) >> 4); };
    if (!inf) {
#pragma unroll 1
        for (int part = 0; part < PARTS; ++part)
#pragma unroll
            for (int t = 0; t < KT + 3; ++t)
#pragma unroll
                for (int ks = 0; ks < 2; ++ks)
                    isr::tc05_mma(d, a_at(part, t, ks), b_at(t, ks), idesc, (part | t | ks) != 0);
    } else {
#pragma unroll 1
        for (int p = 0; p < 4; ++p)
#pragma unroll 1
            for (int part = 0; part < PARTS; ++part)
#pragma unroll 1
                for (int tap = 0; tap < KT; ++tap)
#pragma unroll 1
                    for (int ks = 0; ks < 2; ++ks)
                        isr::tc05_mma(d + 32u * (3 - p), a_at(part, tap + p, ks), b_at(tap + 3, ks), idesc32, (part | tap | ks) != 0);
    }
    isr::tc05_commit(mbar);
}

// Eight channels (group g of this thread's two) of its four positions: registers stay few that way.
constexpr int GC = CH / 4;
using FiQuad = uint32_t[4][GC / 2];   // [position][channel pair], as stored

__device__ __forceinline__ void fi_read(uint32_t tacc, int half, int g, float (&v)[4][GC])
{
    const uint32_t t = isr::tmem_warp_lane_base(tacc) + (uint32_t)(HC * half + GC * g);
#pragma unroll
    for (int p = 0; p < 4; ++p)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[p][0]), "=f"(v[p][1]), "=f"(v[p][2]), "=f"(v[p][3]), "=f"(v[p][4]), "=f"(v[p][5]),
                       "=f"(v[p][6]), "=f"(v[p][7])
                     : "r"(t + 32u * (3 - p)));
#pragma unroll
    for (int p = 0; p < 4; ++p)   // the registers pass through the wait, so that no use moves ahead of it
        asm volatile("tcgen05.wait::ld.sync.aligned;"
                     : "+f"(v[p][0]), "+f"(v[p][1]), "+f"(v[p][2]), "+f"(v[p][3]), "+f"(v[p][4]), "+f"(v[p][5]),
                       "+f"(v[p][6]), "+f"(v[p][7]));
}

// to the planes of row r
__device__ __forceinline__ void fi_to_planes(unsigned char* buf, int r, int half, int g, const FiQuad& q)
{
#pragma unroll
    for (int p = 0; p < 4; ++p)
        *reinterpret_cast<uint4*>(buf + ((2 * half + g) * 4 + p) * FI_PLANE + r * 16) = make_uint4(q[p][0], q[p][1], q[p][2], q[p][3]);
}

// Training forward: the stored activations of four positions pos .. (a multiple of 4, the first `count`
// exist) of row b
__device__ __forceinline__ void fi_to_rows(__nv_bfloat16* __restrict__ h, int b, int L, int pos, int count, int half, int g,
                                           const FiQuad& q)
{
    unsigned short* o = reinterpret_cast<unsigned short*>(h) + ((size_t)b * CH + HC * half + GC * g) * L + pos;
    if ((L & 3) == 0) {   // whole groups of four, 8-byte aligned
#pragma unroll
        for (int c = 0; c < GC; ++c) {
            const uint32_t sel = c & 1 ? 0x7632u : 0x5410u;
            *reinterpret_cast<uint2*>(o + (size_t)c * L) =
                make_uint2(__byte_perm(q[0][c / 2], q[1][c / 2], sel), __byte_perm(q[2][c / 2], q[3][c / 2], sel));
        }
    } else {
#pragma unroll
        for (int p = 0; p < 4; ++p)
            if (p < count)
#pragma unroll
                for (int c = 0; c < GC; ++c) o[(size_t)c * L + p] = (unsigned short)(q[p][c / 2] >> (16 * (c & 1)));
    }
}
// and their ReLU masks (bit co of word (b, i): h[b][co][i] > 0): eight channels of each position into m,
// then this thread's sixteen to memory
__device__ __forceinline__ void fi_mask(uint32_t (&m)[4], int g, const FiQuad& q)
{
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int k = 0; k < GC / 2; ++k) {
            const uint32_t t = __vsetgts2(q[p][k], 0u);   // 1 per half above zero
            m[p] |= ((t | t >> 15) & 3u) << (GC * g + 2 * k);
        }
}
__device__ __forceinline__ void fi_mask_to_rows(uint32_t* __restrict__ bits, int b, int L, int pos, int count, int half,
                                                const uint32_t (&m)[4])
{
    unsigned short* o = reinterpret_cast<unsigned short*>(bits + (size_t)b * L + pos) + half;
#pragma unroll
    for (int p = 0; p < 4; ++p)
        if (p < count) o[2 * p] = (unsigned short)m[p];
}

struct FiFwdSlot {
    uint64_t mbar, drained;
    int last;            // tiles end here; 0 once a wait ran out
    float zm[4];
    int zi[4];
    float mx[4][CH], sum[4][CH];
    int mi[4][CH];
    alignas(16) float z[FI_W];       // logits of the lower channels
    alignas(16) float x[FI_XW];
};
template <int SLOTS>
struct FiFwdShared {
    float w1[CH][12];    // W1[co][0..8], b1[co]
    float bias[3][CH];
    float w5[CH];
    uint32_t tslot;
    FiFwdSlot slot[SLOTS];
};
// tiles in flight per CTA: 80 registers a thread for three in inference; the stores of training need more
template <bool TRAIN> __host__ __device__ constexpr int fi_slots() { return TRAIN ? 2 : 3; }
template <bool TRAIN> __host__ __device__ constexpr int fi_smem()
{
    return FI_OFF_BUF + fi_slots<TRAIN>() * FI_BUF + (int)sizeof(FiFwdShared<fi_slots<TRAIN>()>);
}
static_assert(fi_smem<false>() <= 232448 && fi_smem<true>() <= 232448, "shared memory");
struct FiFwdArgs {
    const float* x;
    const __nv_bfloat16 *w1, *wt;
    const float* theta;
    int L, n_rows, nx;
    float *z, *pmax, *psum, *zmax;
    int *pidx, *zidx;
    __nv_bfloat16* h[4];       // training: h1 .. h4
    uint32_t* bits[3];         // training: ReLU masks of h1 .. h3
    EstWait wait;
};

// DROP (test hook, here and below): no products are issued, so that the waits for them run out
template <bool TRAIN, bool DROP>
__global__ void __launch_bounds__(fi_slots<TRAIN>() * FI_ST, 1) forward_kernel(const __grid_constant__ FiFwdArgs a)
{
    constexpr int SLOTS = fi_slots<TRAIN>(), NT = SLOTS * FI_ST;
    extern __shared__ __align__(128) unsigned char fi_smem_raw[];
    unsigned char* smem = fi_smem_raw;
    auto& sh = *reinterpret_cast<FiFwdShared<SLOTS>*>(smem + FI_OFF_BUF + SLOTS * FI_BUF);
    const int tid = threadIdx.x, slot = tid / FI_ST, st = tid - slot * FI_ST;
    const int lane = tid & 31, w = __shfl_sync(0xffffffffu, st >> 5, 0);   // warp of the slot
    const int half = w >> 2, r = 32 * (w & 3) + lane;
    FiFwdSlot& sl = sh.slot[slot];
    unsigned char* buf = smem + FI_OFF_BUF + slot * FI_BUF;
    const uint32_t mbar = isr::smem_u32(&sl.mbar);
    const int L = a.L, nx = a.nx;

    if (st == 0) {
        isr::mbar_init(mbar, 1);
        isr::mbar_init(isr::smem_u32(&sl.drained), 1);
        sl.last = a.n_rows * a.nx;
    }
    isr::fence_barrier_init();
    if (tid < 32) isr::tmem_alloc(isr::smem_u32(&sh.tslot), fi_cols(SLOTS));
    fi_stage_weights<NT>(smem, a.wt, tid);
    for (int e = tid; e < CH * 12; e += NT) {
        const int co = e / 12, k = e - co * 12;
        sh.w1[co][k] = k < KT ? ld<__nv_bfloat16>(a.w1, (size_t)k * CH + co) : (k == KT ? a.theta[OFF_B1 + co] : 0.f);
    }
    for (int e = tid; e < 3 * CH; e += NT) sh.bias[e / CH][e % CH] = a.theta[b_off(2 + e / CH) + e % CH];
    if (tid < CH) sh.w5[tid] = a.theta[OFF_W5 + tid];
    for (int e = tid; e < SLOTS * FI_BUF / 16; e += NT)   // the last two rows are read, never written
        *reinterpret_cast<uint4*>(smem + FI_OFF_BUF + e * 16) = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    isr::tmem_fence_before_sync();
    __syncthreads();
    isr::tmem_fence_after_sync();
    const uint32_t tacc = sh.tslot + 128u * slot;   // this tile's accumulator
    const float b5 = a.theta[OFF_B5];

    const int n_tiles = a.n_rows * nx, step = gridDim.x * SLOTS;
    // x of a tile: positions i0 - 16 .. , rounded to BF16 as the network reads it
    constexpr int XPER = (FI_XW + FI_ST - 1) / FI_ST;
    float xr[XPER];
    auto load_x = [&](int tile) {
        const int b = tile / nx, i0 = (tile - b * nx) * FI_P;
#pragma unroll
        for (int k = 0; k < XPER; ++k) {
            const int j = st + k * FI_ST, pos = i0 - 16 + j;
            xr[k] = (j < FI_XW && pos >= 0 && pos < L) ? __ldg(a.x + (size_t)b * L + pos) : 0.f;
        }
    };
    uint32_t phase = 0;
    auto stop = [&]() {   // a wait ran out: this is the slot's last tile
        sl.last = 0;
        est_timed_out(a.wait);
    };
    int tile = slot * gridDim.x + blockIdx.x;   // what is left after full rounds goes to different SMs
    if (tile < n_tiles) load_x(tile);
    for (; tile < sl.last; tile += step) {
        const int b = tile / nx, xc = tile - b * nx, i0 = xc * FI_P, end = min(i0 + FI_P, L);
#pragma unroll
        for (int k = 0; k < XPER; ++k) {
            const int j = st + k * FI_ST;
            if (j < FI_XW) sl.x[j] = __bfloat162float(__float2bfloat16_rn(xr[k]));
        }
        fi_slot_or(slot, false);
        if (tile + step < n_tiles) load_x(tile + step);
        // a tile writes out the positions it owns, i0 .. end - 1, of every layer (whole groups of four but
        // at the end of a row)
        auto owned = [&](int pos) { return pos >= i0 && pos < end ? min(4, end - pos) : 0; };
        // zero outside the row
        auto inside = [&](int pos) { return pos >= 0 && pos < L ? ~0u : 0u; };
        // ---- layer 1: positions i0 - 12 + 4 r .. + 3
        bool inf = false;
        {
            float xv[KT + 3];
#pragma unroll
            for (int k = 0; k < KT + 3; k += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&sl.x[4 * r + k]);
                xv[k] = v.x, xv[k + 1] = v.y, xv[k + 2] = v.z, xv[k + 3] = v.w;
            }
            const int pos = i0 - 12 + 4 * r;
            uint32_t top = 0u, mask[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
            for (int g = 0; g < 2; ++g) {
                FiQuad q;
#pragma unroll
                for (int c2 = 0; c2 < GC / 2; ++c2) {
                    float s[2][4];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const float* wr = sh.w1[HC * half + GC * g + 2 * c2 + c];
                        const float4 wa = *reinterpret_cast<const float4*>(wr), wb = *reinterpret_cast<const float4*>(wr + 4);
                        const float2 wc = *reinterpret_cast<const float2*>(wr + 8);
                        const float wk[KT] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w, wc.x};
#pragma unroll
                        for (int p = 0; p < 4; ++p) s[c][p] = wc.y;
#pragma unroll
                        for (int k = 0; k < KT; ++k)
#pragma unroll
                            for (int p = 0; p < 4; ++p) s[c][p] = fmaf(wk[k], xv[p + k], s[c][p]);
                    }
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        q[p][c2] = fi_relu2(s[0][p], s[1][p]) & inside(pos + p);
                        top = fi_max2(top, q[p][c2]);
                    }
                }
                fi_to_planes(buf, r, half, g, q);
                if constexpr (TRAIN) {
                    if (const int n = owned(pos)) fi_to_rows(a.h[0], b, L, pos, n, half, g, q);
                    fi_mask(mask, g, q);
                }
            }
            if constexpr (TRAIN) fi_mask_to_rows(a.bits[0], b, L, pos, owned(pos), half, mask);
            inf = fi_inf2(top);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        inf = fi_slot_or(slot, inf);
        if (!DROP && st == 0) fi_issue<1>(tacc, mbar, buf, smem, inf);
        // relu(accumulator + bias) of layer l + 2, as stored
        auto outputs = [&](int l, int g, FiQuad& q) {
            float v[4][GC];
            fi_read(tacc, half, g, v);
#pragma unroll
            for (int c4 = 0; c4 < GC / 4; ++c4) {
                const float4 bv = *reinterpret_cast<const float4*>(&sh.bias[l][HC * half + GC * g + 4 * c4]);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    q[p][2 * c4] = fi_relu2(v[p][4 * c4] + bv.x, v[p][4 * c4 + 1] + bv.y);
                    q[p][2 * c4 + 1] = fi_relu2(v[p][4 * c4 + 2] + bv.z, v[p][4 * c4 + 3] + bv.w);
                }
            }
        };
        // ---- layers 2 and 3
#pragma unroll 1
        for (int l = 0; l < 2; ++l) {
            if (!isr::mbar_wait(mbar, phase, a.wait.limit)) stop();
            phase ^= 1u;
            isr::tmem_fence_after_sync();
            const int pos = i0 - 8 + 4 * l + 4 * r;
            FiQuad q[2];
            uint32_t top = 0u;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                outputs(l, g, q[g]);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint32_t in = inside(pos + p);
#pragma unroll
                    for (int k = 0; k < GC / 2; ++k) {
                        q[g][p][k] &= in;
                        top = fi_max2(top, q[g][p][k]);
                    }
                }
                fi_to_planes(buf, r, half, g, q[g]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            isr::tmem_fence_before_sync();
            inf = fi_slot_or(slot, fi_inf2(top));
            isr::tmem_fence_after_sync();
            if (!DROP && st == 0) fi_issue<1>(tacc, mbar, buf, smem + (l + 1) * FI_WLAYER, inf);
            if constexpr (TRAIN) {   // beside the next layer's MMAs
                if (const int n = owned(pos)) {
                    uint32_t mask[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        fi_to_rows(a.h[l + 1], b, L, pos, n, half, g, q[g]);
                        fi_mask(mask, g, q[g]);
                    }
                    fi_mask_to_rows(a.bits[l + 1], b, L, pos, n, half, mask);
                }
            }
        }
        // ---- layer 4 stays in registers: the logits (lower channels first, the order of head_chunk_kernel)
        // and the head's statistics
        if (!isr::mbar_wait(mbar, phase, a.wait.limit)) stop();
        phase ^= 1u;
        isr::tmem_fence_after_sync();
        const int pos = i0 + 4 * r, n_own = owned(pos);
        auto logits = [&](int g, const FiQuad& q, float (&s)[4]) {
#pragma unroll
            for (int c4 = 0; c4 < GC / 4; ++c4) {
                const float4 w5 = *reinterpret_cast<const float4*>(&sh.w5[HC * half + GC * g + 4 * c4]);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint32_t p0 = q[p][2 * c4], p1 = q[p][2 * c4 + 1];
                    float part = (L & 7) == 0 ? 0.f : s[p];
                    part = fmaf(w5.x, fi_half(p0, 0), part);
                    part = fmaf(w5.y, fi_half(p0, 1), part);
                    part = fmaf(w5.z, fi_half(p1, 0), part);
                    part = fmaf(w5.w, fi_half(p1, 1), part);
                    s[p] = (L & 7) == 0 ? s[p] + part : part;
                }
            }
        };
        float t[HC];                                   // sums over this thread's positions
        uint32_t key[TRAIN ? HC : HC / 2];             // their maxima (training: with the position)
        FiQuad q[2];
        float s[4] = {b5, b5, b5, b5};
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            outputs(2, g, q[g]);
            if constexpr (TRAIN) {
                if (n_own) fi_to_rows(a.h[3], b, L, pos, n_own, half, g, q[g]);
            }
            if (half == 0) logits(g, q[g], s);
            // other positions count as 0 in the sums and, as every activation is >= 0 and every tile has a
            // position of its own, in the maxima
            FiQuad o;
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int k = 0; k < GC / 2; ++k) o[p][k] = p < n_own ? q[g][p][k] : 0u;
#pragma unroll
            for (int c = 0; c < GC; ++c)
                t[GC * g + c] = (fi_half(o[0][c / 2], c & 1) + fi_half(o[1][c / 2], c & 1)) +
                                (fi_half(o[2][c / 2], c & 1) + fi_half(o[3][c / 2], c & 1));
            if constexpr (TRAIN) {
                // largest value, first position: the value's bits above the position counted down; a
                // position that is not owned has the key 0, below any other's
#pragma unroll
                for (int c = 0; c < GC; ++c) {
                    key[GC * g + c] = 0u;
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const uint32_t bits = c & 1 ? o[p][c / 2] & 0xffff0000u : o[p][c / 2] << 16;
                        key[GC * g + c] = max(key[GC * g + c], p < n_own ? bits | (uint32_t)(FI_W - 1 - 4 * r - p) : 0u);
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < GC / 2; ++k)   // channel pairs
                    key[GC / 2 * g + k] = fi_max2(fi_max2(o[0][k], o[1][k]), fi_max2(o[2][k], o[3][k]));
            }
        }
        isr::tmem_fence_before_sync();
        if (half == 0) *reinterpret_cast<float4*>(&sl.z[4 * r]) = make_float4(s[0], s[1], s[2], s[3]);
        {
            const float cs = fi_scatter(t, lane, [](float u, float v) { return u + v; });
            if ((lane & 1) == 0) sl.sum[w & 3][HC * half + (lane >> 1)] = cs;
            if constexpr (TRAIN) {
                const uint32_t ck = fi_scatter(key, lane, [](uint32_t u, uint32_t v) { return max(u, v); });
                if ((lane & 1) == 0) {
                    const int c = HC * half + (lane >> 1);
                    sl.mx[w & 3][c] = __uint_as_float(ck & 0xffff0000u);
                    sl.mi[w & 3][c] = i0 + FI_W - 1 - (int)(ck & 0xffffu);
                }
            } else {
#pragma unroll
                for (int o = HC / 4; o; o >>= 1) {
                    const bool up = (lane & (4 * o)) != 0;
#pragma unroll
                    for (int k = 0; k < o; ++k) {
                        const uint32_t keep = up ? key[k + o] : key[k], give = up ? key[k] : key[k + o];
                        key[k] = fi_max2(keep, __shfl_xor_sync(0xffffffffu, give, 4 * o));
                    }
                }
                key[0] = fi_max2(key[0], __shfl_xor_sync(0xffffffffu, key[0], 2));
                key[0] = fi_max2(key[0], __shfl_xor_sync(0xffffffffu, key[0], 1));
                if ((lane & 2) == 0) sl.mx[w & 3][HC * half + 2 * (lane >> 2) + (lane & 1)] = fi_half(key[0], lane & 1);
            }
        }
        fi_slot_or(slot, false);
        isr::tmem_fence_after_sync();
        if (half == 1) {
            const float4 s0 = *reinterpret_cast<const float4*>(&sl.z[4 * r]);
            s[0] = s0.x, s[1] = s0.y, s[2] = s0.z, s[3] = s0.w;
            logits(0, q[0], s);
            logits(1, q[1], s);
            float m = -INFINITY;
            int mi = 0x7fffffff;
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (p < n_own && s[p] > m) {
                    m = s[p];
                    mi = pos + p;
                }
            float* zo = a.z + (size_t)b * L + pos;
            if ((L & 3) == 0) {
                if (n_own) *reinterpret_cast<float4*>(zo) = make_float4(s[0], s[1], s[2], s[3]);
            } else {
                for (int p = 0; p < n_own; ++p) zo[p] = s[p];
            }
            for (int o = 16; o; o >>= 1) {
                const float om = __shfl_xor_sync(0xffffffffu, m, o);
                const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
                if (om > m || (om == m && oi < mi)) {
                    m = om;
                    mi = oi;
                }
            }
            if (lane == 0) {
                sl.zm[w & 3] = m;
                sl.zi[w & 3] = mi;
            }
        } else if (w == 0) {
            float m = sl.mx[0][lane], s = sl.sum[0][lane];
            int mi = TRAIN ? sl.mi[0][lane] : 0;
#pragma unroll
            for (int k = 1; k < 4; ++k) {   // ascending positions: ties keep the first
                const float om = sl.mx[k][lane];
                if (om > m) {
                    m = om;
                    if constexpr (TRAIN) mi = sl.mi[k][lane];
                }
                s += sl.sum[k][lane];
            }
            const size_t o = ((size_t)b * nx + xc) * CH + lane;
            a.pmax[o] = m;
            a.psum[o] = s;
            if constexpr (TRAIN) a.pidx[o] = mi;
        }
        if constexpr (!TRAIN) {   // only the prediction asks for the largest logit
            fi_slot_or(slot, false);
            if (st == 0) {
                float best = sl.zm[0];
                int at = sl.zi[0];
                for (int k = 1; k < 4; ++k)   // ascending positions
                    if (sl.zm[k] > best) {
                        best = sl.zm[k];
                        at = sl.zi[k];
                    }
                a.zmax[(size_t)b * nx + xc] = best;
                a.zidx[(size_t)b * nx + xc] = at;
            }
        }
    }
    if (sl.last == 0 && st == 0) {   // what was issued meanwhile completes before the tensor memory goes
        isr::tc05_commit(isr::smem_u32(&sl.drained));
        isr::mbar_wait(isr::smem_u32(&sl.drained), 0u, a.wait.limit);
    }
    isr::tmem_fence_before_sync();
    __syncthreads();
    isr::tmem_fence_after_sync();
    if (tid < 32) isr::tmem_dealloc(sh.tslot, fi_cols(SLOTS));
}

__device__ __forceinline__ float block_sum(float v, float* red)
{
    for (int o = 16; o; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    return t;
}

__device__ __forceinline__ float block_max(float v, float* red)
{
    for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = -INFINITY;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmaxf(t, red[w]);
    return t;
}

// Head backward in two kernels.  head_bwd_row_kernel (per row): softmax statistics of z, the
// loss, the presence-MLP gradients and d(pooled); it leaves per row the scalars the location
// term needs (lse, 1 / sum t, y / B for gates with a line else 0, the line position) and
// d(pooled).  head_bwd_chunk_kernel (CTA = HD_CT positions of one row): dz, the ReLU-masked
// gradient of h4 and the CTA's partial dw5, db5.
constexpr int HB_SCAL = 4;   // per-row scalars: lse, 1 / sum t, y / B (0 without a line), f

__global__ void __launch_bounds__(256) head_bwd_row_kernel(const float* __restrict__ theta, int L, int B,
                                                           const float* __restrict__ z, const float* __restrict__ pooled,
                                                           const float* __restrict__ u, const float* __restrict__ q,
                                                           const float* __restrict__ fpos, const float* __restrict__ pres,
                                                           float* __restrict__ scal, float* __restrict__ dpool,
                                                           float* __restrict__ grad, float* __restrict__ loss)
{
    const int b = blockIdx.x;
    __shared__ float red[8];
    __shared__ float du_s[CH];
    const float* zb = z + (size_t)b * L;
    const float y = pres[b], f = fpos[b];
    // softmax statistics and target normalisation.  Rows of up to 4 x 256 x RV positions (L a
    // multiple of 4) are read once, as float4 pieces all in flight together, and kept in registers
    // for both passes; longer or unaligned rows are read twice with scalar loads.
    constexpr int RV = 5;
    const bool in_regs = (L & 3) == 0 && L <= 4 * 256 * RV;
    float4 zr[RV];
    float m = -INFINITY;
    if (in_regs) {
#pragma unroll
        for (int v = 0; v < RV; ++v) {
            const int i = 4 * (threadIdx.x + 256 * v);
            zr[v] = i < L ? __ldg(reinterpret_cast<const float4*>(zb + i)) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        }
#pragma unroll
        for (int v = 0; v < RV; ++v) m = fmaxf(m, fmaxf(fmaxf(zr[v].x, zr[v].y), fmaxf(zr[v].z, zr[v].w)));
    } else {
        for (int i = threadIdx.x; i < L; i += 256) m = fmaxf(m, zb[i]);
    }
    m = block_max(m, red);
    float se = 0.f, st = 0.f, stz = 0.f;
    auto term = [&](int i, float zi) {
        se += __expf(zi - m);
        const float d = (i - f) / SIGMA_T;
        const float t = __expf(-0.5f * d * d);
        st += t;
        stz += t * zi;
    };
    if (in_regs) {
#pragma unroll
        for (int v = 0; v < RV; ++v) {
            const int i = 4 * (threadIdx.x + 256 * v);
            if (i < L) {
                term(i, zr[v].x);
                term(i + 1, zr[v].y);
                term(i + 2, zr[v].z);
                term(i + 3, zr[v].w);
            }
        }
    } else {
        for (int i = threadIdx.x; i < L; i += 256) term(i, zb[i]);
    }
    se = block_sum(se, red);
    st = block_sum(st, red);
    stz = block_sum(stz, red);
    const float lse = m + logf(se);
    const float invB = 1.f / B;
    const float qb = q[b];
    const float sig = 1.f / (1.f + __expf(-qb));
    const float dq = (sig - y) * invB;
    // the location term exists only for gates with a line (its target may lie anywhere,
    // even outside the band, for gates without one)
    const bool loc = y > 0.f && st > 0.f;
    if (threadIdx.x == 0) {
        // CE = lse - sum t z / sum t ; BCE in the stable form
        const float ce = loc ? y * (lse - stz / st) : 0.f;
        const float bce = fmaxf(qb, 0.f) - qb * y + log1pf(__expf(-fabsf(qb)));
        atomicAdd(loss, (bce + ce) * invB);
        atomicAdd(&grad[OFF_BB], dq);
        float* sc = scal + (size_t)b * HB_SCAL;
        sc[0] = lse;
        sc[1] = loc ? 1.f / st : 0.f;
        sc[2] = loc ? y * invB : 0.f;
        sc[3] = f;
    }
    // presence MLP backward (du by threads 0..31; the 32 x 64 weight gradient by all threads)
    if (threadIdx.x < CH) {
        const int j = threadIdx.x;
        const float uj = u[b * CH + j];
        atomicAdd(&grad[OFF_WB + j], dq * uj);
        const float du = uj > 0.f ? dq * theta[OFF_WB + j] : 0.f;
        du_s[j] = du;
        atomicAdd(&grad[OFF_BA + j], du);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < CH * 2 * CH; e += 256)
        atomicAdd(&grad[OFF_WA + e], du_s[e / (2 * CH)] * pooled[b * 2 * CH + e % (2 * CH)]);
    if (threadIdx.x < 2 * CH) {
        float s = 0.f;
        for (int j = 0; j < CH; ++j) s = fmaf(du_s[j], theta[OFF_WA + j * 2 * CH + threadIdx.x], s);
        dpool[(size_t)b * 2 * CH + threadIdx.x] = s;
    }
}

// warp w: channels 4w .. 4w+3 of the chunk, lanes along the positions (each warp evaluates dz
// itself), so a thread keeps four partial dw5 sums and every warp adds its own channels
template <class T>
__global__ void __launch_bounds__(256, 2) head_bwd_chunk_kernel(const T* __restrict__ h4, const float* __restrict__ theta,
                                                             int L, const float* __restrict__ z,
                                                             const int* __restrict__ amax,
                                                             const float* __restrict__ scal,
                                                             const float* __restrict__ dpool, float* __restrict__ da4,
                                                             float* __restrict__ grad)
{
    const int b = blockIdx.y, i0 = blockIdx.x * HD_CT, iend = min(L, i0 + HD_CT);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float* sc = scal + (size_t)b * HB_SCAL;
    const float lse = sc[0], inv_st = sc[1], ys = sc[2], f = sc[3];
    float w5[4], gmean[4], gmax[4];
    int am[4];
#pragma unroll
    for (int cc = 0; cc < 4; ++cc) {
        const int c = warp * 4 + cc;
        w5[cc] = theta[OFF_W5 + c];
        gmax[cc] = dpool[(size_t)b * 2 * CH + c];
        gmean[cc] = dpool[(size_t)b * 2 * CH + CH + c] / L;
        am[cc] = amax[b * CH + c];
    }
    const float* zb = z + (size_t)b * L;
    const T* hb = h4 + ((size_t)b * CH + warp * 4) * L;
    float* ob = da4 + ((size_t)b * CH + warp * 4) * L;
    // BF16 rows with L a multiple of 8: lane takes positions p = i0 + 8 lane + 256 r, 8 at a time,
    // and every activation load of the chunk is issued here, before dz is computed (iend is a
    // multiple of 8: a piece is whole or absent)
    constexpr int HV = 8;                       // positions per lane and round (one 16-byte BF16 load)
    constexpr int HR = HD_CT / (32 * HV);       // rounds per chunk
    static_assert(HD_CT % (32 * HV) == 0, "whole rounds per chunk");
    bool vec = false;
    if constexpr (std::is_same<T, __nv_bfloat16>::value) vec = (L & 7) == 0;
    uint4 hq[HR][4];
    if (vec) {
#pragma unroll
        for (int r = 0; r < HR; ++r) {
            const int p = i0 + HV * lane + 32 * HV * r;
#pragma unroll
            for (int cc = 0; cc < 4; ++cc)
                hq[r][cc] = p < iend ? *reinterpret_cast<const uint4*>(hb + (size_t)cc * L + p) : make_uint4(0u, 0u, 0u, 0u);
        }
    }
    // dL/dz once per position (every warp needs it for its four channels)
    __shared__ __align__(16) float dz_s[HD_CT];   // read as float4 by the vector path
    float db5 = 0.f;
    for (int i = i0 + threadIdx.x; i < iend; i += 256) {
        const float d = (i - f) / SIGMA_T;
        const float dz = ys != 0.f ? ys * (__expf(zb[i] - lse) - __expf(-0.5f * d * d) * inv_st) : 0.f;
        dz_s[i - i0] = dz;
        db5 += dz;
    }
    __syncthreads();
    float dw5[4] = {0.f, 0.f, 0.f, 0.f};
    // one position's four channels: dw5 += dz h, da4 = (w5 dz + mean and max pooling terms) (h > 0)
    auto position = [&](int i, float dz, const float (&hv)[4], float (&o)[4]) {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            dw5[cc] = fmaf(dz, hv[cc], dw5[cc]);
            float g = w5[cc] * dz + gmean[cc];
            if (i == am[cc]) g += gmax[cc];
            o[cc] = hv[cc] > 0.f ? g : 0.f;
        }
    };
    if constexpr (std::is_same<T, __nv_bfloat16>::value) if (vec) {
#pragma unroll
        for (int r = 0; r < HR; ++r) {
            const int p = i0 + HV * lane + 32 * HV * r;
            if (p >= iend) break;
            const float4 z0 = *reinterpret_cast<const float4*>(&dz_s[p - i0]);
            const float4 z1 = *reinterpret_cast<const float4*>(&dz_s[p - i0 + 4]);
            const float dzv[HV] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
            float o[4][HV];
#pragma unroll
            for (int k = 0; k < HV; ++k) {
                float hv[4], ok[4];
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    const uint32_t w = (&hq[r][cc].x)[k >> 1];
                    hv[cc] = __uint_as_float((k & 1) ? (w & 0xffff0000u) : (w << 16));   // BF16 -> FP32
                }
                position(p + k, dzv[k], hv, ok);
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) o[cc][k] = ok[cc];
            }
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                float4* d = reinterpret_cast<float4*>(ob + (size_t)cc * L + p);
                d[0] = make_float4(o[cc][0], o[cc][1], o[cc][2], o[cc][3]);
                d[1] = make_float4(o[cc][4], o[cc][5], o[cc][6], o[cc][7]);
            }
        }
    }
    if (!vec) {
        for (int i = i0 + lane; i < iend; i += 32) {
            float hv[4], o[4];
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) hv[cc] = ld<T>(hb, (size_t)cc * L + i);
            position(i, dz_s[i - i0], hv, o);
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) ob[(size_t)cc * L + i] = o[cc];
        }
    }
#pragma unroll
    for (int cc = 0; cc < 4; ++cc)
        for (int o = 16; o; o >>= 1) dw5[cc] += __shfl_down_sync(0xffffffffu, dw5[cc], o);
    if (lane == 0) {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) atomicAdd(&grad[OFF_W5 + warp * 4 + cc], dw5[cc]);
    }
    // db5: one sum per CTA (every CTA adds into the same address, so one atomic each, not one per warp)
    __shared__ float db5_s[8];
    for (int o = 16; o; o >>= 1) db5 += __shfl_down_sync(0xffffffffu, db5, o);
    if (lane == 0) db5_s[warp] = db5;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += db5_s[w];
        atomicAdd(&grad[OFF_B5], t);   // the chunk's positions
    }
}

// ---------------------------------------------------------------- fused backward pass (BF16, tcgen05)
// The gradient of the loss from the head down through the three 32-channel layers in one kernel, with the
// tiles, operand layout and slots of forward_kernel: dL/dz and the masked gradient of h4 as
// head_bwd_chunk_kernel forms them, then per layer the convolution with the flipped transposed weights
// on the FP32 gradient split into BF16 hi + lo (48 MMAs), masked by the layer below's ReLU bits.  Every
// masked gradient is written once, in FP32, for the weight gradients, and none is read back: launched
// per layer these passes took 39 + 3 x 55 us for 128 rows x 4608 positions, bound by 75 MB in and out per
// layer and the staging between; together they take 126 us, for 323 MB of which 302 MB are the four
// gradients written (42 us at 7.6 TB/s): two tiles a SM leave the MMAs and the element passes of one
// exposed when the other waits too, and shared memory has no room for a third.  Gradient sums of w5 and
// b5 stay in registers over a CTA's tiles.
constexpr int FB_SLOTS = 2;
struct FiBwdSlot {
    uint64_t mbar;
    float mean[CH], peak[CH], scal[HB_SCAL];   // per channel: pooling gradients of the row
    int at[CH];                                 // position of the channel's maximum
};
struct FiBwdShared {
    float w5[CH];
    uint32_t tslot;
    FiBwdSlot slot[FB_SLOTS];
};
constexpr int FB_OFF_SH = FI_OFF_BUF + FB_SLOTS * 2 * FI_BUF;
constexpr int FB_SMEM = FB_OFF_SH + (int)sizeof(FiBwdShared);
static_assert(FB_SMEM <= 232448 && FB_OFF_SH % 16 == 0, "shared memory");
struct FiBwdArgs {
    const __nv_bfloat16 *h4, *wt;
    const float *theta, *z, *scal, *dpool;
    const int* amax;
    const uint32_t* bits[3];   // masks of h3, h2, h1
    float* da[4];              // masked gradients of h4 .. h1
    float* grad;
    int L, n_rows, nx;
    EstWait wait;
};

template <bool DROP>
__global__ void __launch_bounds__(FB_SLOTS * FI_ST, 1) backward_kernel(const __grid_constant__ FiBwdArgs a)
{
    constexpr int NT = FB_SLOTS * FI_ST;
    extern __shared__ __align__(128) unsigned char fb_smem[];
    auto& sh = *reinterpret_cast<FiBwdShared*>(fb_smem + FB_OFF_SH);
    const int tid = threadIdx.x, slot = tid / FI_ST, st = tid - slot * FI_ST;
    const int lane = tid & 31, w = __shfl_sync(0xffffffffu, st >> 5, 0);
    const int half = w >> 2, r = 32 * (w & 3) + lane;
    FiBwdSlot& sl = sh.slot[slot];
    unsigned char* buf = fb_smem + FI_OFF_BUF + slot * 2 * FI_BUF;   // hi part, lo part
    const uint32_t mbar = isr::smem_u32(&sl.mbar);
    const int L = a.L, nx = a.nx;
    const bool vec = (L & 3) == 0;   // groups of four positions are whole and aligned

    if (st == 0) isr::mbar_init(mbar, 1);
    isr::fence_barrier_init();
    if (tid < 32) isr::tmem_alloc(isr::smem_u32(&sh.tslot), fi_cols(FB_SLOTS));
    fi_stage_weights<NT>(fb_smem, a.wt, tid);
    if (tid < CH) sh.w5[tid] = a.theta[OFF_W5 + tid];
    for (int e = tid; e < FB_SLOTS * 2 * FI_BUF / 16; e += NT)   // the last two rows are read, never written
        *reinterpret_cast<uint4*>(fb_smem + FI_OFF_BUF + e * 16) = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    isr::tmem_fence_before_sync();
    __syncthreads();
    isr::tmem_fence_after_sync();
    const uint32_t tacc = sh.tslot + 128u * slot;

    // v[p][c]: FP32 gradients of eight channels (group g) at four positions -> memory (the first `count`
    // positions) ...
    auto to_rows = [&](float* __restrict__ da, int b, int pos, int count, int g, const float (&v)[4][GC]) {
        float* o = da + ((size_t)b * CH + HC * half + GC * g) * L + pos;
        if (vec) {
            if (count)
#pragma unroll
                for (int c = 0; c < GC; ++c)
                    *reinterpret_cast<float4*>(o + (size_t)c * L) = make_float4(v[0][c], v[1][c], v[2][c], v[3][c]);
        } else {
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (p < count)
#pragma unroll
                    for (int c = 0; c < GC; ++c) o[(size_t)c * L + p] = v[p][c];
        }
    };
    // ... and, split into BF16 hi + lo, to the operand planes; the magnitudes' largest bits into top
    auto to_planes = [&](int g, const float (&v)[4][GC], uint32_t& top) {
        FiQuad hi, lo;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int k = 0; k < GC / 2; ++k) {
                isr::split2<true>(v[p][2 * k], v[p][2 * k + 1], hi[p][k], lo[p][k]);
                top = __vmaxu2(top, hi[p][k] & 0x7fff7fffu);
            }
        fi_to_planes(buf, r, half, g, hi);
        fi_to_planes(buf + FI_BUF, r, half, g, lo);
    };

    const int n_tiles = a.n_rows * nx, step = gridDim.x * FB_SLOTS;
    float dw5[HC], db5 = 0.f;
#pragma unroll
    for (int c = 0; c < HC; ++c) dw5[c] = 0.f;
    uint32_t phase = 0;
    bool failed = false;   // a wait of this slot's threads ran out
    for (int tile = slot * gridDim.x + blockIdx.x; tile < n_tiles && !failed; tile += step) {
        const int b = tile / nx, xc = tile - b * nx, i0 = xc * FI_P, end = min(i0 + FI_P, L);
        auto owned = [&](int pos) { return pos >= i0 && pos < end ? min(4, end - pos) : 0; };
        auto inside = [&](int pos) { return pos >= 0 && pos < L; };
        if (st < CH) {
            sl.peak[st] = a.dpool[(size_t)b * 2 * CH + st];
            sl.mean[st] = a.dpool[(size_t)b * 2 * CH + CH + st] / L;
            sl.at[st] = a.amax[b * CH + st];
        } else if (st < CH + HB_SCAL) {
            sl.scal[st - CH] = a.scal[(size_t)b * HB_SCAL + st - CH];
        }
        fi_slot_or(slot, false);
        // ---- gradient of h4 at positions i0 - 12 + 4 r .. + 3
        uint32_t top = 0u;
        {
            const int pos = i0 - 12 + 4 * r, n_own = owned(pos);
            const float lse = sl.scal[0], inv_st = sl.scal[1], ys = sl.scal[2], f = sl.scal[3];
            float dz[4];
            const float* zb = a.z + (size_t)b * L;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int i = pos + p;
                const float d = (i - f) / SIGMA_T;
                dz[p] = inside(i) && ys != 0.f ? ys * (__expf(zb[i] - lse) - __expf(-0.5f * d * d) * inv_st) : 0.f;
                if (half == 0 && p < n_own) db5 += dz[p];
            }
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const __nv_bfloat16* hb = a.h4 + ((size_t)b * CH + HC * half + GC * g) * L + pos;
                uint2 hq[GC];   // four positions of a channel
#pragma unroll
                for (int c = 0; c < GC; ++c) {
                    hq[c] = make_uint2(0u, 0u);
                    if (vec) {
                        if (inside(pos)) hq[c] = *reinterpret_cast<const uint2*>(hb + (size_t)c * L);
                    } else {
                        const unsigned short* hs = reinterpret_cast<const unsigned short*>(hb) + (size_t)c * L;
                        uint32_t h[4];
#pragma unroll
                        for (int p = 0; p < 4; ++p) h[p] = inside(pos + p) ? hs[p] : 0u;
                        hq[c] = make_uint2(h[0] | h[1] << 16, h[2] | h[3] << 16);
                    }
                }
                float v[4][GC];
#pragma unroll
                for (int c = 0; c < GC; ++c) {
                    const int ch = HC * half + GC * g + c;
                    const float w5 = sh.w5[ch], mean = sl.mean[ch], peak = sl.peak[ch];
                    const int at = sl.at[ch];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const float h = fi_half(p < 2 ? hq[c].x : hq[c].y, p & 1);
                        if (p < n_own) dw5[GC * g + c] = fmaf(dz[p], h, dw5[GC * g + c]);
                        float d = fmaf(w5, dz[p], mean);
                        if (pos + p == at) d += peak;
                        v[p][c] = h > 0.f ? d : 0.f;
                    }
                }
                to_rows(a.da[0], b, pos, n_own, g, v);
                to_planes(g, v, top);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        bool inf = fi_slot_or(slot, fi_inf2(top));
        if (!DROP && st == 0) fi_issue<2>(tacc, mbar, buf, fb_smem + 2 * FI_WLAYER, inf);
        // ---- layers 4, 3, 2: gradients of h3, h2, h1
#pragma unroll 1
        for (int l = 0; l < 3; ++l) {
            const int pos = i0 - 8 + 4 * l + 4 * r, n_own = owned(pos);
            uint32_t m[4] = {0u, 0u, 0u, 0u};   // ReLU masks, on their way during the MMAs
            const uint32_t* mb = a.bits[l] + (size_t)b * L + pos;
            if (vec) {
                if (inside(pos)) {
                    const uint4 q = *reinterpret_cast<const uint4*>(mb);
                    m[0] = q.x, m[1] = q.y, m[2] = q.z, m[3] = q.w;
                }
            } else {
#pragma unroll
                for (int p = 0; p < 4; ++p)
                    if (inside(pos + p)) m[p] = mb[p];
            }
            const bool done = isr::mbar_wait(mbar, phase, a.wait.limit);
            phase ^= 1u;
            isr::tmem_fence_after_sync();
            top = 0u;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                float v[4][GC];
                fi_read(tacc, half, g, v);
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int c = 0; c < GC; ++c)
                        v[p][c] = m[p] >> (HC * half + GC * g + c) & 1u ? v[p][c] : 0.f;
                to_rows(a.da[l + 1], b, pos, n_own, g, v);
                if (l < 2) to_planes(g, v, top);
            }
            isr::tmem_fence_before_sync();
            if (l < 2) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            inf = fi_slot_or(slot, fi_inf2(top) || !done);
            if (inf) {   // one of the two, both of them rare
                if ((failed = fi_slot_or(slot, !done))) break;
                inf = fi_slot_or(slot, fi_inf2(top));
            }
            isr::tmem_fence_after_sync();
            if (!DROP && l < 2 && st == 0) fi_issue<2>(tacc, mbar, buf, fb_smem + (1 - l) * FI_WLAYER, inf);
        }
    }
    if (failed) {
        if (st == 0) est_timed_out(a.wait);
        isr::mbar_wait(mbar, phase ^ 1u, a.wait.limit);
    }
    const float d5 = fi_scatter(dw5, lane, [](float u, float v) { return u + v; });
    if ((lane & 1) == 0) atomicAdd(&a.grad[OFF_W5 + HC * half + (lane >> 1)], d5);
    if (half == 0) {
        for (int o = 16; o; o >>= 1) db5 += __shfl_xor_sync(0xffffffffu, db5, o);
        if (lane == 0) atomicAdd(&a.grad[OFF_B5], db5);
    }
    isr::tmem_fence_before_sync();
    __syncthreads();
    isr::tmem_fence_after_sync();
    if (tid < 32) isr::tmem_dealloc(sh.tslot, fi_cols(FB_SLOTS));
}

// status: set where the gradient is incomplete (tcgen05 engine; else NULL), which then leaves everything as it was
__global__ void adam_kernel(float* __restrict__ theta, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2,
                            const int* __restrict__ status)
{
    if (status && *status) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        theta[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    }
}

}  // namespace

struct isr_est {
    int nfft = 0, lo = 0, L = 0, max_batch = 0, precision = 0, dev = 0;
    cudaStream_t stream = nullptr;
    float *theta = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;
    float* wcopies = nullptr;   // FP32 storage: [WG_COPIES][WG_SIZE] sums of the weight gradients
    int64_t step = 0;
    void* wf = nullptr;       // forward working weights (storage type)
    void* wb = nullptr;       // backward-data working weights
    void* tf = nullptr;       // tensor-core GEMM rows of the forward weights (BF16 only)
    void* tb = nullptr;       // ... and of the backward-data weights
    void* act[5] = {};        // x, h1..h4 (storage type)
    float *z = nullptr, *pooled = nullptr, *u = nullptr, *q = nullptr, *loss = nullptr;
    int* amax = nullptr;
    float *pmax = nullptr, *psum = nullptr;   // head partials per (row, chunk, channel)
    float *hscal = nullptr, *dpool = nullptr; // head backward: per-row scalars and d(pooled)
    float* zmax = nullptr;                    // per (row, chunk): largest location logit ...
    int* zidx = nullptr;                      // ... and its first position
    bool weights_stale = true;                // the working weights need the master copy's values
    int wgrad_slots = 0;                      // resident tensor-core weight-gradient CTAs (all SMs)
    bool conv05 = false;                      // BF16 convolutions on tcgen05 (else mma.sync)
    int sms = 0;                              // multiprocessors of the device
    int* pidx = nullptr;
    float* da[4] = {};                    // masked gradients [da_rows][32][L]: of h4 .. h1 (tcgen05 engine), else two in turn
    int da_rows = 0;                      // rows they hold: max_batch, or fewer on the tcgen05 engine
    // tcgen05 engine: ReLU masks of h1..h3 as written by a training forward pass, [3][B][L] words,
    // bit co of word (b, i) set when h_l[b][co][i] > 0 as stored
    uint32_t* hbits = nullptr;
    // tcgen05 engine: whether a bounded wait ran out, in device memory and in pinned host memory
    int* status = nullptr;
    isr::StatusSlot host_status;
    unsigned wait_limit = 1u << 26;       // polls
    int drop_pass = -1;                   // test hook: the pass that leaves out its products
    EstWait wait() const { return EstWait{wait_limit, status, host_status.word}; }
};

namespace {

using isr::fail;

#define EST_TRY(expr)                                                                                 \
    do {                                                                                              \
        cudaError_t e_ = (expr);                                                                      \
        if (e_ != cudaSuccess)                                                                        \
            return fail(e_ == cudaErrorMemoryAllocation ? ISR_ERR_NO_MEMORY : ISR_ERR_CUDA, "%s: %s", #expr, \
                        cudaGetErrorString(e_));                                                      \
    } while (0)

struct Dev {
    int prev = -1;
    explicit Dev(int d)
    {
        cudaGetDevice(&prev);
        cudaSetDevice(d);
    }
    ~Dev()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

template <bool DROP>
isr_status set_tc05_attrs()
{
    EST_TRY(cudaFuncSetAttribute(forward_kernel<false, DROP>, cudaFuncAttributeMaxDynamicSharedMemorySize, fi_smem<false>()));
    EST_TRY(cudaFuncSetAttribute(forward_kernel<true, DROP>, cudaFuncAttributeMaxDynamicSharedMemorySize, fi_smem<true>()));
    EST_TRY(cudaFuncSetAttribute(backward_kernel<DROP>, cudaFuncAttributeMaxDynamicSharedMemorySize, FB_SMEM));
    EST_TRY(cudaFuncSetAttribute(wgrad_tc05_kernel<DROP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W5_SMEM_LAUNCH));
    return ISR_OK;
}

template <class T>
isr_status set_smem_attrs()
{
    if constexpr (!kTensorConv<T>) {
        EST_TRY(cudaFuncSetAttribute(conv_kernel<true, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem_bytes(16)));
        EST_TRY(cudaFuncSetAttribute(conv_kernel<true, 12>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem_bytes(12)));
        EST_TRY(cudaFuncSetAttribute(conv_kernel<false, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem_bytes(16)));
        EST_TRY(cudaFuncSetAttribute(conv_kernel<false, 12>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem_bytes(12)));
    } else {
        const isr_status st = set_tc05_attrs<false>();
        if (st != ISR_OK) return st;
        EST_TRY(cudaFuncSetAttribute(conv_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes(true)));
        EST_TRY(cudaFuncSetAttribute(conv_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes(false)));
        EST_TRY(cudaFuncSetAttribute(wgrad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)wgrad_tc_smem_bytes()));
    }
    return ISR_OK;
}

HeadArgs head_args(const isr_est* e, int nx, float* pos, float* pres)
{
    return HeadArgs{e->theta, e->L, nx, e->lo, e->pmax, e->psum, e->z, e->zmax, e->pidx, e->zidx, e->amax, e->pooled, e->u, e->q, pos, pres};
}

// Inference on the tcgen05 engine keeps no activations, so the buffers of h1 (logits) and h2 (the rest of
// the head's scratch) hold the head of many more rows than max_batch, and a long prediction takes few
// launches: 1000 rows x 4608 positions in eight launches of 128 rows left a fifth of the last of three
// rounds of tiles idle in each and ran the head's small kernel eight times (506 us with the features;
// 368 us in one launch).  Rows that fit; `a` points into the buffers for n of them.
int predict_rows(const isr_est* e)
{
    const int64_t nx = (e->L + FI_P - 1) / FI_P, bytes = (int64_t)e->max_batch * CH * e->L * 2;
    const int64_t row = 4 * (3 * nx * CH + 2 * nx + CH + 2 * CH + CH + 1);
    return (int)std::max<int64_t>(e->max_batch, std::min<int64_t>({bytes / (4 * (int64_t)e->L), (bytes - 16 * 9) / row, 1 << 16}));
}

void place_head(const isr_est* e, int n, int nx, HeadArgs& a, FiFwdArgs& f)
{
    unsigned char* at = static_cast<unsigned char*>(e->act[2]);
    auto take = [&](int per_row) {
        void* p = at;
        at += ((size_t)4 * n * per_row + 15) / 16 * 16;
        return p;
    };
    a.z = f.z = static_cast<float*>(e->act[1]);
    a.pmax = f.pmax = static_cast<float*>(take(nx * CH));
    a.psum = f.psum = static_cast<float*>(take(nx * CH));
    a.pidx = f.pidx = static_cast<int*>(take(nx * CH));
    a.zmax = f.zmax = static_cast<float*>(take(nx));
    a.zidx = f.zidx = static_cast<int*>(take(nx));
    a.amax = static_cast<int*>(take(CH));
    a.pooled = static_cast<float*>(take(2 * CH));
    a.u = static_cast<float*>(take(CH));
    a.q = static_cast<float*>(take(1));
}

// pos / pres: the prediction outputs (inference), or NULL
template <class T>
isr_status forward_t(isr_est* e, const float* x, int n, float* pos = nullptr, float* pres = nullptr)
{
    const int L = e->L;
    cudaStream_t s = e->stream;
    T* act[5];
    for (int i = 0; i < 5; ++i) act[i] = static_cast<T*>(e->act[i]);
    const size_t nx = (size_t)n * L;
    if (e->weights_stale) {   // working weights follow the master copy only after it changed
        relayout_kernel<T><<<(CH * KT + 3 * CH * CH * KT + 255) / 256, 256, 0, s>>>(
            e->theta, static_cast<T*>(e->wf), static_cast<T*>(e->wb), static_cast<T*>(e->tf), static_cast<T*>(e->tb));
        e->weights_stale = false;
    }
    if constexpr (kTensorConv<T>) {
        if (e->conv05) {
            const int nxi = (L + FI_P - 1) / FI_P, tiles = n * nxi;
            FiFwdArgs a{};
            a.x = x;
            a.w1 = static_cast<const T*>(e->wf);
            a.wt = static_cast<const T*>(e->tf);
            a.theta = e->theta;
            a.L = L;
            a.n_rows = n;
            a.nx = nxi;
            a.z = e->z;
            a.pmax = e->pmax;
            a.psum = e->psum;
            a.zmax = e->zmax;
            a.pidx = e->pidx;
            a.zidx = e->zidx;
            a.wait = e->wait();
            if (pos) {
                HeadArgs ha = head_args(e, nxi, pos, pres);
                if (n > e->max_batch) place_head(e, n, nxi, ha, a);
                auto* k = e->drop_pass == 0 ? forward_kernel<false, true> : forward_kernel<false, false>;
                k<<<std::min(e->sms, tiles), fi_slots<false>() * FI_ST, fi_smem<false>(), s>>>(a);
                head_mlp_kernel<true><<<n, HM_THREADS, 0, s>>>(ha);
            } else {
                // the weight gradient of the first layer reads x as stored
                cast_kernel<T><<<(unsigned)std::min<size_t>((nx + 255) / 256, 4096), 256, 0, s>>>(x, nx, act[0]);
                for (int l = 0; l < 4; ++l) a.h[l] = act[l + 1];
                for (int l = 0; l < 3; ++l) a.bits[l] = e->hbits + (size_t)l * e->max_batch * L;
                auto* k = e->drop_pass == 0 ? forward_kernel<true, true> : forward_kernel<true, false>;
                k<<<std::min(e->sms, tiles), fi_slots<true>() * FI_ST, fi_smem<true>(), s>>>(a);
                head_mlp_kernel<false><<<n, HM_THREADS, 0, s>>>(head_args(e, nxi, nullptr, nullptr));
            }
            EST_TRY(cudaGetLastError());
            return ISR_OK;
        }
    }
    cast_kernel<T><<<(unsigned)std::min<size_t>((nx + 255) / 256, 4096), 256, 0, s>>>(x, nx, act[0]);
    const T* wf = static_cast<const T*>(e->wf);
    conv1_kernel<T><<<dim3((L + L1_CT - 1) / L1_CT, n), 256, 0, s>>>(act[0], wf, e->theta + OFF_B1, L, act[1]);
    for (int l = 2; l <= 4; ++l) {
        if constexpr (kTensorConv<T>)
            conv_tc_kernel<true><<<dim3((L + CF_CT - 1) / CF_CT, n), CF_THREADS, tc_smem_bytes(true), s>>>(
                act[l - 1], static_cast<const T*>(e->tf) + (size_t)(l - 2) * CH * CH * KT, e->theta + b_off(l), nullptr, L,
                act[l]);
        else
            launch_conv<true>(act[l - 1], wf + CH * KT + (size_t)(l - 2) * CH * CH * KT, e->theta + b_off(l), nullptr, L, n,
                              std::max(1, e->sms), act[l], s);
    }
    const int nxh = (L + HD_CT - 1) / HD_CT;
    head_chunk_kernel<T><<<dim3(nxh, n), 256, 0, s>>>(act[4], e->theta, L, nxh, e->z, e->pmax, e->pidx, e->psum,
                                                      e->zmax, e->zidx);
    if (pos) head_mlp_kernel<true><<<n, HM_THREADS, 0, s>>>(head_args(e, nxh, pos, pres));
    else head_mlp_kernel<false><<<n, HM_THREADS, 0, s>>>(head_args(e, nxh, nullptr, nullptr));
    EST_TRY(cudaGetLastError());
    return ISR_OK;
}

template <class T>
isr_status backward_t(isr_est* e, int n, const float* fpos, const float* pres)
{
    const int L = e->L;
    cudaStream_t s = e->stream;
    T* act[5];
    for (int i = 0; i < 5; ++i) act[i] = static_cast<T*>(e->act[i]);
    EST_TRY(cudaMemsetAsync(e->grad, 0, sizeof(float) * NPARAM, s));
    EST_TRY(cudaMemsetAsync(e->loss, 0, sizeof(float), s));
    if constexpr (!kTensorConv<T>) EST_TRY(cudaMemsetAsync(e->wcopies, 0, sizeof(float) * WG_COPIES * WG_SIZE, s));
    head_bwd_row_kernel<<<n, 256, 0, s>>>(e->theta, L, n, e->z, e->pooled, e->u, e->q, fpos, pres, e->hscal,
                                          e->dpool, e->grad, e->loss);
    if constexpr (kTensorConv<T>) {
        if (e->conv05) {
            const int nxi = (L + FI_P - 1) / FI_P;
            for (int r0 = 0; r0 < n; r0 += e->da_rows) {   // rows r0 .. r0 + rows - 1
                const int rows = std::min(e->da_rows, n - r0);
                const size_t at = (size_t)r0 * L;
                FiBwdArgs a{};
                a.h4 = act[4] + at * CH;
                a.wt = static_cast<const T*>(e->tb);
                a.theta = e->theta;
                a.z = e->z + at;
                a.scal = e->hscal + (size_t)r0 * HB_SCAL;
                a.dpool = e->dpool + (size_t)r0 * 2 * CH;
                a.amax = e->amax + (size_t)r0 * CH;
                for (int i = 0; i < 3; ++i) a.bits[i] = e->hbits + (size_t)(2 - i) * e->max_batch * L + at;
                for (int i = 0; i < 4; ++i) a.da[i] = e->da[i];
                a.grad = e->grad;
                a.L = L;
                a.n_rows = rows;
                a.nx = nxi;
                a.wait = e->wait();
                (e->drop_pass == 1 ? backward_kernel<true> : backward_kernel<false>)<<<std::min(e->sms, rows * nxi), FB_SLOTS * FI_ST, FB_SMEM, s>>>(a);
                const int chunks = rows * ((L + W5_CHUNK - 1) / W5_CHUNK), spans = rows * ((L + W1_SPAN - 1) / W1_SPAN);
                W5Args wa{};
                for (int i = 0; i < W5_LAYERS; ++i) {
                    wa.h[i] = act[3 - i] + at * CH;
                    wa.da[i] = e->da[i];
                    wa.dW[i] = e->grad + w_off(4 - i);
                    wa.db[i] = e->grad + b_off(4 - i);
                }
                wa.L = L;
                wa.n_rows = rows;
                wa.wait = e->wait();
                wa.drain = (chunks + std::max(1, e->sms) - 1) / std::max(1, e->sms);
                (e->drop_pass == 2 ? wgrad_tc05_kernel<true> : wgrad_tc05_kernel<false>)<<<std::min(W5_LAYERS * chunks, std::max(W5_LAYERS, e->sms)), W5_BLOCK, W5_SMEM_LAUNCH, s>>>(wa);
                wgrad1_kernel<T><<<std::min(spans, 2 * std::max(1, e->sms)), 256, 0, s>>>(act[0] + at, e->da[3], L, rows,
                                                                                         e->grad + OFF_W1, e->grad + OFF_B1);
            }
            EST_TRY(cudaGetLastError());
            return ISR_OK;
        }
    }
    head_bwd_chunk_kernel<T><<<dim3((L + HD_CT - 1) / HD_CT, n), 256, 0, s>>>(act[4], e->theta, L, e->z, e->amax,
                                                                              e->hscal, e->dpool, e->da[0], e->grad);
    const T* wbk = static_cast<const T*>(e->wb);
    float* da = e->da[0];
    float* dn = e->da[1];
    const int ftile = wgrad_tile(L, n, std::max(1, e->sms)), fspan = wgrad_span(L, n, std::max(1, e->sms), ftile);
    const int span = TC_CT * wgrad_span_chunks(L, n, std::max(1, e->wgrad_slots));
    for (int l = 4; l >= 1; --l) {
        if (l == 1) {
            const int spans = n * ((L + W1_SPAN - 1) / W1_SPAN);
            wgrad1_kernel<T><<<std::min(spans, 2 * std::max(1, e->sms)), 256, 0, s>>>(act[0], da, L, n,
                                                                                     e->grad + OFF_W1, e->grad + OFF_B1);
        } else {
            if constexpr (kTensorConv<T>)
                wgrad_tc_kernel<<<dim3((L + span - 1) / span, n), 256, wgrad_tc_smem_bytes(), s>>>(
                    act[l - 1], da, L, span, e->grad + w_off(l), e->grad + b_off(l));
            else
                (ftile == 96 ? wgrad_kernel<T, 96> : wgrad_kernel<T, 128>)<<<dim3((L + fspan - 1) / fspan, n), 256, 0, s>>>(
                    act[l - 1], da, L, fspan, e->wcopies + (w_off(l) - OFF_W2), e->wcopies + (b_off(l) - OFF_W2));
            // gradient into the layer below, masked by its ReLU: da_{l-1} = (W_l^T * da_l) (h_{l-1} > 0)
            if constexpr (kTensorConv<T>)
                conv_tc_kernel<false><<<dim3((L + CF_CT - 1) / CF_CT, n), CF_THREADS, tc_smem_bytes(false), s>>>(
                    da, static_cast<const T*>(e->tb) + (size_t)(l - 2) * CH * CH * KT, nullptr, act[l - 1], L, dn);
            else
                launch_conv<false>(da, wbk + (size_t)(l - 2) * CH * CH * KT, nullptr, act[l - 1], L, n, std::max(1, e->sms), dn, s);
            std::swap(da, dn);
        }
    }
    if constexpr (!kTensorConv<T>) wgrad_sum_kernel<<<(WG_SIZE + 255) / 256, 256, 0, s>>>(e->wcopies, e->grad + OFF_W2);
    EST_TRY(cudaGetLastError());
    return ISR_OK;
}

bool dev_ptr(const void* p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// ISR_ERR_TIMEOUT, once, if a kernel since the last report gave up waiting.  Between calls it may come late
// (the kernel may still run), after a synchronisation it does not.
isr_status check_waits(isr_est* e)
{
    if (!e->host_status.word || *static_cast<volatile int*>(e->host_status.word) == 0) return ISR_OK;
    EST_TRY(cudaMemsetAsync(e->status, 0, sizeof(int), e->stream));
    EST_TRY(cudaStreamSynchronize(e->stream));
    *static_cast<volatile int*>(e->host_status.word) = 0;
    return fail(ISR_ERR_TIMEOUT, "an estimator kernel timed out waiting for its tensor-core products");
}

isr_status check_batch(isr_est* e, const float* x, int n)
{
    if (!e || !x) return fail(ISR_ERR_INVALID_ARG, "estimator and x must not be NULL");
    if (n < 1 || n > e->max_batch) return fail(ISR_ERR_INVALID_ARG, "batch %d outside [1, %d]", n, e->max_batch);
    if (!dev_ptr(x)) return fail(ISR_ERR_INVALID_ARG, "x must be device memory");
    return ISR_OK;
}

}  // namespace

extern "C" {

isr_status isr_est_create(isr_est** out, int32_t nfft, int32_t band_lo, int32_t band_len, int32_t max_batch,
                          int32_t precision, int32_t device, void* stream)
{
    isr::clear_error();
    if (!out) return fail(ISR_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (nfft < 8 || band_lo < 0 || band_len < 16 || band_lo + band_len > nfft || max_batch < 1)
        return fail(ISR_ERR_INVALID_ARG, "need 0 <= band_lo, band_len >= 16, band_lo + band_len <= nfft, max_batch >= 1");
    if (precision != ISR_EST_FP32 && precision != ISR_EST_BF16 && precision != ISR_EST_BF16_MMASYNC)
        return fail(ISR_ERR_UNSUPPORTED, "unknown precision");
    int dev = device;
    if (dev < 0 && cudaGetDevice(&dev) != cudaSuccess) return fail(ISR_ERR_CUDA, "no current device");
    Dev guard(dev);
    isr_est* e = new (std::nothrow) isr_est();
    if (!e) return fail(ISR_ERR_NO_MEMORY, "host allocation failed");
    e->nfft = nfft;
    e->lo = band_lo;
    e->L = band_len;
    e->max_batch = max_batch;
    e->precision = precision;
    e->conv05 = precision == ISR_EST_BF16;
    e->dev = dev;
    e->stream = static_cast<cudaStream_t>(stream);
    const bool bf16 = precision != ISR_EST_FP32;
    const size_t es = bf16 ? 2 : 4;
    const size_t B = max_batch, L = band_len;
    cudaError_t r = cudaSuccess;
    auto A = [&](void** p, size_t bytes) {
        if (r == cudaSuccess) r = cudaMalloc(p, bytes);
    };
    A((void**)&e->theta, 4 * NPARAM);
    A((void**)&e->m, 4 * NPARAM);
    A((void**)&e->v, 4 * NPARAM);
    A((void**)&e->grad, 4 * NPARAM);
    A(&e->wf, es * (CH * KT + 3 * CH * CH * KT));
    A(&e->wb, es * 3 * CH * CH * KT);
    if (bf16) {
        A(&e->tf, es * 3 * CH * CH * KT);
        A(&e->tb, es * 3 * CH * CH * KT);
    }
    if (!bf16) A((void**)&e->wcopies, sizeof(float) * WG_COPIES * WG_SIZE);
    A(&e->act[0], es * B * L);
    for (int i = 1; i < 5; ++i) A(&e->act[i], es * B * CH * L);
    A((void**)&e->z, 4 * B * L);
    A((void**)&e->pooled, 4 * B * 2 * CH);
    A((void**)&e->u, 4 * B * CH);
    A((void**)&e->q, 4 * B);
    A((void**)&e->loss, 4);
    A((void**)&e->amax, 4 * B * CH);
    const size_t nxh = (L + FI_P - 1) / FI_P;   // head chunks of the fused inference (training has no more)
    static_assert(FI_P <= HD_CT, "head partials");
    A((void**)&e->pmax, 4 * B * nxh * CH);
    A((void**)&e->pidx, 4 * B * nxh * CH);
    A((void**)&e->psum, 4 * B * nxh * CH);
    A((void**)&e->hscal, 4 * B * HB_SCAL);
    A((void**)&e->dpool, 4 * B * 2 * CH);
    A((void**)&e->zmax, 4 * B * nxh);
    A((void**)&e->zidx, 4 * B * nxh);
    if (e->conv05) {
        A((void**)&e->hbits, 4 * 3 * B * L);
        A((void**)&e->status, sizeof(int));
        if (r == cudaSuccess) r = cudaMemset(e->status, 0, sizeof(int));
        if (r == cudaSuccess) r = isr::take_status(e->host_status);
        if (r == cudaSuccess) *e->host_status.word = 0;
    }
    // the tcgen05 engine's backward pass takes as many rows at a time as four gradient buffers fit for: all
    // of them, or where memory is short a half (the two full buffers that the other engines need), and so on
    const int n_da = e->conv05 ? 4 : 2;
    e->da_rows = max_batch;
    while (r == cudaSuccess) {
        for (int i = 0; i < n_da; ++i) A((void**)&e->da[i], (size_t)4 * e->da_rows * CH * L);
        if (r != cudaErrorMemoryAllocation || !e->conv05 || e->da_rows == 1) break;
        cudaGetLastError();
        for (int i = 0; i < n_da; ++i) {
            cudaFree(e->da[i]);
            e->da[i] = nullptr;
        }
        e->da_rows = (e->da_rows + 1) / 2;
        r = cudaSuccess;
    }
    if (r == cudaSuccess) r = cudaMemset(e->theta, 0, 4 * NPARAM);
    if (r == cudaSuccess) r = cudaMemset(e->m, 0, 4 * NPARAM);
    if (r == cudaSuccess) r = cudaMemset(e->v, 0, 4 * NPARAM);
    if (r == cudaSuccess) {
        isr_status st = bf16 ? set_smem_attrs<__nv_bfloat16>() : set_smem_attrs<float>();
        if (st != ISR_OK) {
            isr_est_destroy(e);
            return st;
        }
        int sms = 0;
        r = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        e->sms = std::max(1, sms);
        if (bf16 && r == cudaSuccess) {
            int occ = 0;
            r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, wgrad_tc_kernel, 256, wgrad_tc_smem_bytes());
            e->wgrad_slots = std::max(1, occ) * e->sms;
        }
    }
    if (r != cudaSuccess) {
        isr_est_destroy(e);
        return fail(r == cudaErrorMemoryAllocation ? ISR_ERR_NO_MEMORY : ISR_ERR_CUDA, "allocation failed: %s",
                    cudaGetErrorString(r));
    }
    *out = e;
    return ISR_OK;
}

isr_status isr_est_set_params(isr_est* e, const float* params)
{
    if (!e || !params) return fail(ISR_ERR_INVALID_ARG, "NULL argument");
    Dev guard(e->dev);
    EST_TRY(cudaMemcpyAsync(e->theta, params, 4 * NPARAM, cudaMemcpyDefault, e->stream));
    EST_TRY(cudaMemsetAsync(e->m, 0, 4 * NPARAM, e->stream));
    EST_TRY(cudaMemsetAsync(e->v, 0, 4 * NPARAM, e->stream));
    EST_TRY(cudaStreamSynchronize(e->stream));
    e->step = 0;
    e->weights_stale = true;
    return ISR_OK;
}

isr_status isr_est_get_params(isr_est* e, float* params)
{
    if (!e || !params) return fail(ISR_ERR_INVALID_ARG, "NULL argument");
    Dev guard(e->dev);
    EST_TRY(cudaMemcpyAsync(params, e->theta, 4 * NPARAM, cudaMemcpyDefault, e->stream));
    EST_TRY(cudaStreamSynchronize(e->stream));
    return check_waits(e);
}

isr_status isr_est_features(isr_est* e, const float* spectra, int32_t n, float* x)
{
    if (!e || !spectra || !x || n < 1) return fail(ISR_ERR_INVALID_ARG, "bad arguments");
    Dev guard(e->dev);
    features_kernel<<<n, FT_THREADS, 0, e->stream>>>(spectra, e->nfft, e->lo, e->L, x);
    EST_TRY(cudaGetLastError());
    return ISR_OK;
}

isr_status isr_est_grad(isr_est* e, const float* x, int32_t n, const float* line_bin, const float* present,
                        float* loss, float* grad)
{
    isr_status st = check_batch(e, x, n);
    if (st != ISR_OK) return st;
    if (!line_bin || !present) return fail(ISR_ERR_INVALID_ARG, "labels must not be NULL");
    Dev guard(e->dev);
    st = e->precision != ISR_EST_FP32 ? forward_t<__nv_bfloat16>(e, x, n) : forward_t<float>(e, x, n);
    if (st == ISR_OK)
        st = e->precision != ISR_EST_FP32 ? backward_t<__nv_bfloat16>(e, n, line_bin, present)
                                          : backward_t<float>(e, n, line_bin, present);
    if (st != ISR_OK) return st;
    if (grad) EST_TRY(cudaMemcpyAsync(grad, e->grad, 4 * NPARAM, cudaMemcpyDefault, e->stream));
    if (loss) EST_TRY(cudaMemcpyAsync(loss, e->loss, 4, cudaMemcpyDefault, e->stream));
    EST_TRY(cudaStreamSynchronize(e->stream));
    return check_waits(e);
}

isr_status isr_est_train_step(isr_est* e, const float* x, int32_t n, const float* line_bin, const float* present,
                              float lr, float* loss)
{
    isr_status st = check_batch(e, x, n);
    if (st != ISR_OK) return st;
    if (!line_bin || !present || !(lr > 0.f)) return fail(ISR_ERR_INVALID_ARG, "labels NULL or lr <= 0");
    Dev guard(e->dev);
    st = check_waits(e);
    if (st != ISR_OK) return st;
    st = e->precision != ISR_EST_FP32 ? forward_t<__nv_bfloat16>(e, x, n) : forward_t<float>(e, x, n);
    if (st == ISR_OK)
        st = e->precision != ISR_EST_FP32 ? backward_t<__nv_bfloat16>(e, n, line_bin, present)
                                          : backward_t<float>(e, n, line_bin, present);
    if (st != ISR_OK) return st;
    e->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f / (1.f - powf(b1, (float)e->step)), c2 = 1.f / (1.f - powf(b2, (float)e->step));
    adam_kernel<<<(NPARAM + 255) / 256, 256, 0, e->stream>>>(e->theta, e->grad, e->m, e->v, NPARAM, lr, b1, b2, 1e-8f,
                                                              c1, c2, e->status);
    e->weights_stale = true;
    EST_TRY(cudaGetLastError());
    if (loss) {
        EST_TRY(cudaMemcpyAsync(loss, e->loss, 4, cudaMemcpyDefault, e->stream));
        EST_TRY(cudaStreamSynchronize(e->stream));
        return check_waits(e);
    }
    return ISR_OK;
}

isr_status isr_est_predict(isr_est* e, const float* x, int32_t n, float* line_bin, float* presence)
{
    isr_status st = check_batch(e, x, n);
    if (st != ISR_OK) return st;
    if (!line_bin || !presence) return fail(ISR_ERR_INVALID_ARG, "outputs must not be NULL");
    Dev guard(e->dev);
    st = check_waits(e);
    if (st != ISR_OK) return st;
    return e->precision != ISR_EST_FP32 ? forward_t<__nv_bfloat16>(e, x, n, line_bin, presence)
                                        : forward_t<float>(e, x, n, line_bin, presence);
}

isr_status isr_est_predict_all(isr_est* e, const float* x, int64_t n, float* line_bin, float* presence)
{
    isr_status st = check_batch(e, x, 1);
    if (st != ISR_OK) return st;
    if (n < 1) return fail(ISR_ERR_INVALID_ARG, "n must be >= 1");
    if (!line_bin || !presence) return fail(ISR_ERR_INVALID_ARG, "outputs must not be NULL");
    Dev guard(e->dev);
    st = check_waits(e);
    const int most = e->conv05 ? predict_rows(e) : e->max_batch;
    for (int64_t done = 0; done < n && st == ISR_OK; done += most) {
        const int rows = (int)std::min<int64_t>(most, n - done);
        const float* xr = x + done * e->L;
        st = e->precision != ISR_EST_FP32 ? forward_t<__nv_bfloat16>(e, xr, rows, line_bin + done, presence + done)
                                          : forward_t<float>(e, xr, rows, line_bin + done, presence + done);
    }
    return st;
}

isr_status isr_est_test_drop_products(isr_est* e, int32_t pass, uint32_t polls)
{
    if (!e || pass < -1 || pass > 2 || (pass >= 0 && polls == 0))
        return fail(ISR_ERR_INVALID_ARG, "estimator is NULL, pass not in -1..2 or polls is 0");
    Dev guard(e->dev);
    if (pass >= 0) {
        const isr_status st = set_tc05_attrs<true>();
        if (st != ISR_OK) return st;
    }
    e->drop_pass = pass;
    e->wait_limit = pass >= 0 ? polls : 1u << 26;
    return ISR_OK;
}

void isr_est_destroy(isr_est* e)
{
    if (!e) return;
    Dev guard(e->dev);
    cudaStreamSynchronize(e->stream);
    void* ptrs[] = {e->theta, e->m, e->v, e->grad, e->wcopies, e->wf, e->wb, e->tf, e->tb, e->act[0], e->act[1], e->act[2], e->act[3],
                    e->act[4], e->z, e->pooled, e->u, e->q, e->loss, e->amax, e->da[0], e->da[1], e->da[2], e->da[3],
                    e->pmax, e->pidx, e->psum, e->hscal, e->dpool, e->zmax, e->zidx, e->hbits, e->status};
    for (void* p : ptrs) cudaFree(p);
    isr::give_status(e->host_status);
    cudaGetLastError();
    delete e;
}

}  // extern "C"
