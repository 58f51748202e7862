// isr_ff.cuh -- float-float arithmetic: values held as an unevaluated sum of two FP32 numbers.
//
// This part runs FP64 at about two operations per SM and clock (128 in FP32), so reductions and
// logarithms that need more than 24 bits run on pairs of floats: error-free sums (Knuth's TwoSum,
// Dekker's FastTwoSum) and products (one FMA gives the rounding error), about 2^-47 relative.
#pragma once

#include <cstdint>

namespace isr {

struct ff {
    float h, l;   // value h + l, |l| <= ulp(h) / 2 after ff_norm
};

// s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// the same for |a| >= |b| (or a = 0)
__device__ __forceinline__ ff ff_norm(float a, float b)
{
    const float s = a + b;
    return ff{s, b - (s - a)};
}

__device__ __forceinline__ ff ff_add(ff a, ff b)
{
    float s, e;
    two_sum(a.h, b.h, s, e);
    return ff_norm(s, e + (a.l + b.l));
}

// a + x for a running sum: x enters exactly, the error goes to the low word
__device__ __forceinline__ void ff_acc(ff& a, float x)
{
    float s, e;
    two_sum(a.h, x, s, e);
    a.h = s;
    a.l += e;
}

// a * b
__device__ __forceinline__ ff ff_mul(ff a, ff b)
{
    const float p = __fmul_rn(a.h, b.h);
    const float e = fmaf(a.h, b.h, -p);
    return ff_norm(p, fmaf(a.h, b.l, fmaf(a.l, b.h, e)));
}

__device__ __forceinline__ ff ff_of(double v)
{
    const float h = (float)v;
    return ff{h, (float)(v - (double)h)};
}

__device__ __forceinline__ double ff_to_double(ff a) { return (double)a.h + (double)a.l; }

__device__ __forceinline__ ff ff_shfl_xor(ff a, int o)
{
    return ff{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}

// sum over the warp, in every lane
__device__ __forceinline__ ff ff_warp_sum(ff a)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) a = ff_add(a, ff_shfl_xor(a, o));
    return a;
}

// ---------------------------------------------------------------- logarithm
// ln of a positive normal float to about 2^-44 absolute, after Tang's table-driven scheme
// (ACM TOMS 16, 1990): v = 2^k m, m in [1, 2); a 10-bit c ~ 1 / m from the top 7 mantissa bits;
// ln v = k ln 2 - ln c + ln(1 + r), r = m c - 1 exactly as a pair, |r| < 2^-7.
struct LnTable {
    float c[128];    // 1 / (1 + (i + 1/2) / 128) rounded to a multiple of 2^-10
    float nh[128];   // -ln c, high and low word
    float nl[128];
    // ln x by the series 2 atanh((x - 1) / (x + 1)), x in [1, 2]
    __host__ __device__ static constexpr double ln(double x)
    {
        const double t = (x - 1.0) / (x + 1.0), t2 = t * t;
        double p = 0.0;
        for (int k = 35; k >= 0; --k) p = p * t2 + 1.0 / double(2 * k + 1);
        return 2.0 * t * p;
    }
    __host__ __device__ constexpr LnTable() : c{}, nh{}, nl{}
    {
        for (int i = 0; i < 128; ++i) {
            const double inv = 1.0 / (1.0 + (i + 0.5) / 128.0);
            const double r = double(int(inv * 1024.0 + 0.5)) / 1024.0;
            const double l = ln(1.0 / r);
            c[i] = float(r);
            nh[i] = float(l);
            nl[i] = float(l - double(nh[i]));
        }
    }
};

// t: a copy of LnTable in shared memory
__device__ __forceinline__ ff ff_log(float v, const LnTable& t)
{
    constexpr double kLn2 = LnTable::ln(2.0);
    // ln 2 in three words; the first two carry 14 bits each, so their products with k are exact
    constexpr float l0 = float(int(kLn2 * 16384.0)) / 16384.f;
    constexpr float l1 = float(int((kLn2 - l0) * 268435456.0)) / 268435456.f;
    constexpr float l2 = float(kLn2 - l0 - l1);
    const uint32_t b = __float_as_uint(v);
    const float k = (float)((int)(b >> 23) - 127);
    const int i = (int)((b >> 16) & 127u);
    const float m = __uint_as_float((b & 0x007fffffu) | 0x3f800000u);
    const float c = t.c[i];
    const float p = __fmul_rn(m, c);
    const float rl = fmaf(m, c, -p);
    const float r = p - 1.f;   // exact: p is within 2^-7 of 1
    // ln(1 + r + rl) = r + rl (1 - r + r^2) - r^2 / 2 + r^3 (1/3 - r/4 + r^2/5 - r^3/6 + r^4/7)
    const float q = __fmul_rn(r, r);
    const float qe = fmaf(r, r, -q);
    const float w = fmaf(r, fmaf(r, fmaf(r, fmaf(r, 1.f / 7.f, -1.f / 6.f), 0.2f), -0.25f), 1.f / 3.f);
    float lo = fmaf(__fmul_rn(q, r), w, fmaf(-0.5f, qe, rl * fmaf(r, r - 1.f, 1.f)));
    float s, e;
    two_sum(__fmul_rn(k, l0), t.nh[i], s, e);
    lo += e + t.nl[i];
    two_sum(s, r, s, e);
    lo += e;
    two_sum(s, __fmul_rn(k, l1), s, e);
    lo += e;
    two_sum(s, __fmul_rn(-0.5f, q), s, e);
    lo += fmaf(k, l2, e);
    return ff_norm(s, lo);
}

}  // namespace isr
