// isr_xt.cuh -- the fused kernel for nfft 1024 .. 16384 with the last exchange of the transform in
// tensor memory.
//
// The Stockham kernels of isr_kernel.cuh move every value of a three-pass transform through shared
// memory twice, and their time follows the sum of the issue slots and the shared-memory wavefronts,
// which hardly overlap.  Tensor memory (TMEM) has its own data path: a warp that stores with the
// 16x256b shape and loads with the 32x32b shape trades two of its lane bits for two register bits, and
// the warps that share a lane quarter trade two more through the columns.  Those four index bits are
// what a last pass of up to radix 16 needs, so only the exchange before the middle pass (five bits)
// goes through shared memory.
//
// nfft = N = 32 x 32 x RL (RL = 16, 8, 4, 2, 1 for N = 16384 .. 1024), 32 points per thread, T = N / 32
// threads per gate, A = RL / 4 (at least 1) warps of a gate per lane quarter.  With u = n mod 32 and
// k = n / 32 of the middle pass' butterfly n < T, thread (quarter s, block a < A, lane 4 v + c):
//   pass 0   thread t: 32-point DFT of x[t + T k0], output q0 to shared slot 33 t + q0;
//   middle   RL >= 4: u = s + 4 v, k = c + 4 a; RL = 2: u = (s & 1) + 2 (c >> 1) + 4 v, k = c & 1;
//            RL = 1: u = lane; reads slots 33 k + u + (33 T / 32) k1 (free of bank conflicts),
//            twiddle W_1024^{u k1}, 32-point DFT;
//   exchange output q = m + 4 a' + 4 A e goes to row v + 8 m, columns of block a'; thread (s, a',
//            lane 8 m + v) receives all c and a, and its e < 8 / A;
//   last     RL >= 4: j2 = s + 4 lane + 128 a' + 128 A e, k = c + 4 a; RL = 2: j2 = (s & 1) + 2 (c >> 1) +
//            4 lane + 128 e, k = c & 1; twiddle W_N^{j2 k}, RL-point DFT, bins j2 + 1024 q.
// The twiddles of both passes stand in TMEM too (at 16384 the last of them in shared memory, because
// 256 exchange columns + 64 + 4 x 48 fill the 512 columns).
//
// Measured (binary-phase code, M spectra/s; before: the best Stockham order of that size): nfft 16384
// 31.6 -> 34.2, 8192 66.4 -> 78.9, 4096 147 -> 170, 2048 322 -> 370, 1024 750 -> 842; with a code per IPP
// 16384 18.2 -> 33.9, 2048 190 -> 365, 1024 383 -> 830; complex int16 codes at 4096 105-120 -> 149.  At
// 16384 it issues on 74 % of cycles with the FMA pipe at 55 % and shared-memory wavefronts at 31 %
// (before: 76, 57 and 47 %, with 1,853 instead of 1,668 instructions per warp and transform): one
// transform fills the register file, so its load phases still run beside little else, while the gates of
// the smaller sizes fill each other's.  The paired FP32 instructions on (re, im), an mbarrier in place of
// the barrier at the top of an IPP, and wider TMEM stores (which need copies into consecutive registers)
// each measured slower.
#pragma once

#include "isr_kernel.cuh"

namespace isr {

// ---------------------------------------------------------------- tensor-memory accesses
// One 16x256b group of two complex values: lanes 4 v + c hold (row v, columns 2 c, 2 c + 1) and
// (row v + 8, the same columns).
__device__ __forceinline__ void tmem_st_16x256(uint32_t taddr, float2 z0, float2 z1)
{
    asm volatile("tcgen05.st.sync.aligned.16x256b.x1.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "f"(z0.x), "f"(z0.y),
                 "f"(z1.x), "f"(z1.y)
                 : "memory");
}
// Eight consecutive columns of this thread's lane: store; load and wait.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
                 "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_ld8_wait(uint32_t taddr, float (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6]), "+f"(r[7]));
}

// ---------------------------------------------------------------- twiddles
// Twiddles of group I of a radix-R pass (elements k = I + m R / 4): element I as a complex factor,
// the others as cos (1 + i tan): the tangents are applied with two FMAs each and the cosines ride on
// the first level's additions (sdft_first), two instructions per twiddle fewer than a complex product.
// A vanishing cosine is replaced by 2^-40, which leaves its term's relative error at one rounding.
struct TwGroup {
    float w[8];   // wr, wi of k = I; tangents of m = 1, 2, 3; cos 1, cos 2, cos 3 / cos 1
};

// exp(-2 pi i n / period), period a power of two, rounded from 64 bits
__device__ __forceinline__ float2 unit_root(int n, int period)
{
    double sn, cs;
    sincospi(-2.0 * (double)(n & (period - 1)) / (double)period, &sn, &cs);
    return make_float2((float)cs, (float)sn);
}

// the group of elements I + m R / 4 with the twiddles exp(-2 pi i n k / period)
template <int R>
__device__ __forceinline__ TwGroup tw_group(int I, int n, int period)
{
    TwGroup g;
    float c[4];
    for (int m = 0; m < 4; ++m) {
        const float2 w = unit_root(n * (I + m * (R / 4)), period);
        if (m == 0) {
            g.w[0] = w.x;
            g.w[1] = w.y;
        } else {
            c[m] = fabsf(w.x) < 0x1p-40f ? 0x1p-40f : w.x;
            g.w[1 + m] = w.y / c[m];
        }
    }
    g.w[5] = c[1];
    g.w[6] = c[2];
    g.w[7] = c[3] / c[1];
    return g;
}

// Group I of a radix-R pass from its twiddles: products and the first level of the transform.
template <int R, int I>
__device__ __forceinline__ void tw_first(float2* v, const float (&w)[8])
{
    constexpr int Q = R / 4;
    if constexpr (I > 0) v[I] = cmul(v[I], make_float2(w[0], w[1]));
    static_for<3>([&](auto Mc) {
        constexpr int m = decltype(Mc)::value + 1;
        const float2 x = v[I + m * Q];
        v[I + m * Q] = make_float2(fmaf(-w[1 + m], x.y, x.x), fmaf(w[1 + m], x.x, x.y));
    });
    sdft_first<R, I>(v, w[5], w[6], w[7]);
}

// ---------------------------------------------------------------- decode
// An echo sample as floats (exact): the conversion instruction, or sign extension on the integer pipe
// and a full-width conversion.  The first runs at four lanes per cycle and scheduler, so half of the
// samples take either form (all by the first 33.2, all by the second 33.8, odd ones by the second 33.6,
// the upper half 34.1 M spectra/s at nfft 16384).
template <bool ALU>
__device__ __forceinline__ float2 sample(uint32_t w)
{
    if constexpr (!ALU) {
        return iq_of(w);
    } else {
        int i, q;
        asm("prmt.b32 %0, %1, 0, 0x9910;" : "=r"(i) : "r"(w));   // low half, sign-extended
        asm("shr.s32 %0, %1, 16;" : "=r"(q) : "r"(w));
        return make_float2((float)i, (float)q);
    }
}

// Chip signs of a binary-phase code as thread t of a gate uses them: bit k < 24 set where chip
// t + T k is -1, bits 24 .. 31 the sign of chip k times that of chip k - 16 (sdft_first takes the third
// factor of a group relative to the first).
template <int T>
__device__ __forceinline__ uint32_t chip_signs(const int8_t* row, int t, int code_len)
{
    uint32_t m = 0;
    static_for<32>([&](auto Kc) {
        constexpr int k = decltype(Kc)::value;
        const int pos = t + T * k;
        if (pos < code_len && row[pos] < 0) m |= 1u << k;
    });
    return m ^ ((m << 16) & 0xff000000u);
}

// The same for every row of per-IPP codes, [rows][T] words: one load per thread and IPP in the fused
// kernel instead of 32 byte loads (at nfft 1024 those took as long as the transform).
template <int T>
__global__ void __launch_bounds__(256) pack_signs_kernel(const int8_t* __restrict__ tx, int64_t tx_stride, int code_len,
                                                         int rows, uint32_t* __restrict__ words)
{
    const int64_t n = (int64_t)rows * T;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
        words[i] = chip_signs<T>(tx + (i / T) * tx_stride, (int)(i & (T - 1)), code_len);
}

// ---------------------------------------------------------------- schedule
template <int LOG2N>
struct SchedX {
    static constexpr int N = 1 << LOG2N;
    static constexpr int T = N / 32;            // threads per gate
    static constexpr int G = kThreads / T;      // gates per CTA
    static constexpr int RL = N / 1024;         // radix of the last pass
    static constexpr int NE = 32 / RL;          // its butterflies per thread
    static constexpr int A = RL / 4 > 1 ? RL / 4 : 1;   // warps of a gate per lane quarter
    static constexpr int KSTRIDE = T + T / 32;  // padded distance of slots k1, k1 + 1
    // twiddle groups (8 words): 8 of the middle pass; QL per last-pass butterfly (RL = 2: one per four)
    static constexpr int QL = RL >= 4 ? RL / 4 : 1;
    static constexpr int NGRP = LOG2N == 14 ? 6 : RL >= 4 ? NE * QL : RL == 2 ? 4 : 0;   // last-pass groups in TMEM
    // TMEM columns: the exchange (64 per warp of a quarter), the middle pass' groups, the last pass'
    static constexpr int COL_TW1 = 256, COL_TW2 = 320, TW2 = NGRP * 8;
    static_assert(COL_TW2 + A * TW2 <= 512, "TMEM columns");
    static constexpr int STAGE_WORDS = N + 4;
    static constexpr int OFF_MBAR = 0;          // slot g: the staged window of gate g
    static constexpr int OFF_UNIT = 128;        // XtUnit [G][2]
    static constexpr int OFF_STAGE = OFF_UNIT + 96 * 2 * G;
    static constexpr int OFF_XCH = OFF_STAGE + 4 * STAGE_WORDS * G;
    static constexpr int NPAD = N + N / 32;
    // nfft 16384: groups 0 and 1 of butterfly 1 per thread
    static constexpr int OFF_TWS = OFF_XCH + 8 * NPAD * G;
    static constexpr int SMEM = OFF_TWS + (LOG2N == 14 ? (16 + 8 + 16 + 16) * kThreads : 0);
    static_assert(SMEM <= 232448, "shared memory");
    static_assert(LOG2N >= 10 && LOG2N <= 14, "nfft 1024 .. 16384");
    static_assert(OFF_XCH % 16 == 0 && OFF_STAGE % 16 == 0 && STAGE_WORDS % 4 == 0 && OFF_TWS % 16 == 0, "alignment");
};

// The twiddle groups as the threads of a CTA keep them, [group][half][128 blk + 32 s + lane]: the same for
// every launch, filled once per context (xt_tables_kernel), so that a CTA starts with a few loads
// instead of some forty sines and thirty quotients per thread (a launch of 8 gates x 1 IPP at nfft 16384:
// 17.9 us formed in the kernel, 14.0 us loaded).
template <int LOG2N>
struct XtTables {
    float4 mid[8][2][128];
    float4 last[LOG2N == 14 ? 8 : SchedX<LOG2N>::NGRP + (LOG2N == 10)][2][128 * SchedX<LOG2N>::A];
};
template <int LOG2N>
__device__ XtTables<LOG2N> g_xt_tables;

template <int LOG2N>
__global__ void xt_tables_kernel()
{
    using S = SchedX<LOG2N>;
    constexpr int RL = S::RL, A = S::A;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 8 * 128; i += gridDim.x * blockDim.x) {
        const int I = i / 128, s = i / 32 % 4, lane = i % 32, v4 = 4 * (lane >> 2);
        const int u = RL >= 4 ? s + v4 : RL == 2 ? (s & 1) + (lane & 2) + v4 : lane;
        const TwGroup g = tw_group<32>(I, u, 1024);
        g_xt_tables<LOG2N>.mid[I][0][i % 128] = make_float4(g.w[0], g.w[1], g.w[2], g.w[3]);
        g_xt_tables<LOG2N>.mid[I][1][i % 128] = make_float4(g.w[4], g.w[5], g.w[6], g.w[7]);
    }
    constexpr int NG = LOG2N == 14 ? 8 : S::NGRP;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NG * 128 * A; i += gridDim.x * blockDim.x) {
        const int gr = i / (128 * A), at = i % (128 * A), s = at / 32 % 4, lane = at % 32, blk = at / 128;
        TwGroup g;
        if constexpr (RL >= 4) {
            const int e = gr / S::QL, j2 = s + 4 * lane + 128 * blk + 128 * A * e;
            g = tw_group<RL>(gr % S::QL, j2, S::N);
        } else {
            // radix 2: (tangent, cosine) of butterflies (e, c >> 1) = (2 gr, 0), (2 gr, 1), (2 gr + 1, 0), (2 gr + 1, 1)
            for (int b = 0; b < 4; ++b) {
                const float2 w = unit_root((s & 1) + 4 * lane + 2 * (b & 1) + 128 * (2 * gr + (b >> 1)), S::N);
                const float c = fabsf(w.x) < 0x1p-40f ? 0x1p-40f : w.x;
                g.w[2 * b] = w.y / c;
                g.w[2 * b + 1] = c;
            }
        }
        g_xt_tables<LOG2N>.last[gr][0][at] = make_float4(g.w[0], g.w[1], g.w[2], g.w[3]);
        g_xt_tables<LOG2N>.last[gr][1][at] = make_float4(g.w[4], g.w[5], g.w[6], g.w[7]);
    }
}

// One gate's share of a work unit (some IPPs of one gate), in shared memory: 64 data and 32
// accumulator registers leave few of the 128 for what lives across an IPP.
struct XtUnit {
    const uint32_t* src;     // first staged word of the unit's first row (16-byte boundary)
    int64_t stride;          // words between rows
    const char* tx;          // code of the first row
    int64_t tx_stride;       // bytes between code rows, 0 = one code
    const uint32_t* signs;   // packed chip signs of the first row, [row][T], or NULL
    float* out;              // [N] partial sums; NULL for a gate beyond the last
    uint32_t bytes;          // of a staged window
    int off;                 // the window's first sample within the stage
    int code_len;
    int n;                   // IPPs
    int un;                  // index of the unit in its launch
    uint32_t it0;            // IPPs of this gate before the unit
    int wipe;                // the stage behind the code may hold samples of another unit
    int drop;                // test hook: the IPP that is never staged, -1 = none
    int ok;                  // debug builds: the window lies in its row
};
static_assert(sizeof(XtUnit) <= 96, "OFF_UNIT");

template <int LOG2N>
__device__ __forceinline__ void xt_fill(XtUnit& x, const KArgs& a, int gx, int c, int g, int t)
{
    using S = SchedX<LOG2N>;
    const int r = gx * S::G + g;
    const int64_t s_r = (int64_t)a.range_start + (int64_t)min(r, a.n_ranges - 1) * a.range_step;
    const int p0 = c * a.chunk_len;
    x.off = (int)(s_r & 3);
    x.bytes = (uint32_t)(((x.off + a.code_len + 3) & ~3) * 4);
    x.src = a.echo + (int64_t)p0 * a.echo_stride + (s_r - x.off);
    x.stride = a.echo_stride;
    x.tx_stride = a.tx_stride * a.chip_bytes;
    x.tx = static_cast<const char*>(a.tx) + (int64_t)p0 * x.tx_stride;
    x.signs = a.signs ? a.signs + (int64_t)p0 * S::T : nullptr;
    x.out = r < a.n_ranges ? a.partial + ((int64_t)c * a.n_ranges + r) * S::N : nullptr;
    x.code_len = a.code_len;
    x.n = min(a.chunk_len, a.n_ipp - p0);
    x.drop = a.drop_ipp >= p0 && a.drop_ipp < p0 + x.n ? a.drop_ipp - p0 : -1;
    x.ok = debug_window_ok(a, s_r, x.off, x.bytes, S::STAGE_WORDS, t);
}

// Work of a launch over one window: CTA b takes units b, b + gridDim.x, ... of the (gate group, IPP
// chunk) grid, gate groups first.
struct XtPlanSrc {
    KArgs a;
    // units unit0 .. n_units - 1 of rg gate groups x IPP chunks; unit0 is 0, but without it the kernel is
    // compiled to one that takes 0.3 % longer (nfft 16384: 291.5 -> 292.5 ms for 1000 gates x 10,000 IPPs)
    int rg, unit0, n_units;
    __device__ __forceinline__ int first() const { return unit0 + blockIdx.x; }
    __device__ __forceinline__ int next(int un) const { return un + gridDim.x; }
    __device__ __forceinline__ bool valid(int un) const { return un < n_units; }
    template <int LOG2N>
    __device__ __forceinline__ void fill(XtUnit& x, int un, int g, int t) const
    {
        xt_fill<LOG2N>(x, a, un % rg, un / rg, g, t);
    }
    __device__ __forceinline__ unsigned wait_limit() const { return a.wait_limit; }
    __device__ __forceinline__ int* status() const { return a.status; }
    __device__ __forceinline__ unsigned long long* phase_cycles() const { return a.phase_cycles; }
};

// Work of a batch: CTA b takes units [first[b], first[b + 1]) of windows of one nfft.
struct BatchWin {
    KArgs a;
    int log2n;
    int order;
    int n_gx;   // gate groups
    int n_cy;   // IPP chunks
};
struct BatchUnit {
    int win, gx, cy, pad;
};
struct XtBatchSrc {
    const BatchWin* wins;
    const BatchUnit* units;
    const int* starts;
    unsigned limit;
    int* stat;
    __device__ __forceinline__ int first() const { return __ldg(starts + blockIdx.x); }
    __device__ __forceinline__ int next(int un) const { return un + 1; }
    __device__ __forceinline__ bool valid(int un) const { return un < __ldg(starts + blockIdx.x + 1); }
    template <int LOG2N>
    __device__ __forceinline__ void fill(XtUnit& x, int un, int g, int t) const
    {
        const BatchUnit u = units[un];
        xt_fill<LOG2N>(x, wins[u.win].a, u.gx, u.cy, g, t);
    }
    __device__ __forceinline__ unsigned wait_limit() const { return limit; }
    __device__ __forceinline__ int* status() const { return stat; }
    __device__ __forceinline__ unsigned long long* phase_cycles() const { return nullptr; }
};

// ---------------------------------------------------------------- the kernel
// Persistent, one CTA per SM: the twiddles are set up once per CTA, and the first window of a unit is in
// flight while the unit before it ends.
template <int LOG2N, int TXT, class SRC>
__global__ void __launch_bounds__(kThreads, 1) integrate_kernel_xt(const __grid_constant__ SRC work)
{
    using S = SchedX<LOG2N>;
    constexpr int N = S::N, T = S::T, G = S::G, RL = S::RL, NE = S::NE, A = S::A;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint32_t tslot;
    uint64_t* mbar = reinterpret_cast<uint64_t*>(smem + S::OFF_MBAR);
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int g = warp / (T / 32), t = tid - g * T;
    uint32_t* stage = reinterpret_cast<uint32_t*>(smem + S::OFF_STAGE) + g * S::STAGE_WORDS;
    float2* xch = reinterpret_cast<float2*>(smem + S::OFF_XCH) + g * S::NPAD;
    XtUnit* units = reinterpret_cast<XtUnit*>(smem + S::OFF_UNIT) + 2 * g;   // the current unit and the next
    const uint32_t bar = smem_u32(&mbar[g]);
    auto issue = [&](const XtUnit& x, int i) {   // thread 0 of the gate: the window of the unit's row i
        if (x.ok && i != x.drop) bulk_load(smem_u32(stage), x.src + i * x.stride, x.bytes, bar);
    };

    auto begin = [&](XtUnit& x, int un, uint32_t it0) {   // thread 0 of the gate: unit un, its first window
        work.template fill<LOG2N>(x, un, g, t);
        x.un = un;
        x.it0 = it0;
        // words behind a short code are cleared once, and again after a unit with a longer one
        x.wipe = x.code_len < N && (it0 == 0 || units[&x == units].code_len > x.code_len);
        issue(x, 0);
    };
    const bool any = work.valid(work.first());
    if (t == 0) {   // the first window is on its way while the twiddles are brought
        mbar_init(bar, 1);
        fence_barrier_init();
        if (any) begin(units[0], work.first(), 0u);
    }
    if (warp == kThreads / 32 - 1) tmem_alloc(smem_u32(&tslot), 512);   // all columns: the allocation's base is 0
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();

    // this thread's place in the middle and last passes
    const int s = warp & 3, blk = (warp >> 2) & (A - 1);
    const int c = lane & 3, v4 = 4 * (lane >> 2);
    const int u = RL >= 4 ? s + v4 : RL == 2 ? (s & 1) + (c & 2) + v4 : lane;
    const int k = RL >= 4 ? c + 4 * blk : RL == 2 ? c & 1 : 0;
    const int j2 = RL >= 4 ? s + 4 * lane + 128 * blk : (s & 1) + 4 * lane;
    const uint32_t tq = (uint32_t)(32 * s) << 16;                   // lane quarter of this warp
    const uint32_t t_ld = tq + 64u * (warp >> 2);                   // its exchange columns
    const uint32_t t_st = tq + 64u * ((warp >> 2) - blk) + (uint32_t)(64 / A) * blk;   // + 64 a'
    const uint32_t t_tw1 = tq + S::COL_TW1;
    const uint32_t t_tw2 = tq + S::COL_TW2 + (uint32_t)S::TW2 * blk;

    // twiddle groups, each brought by one of the warps that share it
    float4* tws = reinterpret_cast<float4*>(smem + S::OFF_TWS) + tid;                       // nfft 16384, [3][512]
    float2* tws2 = reinterpret_cast<float2*>(smem + S::OFF_TWS + 48 * kThreads) + tid;
    const int at = 32 * s + lane;
    auto bring = [&](uint32_t col, const float4 (&p)[2][128 * A], int i) {
        const float4 a0 = __ldg(&p[0][i]), a1 = __ldg(&p[1][i]);
        const float w[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        tmem_st8(col, w);
    };
    static_for<2>([&](auto Hc) {
        const int I = (warp >> 2) + 4 * decltype(Hc)::value;
        const float4 a0 = __ldg(&g_xt_tables<LOG2N>.mid[I][0][at]), a1 = __ldg(&g_xt_tables<LOG2N>.mid[I][1][at]);
        const float w[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        tmem_st8(t_tw1 + 8 * I, w);
    });
    if constexpr (LOG2N == 14) {
        static_for<6>([&](auto Ic) {
            constexpr int i = decltype(Ic)::value;
            bring(t_tw2 + 8 * i, g_xt_tables<LOG2N>.last[i < 4 ? i : i + 2], at + 128 * blk);
        });
        const auto& p = g_xt_tables<LOG2N>.last;
        const float4 a0 = __ldg(&p[4][0][at + 128 * blk]), a1 = __ldg(&p[4][1][at + 128 * blk]);
        tws[0] = make_float4(a0.z, a0.w, a1.x, a1.y);
        *tws2 = make_float2(a1.z, a1.w);
        tws[kThreads] = __ldg(&p[5][0][at + 128 * blk]);
        tws[2 * kThreads] = __ldg(&p[5][1][at + 128 * blk]);
    } else if constexpr (RL >= 2) {
        static_for<S::NGRP / (4 / A)>([&](auto Ic) {
            const int i = (warp >> 2) / A + (4 / A) * decltype(Ic)::value;
            bring(t_tw2 + 8 * i, g_xt_tables<LOG2N>.last[i], at + 128 * blk);
        });
    }
    tmem_wait_st();
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();

    auto gsync = [&]() {
        if constexpr (T == 32) __syncwarp();
        else if constexpr (G == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(T) : "memory");
    };
    auto gsync_or = [&](bool pred) -> bool {
        if constexpr (T == 32) {
            return __any_sync(0xffffffffu, pred);
        } else if constexpr (G == 1) {
            return __syncthreads_or(pred) != 0;
        } else {
            uint32_t any;
            asm volatile(
                "{\n\t.reg .pred p, q;\n\t"
                "setp.ne.u32 p, %1, 0;\n\t"
                "bar.red.or.pred q, %2, %3, p;\n\t"
                "selp.u32 %0, 1, 0, q;\n\t}"
                : "=r"(any)
                : "r"((uint32_t)pred), "r"(1 + g), "n"(T)
                : "memory");
            return any != 0;
        }
    };
    // the A warps of a gate that share a lane quarter
    auto qsync = [&]() {
        if constexpr (A > 1) asm volatile("bar.sync %0, %1;" ::"r"((G == 1 ? 1 : 1 + G) + 4 * g + s), "n"(32 * A) : "memory");
    };

    const float2* x_ld = xch + 33 * k + u;
    bool timed_out = false;
    uint32_t it = 0;   // IPPs of this gate so far; units alternate between the two slots
    uint32_t signs = 0;
#ifdef ISR_DEBUG
    long long ph[4] = {0, 0, 0, 0}, tq0 = 0, tq1 = 0, tq2 = 0, n_ph = 0;
#endif
    const XtUnit* x = units;
    bool more = any;
    while (more) {
        if constexpr (TXT == TX_PM1) {
            if (x->signs) signs = __ldg(x->signs + t);
            else signs = chip_signs<T>(reinterpret_cast<const int8_t*>(x->tx), t, x->code_len);
        }
        float acc[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = 0.f;

        for (; it - x->it0 != (uint32_t)x->n; ++it) {
#ifdef ISR_DEBUG
            const long long tz = clock64();
#endif
            const bool ok = mbar_wait(bar, it & 1u, work.wait_limit());
            gsync();   // the previous IPP's middle-pass reads of xch precede this IPP's stores
#ifdef ISR_DEBUG
            tq0 = clock64();
            ph[0] += tq0 - tz;
#endif
            float2 v[32];
            {
                // ---- pass 0: decode, 32-point DFT.  The samples behind a code shorter than nfft read as
                // zeros: a unit's first IPP clears them all if need be, and as copies are rounded to 16
                // bytes, every IPP what that left behind the last chip (at most 6 words).  A thread
                // clears the words that it alone reads.
                uint32_t* win = stage + x->off + t;
                const int L = x->code_len;
                if (L != N) {
                    const int d = (t - L) & (T - 1);
                    if (x->wipe && it == x->it0) {
                        for (int pos = L + d; pos < N; pos += T) win[pos - t] = 0u;
                        // the words that a unit with a larger offset reads beyond these
                        if (t < 4 && N + t >= x->off + L) stage[N + t] = 0u;
                        fence_proxy_async();
                    } else if (d < 6 && L + d < N) {
                        win[L + d - t] = 0u;
                        fence_proxy_async();
                    }
                }
                if constexpr (TXT == TX_PM1) {
                    static_for<8>([&](auto Ic) {
                        constexpr int I = decltype(Ic)::value;
                        auto bit = [&](int b) { return (signs << (31 - b)) & 0x80000000u; };
                        auto one = [&](int b) { return __uint_as_float(bit(b) ^ 0x3f800000u); };
                        static_for<4>([&](auto Mc) {
                            constexpr int kk = I + 8 * decltype(Mc)::value;
                            v[kk] = sample<(kk >= 16)>(win[T * kk]);
                        });
                        v[I].x = __uint_as_float(__float_as_uint(v[I].x) ^ bit(I));
                        v[I].y = __uint_as_float(__float_as_uint(v[I].y) ^ bit(I));
                        sdft_first<32, I>(v, one(I + 8), one(I + 16), one(I + 24));
                    });
                    sdft_rest<32>(v);
                } else {
                    const char* row = x->tx + (int64_t)(it - x->it0) * x->tx_stride;
                    static_for<32>([&](auto Kc) {
                        constexpr int kk = decltype(Kc)::value;
                        const int pos = t + T * kk;
                        // chips at or past code_len are the zero padding and are never read
                        float2 e = make_float2(0.f, 0.f);
                        if constexpr (TXT == TX_CI16) {
                            const uint32_t w = pos < L ? __ldg(reinterpret_cast<const uint32_t*>(row) + pos) : 0u;
                            e = sample<true>(w);
                        } else {
                            if (pos < L) e = __ldg(reinterpret_cast<const float2*>(row) + pos);
                        }
                        const float2 m = sample<(kk >= 16)>(win[T * kk]);
                        // conj(e) * m
                        v[kk] = make_float2(fmaf(e.x, m.x, e.y * m.y), fmaf(e.x, m.y, -e.y * m.x));
                    });
                    sdft<32>(v);
                }
            }
            store_strided<1, 32, 32>(xch, 32 * t, v);

            // window consumed, pass-0 outputs visible, and the vote on the window's wait
            if (gsync_or(!ok)) {
                timed_out = true;
                break;
            }
            if (t == 0) {
                const int i1 = (int)(it + 1 - x->it0);
                if (i1 < x->n) {
                    fence_proxy_async();
                    issue(*x, i1);
                } else if (work.valid(work.next(x->un))) {
                    fence_proxy_async();
                    begin(units[x == units], work.next(x->un), it + 1);
                }
            }
            if constexpr (TXT == TX_PM1) {
                if (x->tx_stride != 0 && (int)(it + 1 - x->it0) < x->n) {   // the next IPP's chips
                    const int64_t i1 = (int64_t)(it + 1 - x->it0);
                    if (x->signs) signs = __ldg(x->signs + i1 * T + t);
                    else signs = chip_signs<T>(reinterpret_cast<const int8_t*>(x->tx + i1 * x->tx_stride), t, x->code_len);
                }
            }
#ifdef ISR_DEBUG
            tq1 = clock64();
            ph[1] += tq1 - tq0;
#endif
            // ---- middle pass
            static_for<32>([&](auto Kc) {
                constexpr int kk = decltype(Kc)::value;
                v[kk] = x_ld[kk * S::KSTRIDE];
            });
            static_for<8>([&](auto Ic) {
                constexpr int I = decltype(Ic)::value;
                float w[8];
                tmem_ld8_wait(t_tw1 + 8 * I, w);
                tw_first<32, I>(v, w);
            });
            sdft_rest<32>(v);
            if constexpr (RL == 1) {
                static_for<32>([&](auto Qc) {
                    constexpr int q = decltype(Qc)::value;
                    const float2 X = v[BitRev<32>::at(q)];
                    acc[q] = fmaf(X.x, X.x, fmaf(X.y, X.y, acc[q]));
                });
#ifdef ISR_DEBUG
                tq2 = tq1;
#endif
            } else {
                // ---- exchange: output q = m + 4 b + 4 A e to row v + 8 m of block b
                static_for<A>([&](auto Bc) {
                    constexpr int b = decltype(Bc)::value;
                    static_for<2 * (8 / A)>([&](auto Hc) {
                        constexpr int h = decltype(Hc)::value & 1, e = decltype(Hc)::value >> 1;
                        constexpr int q = 2 * h + 4 * b + 4 * A * e;
                        tmem_st_16x256(t_st + 64u * b + 8u * e + ((uint32_t)(16 * h) << 16), v[BitRev<32>::at(q)],
                                       v[BitRev<32>::at(q + 1)]);
                    });
                });
                tmem_wait_st();
                if constexpr (A > 1) {
                    tmem_fence_before_sync();
                    qsync();
                    tmem_fence_after_sync();
                }
#ifdef ISR_DEBUG
                tq2 = clock64();
                ph[2] += tq2 - tq1;
#endif
                // ---- last pass: value (a, e, c) at complex column a (32 / A) + 4 e + c
                uint32_t w0[32], w1[32];
                tmem_ld32(t_ld, w0);
                tmem_ld32(t_ld + 32, w1);
                tmem_wait_ld32(w0);
                tmem_wait_ld32(w1);
                static_for<32>([&](auto Ic) {
                    constexpr int j = decltype(Ic)::value;
                    constexpr int ca = j / (32 / A), e = (j / 4) % (8 / A), cc = j & 3;
                    // RL >= 4: butterfly e, element k = c + 4 a; RL = 2: butterfly (e, c >> 1), element c & 1
                    constexpr int at = RL >= 4 ? e * RL + cc + 4 * ca : 4 * e + cc;
                    if constexpr (j < 16) v[at] = make_float2(__uint_as_float(w0[2 * j]), __uint_as_float(w0[2 * j + 1]));
                    else v[at] = make_float2(__uint_as_float(w1[2 * j - 32]), __uint_as_float(w1[2 * j - 31]));
                });
                if constexpr (RL == 2) {
                    static_for<4>([&](auto Gc) {
                        constexpr int gr = decltype(Gc)::value;
                        float w[8];
                        tmem_ld8_wait(t_tw2 + 8 * gr, w);
                        static_for<4>([&](auto Bc) {
                            constexpr int b = decltype(Bc)::value, at = 8 * gr + 2 * b;   // butterfly at / 2
                            const float2 x0 = v[at], x1 = v[at + 1];
                            const float2 y = make_float2(fmaf(-w[2 * b], x1.y, x1.x), fmaf(w[2 * b], x1.x, x1.y));
                            const float2 p = make_float2(fmaf(w[2 * b + 1], y.x, x0.x), fmaf(w[2 * b + 1], y.y, x0.y));
                            const float2 m = make_float2(fmaf(-w[2 * b + 1], y.x, x0.x), fmaf(-w[2 * b + 1], y.y, x0.y));
                            acc[at] = fmaf(p.x, p.x, fmaf(p.y, p.y, acc[at]));
                            acc[at + 1] = fmaf(m.x, m.x, fmaf(m.y, m.y, acc[at + 1]));
                        });
                    });
                } else {
                    static_for<NE>([&](auto Ec) {
                        constexpr int e = decltype(Ec)::value;
                        float2* z = v + e * RL;
                        static_for<S::QL>([&](auto Ic) {
                            constexpr int I = decltype(Ic)::value;
                            float w[8];
                            if constexpr (LOG2N == 14 && e == 1 && I == 0) {
                                const float4 p = tws[0];
                                const float2 q = *tws2;
                                w[2] = p.x, w[3] = p.y, w[4] = p.z, w[5] = p.w, w[6] = q.x, w[7] = q.y;
                            } else if constexpr (LOG2N == 14 && e == 1 && I == 1) {
                                const float4 p = tws[kThreads], q = tws[2 * kThreads];
                                w[0] = p.x, w[1] = p.y, w[2] = p.z, w[3] = p.w, w[4] = q.x, w[5] = q.y, w[6] = q.z, w[7] = q.w;
                            } else {
                                tmem_ld8_wait(t_tw2 + 8 * (LOG2N == 14 ? (e == 0 ? I : 2 + I) : e * S::QL + I), w);
                            }
                            tw_first<RL, I>(z, w);
                        });
                        sdft_rest<RL>(z);
                        static_for<RL>([&](auto Qc) {
                            constexpr int q = decltype(Qc)::value;
                            const float2 X = z[BitRev<RL>::at(q)];
                            acc[e * RL + q] = fmaf(X.x, X.x, fmaf(X.y, X.y, acc[e * RL + q]));
                        });
                    });
                }
            }
#ifdef ISR_DEBUG
            ph[3] += clock64() - tq2;
            ++n_ph;
#endif
        }
        if (timed_out) break;

        // ---- chunk partials to coalesced rows: bins lane + 32 q (RL = 1) straight from the registers,
        // else bins j2 + ... through the exchange buffer, one pad word per 32 against the stride of 4
        float* out = x->out;
        if constexpr (RL == 1) {
            gsync();
            if (out) {
#pragma unroll
                for (int q = 0; q < 32; ++q) out[lane + 32 * q] = acc[q];
            }
        } else {
            float* fx = reinterpret_cast<float*>(xch);
            gsync();
            float* fj = fx + j2 + (j2 >> 5);
            static_for<32>([&](auto Ic) {
                constexpr int b = decltype(Ic)::value;
                // RL >= 4: acc[e RL + q]; RL = 2: acc[4 e + 2 (c >> 1) + q]
                constexpr int o = RL >= 4 ? 128 * A * (b / RL) + 1024 * (b % RL) : 128 * (b >> 2) + 1024 * (b & 1);
                constexpr int d = RL == 2 ? b & 2 : 0;   // stays inside a group of four bins: no pad in between
                fj[o + o / 32 + d] = acc[b];
            });
            gsync();
            if (out) {
#pragma unroll
                for (int q = 0; q < 32; ++q) out[t + T * q] = fx[t + (t >> 5) + q * S::KSTRIDE];
            }
        }
        more = work.valid(work.next(x->un));
        x = units + (x == units);
    }
#ifdef ISR_DEBUG
    if (!timed_out && work.phase_cycles() && tid == 0 && n_ph > 0) {
        for (int i = 0; i < 4; ++i) atomicAdd(work.phase_cycles() + i, (unsigned long long)ph[i]);
        atomicAdd(work.phase_cycles() + 4, (unsigned long long)n_ph);
    }
#endif
    if (timed_out) {
        if (t == 0) atomicOr(work.status(), 1);
        // let the copy still in flight land before the CTA's shared memory is released
        mbar_wait(bar, it & 1u, work.wait_limit());
    }
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    if (warp == kThreads / 32 - 1) tmem_dealloc(tslot, 512);
}

}  // namespace isr
