// isr_kernels.cuh -- kernel registry shared by the instantiation units and the host API.
#pragma once

#include <algorithm>

#include "isr.h"
#include "isr_kernel.cuh"
#include "isr_paired.cuh"
#include "isr_xt.cuh"

namespace isr {

// record a one-line reason for isr_last_error() and return st (defined in isr_api.cu)
isr_status fail(isr_status st, const char* fmt, ...);
void clear_error();

// radix orders: 0 and 6 the tensor-memory exchange (isr_xt.cuh), 1-2 Stockham, 3 warp-local, 4-5 paired
// FP32, 7-8 orders 1-2 with the inter-pass twiddles in tensor memory, 9 the warp-local schedule with its
// twiddles in tensor memory
constexpr int kNumOrders = 10;

struct KernelEntry {
    const void* fn;   // nfft < 1024: integrate_kernel<LOG2N, TXT>
    const void* fn_order[kNumOrders];  // nfft < 1024: [0] the same for code_len == nfft; else the radix
                                       // orders 1-9 of full-length binary phase but 6 (1-3: nfft >= 2048)
    int smem_order[kNumOrders];        // their shared memory
    const void* fn_tc[9];     // [mode] tensor-core first pass (nfft 16384, binary phase): 1-4 mma.sync,
                              // 5-8 tcgen05; [0] unused
    int smem_tc;
    int smem;         // of fn (bytes)
    int gates;        // range gates per CTA (G)
    int threads;      // threads per CTA
    // nfft >= 1024: the kernel with its last exchange in tensor memory (isr_xt.cuh), persistent, launched
    // by launch_integrate; pack forms its sign words of per-IPP binary-phase codes
    const void* fn_xt = nullptr;
    const void* fn_xt_batch = nullptr;   // the same kernel over the units of a batch (binary phase, nfft >= 2048)
    const void* fn_pack = nullptr;
    const void* fn_tables = nullptr;   // fills the twiddle tables of the current device
    int smem_xt = 0;
};

template <int L>
KernelEntry entry_for(int txt)
{
    using S = Sched<L>;
    KernelEntry e{};
    e.gates = S::G;
    e.threads = kThreads;
    if constexpr (L < 10) {
        e.fn = txt == TX_CI16 ? (const void*)integrate_kernel<L, TX_CI16>
             : txt == TX_C32  ? (const void*)integrate_kernel<L, TX_C32>
                              : (const void*)integrate_kernel<L, TX_PM1>;
        e.fn_order[0] = txt == TX_PM1 ? (const void*)integrate_kernel<L, TX_PM1, true> : e.fn;
        e.smem = e.smem_order[0] = S::SMEM;
    }
    if constexpr (L >= 10) {
        e.fn_xt = txt == TX_CI16 ? (const void*)integrate_kernel_xt<L, TX_CI16, XtPlanSrc>
                : txt == TX_C32  ? (const void*)integrate_kernel_xt<L, TX_C32, XtPlanSrc>
                                 : (const void*)integrate_kernel_xt<L, TX_PM1, XtPlanSrc>;
        e.fn_pack = txt == TX_PM1 ? (const void*)pack_signs_kernel<SchedX<L>::T> : nullptr;
        if constexpr (L >= 11)
            if (txt == TX_PM1) e.fn_xt_batch = (const void*)integrate_kernel_xt<L, TX_PM1, XtBatchSrc>;
        e.fn_tables = (const void*)xt_tables_kernel<L>;
        e.smem_xt = SchedX<L>::SMEM;
    }
    if constexpr (L >= 11) {
        if (txt == TX_PM1) {
            e.fn_order[1] = (const void*)integrate_kernel<L, TX_PM1, true, 1>;
            e.fn_order[2] = (const void*)integrate_kernel<L, TX_PM1, true, 2>;
            e.fn_order[3] = (const void*)integrate_kernel_wl<L, TX_PM1, true>;
            e.smem_order[1] = Sched<L, 1>::SMEM;
            e.smem_order[2] = Sched<L, 2>::SMEM;
            e.smem_order[3] = SchedWL<L>::SMEM;
        }
    }
    if constexpr (L == 14) {
        if (txt == TX_PM1) {
            e.fn_order[4] = (const void*)integrate_kernel_p<true>;
            e.smem_order[4] = SchedP::SMEM;
            e.fn_order[5] = (const void*)integrate_kernel_q<true>;
            e.smem_order[5] = SchedQ::SMEM;
            e.fn_order[7] = (const void*)integrate_kernel_tm<14, TX_PM1, true, 1>;
            e.smem_order[7] = Sched<14, 1, true>::SMEM;
            e.fn_order[8] = (const void*)integrate_kernel_tm<14, TX_PM1, true, 2>;
            e.smem_order[8] = Sched<14, 2, true>::SMEM;
            e.fn_order[9] = (const void*)integrate_kernel_wl_tm<14, TX_PM1, true>;
            e.smem_order[9] = SchedWL<14>::SMEM;
            e.fn_tc[1] = (const void*)integrate_kernel<14, TX_PM1, true, 1, P0_BF16_SPLIT>;
            e.fn_tc[2] = (const void*)integrate_kernel<14, TX_PM1, true, 1, P0_FP16_SPLIT>;
            e.fn_tc[3] = (const void*)integrate_kernel<14, TX_PM1, true, 1, P0_BF16>;
            e.fn_tc[4] = (const void*)integrate_kernel<14, TX_PM1, true, 1, P0_FP16>;
            e.fn_tc[5] = (const void*)integrate_kernel_tc05<P0_TC05_BF16_SPLIT>;
            e.fn_tc[6] = (const void*)integrate_kernel_tc05<P0_TC05_FP16_SPLIT>;
            e.fn_tc[7] = (const void*)integrate_kernel_tc05<P0_TC05_BF16>;
            e.fn_tc[8] = (const void*)integrate_kernel_tc05<P0_TC05_FP16>;
            e.smem_tc = Sched<14, 1>::SMEM + kTcAfragBytes;
        }
    }
    return e;
}

// defined in the instantiation units (one per group of sizes, compiled in parallel)
KernelEntry entry_small(int log2n, int txt);  // nfft 8 .. 512
KernelEntry entry_mid(int log2n, int txt);    // nfft 1024 .. 4096
KernelEntry entry_8192(int txt);
KernelEntry entry_16384(int txt);

inline KernelEntry kernel_entry(int log2n, int txt)
{
    if (log2n <= 9) return entry_small(log2n, txt);
    if (log2n <= 12) return entry_mid(log2n, txt);
    if (log2n == 13) return entry_8192(txt);
    return entry_16384(txt);
}

// Ready the entry's kernels on the current device (once per plan): opt them into their shared memory and
// fill the twiddle tables if its context does not have them (synchronises `stream`).
cudaError_t prepare_entry(const KernelEntry& ke, int log2n, cudaStream_t stream);

// A word of pinned host memory for a handle's status, from a page that the current context's handles share.
struct StatusSlot {
    unsigned long long pool = 0;   // 0: the word is an allocation of its own
    int* word = nullptr;
};
cudaError_t take_status(StatusSlot& slot);
void give_status(const StatusSlot& slot);

// whether launch_integrate takes the tensor-memory kernel: for every code and order that has no kernel of
// its own, which only the orders 1-5 and 7-9 of full-length binary phase have
inline bool takes_xt(const KernelEntry& ke, bool full, int order) { return ke.fn_xt && (!full || !ke.fn_order[order]); }

// IPP chunks of a launch over n IPPs and rg gate groups on sm_count SMs, c_min .. c_max of them.  One CTA
// per SM works through rg x C units of ceil(n / C) IPPs each; a unit costs its IPPs (about 4.3 us each
// for any nfft) and a third of one more for its start and its partial sums, and every chunk's partials
// (bins floats) are written and read once.  The C with the least sum is taken: about two waves, the
// rule before, left up to a third of the SMs idle in the last one (777 gates x 333 IPPs at nfft 2048:
// four chunks made 392 units, three rounds of 84 IPPs; three make two of 111).  Weighed are the few
// least counts, which many gate groups want, and the most chunks that fit in each of the next 16 numbers
// of rounds; with no more than four units per SM to choose from, 500 gates x 200 IPPs at nfft 4096 had no
// split better than one chunk on 125 of the SMs (843 us; six chunks, five rounds of 34 IPPs: 726 us).
inline int64_t pick_chunks(int64_t n, int64_t rg, int64_t sm_count, int64_t c_min, int64_t c_max, int64_t bins)
{
    constexpr double kUnitIpps = 0.33, kChunkIppsPerBin = 8.0 / (6.5e6 * 4.3);   // 8 bytes at 6.5 MB per us
    c_max = std::min(c_max, n);
    c_min = std::min(c_min, c_max);
    int64_t best = c_min;
    double best_cost = -1;
    auto weigh = [&](int64_t c) {
        c = std::max(c_min, std::min(c, c_max));
        const int64_t chunk = (n + c - 1) / c, real = (n + chunk - 1) / chunk;
        const int64_t rounds = (rg * real + sm_count - 1) / sm_count;
        const double cost = (double)rounds * ((double)chunk + kUnitIpps) + (double)real * (double)bins * kChunkIppsPerBin;
        if (best_cost < 0 || cost < best_cost) {
            best = c;
            best_cost = cost;
        }
    };
    for (int64_t c = c_min; c < c_min + 4; ++c) weigh(c);
    const int64_t rounds_min = (rg * c_min + sm_count - 1) / sm_count;
    for (int64_t k = rounds_min; k < rounds_min + 16; ++k) weigh(k * sm_count / rg);
    return best;
}

// One launch over rg gate groups x n_chunks IPP chunks of `a` with radix order `order`.
inline cudaError_t launch_integrate(const KernelEntry& ke, KArgs a, bool full, int order, int rg, int n_chunks,
                                    int sm_count, cudaStream_t stream)
{
    if (takes_xt(ke, full, order)) {
        XtPlanSrc src{a, rg, 0, rg * n_chunks};
        void* args[] = {&src};
        const int grid = std::min(src.n_units, sm_count);   // persistent: one CTA per SM
        return cudaLaunchKernel(ke.fn_xt, dim3((unsigned)grid), dim3(kThreads), args, (size_t)ke.smem_xt, stream);
    }
    void* args[] = {&a};
    return cudaLaunchKernel(full ? ke.fn_order[order] : ke.fn, dim3((unsigned)rg, (unsigned)n_chunks),
                            dim3((unsigned)ke.threads), args, (size_t)(full ? ke.smem_order[order] : ke.smem), stream);
}

}  // namespace isr
