// Sparse server apply of one B-FASGD push (paper Sec. 2.3 with unsent
// entries dropped): for i < count, parameter p = idx[i] receives gradient
// entry val[i] through the same per-element rule as the dense pass
// (Eq. 1-2 or Eq. 4-8); parameters not in the list are not touched.
//
// Indices in one list are strictly ascending, so no two threads touch the
// same parameter and no atomics are needed.  The count is read on the device
// (it was produced there by the select kernels), so no host round trip sits
// between select and apply.  A persistent grid walks the list; each warp takes
// 32 kUnroll consecutive entries per iteration, so the index and value loads are
// coalesced and kUnroll gathers per array are in flight per thread.
//
// Bound by HBM at the granularity of sectors: at 20 % kept almost every sector
// of theta, n, b, v is read and most are written (25M: 721 MB in about 120 us, 6.0
// TB/s), and by latency for small models: with the first list entries asked for
// beside the count and two entries per thread instead of four, four exchanges
// take 107 instead of 112 us at 1.29M, 154 instead of 177 at 3M, 271 instead of
// 277 at 6M (launch_rule has the forms and their figures).

#include "kernels.cuh"
#include "pdl.cuh"
#include "update.cuh"

namespace fasgd {
namespace {

constexpr int kSparseThreads = 256;

// AHEAD: the first step's list entries are loaded beside the count.  BLOCKS: blocks
// per SM that the registers are held to.
template <int RULE, bool EXACT, int kUnroll, bool AHEAD, int BLOCKS>
__global__ void __launch_bounds__(kSparseThreads, BLOCKS) fasgd_sparse_kernel(const __grid_constant__ SparseArgs a) {
    constexpr bool FAS = RULE != kRuleSgd;
    const int lane = threadIdx.x & 31;
    int64_t warp_id = ((int64_t)blockIdx.x * kSparseThreads + threadIdx.x) >> 5;
    int64_t nwarps = ((int64_t)gridDim.x * kSparseThreads) >> 5;
    pdl_wait();
    pdl_trigger();
    int64_t count = a.count_max;
    if (a.count_dev != nullptr) count = *a.count_dev;
    int32_t p[kUnroll], prev[kUnroll];
    float g[kUnroll];
    // This lane's entries of the step at `from`, those below `end`.
    const auto load = [&](int64_t from, int64_t end) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int64_t i = from + u * 32 + lane;
            if (i < end) {
                p[u] = a.idx[i];
                g[u] = a.val[i];
                prev[u] = i > 0 ? a.idx[i - 1] : -1;
            }
        }
    };
    if (AHEAD) load(warp_id * (32 * kUnroll), a.count_max);
    if (a.count_dev != nullptr && (count < 0 || count > a.count_max)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.err, 1);
        count = count < 0 ? 0 : a.count_max;
    }
    if constexpr (!AHEAD) {
        if (count < a.half_below) {   // half or a quarter of each block's warps
            const int part = count < a.quarter_below ? 4 : 2;
            if (threadIdx.x >= kSparseThreads / part) return;
            warp_id = ((int64_t)blockIdx.x * (kSparseThreads / part) + threadIdx.x) >> 5;
            nwarps /= part;
        }
    }
    const int64_t first = warp_id * (32 * kUnroll);
    for (int64_t base = first; base < count; base += nwarps * (32 * kUnroll)) {
        bool ok[kUnroll];
        if (!AHEAD || base != first) load(base, count);
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            ok[u] = base + u * 32 + lane < count;
            if (ok[u]) {
                if (p[u] < 0 || (int64_t)p[u] >= a.P) {
                    atomicOr(a.err, 2);
                    ok[u] = false;
                } else if (p[u] <= prev[u]) {
                    atomicOr(a.err, 4);
                    ok[u] = false;
                }
            }
        }
        float th[kUnroll], n[kUnroll], b[kUnroll], v[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (ok[u]) {
                th[u] = a.theta[p[u]];
                if (FAS) {
                    n[u] = a.n[p[u]];
                    b[u] = a.b[p[u]];
                    v[u] = a.v[p[u]];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            if (ok[u]) {
                if (FAS) {
                    rule_update<EXACT ? kArithExact : kArithApprox, RULE == kRuleFasgdStd>(
                        th[u], n[u], b[u], v[u], g[u], a.coef, a.sp);
                    a.n[p[u]] = n[u];
                    a.b[p[u]] = b[u];
                    a.v[p[u]] = v[u];
                } else {
                    sgd_update(th[u], g[u], a.coef);
                }
                a.theta[p[u]] = th[u];
            }
        }
    }
}

template <int RULE, bool EXACT, int kUnroll, bool AHEAD, int BLOCKS>
cudaError_t launch_form(const SparseArgs& a, int num_sms, cudaStream_t stream) {
    // Enough warps for the host-side bound on the count, at most one full wave.
    const int64_t per_block = (int64_t)kSparseThreads * kUnroll;
    int64_t want = (a.count_max + per_block - 1) / per_block;
    const int64_t cap = (int64_t)num_sms * BLOCKS;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    return launch_pdl(fasgd_sparse_kernel<RULE, EXACT, kUnroll, AHEAD, BLOCKS>, (unsigned)want, kSparseThreads, 0, stream, a);
}

// FASGD rules, up to 7M entries at most: two per thread, the first step's ahead of
// the count, as many warps as fit (latency shows there).  Beyond: four per thread,
// four blocks per SM, and of each block's warps all, half or a quarter, by the
// list's density.  Scattered sectors HBM serves faster with fewer bytes in flight
// (under 45 % kept half the warps, under 14 % a quarter), a dense list, whose
// gathers are coalesced, needs all of them.  (Part of each block, since the first
// blocks of a larger grid do not spread over the SMs: 20 % at 25M 138 us so.)  One
// apply in us, the forms it replaces -- four per thread and 48 registers at every
// size, then the small form up to 10M and 83 registers beyond, which left two
// blocks per SM at any density -- and this:
//   kept        5 %                  20 %                  60 %                  100 %
//   25M    111.6, 106.5, 93.1   127.6, 123.2, 124.1   150.5, 168.5, 148.2   160.8, 196.8, 153.2
//   12M     46.1,  48.2, 44.1    66.2,  61.2,  61.3    74.7,  82.6,  72.7    79.5,  96.8,  76.8
//   9M      26.4,  28.0, 24.4    44.4,  45.1,  44.7    56.4,  55.7,  55.1    60.5,  57.0,  57.4
// At 6M the two forms are within 4 % (10 % kept 17.4 small, 18.1 large; 60 %
// 31.6, 30.9).
// ASGD/SASGD gather one array: four per thread, five blocks per SM, all the warps
// (25M: half would take 41 against 34 us at 20 %, 118 against 68 at 100 %) but for
// large models under 6 % kept (15.5 -> 13.3 at 5 %); at 3M and 6M, all kept, 5.6
// and 10.0 against 7.1 and 13.5 in the small form.
template <int RULE, bool EXACT>
cudaError_t launch_rule(SparseArgs a, int num_sms, cudaStream_t stream) {
    const bool large = a.count_max > 7'000'000;
    if constexpr (RULE == kRuleSgd) {
        a.half_below = large ? a.P / 16 : 0;
        a.quarter_below = 0;
        return launch_form<RULE, EXACT, 4, false, 5>(a, num_sms, stream);
    } else {
        a.half_below = a.P / 20 * 9;
        a.quarter_below = a.P / 7;
        return large ? launch_form<RULE, EXACT, 4, false, 4>(a, num_sms, stream)
                     : launch_form<RULE, EXACT, 2, true, EXACT ? 6 : 8>(a, num_sms, stream);
    }
}

constexpr int kScatterUnroll = 8;

// Client side of a B-FASGD fetch: theta[idx[i]] = val[i] for i < count.
// Indices come from one compaction, so they are distinct and no two threads
// write the same parameter; an index outside [0, P) is skipped and flagged.
__global__ void __launch_bounds__(kSparseThreads) fetch_scatter_kernel(const __grid_constant__ ScatterArgs a) {
    pdl_wait();
    pdl_trigger();
    int64_t count = a.count_max;
    if (a.count_dev != nullptr) {
        const int64_t c = *a.count_dev;
        count = c;
        if (c < 0 || c > a.count_max) {
            if (blockIdx.x == 0 && threadIdx.x == 0 && a.err != nullptr) atomicOr(a.err, 1);
            count = c < 0 ? 0 : a.count_max;
        }
    }
    // kScatterUnroll entries per thread per step (consecutive lanes, coalesced
    // list loads), every load of a step issued before its stores.
    const int64_t span = (int64_t)kSparseThreads * kScatterUnroll;
    for (int64_t base = (int64_t)blockIdx.x * span; base < count; base += (int64_t)gridDim.x * span) {
        int32_t p[kScatterUnroll];
        float x[kScatterUnroll];
#pragma unroll
        for (int k = 0; k < kScatterUnroll; ++k) {
            const int64_t i = base + k * kSparseThreads + threadIdx.x;
            p[k] = 0;
            x[k] = 0.f;
            if (i < count) {
                p[k] = a.idx[i];
                x[k] = a.val[i];
            }
        }
#pragma unroll
        for (int k = 0; k < kScatterUnroll; ++k) {
            const int64_t i = base + k * kSparseThreads + threadIdx.x;
            if (i >= count) continue;
            if (p[k] < 0 || (int64_t)p[k] >= a.P) {
                if (a.err != nullptr) atomicOr(a.err, 2);
                continue;
            }
            a.theta[p[k]] = x[k];
        }
    }
}

}  // namespace

cudaError_t launch_scatter(const ScatterArgs& a, int num_sms, cudaStream_t stream) {
    int64_t want = (a.count_max + kSparseThreads - 1) / kSparseThreads;
    const int64_t cap = (int64_t)(num_sms > 0 ? num_sms : 1) * 8;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    return launch_pdl(fetch_scatter_kernel, (unsigned)want, kSparseThreads, 0, stream, a);
}

cudaError_t launch_sparse(const SparseArgs& a, int rule, bool exact, int num_sms,
                          cudaStream_t stream, int64_t* launches) {
    cudaError_t st;
    if (rule == kRuleSgd)
        st = launch_rule<kRuleSgd, false>(a, num_sms, stream);
    else if (rule == kRuleFasgd)
        st = exact ? launch_rule<kRuleFasgd, true>(a, num_sms, stream)
                   : launch_rule<kRuleFasgd, false>(a, num_sms, stream);
    else
        st = exact ? launch_rule<kRuleFasgdStd, true>(a, num_sms, stream)
                   : launch_rule<kRuleFasgdStd, false>(a, num_sms, stream);
    if (st == cudaSuccess) ++*launches;
    return st;
}

}  // namespace fasgd
