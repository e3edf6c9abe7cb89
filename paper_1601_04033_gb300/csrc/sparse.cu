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
// of theta, n, b, v is read and most are written (25M: 725 MB in about 117 us, 6.2
// TB/s), and by latency for small models: with the first list entries asked for
// beside the count and two entries per thread instead of four, four exchanges
// take 107 instead of 112 us at 1.29M, 154 instead of 177 at 3M, 271 instead of
// 277 at 6M.

#include <atomic>

#include "kernels.cuh"
#include "pdl.cuh"
#include "update.cuh"

namespace fasgd {
namespace {

constexpr int kSparseThreads = 256;

// AHEAD: the first step's list entries are loaded beside the count.
template <int RULE, bool EXACT, int kUnroll, bool AHEAD>
__global__ void __launch_bounds__(kSparseThreads, !AHEAD ? 1 : EXACT ? 6 : 8) fasgd_sparse_kernel(const __grid_constant__ SparseArgs a) {
    constexpr bool FAS = RULE != kRuleSgd;
    const int lane = threadIdx.x & 31;
    const int64_t warp_id = ((int64_t)blockIdx.x * kSparseThreads + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * kSparseThreads) >> 5;
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
    const int64_t first = warp_id * (32 * kUnroll);
    if (AHEAD) load(first, a.count_max);
    if (a.count_dev != nullptr && (count < 0 || count > a.count_max)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.err, 1);
        count = count < 0 ? 0 : a.count_max;
    }
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

template <int RULE, bool EXACT, int kUnroll, bool AHEAD>
cudaError_t launch_form(const SparseArgs& a, int num_sms, cudaStream_t stream) {
    // Resident blocks per SM, looked up once (the grid is only capped by it).
    static std::atomic<int> cached{0};
    int blocks_per_sm = cached.load(std::memory_order_relaxed);
    if (blocks_per_sm == 0) {
        cudaError_t st = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &blocks_per_sm, fasgd_sparse_kernel<RULE, EXACT, kUnroll, AHEAD>, kSparseThreads, 0);
        if (st != cudaSuccess) return st;
        if (blocks_per_sm < 1) blocks_per_sm = 1;
        cached.store(blocks_per_sm, std::memory_order_relaxed);
    }
    // Enough warps for the host-side bound on the count, at most one full wave.
    const int64_t per_block = (int64_t)kSparseThreads * kUnroll;
    int64_t want = (a.count_max + per_block - 1) / per_block;
    const int64_t cap = (int64_t)num_sms * blocks_per_sm;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    return launch_pdl(fasgd_sparse_kernel<RULE, EXACT, kUnroll, AHEAD>, (unsigned)want, kSparseThreads, 0, stream, a);
}

// Models up to 10M parameters: two entries per thread, the first step's ahead of
// the count, as many warps as fit (latency shows there).  Larger ones: four after
// it and registers to hold them, two blocks per SM: with fewer bytes in flight
// HBM serves the scattered sectors faster (four exchanges at 25M: 957 us against
// 980 with the small form and 975 with six blocks; 7M 319 against 313; 12M 499
// against 502; 16M 640 against 650).
template <int RULE, bool EXACT>
cudaError_t launch_rule(const SparseArgs& a, int num_sms, cudaStream_t stream) {
    return a.count_max <= 10'000'000 ? launch_form<RULE, EXACT, 2, true>(a, num_sms, stream)
                                     : launch_form<RULE, EXACT, 4, false>(a, num_sms, stream);
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
