// Fused dense server pass: K pending pushes applied in one sweep over P.
//
// Every parameter's theta (and n, b, v for FASGD) is read once, the K
// gradient slices are read once, all K pushes are applied in arrival order
// with the state held in registers, and the state is written once.  The pass
// therefore moves (8 + 4K) bytes per parameter for ASGD/SASGD and (32 + 4K)
// for FASGD, the minimum for K pushes (paper Sec. 2.1 protocol, Eq. 1-2 and
// Eq. 4-8 applied K times).
//
// Structure: a persistent kernel, one block per SM (or two smaller ones), one
// producer warp and 16 consumer warps.  The parameter range is cut into tiles
// of 2048; the producer's elected lane stages each tile's state slices and up
// to CH gradient slices into a shared-memory ring with 1-D bulk async copies
// (cp.async.bulk, completion counted on an mbarrier), while the consumer
// warps compute on the previous stage: each thread takes four consecutive
// parameters (128-bit shared loads), frees the stage as soon as its inputs
// are in registers, applies the pushes, and stores the state with 128-bit
// global stores.  A larger K runs as several stages per tile (the state travels
// with the first one only).  Every block has an equal piece of what the whole
// tiles leave over and the same number of tiles (BlockShare); the last P mod 4
// parameters go through plain loads.  Passes of fewer than 8 tiles per SM use a plain grid
// instead (one quad of parameters per thread, fasgd_direct_kernel).
//
// With SUMS (one push, a.msg.partial set) the pass applies a per-message push
// whose Eq. 9 decision was taken by the kernel before it, or, where the
// statistic had to be formed afresh, takes it itself from the sums
// (message_decide, in every block's warp 0): transmitted, it applies the pushed
// gradient while copying it into the client's cache slot; dropped, it applies
// the slot.  It also leaves every block's float-float sum of the new v, formed
// in registers, so the next decision needs no pass over v (message.cu).
//
// Both kernels are launched as programmatic dependents (pdl.cuh): a pass is
// scheduled while the kernel before it on the stream drains, sets up its
// barriers, and waits (griddepcontrol.wait) before it touches memory.
//
// Every wait on an mbarrier is bounded (about one second of wall clock);
// on expiry the block sets flag 8 of the error word, waits (bounded) for its
// own copies in flight, and returns.  Elements are independent, so the
// result does not depend on the grid or on which path handled an element.

#include <atomic>
#include <type_traits>

#include "kernels.cuh"
#include "message.cuh"
#include "pdl.cuh"
#include "twosum.cuh"
#include "update.cuh"
#include "wait.cuh"

namespace fasgd {
namespace {

// Ring geometry per consumer count CONS (threads that compute; 512 or 256):
// tiles of 4 CONS parameters, CONS + 32 threads per block (one producer
// warp), 512 / CONS blocks per SM sharing 220 KB of shared memory.  A stage
// holds the state's slices and min(K, CH) gradients'; how many stages a pass
// uses is chosen with CH (launch_rule).
template <int CONS> struct Geom {
    static constexpr int kTile = 4 * CONS;
    static constexpr int kThreads = CONS + 32;
    static constexpr int kBlocksPerSm = 512 / CONS;
    static constexpr int kMaxStages = 8;
    static constexpr int kSmemBudget = 220 * 1024 / kBlocksPerSm;   // ring + barriers, per block
};
constexpr int kTile = Geom<512>::kTile;         // the reference tile (2048 parameters)

// ---- bulk async copy (the mbarrier wrappers and bounded waits: wait.cuh) ----
// 1-D bulk copy global -> shared (16-byte aligned, size a multiple of 16),
// completion signalled on `bar` as transaction bytes.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// A quad whose exact arithmetic left the range of its fast form.
template <int RULE>
__device__ __forceinline__ void redo_quad(const DenseArgs& a, const float* g0, int64_t e, float4& th,
                                          float4& n, float4& b, float4& v) {
    const QuadState q = exact_quad<RULE == kRuleFasgdStd>(a.theta, a.n, a.b, a.v, g0, a.grad, a.coef, a.K, e, a.sp);
    th = q.th;
    n = q.n;
    b = q.b;
    v = q.v;
}

// The last P mod 4 parameters, thread i < P mod 4 taking one; returns the new
// v of its parameter (0 for the other threads).
template <int RULE, int ARITH>
__device__ __forceinline__ float apply_ragged(const DenseArgs& a, int tid, const float* g0, float* copy_to) {
    constexpr bool FAS = RULE != kRuleSgd;
    const int64_t p = (a.P & ~int64_t(3)) + tid;
    if (p >= a.P) return 0.f;
    float th = a.theta[p], n = 0.f, b = 0.f, v = 0.f;
    if (FAS) {
        n = a.n[p];
        b = a.b[p];
        v = a.v[p];
    }
    for (int k = 0; k < a.K; ++k) {
        const float g = (k == 0 ? g0 : a.grad[k])[p];
        if (k == 0 && copy_to != nullptr) copy_to[p] = g;
        if (FAS)
            rule_update<ARITH, RULE == kRuleFasgdStd>(th, n, b, v, g, a.coef[k], a.sp);
        else
            sgd_update(th, g, a.coef[k]);
    }
    a.theta[p] = th;
    if (FAS) {
        a.n[p] = n;
        a.b[p] = b;
        a.v[p] = v;
    }
    return v;
}

struct Ring {
    int stages;     // stages in the ring
    int chunks;     // stages per tile: ceil(K / CH)
    int floats;     // floats per stage
};

// RULE: kRuleSgd / kRuleFasgd / kRuleFasgdStd; ARITH: kArithApprox /
// kArithApproxFtz / kArithExact (see update.cuh); CH: gradient slices per stage;
// SUMS: also leave the blocks' sums of the new v (FASGD rules, K = 1); CONS:
// consumer threads per block (the ring geometry, Geom).
template <int RULE, int ARITH, int CH, bool SUMS, int CONS>
__global__ void __launch_bounds__(Geom<CONS>::kThreads, Geom<CONS>::kBlocksPerSm)
fasgd_dense_kernel(const __grid_constant__ DenseArgs a, const Ring ring) {
    using G = Geom<CONS>;
    constexpr bool FAS = RULE != kRuleSgd;
    constexpr int kState = FAS ? 4 : 1;              // theta (, n, b, v)
    constexpr int kTile = G::kTile, kConsumerWarps = CONS / 32;
    extern __shared__ __align__(128) unsigned char smem[];
    float* buf = reinterpret_cast<float*>(smem);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)ring.stages * ring.floats * 4);
    uint64_t* empty = full + ring.stages;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const BlockShare share(a.P & ~int64_t(3), kTile, gridDim.x, blockIdx.x);

    if (threadIdx.x == 0) {
        for (int s = 0; s < ring.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], kConsumerWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const auto load_state = [&](float* st, int64_t off, uint32_t bytes, uint64_t* bar) {
        bulk_load(st, a.theta + off, bytes, bar);
        if (FAS) {
            bulk_load(st + 1 * kTile, a.n + off, bytes, bar);
            bulk_load(st + 2 * kTile, a.b + off, bytes, bar);
            bulk_load(st + 3 * kTile, a.v + off, bytes, bar);
        }
    };
    // A message push (SUMS) follows its own decision kernel, which only reads v
    // or its sums and started after every earlier kernel had finished, so the
    // state may be read before that kernel is complete: the first stages' state
    // is on its way while the decision is taken.
    int64_t early = 0;
    if (SUMS && warp == kConsumerWarps && lane == 0) {
        early = share.tiles < ring.stages ? share.tiles : ring.stages;
        for (int i = 0; i < (int)early; ++i) {
            const uint32_t bytes = (uint32_t)share.length(i) * 4;
            mbar_arrive_expect_tx(&full[i], (kState + 1) * bytes);
            load_state(buf + (size_t)i * ring.floats, share.offset(i), bytes, &full[i]);
        }
    }
    pdl_wait();      // the kernel before this one on the stream is complete
    pdl_trigger();
    // Transmitted: apply the pushed gradient and copy it into the client's cache
    // slot; dropped: apply the slot.
    const float* g0 = a.grad[0];
    float* copy_to = nullptr;
    if constexpr (SUMS) {
        uint32_t send;
        if (a.msg.decided != nullptr) {
            send = *a.msg.decided;
        } else {     // the statistic was formed afresh: decide from its sums
            __shared__ uint32_t s_send;
            if (warp == 0) {
                float vbar;
                const uint32_t d = message_decide(a.msg.fresh, a.msg.nblocks, a.P, a.msg.c, a.msg.eps_b,
                                                  a.msg.round_key0, a.msg.round_key1, a.msg.client_word,
                                                  a.msg.n_lo, a.msg.n_hi, &vbar);
                if (lane == 0) {
                    s_send = d;
                    if (blockIdx.x == 0 && a.msg.flag_out != nullptr) *a.msg.flag_out = (int32_t)d;
                }
            }
            __syncthreads();
            send = s_send;
        }
        if (send) {
            g0 = a.msg.src;
            copy_to = a.msg.slot;
        }
    }

    if (warp == kConsumerWarps) {
        // ---------------- producer: one elected lane ----------------
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            uint32_t issued = 0;            // bit s: stage s has been filled
            uint32_t issued_phase = 0;      // bit s: the phase parity of its last fill
            for (int64_t t = 0; t < share.tiles && ok; ++t) {
                const int64_t off = share.offset(t);
                const uint32_t bytes = (uint32_t)share.length(t) * 4;
                for (int c = 0; c < ring.chunks; ++c) {
                    ok = wait_one(&empty[s], ph ^ 1u, a.err);
                    if (!ok) break;
                    const int k0 = c * CH, ng = min(CH, a.K - k0);
                    float* st = buf + (size_t)s * ring.floats;
                    if (t >= early) {               // else armed, and its state asked for, above
                        mbar_arrive_expect_tx(&full[s], (uint32_t)((c == 0 ? kState : 0) + ng) * bytes);
                        if (c == 0) load_state(st, off, bytes, &full[s]);
                    }
                    for (int j = 0; j < ng; ++j)
                        bulk_load(st + (kState + j) * kTile, (k0 + j == 0 ? g0 : a.grad[k0 + j]) + off,
                                  bytes, &full[s]);
                    issued |= 1u << s;
                    issued_phase = (issued_phase & ~(1u << s)) | (ph << s);
                    if (++s == ring.stages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            // Every fill issued by this block has landed before it exits.
            for (int i = 0; i < ring.stages; ++i)
                if (issued & (1u << i)) wait_one(&full[i], (issued_phase >> i) & 1u, a.err);
        }
        return;
    }

    // ---------------- consumers ----------------
    const int tid = threadIdx.x;
    int s = 0;
    uint32_t ph = 0;
    VSum vsum;
    // One tile from `off`; whole: all of its threads have a quad, else those
    // below `length`.
    const auto tile = [&](auto whole, int64_t off, int length) {
        const bool mine = whole.value || 4 * tid < length;
        const int64_t e = off + 4 * (int64_t)tid;
        float4 th = make_float4(0.f, 0.f, 0.f, 0.f), n = th, b = th, v = th;
        Guard<ARITH> guard;
        for (int c = 0; c < ring.chunks; ++c) {
            if (!wait_warp(&full[s], ph, a.err)) return false;
            const float4* st = reinterpret_cast<const float4*>(buf + (size_t)s * ring.floats) + tid;
            float4 g[CH];
            const int k0 = c * CH, ng = min(CH, a.K - k0);
            if (mine) {
                if (c == 0) {
                    th = st[0];
                    if (FAS) {
                        n = st[1 * (kTile / 4)];
                        b = st[2 * (kTile / 4)];
                        v = st[3 * (kTile / 4)];
                    }
                }
                if (ng == CH) {
#pragma unroll
                    for (int j = 0; j < CH; ++j) g[j] = st[(kState + j) * (kTile / 4)];
                } else {
#pragma unroll
                    for (int j = 0; j < CH; ++j)
                        if (j < ng) g[j] = st[(kState + j) * (kTile / 4)];
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);   // inputs are in registers
            if (++s == ring.stages) {
                s = 0;
                ph ^= 1u;
            }
            if (!mine) continue;
            if (SUMS && copy_to != nullptr)          // a transmitted message refreshes its slot
                *reinterpret_cast<float4*>(copy_to + e) = g[0];
            if (ng == CH) {
#pragma unroll
                for (int j = 0; j < CH; ++j) update4<RULE, ARITH>(th, n, b, v, g[j], a.coef[k0 + j], a.sp, guard);
            } else {
#pragma unroll
                for (int j = 0; j < CH; ++j)
                    if (j < ng) update4<RULE, ARITH>(th, n, b, v, g[j], a.coef[k0 + j], a.sp, guard);
            }
        }
        if (!mine) return true;
        if (!guard.ok()) redo_quad<RULE>(a, g0, e, th, n, b, v);
        *reinterpret_cast<float4*>(a.theta + e) = th;
        if (FAS) {
            *reinterpret_cast<float4*>(a.n + e) = n;
            *reinterpret_cast<float4*>(a.b + e) = b;
            *reinterpret_cast<float4*>(a.v + e) = v;
        }
        if (SUMS) vsum.add(v);
        return true;
    };
    bool ok = share.piece == 0 || tile(std::false_type{}, share.piece_start, share.piece);
    for (int64_t t = 0; t < share.whole && ok; ++t) ok = tile(std::true_type{}, share.first + t * share.step, kTile);
    if (ok && blockIdx.x == gridDim.x - 1) {
        const float v = apply_ragged<RULE, ARITH>(a, tid, g0, copy_to);
        if (SUMS && tid < (int)(a.P & 3)) vsum.add(make_float4(v, 0.f, 0.f, 0.f));
    }
    if constexpr (SUMS) {
        __shared__ float2 s_sum[kConsumerWarps];
        const float2 w = vsum.warp_total();
        if (lane == 0) s_sum[warp] = w;
        asm volatile("bar.sync 1, %0;" ::"n"(CONS) : "memory");   // the consumers
        if (tid == 0) a.msg.partial[blockIdx.x] = ordered_total<kConsumerWarps>(s_sum);
    }
}

// A pass with up to `stages` stages in the ring.
template <int RULE, int ARITH, int CH, bool SUMS = false, int CONS = 512>
cudaError_t launch_ch(const DenseArgs& a, int stages, int num_sms, cudaStream_t stream) {
    using G = Geom<CONS>;
    constexpr int kState = RULE != kRuleSgd ? 4 : 1;
    Ring ring;
    ring.chunks = (a.K + CH - 1) / CH;
    ring.floats = (kState + (a.K < CH ? a.K : CH)) * G::kTile;
    ring.stages = (G::kSmemBudget - 2 * G::kMaxStages * 8) / (ring.floats * 4);
    if (ring.stages > stages) ring.stages = stages;
    const size_t smem = (size_t)ring.stages * ring.floats * 4 + 2 * ring.stages * sizeof(uint64_t);
    // The shared-memory limit is a per-device attribute of the kernel: set it
    // once per device (bit d of the mask) and instantiation.
    static std::atomic<uint64_t> configured{0};
    int dev = 0;
    cudaError_t st = cudaGetDevice(&dev);
    if (st != cudaSuccess) return st;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0;
    if (bit == 0 || !(configured.load(std::memory_order_acquire) & bit)) {
        st = cudaFuncSetAttribute(fasgd_dense_kernel<RULE, ARITH, CH, SUMS, CONS>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmemBudget);
        if (st != cudaSuccess) return st;
        configured.fetch_or(bit, std::memory_order_acq_rel);
    }
    return launch_pdl(fasgd_dense_kernel<RULE, ARITH, CH, SUMS, CONS>,
                      (unsigned)(SUMS ? kMessageBlocks : G::kBlocksPerSm * num_sms), G::kThreads, smem, stream, a, ring);
}

// ---- small passes ------------------------------------------------------------
// With few tiles per SM the ring's staging does not pay: its blocks stage,
// compute and store a handful of tiles each, and the last then runs the tail.
// A plain grid with one quad of parameters per thread and all of a thread's
// loads issued before its arithmetic makes one round trip to memory instead.
// Measured per pass (graph replay, K = 1 / 8): equal or faster up to
// 2.5M parameters (7,850: 2.1 / 3.4 us against 3.4 / 6.7 us; 1.29M: 5.0 /
// 10.7 us against 5.5 / 13.1 us), behind the ring from about 5M (K = 1:
// 23.5 against 18.1 us), so it takes passes below 8 tiles per SM.  Such
// working sets stay in L2 between passes, so the gradient loads keep the
// default cache policy here.
constexpr int kDirectThreads = 128;
constexpr int kDirectTilesPerSm = 8;
// Blocks of the grid at most, per SM: up to 1.25M parameters a thread has one
// quad, beyond that the last round is short.  The kernel is built for K = 1, up
// to 4 and up to 8 gradients at a time: 40 registers instead of 64 at K = 1, so
// 12 blocks per SM are resident instead of 8.  Push + apply + pull at 1.29M, with
// 8 blocks per SM and one kernel for all K -> now: K = 1 10.7 -> 8.3 us, K = 3
// 13.8 -> 12.4, K = 8 18.8 -> 18.0, exact K = 1 12.3 -> 9.2.
constexpr int kDirectBlocksPerSm = 16;

template <int RULE, int ARITH, int KMAX>
__global__ void __launch_bounds__(kDirectThreads)
fasgd_direct_kernel(const __grid_constant__ DenseArgs a) {
    constexpr bool FAS = RULE != kRuleSgd;
    constexpr bool STD = RULE == kRuleFasgdStd;
    pdl_wait();
    pdl_trigger();
    const int64_t nq = (a.P + 3) / 4;  // quads; the last may be partial
    for (int64_t q = (int64_t)blockIdx.x * kDirectThreads + threadIdx.x; q < nq;
         q += (int64_t)gridDim.x * kDirectThreads) {
        const int64_t e = 4 * q;
        if (e + 4 <= a.P) {
            float4 th = *reinterpret_cast<const float4*>(a.theta + e);
            float4 n = make_float4(0.f, 0.f, 0.f, 0.f), b = n, v = n;
            if (FAS) {
                n = *reinterpret_cast<const float4*>(a.n + e);
                b = *reinterpret_cast<const float4*>(a.b + e);
                v = *reinterpret_cast<const float4*>(a.v + e);
            }
            Guard<ARITH> guard;
            for (int k0 = 0; k0 < (KMAX == 1 ? 1 : a.K); k0 += KMAX) {
                float4 g[KMAX];
#pragma unroll
                for (int j = 0; j < KMAX; ++j)
                    if (KMAX == 1 || k0 + j < a.K) g[j] = *reinterpret_cast<const float4*>(a.grad[k0 + j] + e);
#pragma unroll
                for (int j = 0; j < KMAX; ++j)
                    if (KMAX == 1 || k0 + j < a.K) update4<RULE, ARITH>(th, n, b, v, g[j], a.coef[k0 + j], a.sp, guard);
            }
            if (!guard.ok()) redo_quad<RULE>(a, a.grad[0], e, th, n, b, v);
            *reinterpret_cast<float4*>(a.theta + e) = th;
            if (FAS) {
                *reinterpret_cast<float4*>(a.n + e) = n;
                *reinterpret_cast<float4*>(a.b + e) = b;
                *reinterpret_cast<float4*>(a.v + e) = v;
            }
        } else {
            for (int64_t p = e; p < a.P; ++p) {
                float th = a.theta[p], n = 0.f, b = 0.f, v = 0.f;
                if (FAS) {
                    n = a.n[p];
                    b = a.b[p];
                    v = a.v[p];
                }
                for (int k = 0; k < a.K; ++k) {
                    if (FAS)
                        rule_update<ARITH, STD>(th, n, b, v, a.grad[k][p], a.coef[k], a.sp);
                    else
                        sgd_update(th, a.grad[k][p], a.coef[k]);
                }
                a.theta[p] = th;
                if (FAS) {
                    a.n[p] = n;
                    a.b[p] = b;
                    a.v[p] = v;
                }
            }
        }
    }
}

template <int RULE, int ARITH>
cudaError_t launch_direct(const DenseArgs& a, int num_sms, cudaStream_t stream) {
    const int64_t nq = (a.P + 3) / 4;
    int64_t grid = (nq + kDirectThreads - 1) / kDirectThreads;
    if (grid > kDirectBlocksPerSm * (int64_t)num_sms) grid = kDirectBlocksPerSm * (int64_t)num_sms;
    const auto kernel = a.K == 1   ? fasgd_direct_kernel<RULE, ARITH, 1>
                        : a.K <= 4 ? fasgd_direct_kernel<RULE, ARITH, 4>
                                   : fasgd_direct_kernel<RULE, ARITH, 8>;
    return launch_pdl(kernel, (unsigned)grid, kDirectThreads, 0, stream, a);
}

template <int RULE, int ARITH>
cudaError_t launch_rule(const DenseArgs& a, int num_sms, cudaStream_t stream) {
    if constexpr (RULE != kRuleSgd) {
        if (a.msg.partial != nullptr) {
            if (a.K != 1) return cudaErrorInvalidValue;
            // State within L2 (16 bytes per parameter, 129 MB): all five
            // stages, since the decision's latency in front of the pass counts
            // (eight pushes and fetches at 5M: 233 against 269 us with two).
            // Beyond it two, as below (25M: 1237 against 1264 us).
            const bool in_l2 = a.P <= 7'000'000;
            return launch_ch<RULE, ARITH, 1, true>(a, in_l2 ? 5 : 2, num_sms, stream);
        }
    }
    if (a.P / kTile < kDirectTilesPerSm * num_sms) return launch_direct<RULE, ARITH>(a, num_sms, stream);
    // How many gradient slices a stage takes (CH) and how many stages: a tile's
    // first stage holds its state and CH gradients, the others CH each.
    //
    // From HBM (everything the pass touches is more than L2 holds) the pass
    // streams best with some 80 to 160 KB per SM in flight, less than the
    // shared memory would hold (reads that run further ahead only push the
    // writes together).  Sweep of CH = 1, 2, 4, 8 (512 consumers; also 4, 8
    // with two blocks of 256) by 2 to 8 stages, push + apply + pull in us at
    // 25M parameters, as before (CH = K rounded up to a power of two, every
    // stage that fits; K > 8 two blocks of 256, CH = 8) -> as chosen; the same
    // choices were best or within 1 % at 8M, 10M, 12M and 50M:
    //   FASGD  K = 1: 172.6 -> 164   2: 185 -> 176     3: 201 -> 190
    //          4: 215 -> 206         5: 231 -> 217     6: 244 -> 229
    //          8: 253 -> 254         12: 316 -> 312    16: 375 (same)   32: 631 -> 601
    //   exact  3: 204 -> 190         4: 223 -> 207     5: 222 (same)
    //          6: 238 -> 232         7: 260 -> 247     8: 273     16: 494
    //          (with the present guard of the quotient 5: 221, 6: 232, 7: 257, 16: 491)
    //   SGD    K = 3: 103 -> 102     5: 133.4 -> 131.6 6: 148 -> 146     8: 182 -> 174
    //          12: 242 -> 232        16: 300 -> 287    32: 531 -> 512
    //
    // Out of L2 latency counts instead, and more bytes in flight pay: stages of
    // all K gradients, as many as 192 KB per SM hold, in two blocks of 256
    // consumers (SGD: one of 512, every stage that fits).  Push + apply in us,
    // the choice for HBM -> this one:
    //   FASGD  K = 1: 5M 23.5 -> 20.0, 6M 33.3 -> 31.0    2: 4M 18.6 -> 16.6, 6M 38.1 -> 36.3
    //          3: 4M 24.3 -> 21.2    4: 2.6M 13.8 -> 12.7, 4M 27.5 -> 25.2
    //          5: 4M 31.0 -> 28.2    6: 2.6M 19.4 -> 17.4  8: 2.6M 24.0 -> 22.3
    //   exact  K = 1: 5M 23.7 -> 20.1   2: 4M 19.8 -> 17.2   3: 4M 26.0 -> 23.1
    //          4: 4M 28.9 -> 27.2    5: 4M 34.0 -> 32.9   (6, 7, 8: 2.6M 24.5, 27.5, 30.8 -> 24.7, 28.0, 31.7)
    //   SGD    K = 4: 5M 14.3 -> 13.5, 6M 22.0 -> 21.0    6: 4M 17.9 -> 17.0    8: 2.6M 11.6 -> 10.3
    //          K = 1 alone the same, behind other kernels less: with a pull 8M 19.2 -> 17.0,
    //          dropped message pushes at 12M 23.7 -> 18.3, with a budget push at 5M 21.5 -> 19.7
    // The line is at what the pass touches, a little above L2's 129 MB, where
    // the two cross: FASGD K = 2 at 6M (144 MB) 38.1 -> 36.3, at 7M (168 MB)
    // 43.3 -> 44.4; K = 3 at 5.5M (154 MB) 36.9 -> 36.7; SGD K = 4 at 7M
    // (140 MB) 25.9 -> 26.8.
    const int64_t touched = 4 * a.P * ((RULE != kRuleSgd ? 4 : 1) + a.K);
    const bool in_l2 = touched <= (RULE != kRuleSgd ? 150'000'000 : 130'000'000);
    if constexpr (RULE == kRuleSgd) {
        if (a.K == 1) return launch_ch<RULE, ARITH, 1>(a, in_l2 ? 8 : 5, num_sms, stream);
        if (a.K == 2) return launch_ch<RULE, ARITH, 2>(a, 5, num_sms, stream);
        if (a.K <= 4) return launch_ch<RULE, ARITH, 4>(a, a.K == 3 ? 4 : in_l2 ? 5 : 3, num_sms, stream);
        if (a.K <= 8 || a.K > 14) return launch_ch<RULE, ARITH, 8>(a, a.K == 5 || (a.K <= 8 && in_l2) ? 3 : 2, num_sms, stream);
        return launch_ch<RULE, ARITH, 4>(a, 4, num_sms, stream);
    } else {
        if (in_l2 && a.K <= (ARITH == kArithExact ? 5 : 8)) {
            if (a.K == 1) return launch_ch<RULE, ARITH, 1, false, 256>(a, 4, num_sms, stream);
            if (a.K == 2) return launch_ch<RULE, ARITH, 2, false, 256>(a, 4, num_sms, stream);
            if (a.K <= 4) return launch_ch<RULE, ARITH, 4, false, 256>(a, 3, num_sms, stream);
            return launch_ch<RULE, ARITH, 8, false, 256>(a, 2, num_sms, stream);
        }
        if (a.K == 1) return launch_ch<RULE, ARITH, 1>(a, 2, num_sms, stream);
        if (a.K == 2) return launch_ch<RULE, ARITH, 1>(a, 3, num_sms, stream);
        if (a.K <= 4) return launch_ch<RULE, ARITH, 2>(a, 3, num_sms, stream);
        if constexpr (ARITH == kArithExact) {
            // More values per push: four slices at a time leave them the registers.
            if (a.K == 5) return launch_ch<RULE, ARITH, 2>(a, 4, num_sms, stream);
            if (a.K <= 7) return launch_ch<RULE, ARITH, 8>(a, 2, num_sms, stream);
            return launch_ch<RULE, ARITH, 4>(a, 3, num_sms, stream);
        } else {
            if (a.K <= 6) return launch_ch<RULE, ARITH, 2>(a, 4, num_sms, stream);
            if (a.K <= 8) return launch_ch<RULE, ARITH, 4>(a, 3, num_sms, stream);
            if (a.K <= 12) return launch_ch<RULE, ARITH, 4, false, 256>(a, 3, num_sms, stream);
            return launch_ch<RULE, ARITH, 8, false, 256>(a, 2, num_sms, stream);
        }
    }
}

}  // namespace

cudaError_t launch_dense(const DenseArgs& a, int rule, bool exact, int num_sms,
                         cudaStream_t stream, int64_t* launches) {
    const bool ftz = a.sp.eps >= kFtzSafeEps;
    cudaError_t st;
    if (rule == kRuleSgd)
        st = launch_rule<kRuleSgd, kArithApprox>(a, num_sms, stream);  // exact in every mode
    else if (rule == kRuleFasgd)
        st = exact ? launch_rule<kRuleFasgd, kArithExact>(a, num_sms, stream)
             : ftz ? launch_rule<kRuleFasgd, kArithApproxFtz>(a, num_sms, stream)
                   : launch_rule<kRuleFasgd, kArithApprox>(a, num_sms, stream);
    else
        st = exact ? launch_rule<kRuleFasgdStd, kArithExact>(a, num_sms, stream)
             : ftz ? launch_rule<kRuleFasgdStd, kArithApproxFtz>(a, num_sms, stream)
                   : launch_rule<kRuleFasgdStd, kArithApprox>(a, num_sms, stream);
    if (st == cudaSuccess) ++*launches;
    return st;
}

}  // namespace fasgd
