// B-FASGD transmission decisions, per parameter (paper Sec. 2.3, Eq. 9): the
// send (push) or fetch decision and the compaction of the kept entries into
// an ascending index list and the matching values (the push's gradient, or
// the server's theta for a fetch).  Push and fetch draws come from separate
// Philox counter streams (bit 31 of the client word).
//
// Two kernels, on the caller's stream:
//   1. decide:  per tile of 4096 parameters (one block), draw u_p
//               (Philox4x32-10), take the Eq. 9 decision against v_p, store one
//               bit per parameter and the tile's count of kept entries;
//   2. compact: per tile, the sum of the earlier tiles' counts gives its place
//               in the lists; the kept entries are written there in order.
// (Beyond 8192 tiles a scan kernel between them forms those sums once, so that
// the tiles do not each read all the counts before theirs.)  The order of the
// output is the order of p, so the result is unique and does not depend on the
// launch; no atomics, and no block waits for another.
//
// Bounds.  decide: the multiply and ALU pipes (ncu at 25M: 24.3 us, the fused
// multiply-add heavy pipe 67 % and the ALU 57 % busy, DRAM 4.1 TB/s):
// Philox4x32-10 is some 15 instructions per parameter, the test 4, on packed
// fp32 pairs, and one funnel shift takes its sign bit into the lane's word.
// compact: HBM and latency (23.6 us for 103 MB read and 40 MB written).
// Each lane decides quads 32 it + lane (it = 0 .. 7) of its warp's 1024, so its
// bits are in another order than the parameters': an 8 x 8 transposition of
// nibbles among eight lanes (three shuffles) and one more shuffle give lane l
// the 32 bits of parameters 32 l .. 32 l + 31.  Each lane then writes its set
// bits' offsets at their ranks into shared memory (one step per kept entry
// instead of tests per parameter: 0.46 instead of 0.69 warp instructions per
// parameter at 20 % kept), and consecutive lanes fetch the kept values, so that
// only their sectors are read, and write consecutive entries.  A warp that keeps
// more than a third of its 1024 reads all of them, in the decision's quads, and
// orders 128 parameters at a time (kDenseSpan).
// Tiles of 4096, blocks of 128 threads (the decision: eight per SM, for mid-sized
// models 256 or 512 threads; the compaction: ten, as many as hold its registers):
// short last waves, and work for every SM from 0.6M parameters on.
// The whole select of 25M parameters at 20 % kept: 57 -> about 46 us with the
// scan kernel gone (exchange of four clients 1068 -> 976 us).
//
// Tried as one kernel (the compaction's memory time under the decision's ALU
// time): warps that wait for the counts of earlier tiles took 140 us per 25M
// one tile each (the polls of the same few words), and 57 us persistent with
// three decided tiles in hand (tickets for the tiles, one address, cost 2.3 ns
// an atomic).  Values prefetched into L2 by decide: 1014 against 986 us.

#include <type_traits>

#include "eq9.cuh"
#include "kernels.cuh"
#include "pdl.cuh"
#include "update.cuh"

namespace fasgd {
namespace {

// A span of 1024 parameters is one word of bits per lane of a warp.  compact: a
// span per warp.  decide: QUADS quads per lane, so that a warp takes a span (8),
// a half or a quarter of one.
constexpr int kSpan = 1024;
constexpr int kThreads = kSelectTile / 32;
constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xffffffffu;
// Entries kept from which on a span is read whole (copy_dense_span).  The serial
// step per kept entry and the scattered fetches behind the first 256 cost more
// than the tests per parameter from about a third on.  The whole select, all
// spans the sparse way -> as it is: 25M at 35 % kept 56.4 -> 53.3 us, 60 %
// 82.2 -> 60.2, 100 % 127.5 -> 70.8 (300 MB at 6.5 TB/s behind the decision's
// 25 us); 1.29M 8.4 -> 7.6, 11.0 -> 7.3, 18.4 -> 8.4; below 30 % kept within
// 3 % either way.
constexpr int kDenseSpan = 340;

__device__ __forceinline__ uint32_t smem_address(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// This lane's quads of v in the warp's parameters from `start` (zero past P).
template <int QUADS>
__device__ __forceinline__ void load_quads(float4 (&q)[QUADS], const float* v, int64_t start, int64_t P,
                                          int lane) {
    const int64_t e = start + 4 * lane;
    if (start + 128 * QUADS <= P) {
#pragma unroll
        for (int it = 0; it < QUADS; ++it) q[it] = __ldcs(reinterpret_cast<const float4*>(v + e + 128 * it));
    } else {
#pragma unroll
        for (int it = 0; it < QUADS; ++it) {
            const int64_t p = e + 128 * it;
            q[it].x = p < P ? v[p] : 0.f;
            q[it].y = p + 1 < P ? v[p + 1] : 0.f;
            q[it].z = p + 2 < P ? v[p + 2] : 0.f;
            q[it].w = p + 3 < P ? v[p + 3] : 0.f;
        }
    }
}

// The sign of u d - a 2^24 for two parameters (send_test's difference, as
// packed operations): negative means sent.
template <bool SCALE_D>
__device__ __forceinline__ void send_difference(uint32_t w0, uint32_t w1, float v0, float v1, Pair c,
                                                Pair eps_b, float& s0, float& s1) {
    const Pair a = add2(pair(v0, v1), eps_b);
    const Pair d = add2(a, c);
    const Pair u = pair((float)(w0 >> 8), (float)(w1 >> 8));   // exact: below 2^24
    if (SCALE_D) {
        const Pair scale = pair(5.9604644775390625e-8f, 5.9604644775390625e-8f);
        unpack(fma2(u, mul2(d, scale), mul2(a, pair(-1.f, -1.f))), s0, s1);
    } else {
        unpack(fma2(u, d, mul2(a, pair(-16777216.0f, -16777216.0f))), s0, s1);
    }
}

// Bit 4 it + j: parameter start + 128 it + 4 lane + j is sent.
template <bool SCALE_D, int QUADS>
__device__ __forceinline__ uint32_t quad_bits(const SelectArgs& a, const float4 (&v)[QUADS], uint32_t start,
                                              int lane) {
    const Pair c = pair(a.c, a.c), eps_b = pair(a.eps_b, a.eps_b);
    uint32_t bits = 0;
#pragma unroll
    for (int it = QUADS - 1; it >= 0; --it) {
        const uint32_t e = start + 128 * it + 4 * lane;   // P < 2^31
        const Philox4 r = philox4x32_10(e >> 2, a.client_word, a.push_lo, a.push_hi, a.round_key0, a.round_key1);
        float s[4];
        send_difference<SCALE_D>(r.x[0], r.x[1], v[it].x, v[it].y, c, eps_b, s[0], s[1]);
        send_difference<SCALE_D>(r.x[2], r.x[3], v[it].z, v[it].w, c, eps_b, s[2], s[3]);
#pragma unroll
        for (int j = 3; j >= 0; --j) {
            if (SCALE_D)   // c = +inf can make a NaN: not sent
                bits = 2 * bits + (s[j] < 0.f ? 1u : 0u);
            else           // one funnel shift takes the sign in
                bits = __funnelshift_l(__float_as_uint(s[j]), bits, 1);
        }
    }
    return bits;
}

// From this lane's quads' bits (nibble it: quad 32 it + lane) to the bits of
// parameters 32 lane .. 32 lane + 31 of the span.
__device__ __forceinline__ uint32_t lane_word(uint32_t x, int lane) {
    // Nibble (lane & 7, it) <-> (it, lane & 7) within each group of eight lanes.
    uint32_t y = __shfl_xor_sync(kFull, x, 4);
    x = __byte_perm(x, y, (lane & 4) ? 0x3276 : 0x5410);
    y = __shfl_xor_sync(kFull, x, 2);
    x = __byte_perm(x, y, (lane & 2) ? 0x3715 : 0x6240);
    y = __shfl_xor_sync(kFull, x, 1);
    x = (lane & 1) ? (x & 0xf0f0f0f0u) | ((y >> 4) & 0x0f0f0f0fu) : (x & 0x0f0f0f0fu) | ((y << 4) & 0xf0f0f0f0u);
    // Lane 8 a + b now holds word 4 b + a.
    return __shfl_sync(kFull, x, 8 * (lane & 3) + (lane >> 2));
}

// SCALE_D: the form of the Eq. 9 test for this call's c (send_form).
template <bool SCALE_D, int QUADS>
__global__ void __launch_bounds__(kSelectTile / (4 * QUADS), QUADS) bfasgd_decide_kernel(const __grid_constant__ SelectArgs a) {
    constexpr int kDecideWarps = kSelectTile / (128 * QUADS), kParts = 8 / QUADS;   // warps per span
    __shared__ int32_t warp_cnt[kDecideWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t start = (int64_t)blockIdx.x * kSelectTile + warp * (128 * QUADS);
    pdl_wait();
    pdl_trigger();
    float4 v[QUADS];
    load_quads(v, a.v, start, a.P, lane);
    uint32_t bits = quad_bits<SCALE_D>(a, v, (uint32_t)start, lane);
    if (start + 128 * QUADS > a.P) {   // parameters past P are never sent
#pragma unroll
        for (int it = 0; it < QUADS; ++it) {
            const int64_t left = a.P - (start + 128 * it + 4 * lane);
            const uint32_t keep = left >= 4 ? 0xfu : left <= 0 ? 0u : (1u << left) - 1u;
            bits &= ~((~keep & 0xfu) << (4 * it));
        }
    }
    // This warp's part of the lane's word of the span (quads 32 it + lane).
    using Part = typename std::conditional<QUADS == 8, uint32_t,
                                           typename std::conditional<QUADS == 4, uint16_t, uint8_t>::type>::type;
    reinterpret_cast<Part*>(a.mask)[kParts * ((start >> 10) * 32 + lane) + warp % kParts] = (Part)bits;
    const int n = (int)__reduce_add_sync(kFull, (uint32_t)__popc(bits));
    if (lane == 0) warp_cnt[warp] = n;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t t = 0;
#pragma unroll
        for (int w = 0; w < kDecideWarps; ++w) t += warp_cnt[w];
        a.tile_count[blockIdx.x] = (uint16_t)t;
    }
}

template <int QUADS>
cudaError_t launch_decide(const SelectArgs& a, cudaStream_t stream) {
    const auto kernel = send_form(a.c) ? bfasgd_decide_kernel<true, QUADS> : bfasgd_decide_kernel<false, QUADS>;
    return launch_pdl(kernel, (unsigned)a.ntiles, kSelectTile / (4 * QUADS), 0, stream, a);
}

constexpr int kScanThreads = 1024;
// More tiles than this (33.5M parameters): their bases come from the scan
// kernel (4 us); up to there each tile reads the counts before its own (16 KB
// at most, on average half, from L2), in the shadow of its other loads.
constexpr int kScanTiles = 8192;

__global__ void __launch_bounds__(kScanThreads) bfasgd_scan_kernel(const __grid_constant__ SelectArgs a) {
    __shared__ int64_t warp_sum[kScanThreads / 32];
    pdl_wait();
    pdl_trigger();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (a.ntiles + kScanThreads - 1) / kScanThreads;
    const int lo = tid * per;
    const int hi = min(lo + per, a.ntiles);
    // Up to four counts per thread (P up to 32M) are loaded at once and kept.
    constexpr int kKeep = 4;
    int32_t kept[kKeep];
    int64_t local = 0;
    if (per <= kKeep) {
#pragma unroll
        for (int k = 0; k < kKeep; ++k) kept[k] = lo + k < hi ? (int32_t)a.tile_count[lo + k] : 0;
#pragma unroll
        for (int k = 0; k < kKeep; ++k) local += kept[k];
    } else {
        for (int t = lo; t < hi; ++t) local += a.tile_count[t];
    }
    // Inclusive scan of the per-thread sums across the block.
    int64_t incl = local;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t s = warp_sum[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int64_t y = __shfl_up_sync(kFull, s, off);
            if (lane >= off) s += y;
        }
        warp_sum[lane] = s;  // inclusive over warps
    }
    __syncthreads();
    int64_t run = incl - local + (warp > 0 ? warp_sum[warp - 1] : 0);  // exclusive prefix
    if (per <= kKeep) {
#pragma unroll
        for (int k = 0; k < kKeep; ++k)
            if (lo + k < hi) {
                a.tile_base[lo + k] = run;
                run += kept[k];
            }
    } else {
        for (int t = lo; t < hi; ++t) {
            a.tile_base[t] = run;
            run += a.tile_count[t];
        }
    }
    if (tid == kScanThreads - 1) *a.count = warp_sum[kScanThreads / 32 - 1];
}

// A span with few entries kept (below kDenseSpan): each lane writes its set bits'
// offsets at their ranks into shared memory, and consecutive lanes fetch the kept
// values, kHeld of them per lane ahead of the barrier behind which the place in
// the lists is known.
constexpr int kHeld = 8;
struct SparseSpan {
    float x[kHeld];
    int o[kHeld];
    // word: the bits of parameters 32 lane .. 32 lane + 31; incl: the entries
    // kept up to those.
    __device__ __forceinline__ void load(const float* src, uint32_t word, int incl, int kept, int lane,
                                         uint16_t* off) {
        // From the highest bit down: one step per kept entry.
        for (int r = incl - 1; word != 0; --r) {
            const int b = 31 - __clz((int)word);
            off[r] = (uint16_t)(32 * lane + b);
            word ^= 1u << b;
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            const int k = lane + 32 * i;
            if (k < kept) {
                o[i] = off[k];
                x[i] = __ldcs(src + o[i]);
            }
        }
    }
    __device__ __forceinline__ void store(const SelectArgs& a, int kept, int64_t start, int lane,
                                          const uint16_t* off, int32_t out) const {
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            const int k = lane + 32 * i;
            if (k < kept) {
                a.idx[out + k] = (int32_t)start + o[i];
                a.val[out + k] = x[i];
            }
        }
        for (int k = lane + 32 * kHeld; k < kept; k += 32) {
            const int p = off[k];
            a.idx[out + k] = (int32_t)start + p;
            a.val[out + k] = __ldcs(a.values + start + p);
        }
    }
};

// A span with many: every value is read, in the quads that the lane's bits are
// of (nibble it: quad 32 it + lane), and each pass of 128 parameters puts its
// kept entries in order in shared memory (two passes' room: one wait per pass)
// for coalesced stores.
__device__ __forceinline__ void copy_dense_span(const SelectArgs& a, uint32_t bits, int64_t start, int lane,
                                                uint2* stage, int32_t out) {
    // Kept entries per nibble, then their running sums over the lanes, four
    // passes to a word (a pass keeps 128 at most): even passes, odd passes.
    uint32_t n = bits - ((bits >> 1) & 0x55555555u);
    n = (n & 0x33333333u) + ((n >> 2) & 0x33333333u);
    uint32_t even = n & 0x0f0f0f0fu, odd = (n >> 4) & 0x0f0f0f0fu;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t e = __shfl_up_sync(kFull, even, d), o = __shfl_up_sync(kFull, odd, d);
        if (lane >= d) {
            even += e;
            odd += o;
        }
    }
    constexpr int kAtOnce = 4;   // quads per lane in flight: eight would cost the kernel a third of its warps
    float4 q[kAtOnce];
    const uint32_t all_even = __shfl_sync(kFull, even, 31), all_odd = __shfl_sync(kFull, odd, 31);
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        if (it % kAtOnce == 0) load_quads(q, a.values, start + 128 * it, a.P, lane);
        const int sh = 8 * (it >> 1);
        const int total = (int)(((it & 1) ? all_odd : all_even) >> sh & 0xffu);
        int r = (int)(((it & 1) ? odd : even) >> sh & 0xffu) - (int)(n >> (4 * it) & 0xfu);
        const uint32_t e = (uint32_t)start + 128 * it + 4 * lane;   // P < 2^31
        const float4 v = q[it % kAtOnce];
        const uint32_t x[4] = {__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w)};
        uint2* s = stage + 128 * (it & 1);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (bits >> (4 * it + j) & 1u) s[r++] = make_uint2(e + j, x[j]);
        __syncwarp();
        for (int k = lane; k < total; k += 32) {
            const uint2 y = s[k];
            a.idx[out + k] = (int32_t)y.x;
            a.val[out + k] = __uint_as_float(y.y);
        }
        out += total;
    }
}

// SCANNED: tile_base holds the sums (bfasgd_scan_kernel), else the block adds
// the counts before its tile.
template <bool SCANNED>
__global__ void __launch_bounds__(kThreads, 10) bfasgd_compact_kernel(const __grid_constant__ SelectArgs a) {
    __shared__ __align__(16) unsigned char s_span[kWarps][2 * kSpan];
    __shared__ int32_t warp_cnt[kWarps], warp_sum[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t start = (int64_t)blockIdx.x * kSelectTile + warp * kSpan;
    pdl_wait();
    pdl_trigger();
    const uint32_t bits = a.mask[(start >> 5) + lane];
    int32_t tile_out = 0;   // places in the lists are below P < 2^31
    int32_t before = 0;
    if (SCANNED) {
        tile_out = (int32_t)a.tile_base[blockIdx.x];
    } else {
        // Eight counts per load; the last load's own and later ones are left out.
        for (int t = 8 * threadIdx.x; t < (int)blockIdx.x; t += 8 * kThreads) {
            const uint4 q = *reinterpret_cast<const uint4*>(a.tile_count + t);
            const uint32_t c[4] = {q.x, q.y, q.z, q.w};
            const int left = (int)blockIdx.x - t;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (2 * i < left) before += (int32_t)(c[i] & 0xffffu);
                if (2 * i + 1 < left) before += (int32_t)(c[i] >> 16);
            }
        }
    }
    const uint32_t word = lane_word(bits, lane);
    int incl = __popc(word);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) warp_cnt[warp] = incl;
    if (!SCANNED) {
        before = (int32_t)__reduce_add_sync(kFull, (uint32_t)before);
        if (lane == 0) warp_sum[warp] = before;
    }
    const int kept = __shfl_sync(kFull, incl, 31);
    const bool sparse = kept < kDenseSpan;   // the whole warp's
    uint16_t* off = reinterpret_cast<uint16_t*>(s_span[warp]);
    SparseSpan span;
    if (sparse) span.load(a.values + start, word, incl, kept, lane, off);
    __syncthreads();
    int32_t ahead = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        if (!SCANNED) ahead += warp_sum[w];
        if (w < warp) ahead += warp_cnt[w];
    }
    const int32_t out = tile_out + ahead;
    if (sparse)
        span.store(a, kept, start, lane, off, out);
    else
        copy_dense_span(a, bits, start, lane, reinterpret_cast<uint2*>(s_span[warp]), out);
    if (!SCANNED && blockIdx.x == gridDim.x - 1 && warp == kWarps - 1 && lane == 0) *a.count = (int64_t)out + kept;
}

}  // namespace

void select_key_schedule(SelectArgs& a, uint64_t seed) {
    philox_key_schedule(seed, a.round_key0, a.round_key1);
}

cudaError_t launch_select(const SelectArgs& a, cudaStream_t stream, int64_t* launches) {
    // Quads per lane: from 1.4 to 7.2 tiles per SM shorter chains of draws per
    // warp (and more warps) pay; below that a tile's 16 warps would crowd one SM
    // while others idle, above it the SMs are full anyway.  Four exchanges
    // without a pull, one after the other on the same buffers, with 2 / 4 / 8
    // (the compaction then as it was before kDenseSpan), us: 600,000 78 / 72 / 72, 800,000 83 / 84 / 80,
    // 1.0M 88 / 92 / 93, 1.29M 90 / 101 / 107, 1.6M 109 / 109 / 119, 2M 122 /
    // 117 / 127, 4M 207 / 196 / 196, 8M 372 / 356 / 350.
    cudaError_t st = a.P > 850'000 && a.P <= 1'500'000     ? launch_decide<2>(a, stream)
                     : a.P > 1'500'000 && a.P <= 4'500'000 ? launch_decide<4>(a, stream)
                                                           : launch_decide<8>(a, stream);
    if (st != cudaSuccess) return st;
    ++*launches;
    const bool scan = a.ntiles > kScanTiles;
    if (scan) {
        st = launch_pdl(bfasgd_scan_kernel, 1, kScanThreads, 0, stream, a);
        if (st != cudaSuccess) return st;
        ++*launches;
    }
    const auto compact = scan ? bfasgd_compact_kernel<true> : bfasgd_compact_kernel<false>;
    st = launch_pdl(compact, (unsigned)a.ntiles, kThreads, 0, stream, a);
    if (st != cudaSuccess) return st;
    ++*launches;
    return cudaSuccess;
}

}  // namespace fasgd

// ---------------------------------------------------------------------------
// Allocation-free variant of bfasgd_select_compact for callers that may not
// allocate device memory (see include/fasgd.h).  The same kernels run
// with their scratch in one fixed static device array instead of handle-owned
// buffers.
// ---------------------------------------------------------------------------
#include <cmath>
#include <cstdio>
#include <mutex>

namespace fasgd {
void set_handleless_error(const char* msg);  // defined in runtime.cu
}

namespace {

constexpr int64_t kNoallocTiles = BFASGD_NOALLOC_PMAX / fasgd::kSelectTile;          
constexpr int64_t kNoallocMaskBytes = kNoallocTiles * fasgd::kSelectTileWords * 4;  // 2 MiB
constexpr int64_t kNoallocCountBytes = kNoallocTiles * 2;
static_assert(kNoallocMaskBytes + kNoallocCountBytes <= BFASGD_NOALLOC_SCRATCH_BYTES,
              "scratch size in fasgd.h out of date");
static_assert(kNoallocMaskBytes % 256 == 0 && kNoallocTiles % 8 == 0, "scratch layout");
static_assert(kNoallocTiles <= fasgd::kScanTiles, "no tile bases here");

// Mask words, then 16-bit tile counts.
static __device__ __align__(256) unsigned char g_noalloc_scratch[BFASGD_NOALLOC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
void* g_noalloc_addr[kMaxDevices] = {};

// Device address of the static scratch on the current device, looked up once
// per device.  Host code cannot use the symbol itself as a device pointer.
// The look-up is a runtime call that does not belong in a stream capture:
// if it is still to be made while `stream` is capturing, *capturing is set
// and nothing is done.
cudaError_t noalloc_scratch(cudaStream_t stream, unsigned char** out, bool* capturing) {
    *capturing = false;
    int dev = 0;
    cudaError_t st = cudaGetDevice(&dev);
    if (st != cudaSuccess) return st;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (g_noalloc_addr[dev] == nullptr) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        st = cudaStreamIsCapturing(stream, &cs);
        if (st != cudaSuccess) return st;
        if (cs != cudaStreamCaptureStatusNone) {
            *capturing = true;
            return cudaSuccess;
        }
        void* p = nullptr;
        st = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (st != cudaSuccess) return st;
        g_noalloc_addr[dev] = p;
    }
    *out = static_cast<unsigned char*>(g_noalloc_addr[dev]);
    return cudaSuccess;
}

bool aligned_to(const void* p, uintptr_t a) {
    return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0;
}

int noalloc_fail(int code, const char* msg) {
    fasgd::set_handleless_error(msg);
    return code;
}

}  // namespace

extern "C" int bfasgd_select_compact_noalloc(int64_t P, const float* grad, const float* v,
                                             float c, float eps_b, uint64_t seed, int32_t client,
                                             uint64_t push_no, int32_t* idx, float* val,
                                             int64_t* n_dev, void* stream) {
    if (P < 1 || P > BFASGD_NOALLOC_PMAX) {
        char buf[160];
        snprintf(buf, sizeof buf,
                 "bfasgd_select_compact_noalloc: P=%lld outside [1, %lld], the size of its "
                 "static scratch", (long long)P, (long long)BFASGD_NOALLOC_PMAX);
        return noalloc_fail(FASGD_EINVAL, buf);
    }
    if (client < 0) return noalloc_fail(FASGD_EINVAL, "bfasgd_select_compact_noalloc: client < 0");
    if (grad == nullptr || v == nullptr || !aligned_to(grad, 16) || !aligned_to(v, 16))
        return noalloc_fail(FASGD_EINVAL,
                            "bfasgd_select_compact_noalloc: grad and v must be non-NULL "
                            "16-byte aligned device pointers");
    if (idx == nullptr || val == nullptr || n_dev == nullptr || !aligned_to(idx, 4) ||
        !aligned_to(val, 4) || !aligned_to(n_dev, 8))
        return noalloc_fail(FASGD_EINVAL,
                            "bfasgd_select_compact_noalloc: idx, val, n_dev must be non-NULL "
                            "and aligned");
    if (!(c >= 0.f) || !(eps_b >= 0.f) || !std::isfinite(eps_b))
        return noalloc_fail(FASGD_EINVAL,
                            "bfasgd_select_compact_noalloc: need c >= 0 and finite eps_b >= 0");
    unsigned char* scratch = nullptr;
    bool capturing = false;
    cudaError_t st = noalloc_scratch(static_cast<cudaStream_t>(stream), &scratch, &capturing);
    if (st != cudaSuccess)
        return noalloc_fail(FASGD_ECUDA, "bfasgd_select_compact_noalloc: cannot address the "
                                         "static scratch on this device");
    if (capturing)
        return noalloc_fail(FASGD_EINVAL,
                            "bfasgd_select_compact_noalloc: the first call on a device looks up "
                            "its static scratch and must come before any stream capture");
    fasgd::SelectArgs a;
    a.values = grad;
    a.v = v;
    a.idx = idx;
    a.val = val;
    a.count = n_dev;
    a.mask = reinterpret_cast<uint32_t*>(scratch);
    a.tile_count = reinterpret_cast<uint16_t*>(scratch + kNoallocMaskBytes);
    a.tile_base = nullptr;   // too few tiles for the scan kernel
    a.P = P;
    a.ntiles = fasgd::select_tiles(P);
    a.c = c;
    a.eps_b = eps_b;
    fasgd::select_key_schedule(a, seed);
    a.client_word = (uint32_t)client;
    a.push_lo = (uint32_t)push_no;
    a.push_hi = (uint32_t)(push_no >> 32);
    int64_t launches = 0;
    st = fasgd::launch_select(a, static_cast<cudaStream_t>(stream), &launches);
    if (st != cudaSuccess)
        return noalloc_fail(FASGD_ECUDA, cudaGetErrorString(st));
    return FASGD_OK;
}
