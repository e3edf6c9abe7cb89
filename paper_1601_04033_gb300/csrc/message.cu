// The paper's literal B-FASGD (Sec. 2.3): one Eq. 9 decision per
// transmission opportunity, taken against v = the mean over all parameters
// of the server's moving averages.
//
// The statistic is kept as one float-float sum of v per block of the dense
// pass: the pass of a message push adds its blocks' new v up in registers
// (VSum) as it stores them, each thread its quads of the block's share in
// order, then a fixed tree.  After any other change of v, vbar_partial_kernel
// forms the same sums from v (same shares, same order, same bits).  The shares
// depend on P alone (kMessageBlocks), so a decision depends neither on which
// kernel formed the sums nor on the GPU.  A decision (message_decide, one warp) adds the
// sums in a fixed order, forms vbar = fl32(sum / P) (ff_div_int), draws u
// (Philox4x32-10, word 0 at counter (2^32-1, client + 2^31 * stream, n)) and
// takes the exact Eq. 9 test.
//
//   - A push under the FASGD rules: message_decide_kernel takes the decision
//     while the pass behind it already loads its first tiles' state; the pass
//     applies the pushed gradient, refreshing the client's cache slot as it
//     streams, or the slot.  If the sums had to be formed afresh, the pass takes
//     the decision itself from them (message.cuh), so a push is two kernels.
//   - A fetch, an ASGD/SASGD push and the statistic query:
//     message_resolve_kernel, every block of which takes the decision and, if
//     the message is transmitted, copies src to dst (for a push: the gradient to
//     the client's slot of the server's gradient cache, which the pass that
//     follows reads; for a fetch: theta to the client's copy).
//
// Measured at 25M parameters (eight pushes, eight fetches, a pull): sums per
// 128-parameter chunk with a kernel per decision to combine them 1355 us, these
// 1237 us.  A warp's tree per chunk cost 27 instructions per parameter,
// the running sums 11.

#include "eq9.cuh"
#include "kernels.cuh"
#include "message.cuh"
#include "pdl.cuh"
#include "twosum.cuh"

namespace fasgd {
namespace {

constexpr int kMsgThreads = 256;

constexpr int kSumThreads = 512;   // as the dense pass's consumers: a tile is one quad of each

// The sums the dense pass would leave, from v: thread t of block b adds quad t
// of each tile of the block's share in order (four tiles' loads in flight).
__global__ void __launch_bounds__(kSumThreads) vbar_partial_kernel(const __grid_constant__ MessageArgs a) {
    __shared__ float2 s_sum[kSumThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const BlockShare share(a.P & ~int64_t(3), 4 * kSumThreads, gridDim.x, blockIdx.x);
    pdl_wait();
    pdl_trigger();
    VSum sum;
    for (int64_t t = 0; t < share.tiles; t += 4) {
        float4 x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (t + k < share.tiles && 4 * tid < share.length(t + k))
                x[k] = reinterpret_cast<const float4*>(a.v + share.offset(t + k))[tid];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (t + k < share.tiles && 4 * tid < share.length(t + k)) sum.add(x[k]);
    }
    if (blockIdx.x == gridDim.x - 1 && tid < (int)(a.P & 3))
        sum.add(make_float4(a.v[(a.P & ~int64_t(3)) + tid], 0.f, 0.f, 0.f));
    const float2 w = sum.warp_total();
    if (lane == 0) s_sum[warp] = w;
    __syncthreads();
    if (tid == 0) a.partial[blockIdx.x] = ordered_total<kSumThreads / 32>(s_sum);
}

// One warp: the decision of a push, for the pass behind it (which starts on its
// state meanwhile: this kernel touches none of it).
__global__ void __launch_bounds__(32) message_decide_kernel(const __grid_constant__ MessageArgs a) {
    pdl_wait();
    pdl_trigger();
    float vbar;
    const uint32_t send = message_decide(a.partial, a.nblocks, a.P, a.c, a.eps_b, a.round_key0,
                                         a.round_key1, a.client_word, a.n_lo, a.n_hi, &vbar);
    if (threadIdx.x == 0) {
        *a.decided = send;
        if (a.flag_out != nullptr) *a.flag_out = (int32_t)send;
    }
}

__global__ void __launch_bounds__(kMsgThreads) message_resolve_kernel(const __grid_constant__ MessageArgs a) {
    __shared__ uint32_t s_send;
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x < 32) {
        float vbar;
        const uint32_t send = message_decide(a.partial, a.nblocks, a.P, a.c, a.eps_b,
                                             a.round_key0, a.round_key1, a.client_word, a.n_lo,
                                             a.n_hi, &vbar);
        if (threadIdx.x == 0) {
            s_send = send;
            if (blockIdx.x == 0 && a.flag_out != nullptr) *a.flag_out = (int32_t)send;
            if (blockIdx.x == 0 && a.vbar_out != nullptr) *a.vbar_out = vbar;
        }
    }
    __syncthreads();
    if (!s_send || a.src == nullptr) return;
    const int64_t nq = a.P >> 2;
    const int64_t stride = (int64_t)gridDim.x * kMsgThreads;
    for (int64_t q = (int64_t)blockIdx.x * kMsgThreads + threadIdx.x; q < nq; q += stride)
        reinterpret_cast<float4*>(a.dst)[q] = __ldcs(reinterpret_cast<const float4*>(a.src) + q);
    if (blockIdx.x == 0 && threadIdx.x < (int)(a.P & 3))
        a.dst[4 * nq + threadIdx.x] = a.src[4 * nq + threadIdx.x];
}

}  // namespace

cudaError_t launch_message_sums(const MessageArgs& a, cudaStream_t stream, int64_t* launches) {
    const cudaError_t st = launch_pdl(vbar_partial_kernel, kMessageBlocks, kSumThreads, 0, stream, a);
    if (st == cudaSuccess) ++*launches;
    return st;
}

cudaError_t launch_message_decide(const MessageArgs& a, cudaStream_t stream, int64_t* launches) {
    const cudaError_t st = launch_pdl(message_decide_kernel, 1, 32, 0, stream, a);
    if (st == cudaSuccess) ++*launches;
    return st;
}

cudaError_t launch_message(const MessageArgs& a, int num_sms, cudaStream_t stream,
                           int64_t* launches) {
    cudaError_t st;
    int64_t grid = ((a.P >> 2) + kMsgThreads - 1) / kMsgThreads;
    const int64_t cap = (int64_t)(num_sms > 0 ? num_sms : 1) * 8;
    if (grid > cap) grid = cap;
    if (grid < 1) grid = 1;
    st = launch_pdl(message_resolve_kernel, (unsigned)grid, kMsgThreads, 0, stream, a);
    if (st != cudaSuccess) return st;
    ++*launches;
    return cudaSuccess;
}

}  // namespace fasgd
