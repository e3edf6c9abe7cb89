// Device-to-device copies of the server's arrays into a caller's buffers
// (fasgd_pull, fasgd_get_state) on the handle's own stream.
//
// Bound by HBM (8 bytes per value) for large arrays and by launch latency for
// small ones.  A kernel on the handle's stream, launched as a programmatic
// dependent of the pass before it, replaces a cudaMemcpyAsync on a second
// stream between two event waits (a stream hop each way), and the arrays of a
// checkpoint go in one launch.  Measured per step from Python, before / now:
// push + apply + pull at P = 7,850 8.9 / 7.3 us, at 1.29M 20.4 / 11.0 us, K = 8
// at 25M 264 / 252 us; five pushes + apply + pull + whole state at 5M
// 127 / 89 us.

#include "kernels.cuh"
#include "pdl.cuh"

namespace fasgd {
namespace {

constexpr int kCopyThreads = 256;

// UNROLL quads per thread, every load issued before the stores; blockIdx.y
// names the array.  VEC: dst is 16-byte aligned (src always is).
template <int UNROLL, bool VEC>
__global__ void __launch_bounds__(kCopyThreads) copy_kernel(const __grid_constant__ CopyArgs a) {
    pdl_wait();
    pdl_trigger();
    const float* src = a.src[blockIdx.y];
    float* dst = a.dst[blockIdx.y];
    const int64_t n = VEC ? a.P >> 2 : a.P;   // quads, or values
    const int64_t i0 = (int64_t)blockIdx.x * (kCopyThreads * UNROLL) + threadIdx.x;
    if constexpr (VEC) {
        float4 x[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (i0 + u * kCopyThreads < n) x[u] = reinterpret_cast<const float4*>(src)[i0 + u * kCopyThreads];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (i0 + u * kCopyThreads < n) reinterpret_cast<float4*>(dst)[i0 + u * kCopyThreads] = x[u];
        const int64_t p = 4 * n + threadIdx.x;   // the last P mod 4 values
        if (blockIdx.x == 0 && p < a.P) dst[p] = src[p];
    } else {
        float x[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (i0 + u * kCopyThreads < n) x[u] = src[i0 + u * kCopyThreads];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (i0 + u * kCopyThreads < n) dst[i0 + u * kCopyThreads] = x[u];
    }
}

template <int UNROLL, bool VEC>
cudaError_t launch(const CopyArgs& a, cudaStream_t stream) {
    const int64_t n = VEC ? a.P >> 2 : a.P;
    const int64_t per = (int64_t)kCopyThreads * UNROLL;
    int64_t grid = (n + per - 1) / per;
    if (grid < 1) grid = 1;
    return launch_pdl(copy_kernel<UNROLL, VEC>, dim3((unsigned)grid, (unsigned)a.count),
                      kCopyThreads, 0, stream, a);
}

}  // namespace

cudaError_t launch_copy(const CopyArgs& a, int num_sms, cudaStream_t stream) {
    bool vec = true;
    for (int i = 0; i < a.count; ++i) vec = vec && (reinterpret_cast<uintptr_t>(a.dst[i]) & 15) == 0;
    if (!vec) return launch<4, false>(a, stream);
    // One quad per thread while that fits one wave of eight blocks per SM (the
    // fewest loads in a row), else four loads in flight per thread.
    const bool small = (a.P >> 2) * a.count <= (int64_t)num_sms * 8 * kCopyThreads;
    return small ? launch<1, true>(a, stream) : launch<4, true>(a, stream);
}

}  // namespace fasgd
