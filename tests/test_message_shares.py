"""The partition of the per-message statistic is a function of P alone: the
launches of a message push's pass and of the kernel that forms its sums,
recorded on the host for GPUs of several sizes (no GPU needed), have one grid,
while a pass that leaves no sums follows the number of SMs."""

import subprocess

from paper_1601_04033_gb300 import build

SRC = r"""
#include <cstdio>
#include <cstring>
#include "pdl.cuh"
namespace fasgd {
static unsigned grids[8];
static int recorded = 0;
template <typename K, typename... A>
cudaError_t record_launch(K, dim3 grid, dim3, size_t, cudaStream_t, A&&...) {
    grids[recorded++ & 7] = grid.x;
    return cudaSuccess;
}
}  // namespace fasgd
#define launch_pdl record_launch
#define cudaGetDevice(p) (*(p) = 0, cudaSuccess)
#define cudaFuncSetAttribute(...) cudaSuccess
#include "dense.cu"
#include "message.cu"

int main() {
    using namespace fasgd;
    int64_t launches = 0;
    for (int64_t P : {int64_t(5), int64_t(311299), int64_t(25000000)})
        for (int sms : {100, 132, 148, 152, 160}) {
            DenseArgs a;
            std::memset(&a, 0, sizeof a);
            a.P = P;
            a.K = 1;
            float2 sums;
            a.msg.partial = &sums;
            recorded = 0;
            for (int rule : {kRuleFasgd, kRuleFasgdStd})
                for (bool exact : {false, true})
                    if (launch_dense(a, rule, exact, sms, nullptr, &launches) != cudaSuccess) return 1;
            MessageArgs m;
            std::memset(&m, 0, sizeof m);
            m.P = P;
            if (launch_message_sums(m, nullptr, &launches) != cudaSuccess) return 1;
            for (int i = 0; i < 5; ++i)
                if (recorded != 5 || grids[i] != grids[0] || grids[0] != 152)
                    return std::printf("P = %lld, %d SMs: grid %u\n", (long long)P, sms, grids[i]), 1;
            a.msg.partial = nullptr;
            recorded = 0;
            if (P > 20000000 && (launch_dense(a, kRuleFasgd, false, sms, nullptr, &launches) != cudaSuccess || grids[0] != (unsigned)sms))
                return std::printf("plain pass on %d SMs: grid %u\n", sms, grids[0]), 1;
        }
    return 0;
}
"""


def test_one_partition_whatever_the_gpu(tmp_path):
    src, exe = tmp_path / "shares.cu", tmp_path / "shares"
    src.write_text(SRC)
    # Host code only matters here: device code stops at PTX, unoptimised.
    r = subprocess.run([build.nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-O0",
                        f"-I{build.INCLUDE}", f"-I{build.CSRC}", str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
