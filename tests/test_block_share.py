"""Every parameter of a dense pass belongs to exactly one block's share: the
geometry of the ring's tiles and pieces (kernels.cuh, BlockShare), compiled for
the host and checked over sizes around its edges."""

import os
import subprocess

from paper_1601_04033_gb300 import build

SRC = r"""
#include <cstdio>
#include <vector>
#include "kernels.cuh"
int main() {
    const int64_t sizes[] = {0, 4, 124, 128, 132, 1024, 19456, 19460, 152 * 128, 152 * 128 + 4,
                             152 * 2048 - 4, 152 * 2048, 152 * 2048 + 4, 152 * 2048 * 3 + 127 * 4,
                             5000000, 1290508, 7848, 304 * 1024 * 2 + 8, 20000004};
    for (int64_t P : sizes)
        for (int shape = 0; shape < 3; ++shape) {
            const int tile = shape == 1 ? 1024 : 2048;
            const int64_t blocks = shape == 0 ? 152 : shape == 1 ? 304 : 7;
            std::vector<unsigned char> seen(P / 4, 0);
            for (int64_t b = 0; b < blocks; ++b) {
                const fasgd::BlockShare s(P, tile, blocks, b);
                for (int64_t t = 0; t < s.tiles; ++t) {
                    const int64_t o = s.offset(t), n = s.length(t);
                    if (o < 0 || n < 1 || n > tile || o + n > P || o % 4 || n % 4) return std::printf("bounds %lld\n", (long long)P), 1;
                    for (int64_t q = o / 4; q < (o + n) / 4; ++q) ++seen[q];
                }
            }
            for (unsigned char c : seen)
                if (c != 1) return std::printf("cover %lld\n", (long long)P), 1;
        }
    return 0;
}
"""


def test_every_quad_has_one_owner(tmp_path):
    src, exe = tmp_path / "share.cu", tmp_path / "share"
    src.write_text(SRC)
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-O1", f"-I{build.INCLUDE}", f"-I{build.CSRC}",
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, env=dict(os.environ))
    assert r.returncode == 0, r.stdout
