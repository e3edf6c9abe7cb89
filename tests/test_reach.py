"""The host's range check in front of copies that a kernel makes (reach.cuh),
compiled for the host over made-up allocations: inside one, to its last byte,
one byte past it, over neighbours, over a gap, and outside every one."""

import subprocess

from paper_1601_04033_gb300 import build

SRC = r"""
#include <cstdio>
#include "reach.cuh"
struct Block { uintptr_t base; size_t size; };
static const Block blocks[] = {{4096, 1000}, {8192, 512}, {8704, 512}, {9216, 256}, {16384, 64}};
static bool find(uintptr_t p, uintptr_t* base, size_t* size) {
    for (const Block& b : blocks)
        if (p >= b.base && p - b.base < b.size) return *base = b.base, *size = b.size, true;
    return false;
}
int main() {
    using namespace fasgd;
    struct { uintptr_t p; size_t bytes; Reach want; } cases[] = {
        {4096, 1000, kReachOne},    {4096, 1001, kReachShort},   {4100, 996, kReachOne},
        {4100, 997, kReachShort},   {5095, 1, kReachOne},        {5096, 1, kReachUnknown},
        {4095, 1, kReachUnknown},   {8192, 512, kReachOne},      {8192, 513, kReachSeveral},
        {8192, 1280, kReachSeveral}, {8192, 1281, kReachShort},  {8700, 517, kReachSeveral},
        {9000, 4096, kReachShort},  {0, 16, kReachUnknown},      {16384, 64, kReachOne},
        {16384, ~size_t(0), kReachShort}};
    int n = 0;
    for (const auto& c : cases) {
        const Reach got = reach(c.p, c.bytes, find);
        if (got != c.want) std::printf("%zu + %zu: %d, want %d\n", (size_t)c.p, c.bytes, got, c.want), ++n;
    }
    return n;
}
"""


def test_reach_over_allocations(tmp_path):
    src, exe = tmp_path / "reach.cpp", tmp_path / "reach"
    src.write_text(SRC.replace("reach.cuh", f"{build.CSRC}/reach.cuh"))
    r = subprocess.run(["g++", "-std=c++17", "-Wall", "-Wextra", str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
