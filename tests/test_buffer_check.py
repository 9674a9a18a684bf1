"""Decision on a caller's buffer, whether a kernel accesses it directly, on the
host over a made-up table of allocations (no device, no launch)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2301_10674_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "buffer_check.h"
using namespace fsl;
// device 0: [4096, 8192), directly behind it [8192, 12288), after a gap
// [16384, 20480); host [20480, 24576); device 1: [32768, 36864)
static bool lookup(const void* p, BufferInfo& b) {
    static const BufferInfo table[] = {
        {true, 0, 4096, 4096}, {true, 0, 8192, 4096}, {true, 0, 16384, 4096}, {false, 0, 20480, 4096}, {true, 1, 32768, 4096}};
    for (const BufferInfo& t : table)
        if ((std::uintptr_t)p >= t.base && (std::uintptr_t)p - t.base < t.size) {
            b = t;
            return true;
        }
    return false;
}
int main() {
    struct { std::uintptr_t at; std::size_t bytes, align; } q[] = {
        {4096, 4096, 8}, {4104, 4088, 8}, {8192, 16, 8},     // inside one allocation: yes
        {4104, 4096, 8},     // into the next one
        {8192, 12288, 8},    // over a gap, both ends device memory
        {16384, 4104, 8},    // into host memory
        {4100, 8, 8},        // misaligned
        {0, 8, 8}, {20480, 8, 8}, {32768, 8, 8},             // unknown, host, another device
        {4096, ~(std::size_t)0 - 4095, 8}};                  // a size that wraps around
    for (auto& e : q) std::putchar(kernel_may_access((const void*)e.at, e.bytes, e.align, 0, lookup) ? '1' : '0');
    return 0;
}
"""


def test_only_a_range_inside_one_allocation_is_accessed(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert out == "111" + "0" * 8
