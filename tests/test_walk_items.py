"""The item numbers of a walk, level x case block, beyond 32 bits: the function
that the evaluators number their items with, compiled for the host and driven
across 2^32 against 64-bit arithmetic."""
import os
import subprocess

SRC = r"""
#include "common.cuh"
#include <cstdio>
int main() {
    for (uint32_t ncb : {1u, 2u, 3u, 75u, 256u}) {
        WalkItem a{0u, 0u, 0u};
        uint64_t n = 0, x = 12345;
        for (long step = 0; step < 4000000; ++step) {
            x = x * 6364136223846793005ull + 1442695040888963407ull;
            n += 1 + (x >> 33) % (33u * ncb + 8u);            // what other evaluators took meanwhile
            if (step % 1000 == 0) {                           // far ahead: the same place, other high bits
                const uint64_t far = n + 0x3FFFFF00ull;
                for (; n < far; n += 0x0FFFFFC0ull) {
                    a.take((uint32_t)n, ncb);
                    if (a.level != (uint32_t)(n / ncb) || a.cb != n % ncb) { printf("%llu %u\n", (unsigned long long)n, ncb); return 1; }
                }
            }
            a.take((uint32_t)n, ncb);
            if (a.level != (uint32_t)(n / ncb) || a.cb != n % ncb) { printf("%llu %u\n", (unsigned long long)n, ncb); return 1; }
        }
        if (n >> 33 == 0) return 2;
    }
    return 0;
}
"""


def test_items_beyond_32_bits(tmp_path):
    from paper_2205_03251_gb300 import _build
    (tmp_path / "items.cu").write_text(SRC)
    exe = tmp_path / "items"
    subprocess.check_call([_build._nvcc(), "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                           _build.INCLUDE, "-I", _build.CSRC, "-o", str(exe), str(tmp_path / "items.cu")])
    subprocess.check_call([str(exe)])
