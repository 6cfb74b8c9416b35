"""The wait of the radix passes' look-back (csrc/lookback.cuh), compiled for the
host and run against words that are published while it polls."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2510_12174_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include <initializer_list>
#include <vector>
#include "lookback.cuh"
// Chunk p holds the count p + 1 and is published once its word was polled
// `after` times (never: chunk `lost`); multiples of `inclusive` publish their prefix.
static int walk(int64_t chunk, int after, int64_t inclusive, int64_t lost, uint32_t* sum) {
    std::vector<int> polled(chunk, 0);
    auto load = [&](int64_t p) -> unsigned long long {
        if (p == lost || polled[p]++ < after) return (6ull << 2 | 2) << 32;
        const bool pre = p % inclusive == 0;
        const unsigned long long c = pre ? (p + 1) * (p + 2) / 2 : p + 1;
        return (7ull << 2 | (pre ? 2 : 1)) << 32 | c;
    };
    return unigs::look_back_walk<8>(load, chunk, 7u, 100u, sum);
}
int main() {
    for (int64_t chunk : {1, 2, 7, 8, 9, 64, 1000})
        for (int after : {0, 1, 90})
            for (int64_t inclusive : {1, 5, 4096}) {
                uint32_t sum = 0;
                const int ok = walk(chunk, after, inclusive, -1, &sum);
                if (!ok || sum != chunk * (chunk + 1) / 2) {
                    printf("chunk %lld after %d inclusive %lld: %d %u\n", (long long)chunk,
                           after, (long long)inclusive, ok, sum);
                    return 1;
                }
            }
    uint32_t sum = 12345;
    if (walk(9, 0, 4096, 7, &sum) || sum != 12345) {
        printf("no give-up\n");
        return 1;
    }
    return 0;
}
"""


def test_limit_is_on_the_wait_for_one_word(tmp_path):
    """Each of up to 1000 predecessors is published once it was polled 90 times:
    no wait reaches the limit of 100, and the walk returns the sum.  A word that
    is never published ends it."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "walk.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "walk"
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
