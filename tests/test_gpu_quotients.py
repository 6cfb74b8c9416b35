"""The kernels' quotients by a reciprocal against the general division, bit for
bit, on the device: a driver compiled from the library's own headers."""
import os
import subprocess

import pytest

from paper_2510_12174_gb300 import build as b

pytestmark = pytest.mark.gpu

DRIVER = r"""
#include <cstdio>
#include "unigs_internal.cuh"
#include "bwd_pair.cuh"
using namespace unigs;

__device__ uint64_t mix(uint64_t x) {
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}
// 2^e (1 + m 2^-23); a quarter of the mantissas within 16 of 0 or of all ones
__device__ float make(int e, uint64_t r) {
    uint32_t m = (uint32_t)r & 0x7fffffu;
    if ((r >> 60) < 2) m &= 15u;
    if ((r >> 60) == 2 || (r >> 60) == 3) m |= 0x7ffff0u;
    return __uint_as_float((uint32_t)(e + 127) << 23 | m);
}
__global__ void check(unsigned long long per, unsigned long long* out) {
    const unsigned long long id = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    unsigned long long bad_tile = 0, bad_T = 0, seen = 0;
    for (unsigned long long i = 0; i < per; ++i) {
        const uint64_t a = mix(2 * (id * per + i)), c = mix(2 * (id * per + i) + 1);
        // the tile test: diagonals of the conic in [2^-60, 2^60], all of them
        // with a reciprocal; |n| from 2^-100 to 2^92
        const float d = make((int)((a >> 32) % 120) - 60, a ^ c << 7);
        const float n = copysignf(make((int)((c >> 32) % 192) - 100, c), (a >> 31) & 1 ? 1.f : -1.f);
        const float cr[CULL_FLOATS] = {0.f, 0.f, d, 0.f, d, 0.f, 0.f, 0.f};
        const CullTest t = cull_test(cr);
        const float q = __fdiv_rn(n, d);
        if (t.yA == 0.f || t.yC != t.yA) ++bad_tile;
        if (fabsf(q) >= 0x1p-125f && fabsf(q) < 0x1p127f) {
            ++seen;
            if (__float_as_uint(div_recip(n, d, t.yA)) != __float_as_uint(q)) ++bad_tile;
        }
        // the transmittance: 1 - alpha in [2^-24, 1], T in [2^-100, 1)
        const float alpha = i & 1 ? (float)(a >> 40) * 0x1p-24f : 1.f - make(-1 - (int)(a >> 40) % 24, c);
        const float om = 1.f - alpha;
        const float T = make(-(int)((c >> 40) % 100) - 1, a ^ c);
        if (om > 0.f &&
            __float_as_uint(restored_T(T, om, rcp_ftz(om))) != __float_as_uint(__fdiv_rn(T, om)))
            ++bad_T;
    }
    atomicAdd(out, bad_tile);
    atomicAdd(out + 1, bad_T);
    atomicAdd(out + 2, seen);
}
int main() {
    unsigned long long *d, h[3];
    cudaMalloc(&d, sizeof(h));
    cudaMemset(d, 0, sizeof(h));
    check<<<1216, 256>>>(1000, d);
    if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu %llu %llu\n", h[0], h[1], h[2]);
    return h[0] || h[1] || h[2] < 200000000ull;
}
"""


def test_quotients_are_the_rounded_ones(tmp_path):
    """311M pairs of each kind, divisors next to powers of two among them."""
    src, exe = tmp_path / "quotients.cu", tmp_path / "quotients"
    src.write_text(DRIVER)
    subprocess.run([b._nvcc(), *b.NVCC_FLAGS, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, "tile test, transmittance, compared: " + r.stdout
