"""The device forms of the integer-instruction float64 operations
(csrc/softf64.cuh: the carry-chain rounding and the hardware's seeds, which the
host's check does not run) against the FP64 instructions, bit for bit, over
operands of structured significands and every exponent: prod, root and recip of
any operands, prod_z and prod_nz of operands in their range."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2206_05761_gb300", "csrc")
OUT = os.path.join(ROOT, "paper_2206_05761_gb300", "_build", "softf64_check")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "softf64.cuh"
using namespace hwfv1;

struct Rng {
    uint64_t s;
    __device__ uint64_t next() {
        s ^= s << 13; s ^= s >> 7; s ^= s << 17;
        return s * 0x2545F4914F6CDD1Dull;
    }
};
__device__ uint64_t operand(Rng& r) {
    uint64_t f = r.next() >> 12;
    switch (r.next() % 8) {
        case 0: f = 0; break;
        case 1: f = (1ull << 52) - 1 - r.next() % 8; break;
        case 2: f = r.next() % 16; break;
        case 3: f = (r.next() & 0xFFFFF) << 32; break;
        case 4: f = 1ull << (r.next() % 52); break;
    }
    uint64_t e = r.next() % 4 ? 983 + r.next() % 80 : r.next() % 2048;
    if (r.next() % 64 == 0) e = r.next() % 2 ? r.next() % 3 : 2044 + r.next() % 4;
    return (r.next() & 1) << 63 | e << 52 | f;
}
__device__ double val(uint64_t b) { return __longlong_as_double((long long)b); }
__device__ uint64_t bits(double x) { return (uint64_t)__double_as_longlong(x); }
// differ: not the same bits (two NaNs count as the same)
__device__ bool differ(double got, double want) { return bits(got) != bits(want) && !(isnan(got) && isnan(want)); }

enum { kProd, kProdZ, kProdNz, kRoot, kRecip, kOps };
__global__ void check(uint64_t seed, int n, unsigned long long* wrong, unsigned long long* done) {
    Rng r = {(seed + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) * 0x9E3779B97F4A7C15ull | 1ull};
    for (int k = 0; k < 4; ++k) r.next();
    unsigned long long bad[kOps] = {}, cnt[kOps] = {};
    auto tell = [&](int op, double got, double want) {
        ++cnt[op];
        if (differ(got, want)) ++bad[op];
    };
    for (int i = 0; i < n; ++i) {
        uint64_t p = operand(r), q = operand(r);
        if (i % 4 == 2) {                      // 27-bit factors: products of 53 and 54 bits, ties among them
            p = (p & 0xFFF0000000000000ull) | (r.next() & 0x3FFFFFF) << 26;
            q = (q & 0xFFF0000000000000ull) | (r.next() & 0x3FFFFFF) << (24 + r.next() % 3);
        }
        tell(kProd, prod(val(p), val(q)), __dmul_rn(val(p), val(q)));
        if (mul_in_range((uint32_t)(p >> 32), (uint32_t)(q >> 32))) {
            tell(kProdNz, prod_nz(val(p), val(q)), __dmul_rn(val(p), val(q)));
            uint64_t a = p, b = q;
            if (r.next() % 4 == 0) a &= 1ull << 63;      // signed zeros beside factors in range
            if (r.next() % 4 == 0) b &= 1ull << 63;
            tell(kProdZ, prod_z(val(a), val(b)), __dmul_rn(val(a), val(b)));
        }
        uint64_t x = p;
        if (i % 4 == 1) {                      // next to the square of a 27-bit integer
            const double m = (double)((1ull << 26) | (r.next() & ((1ull << 26) - 1)));
            x = bits(__dmul_rn(__dmul_rn(m, m), r.next() % 2 ? 1.0 : 4.0)) + r.next() % 5 - 2;
        } else if (i % 8 == 3) {               // next to a rounded square
            const double m = val(1023ull << 52 | r.next() >> 12);
            x = bits(__dmul_rn(m, m)) + r.next() % 3 - 1;
        }
        tell(kRoot, root(val(x)), __dsqrt_rn(val(x)));
        x = i % 4 == 1 ? bits(__drcp_rn(val(q))) + r.next() % 5 - 2 : q;
        tell(kRecip, recip(val(x)), __drcp_rn(val(x)));
    }
    for (int o = 0; o < kOps; ++o) {
        atomicAdd(wrong + o, bad[o]);
        atomicAdd(done + o, cnt[o]);
    }
}

int main() {
    unsigned long long *d = nullptr, h[2 * kOps];
    if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 2;
    check<<<152, 256>>>(20, 512, d, d + kOps);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    cudaFree(d);
    const char* name[kOps] = {"prod", "prod_z", "prod_nz", "root", "recip"};
    int bad = 0;
    for (int o = 0; o < kOps; ++o) {
        std::printf("%s: %llu of %llu wrong\n", name[o], h[o], h[kOps + o]);
        bad |= h[o] != 0 || h[kOps + o] < 1000000ull;
    }
    return bad;
}
"""


def test_device_forms_match_the_fp64_instructions():
    from paper_2206_05761_gb300 import _build
    os.makedirs(OUT, exist_ok=True)
    src, exe = os.path.join(OUT, "device.cu"), os.path.join(OUT, "device")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([_build._nvcc(), *_build.ARCH, "-O3", "-std=c++17", "--fmad=false", "-I" + CSRC, src, "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
