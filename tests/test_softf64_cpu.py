"""The integer-instruction float64 operations (csrc/softf64.cuh) against the
host's IEEE operations, bit for bit, on the operands where a rounding can go
wrong: exact squares and their neighbours, powers of two, all-ones
significands, reciprocals of reciprocals, products next to ties, signed
zeros, every exponent parity, the range's edges; with seeds off by more than
the device's approximations are."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2206_05761_gb300", "csrc")
OUT = os.path.join(ROOT, "paper_2206_05761_gb300", "_build", "softf64_check")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "softf64.cuh"
using namespace hwfv1;

static uint64_t state = 0x9E3779B97F4A7C15ull;
static uint64_t rnd() {
    state ^= state << 13; state ^= state >> 7; state ^= state << 17;
    return state * 0x2545F4914F6CDD1Dull;
}
static double val(uint64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
static uint64_t bits(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
static float fval(uint32_t b) { float x; std::memcpy(&x, &b, 4); return x; }
static uint32_t fbits(float x) { uint32_t b; std::memcpy(&b, &x, 4); return b; }

// a double of structured significand and any exponent
static uint64_t operand() {
    uint64_t f = rnd() >> 12;
    switch (rnd() % 8) {
        case 0: f = 0; break;
        case 1: f = (1ull << 52) - 1 - rnd() % 8; break;
        case 2: f = rnd() % 16; break;
        case 3: f = (rnd() & 0xFFFFF) << 32; break;
        case 4: f = 1ull << (rnd() % 52); break;
    }
    uint64_t e = rnd() % 4 ? 983 + rnd() % 80 : rnd() % 2048;
    if (rnd() % 64 == 0) e = rnd() % 2 ? rnd() % 3 : 2044 + rnd() % 4;
    return (rnd() & 1) << 63 | e << 52 | f;
}

static long fails = 0;
static void check(const char* what, uint64_t x, uint64_t got, double want) {
    if (got != bits(want) && fails++ < 10)
        std::printf("%s(%016llx) = %016llx, want %016llx\n", what, (unsigned long long)x, (unsigned long long)got,
                    (unsigned long long)bits(want));
}

int main(int, char** argv) {
    const long n = std::atol(argv[1]);
    const int off = std::atoi(argv[2]);        // seeds off by up to this many units of the last place
    for (long i = 0; i < n; ++i) {
        const uint64_t a = operand();
        const int d = (int)(rnd() % (2 * off + 1)) - off;
        uint64_t x = a & 0x7FFFFFFFFFFFFFFFull;
        if (i % 4 == 1) {                      // next to the square of a 27-bit integer
            const double m = (double)((1ull << 26) | (rnd() & ((1ull << 26) - 1)));
            x = bits(m * m * (rnd() % 2 ? 1.0 : 4.0)) + rnd() % 5 - 2;
        } else if (i % 8 == 3) {               // next to a rounded square
            const double q = val(1023ull << 52 | rnd() >> 12);
            x = bits(q * q) + rnd() % 3 - 1;
        }
        uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
        if (sqrt_in_range(hi)) {
            const uint32_t y = fbits((float)(1.0 / std::sqrt((double)fval(sqrt_seed_arg(lo, hi))))) + d;
            check("sqrt", x, sqrt_bits(lo, hi, y), std::sqrt(val(x)));
        } else if (x > 0x000FFFFFFFFFFFFFull && x < 0x7FF0000000000000ull) {
            ++fails;                           // every positive normal number is in range
        }
        x = a;
        if (i % 4 == 1) x = bits(1.0 / val(a)) + rnd() % 5 - 2;
        lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
        if (rcp_in_range(hi)) {
            const uint32_t y = fbits((float)(1.0 / (double)fval(rcp_seed_arg(lo, hi)))) + d;
            check("rcp", x, rcp_bits(lo, hi, y), 1.0 / val(x));
        }
        if (a << 1 <= 0x7FF0000000000000ull << 1) {            // (not a NaN)
            check("2 x", a, pow2_bits<1>(a), 2.0 * val(a));
            check("x / 2", a, pow2_bits<-1>(a), 0.5 * val(a));
            check("x / 4", a, pow2_bits<-2>(a), 0.25 * val(a));
        }
        uint64_t p = a, q = operand();
        if (i % 4 == 2) {                      // 27-bit factors: products of 53 and 54 bits, ties among them
            p = (p & 0xFFF0000000000000ull) | (rnd() & 0x3FFFFFF) << 26;
            q = (q & 0xFFF0000000000000ull) | (rnd() & 0x3FFFFFF) << (24 + rnd() % 3);
        }
        const bool in = mul_in_range((uint32_t)(p >> 32), (uint32_t)(q >> 32));
        const double pq = val(p) * val(q);
        const uint64_t m = bits(pq) & 0x7FFFFFFFFFFFFFFFull;
        if (in) {
            check("mul", p, mul_bits<false>((uint32_t)p, (uint32_t)(p >> 32), (uint32_t)q, (uint32_t)(q >> 32)), pq);
            if (rnd() % 2) p &= 1ull << 63;    // signed zeros beside normal factors
            if (rnd() % 2) q &= 1ull << 63;
            check("mul with zeros", p, mul_bits<true>((uint32_t)p, (uint32_t)(p >> 32), (uint32_t)q, (uint32_t)(q >> 32)),
                  val(p) * val(q));
        } else if (m > 0x002FFFFFFFFFFFFFull && m < 0x7FD0000000000000ull &&
                   (p & 0x7FF0000000000000ull) && (q & 0x7FF0000000000000ull)) {
            ++fails;                           // normal factors, a product well inside the normal range
        }
    }
    std::printf("%ld wrong\n", fails);
    return fails != 0;
}
"""


@pytest.fixture(scope="module")
def program():
    os.makedirs(OUT, exist_ok=True)
    src, exe = os.path.join(OUT, "check.cu"), os.path.join(OUT, "check")
    with open(src, "w") as f:
        f.write(PROGRAM)
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    subprocess.run([nvcc if os.path.exists(nvcc) else "nvcc", "-O2", "-std=c++17", "-I" + CSRC, src, "-o", exe],
                   check=True, capture_output=True)
    return exe


# the device's approximations are within 1 (reciprocal) and 2 (inverse square
# root) units of the last place
@pytest.mark.parametrize("off", [0, 4])
def test_integer_float64_operations_match_ieee(program, off):
    r = subprocess.run([program, "8000000", str(off)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
