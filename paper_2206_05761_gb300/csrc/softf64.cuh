// softf64.cuh -- float64 operations in integer instructions, rounded to
// nearest (ties to even) bit for bit as the FP64 instructions round them.
//
// The FP64 pipe takes about 77 cycles per warp and sub-partition for one
// addition or multiplication (0.53 T/s on the whole GPU), the integer pipes
// 1-2 for an instruction, and the two work at the same time.  A square root or
// reciprocal, which the FP64 pipe builds from several of its instructions, is
// far cheaper in some forty integer instructions; a product costs less too
// and leaves the FP64 pipe to the sums.  Measured, cycles per warp and
// sub-partition with 48-64 warps per SM: square root 86-90 against 620 on the
// FP64 pipe, reciprocal 67-71 against 362, product 46 (57 where a factor may be
// zero, 66 with a check of its range) against 77; a product followed by a sum
// takes the time of the sum.
//
// The methods are the usual ones of exact arithmetic: a float seed refined by
// Newton steps in fixed point, each with the residual taken modulo 2^64 (it
// is small, so the low words determine it), and the last bit decided by the
// sign of the exact residual at the midpoint of two neighbouring results.
// A seed only has to be within 2^-20 (reciprocal) or 2^-21 (square root)
// relative of the value it stands for.
//
// Qn below: an integer v stands for v / 2^n.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace hwfv1 {

#ifdef __CUDA_ARCH__
#define HWFV1_FSHL(lo, hi, s) __funnelshift_l(lo, hi, s)
#define HWFV1_FSHR(lo, hi, s) __funnelshift_r(lo, hi, s)
#else
#define HWFV1_FSHL(lo, hi, s) ((uint32_t)(((((uint64_t)(hi) << 32) | (lo)) << (s)) >> 32))
#define HWFV1_FSHR(lo, hi, s) ((uint32_t)((((uint64_t)(hi) << 32) | (lo)) >> (s)))
#endif

__host__ __device__ __forceinline__ uint32_t mulhi_u(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
__host__ __device__ __forceinline__ int32_t mulhi_s(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}

// A positive float in [0.25, 2) as a Q24 integer, exact in [0.5, 1] and within
// 2^-23 relative next to those bounds.
__host__ __device__ __forceinline__ uint32_t seed_q24(uint32_t y) { return y - (125u << 23); }

// ---- square root -----------------------------------------------------------
// x positive and normal.  M = x's significand, an integer in Q52 in [1, 4)
// (an odd exponent doubles it): sqrt(M) is in [1, 2).
__host__ __device__ __forceinline__ bool sqrt_in_range(uint32_t hi) { return hi - 0x00100000u < 0x7FE00000u; }
// the float near M whose inverse square root seeds the iteration
__host__ __device__ __forceinline__ uint32_t sqrt_seed_arg(uint32_t lo, uint32_t hi) {
    return (HWFV1_FSHL(lo, hi, 3) & 0x007FFFFFu) | ((hi & 0x00100000u) ? 0x3F800000u : 0x40000000u);
}
__host__ __device__ __forceinline__ uint64_t sqrt_bits(uint32_t lo, uint32_t hi, uint32_t seed) {
    const uint32_t odd = (hi & 0x00100000u) ? 0u : 1u;
    const uint32_t mh = (hi & 0x000FFFFFu) | 0x00100000u;
    const uint32_t Ml = lo << odd, Mh = HWFV1_FSHL(lo, mh, odd);
    const uint32_t y24 = seed_q24(seed);
    // s0 = M y in Q23, within 2^-21 of the root
    const uint32_t s0 = mulhi_u(HWFV1_FSHR(Ml, Mh, 22), y24 << 6) >> 5;
    // s1 = s0 + (M - s0^2) y / 2 in Q46: within 2^-42
    const int32_t r0 = (int32_t)(HWFV1_FSHR(Ml, Mh, 5) - 2u * s0 * s0);     // Q47, modulo 2^32
    const int32_t d0 = mulhi_s(r0, (int32_t)(y24 << 6));                     // r y / 2 in Q46
    const uint64_t s1 = ((uint64_t)s0 << 23) + (uint64_t)(int64_t)d0;
    const uint32_t s1l = (uint32_t)s1, s1h = (uint32_t)(s1 >> 32);
    // M - s1^2, the high word of its low 64 bits in Q92: Q60
    const int32_t r1 = (int32_t)((Ml << 8) - 2u * s1h * s1l - mulhi_u(s1l, s1l));
    // k = floor of the root so far in Q52: the root lies in [k - 1/4, k + 5/4)
    const int32_t d1 = mulhi_s(r1, (int32_t)(y24 >> 1));                     // r y / 2 in Q52
    const uint64_t k = (s1 << 6) + (uint64_t)(int64_t)d1;
    // the midpoint c = k + 1/2 in Q53: M > c^2?  (c is odd, so the low word
    // of c^2 is never 0 and always borrows; equality cannot occur)
    const uint32_t cl = ((uint32_t)k << 1) | 1u, ch = (uint32_t)(k >> 31);
    const int32_t t = (int32_t)((Ml << 22) + ~(mulhi_u(cl, cl) + 2u * ch * cl));
    const uint64_t s = k + (uint64_t)(t >= 0 ? 1 : 0);
    const uint32_t eo = ((hi + (1023u << 20)) >> 1) & 0x7FF00000u;           // (e + 1023) / 2
    return s + ((uint64_t)(eo - 0x00100000u) << 32);
}

// ---- reciprocal ------------------------------------------------------------
// x normal with |x| < 2^1022 (its reciprocal is then normal too)
__host__ __device__ __forceinline__ bool rcp_in_range(uint32_t hi) {
    return (hi & 0x7FFFFFFFu) - 0x00100000u < 0x7FD00000u - 0x00100000u;
}
// the float near the significand in [1, 2) whose reciprocal seeds
__host__ __device__ __forceinline__ uint32_t rcp_seed_arg(uint32_t lo, uint32_t hi) {
    return (HWFV1_FSHL(lo, hi, 3) & 0x007FFFFFu) | 0x3F800000u;
}
__host__ __device__ __forceinline__ uint64_t rcp_bits(uint32_t lo, uint32_t hi, uint32_t seed) {
    const uint32_t mh = (hi & 0x000FFFFFu) | 0x00100000u;                    // m = mh:lo in Q52, [1, 2)
    const uint32_t y24 = seed_q24(seed);
    // 1 - m y, the high word of its low 64 bits in Q76: Q44
    const uint32_t p0 = mulhi_u(lo, y24) + mh * y24;
    // y1 = y + y (1 - m y) in Q43: within 2^-39
    const int32_t d0 = mulhi_s((int32_t)(0u - (p0 << 7)), (int32_t)y24);
    const uint64_t y1 = ((uint64_t)y24 << 19) + (uint64_t)(int64_t)d0;
    const uint32_t yl = (uint32_t)y1, yh = (uint32_t)(y1 >> 32);
    // 1 - m y1, the high word of its low 64 bits in Q95: Q63
    const uint32_t p1 = mulhi_u(lo, yl) + lo * yh + mh * yl;
    // k = floor of the reciprocal so far in Q53
    const int32_t d1 = mulhi_s((int32_t)(0u - p1), (int32_t)(y24 >> 2));
    const uint64_t k = (y1 << 10) + (uint64_t)(int64_t)d1;
    // the midpoint c = k + 1/2 in Q54: m c < 1?  (m c = 1 cannot occur, c is
    // odd; the sign of m c - 1 is that of its low 64 bits)
    const uint32_t cl = ((uint32_t)k << 1) | 1u, ch = (uint32_t)(k >> 31);
    const uint32_t p2 = mulhi_u(lo, cl) + lo * ch + mh * cl;
    const uint64_t q = k + (uint64_t)(p2 >> 31);
    // exponent 2045 - e (one more, by the carry, for a power of two)
    const uint32_t eo = (2045u << 20) - (hi & 0x7FF00000u) - 0x00100000u;
    return (q + ((uint64_t)eo << 32)) | ((uint64_t)(hi & 0x80000000u) << 32);
}

// ---- product ---------------------------------------------------------------
// true when both factors are normal and so is the product before rounding
__host__ __device__ __forceinline__ bool mul_in_range(uint32_t ah, uint32_t bh) {
    const uint32_t ea = ah & 0x7FF00000u, eb = bh & 0x7FF00000u;
    // ea, eb in [1, 2046] (neither 0 nor 2047) and ea + eb - 1023 in [1, 2044]
    const bool na = ((ah + 0x00100000u) & 0x7FE00000u) != 0u, nb = ((bh + 0x00100000u) & 0x7FE00000u) != 0u;
    return na && nb && ea + eb - (1024u << 20) < (2044u << 20);
}
// The product of two factors in range; with Z, of factors in range or +-0 (a
// zero factor gives a signed zero).
template <bool Z>
__host__ __device__ __forceinline__ uint64_t mul_bits(uint32_t al, uint32_t ah, uint32_t bl, uint32_t bh) {
    const uint32_t ma = (ah & 0x000FFFFFu) | 0x00100000u, mb = (bh & 0x000FFFFFu) | 0x00100000u;
    // 105 or 106 bits, w3:w2:w1:w0; the two middle products and the carries
    // into them fit 64 bits
    const uint64_t p00 = (uint64_t)al * bl;
    const uint64_t mid = (uint64_t)ma * bl + ((uint64_t)al * mb + (p00 >> 32));
    const uint64_t top = (uint64_t)ma * mb + (mid >> 32);
    const uint32_t w3 = (uint32_t)(top >> 32), w2 = (uint32_t)top, w1 = (uint32_t)mid, w0 = (uint32_t)p00;
    // the significand kh:kl is the top 53 bits: z = 11 with 106 bits (the
    // product of the significands is 2 or more), 12 with 105
    const uint32_t z = (6655u - w3) >> 9;
    const uint32_t kl = HWFV1_FSHL(w1, w2, z), kh = HWFV1_FSHL(w2, w3, z);
    // the bits below, rounded into kl by the carry of an addition: more than
    // half a unit (w0 only matters as "not 0"), or half and an odd kl
    const uint32_t f = HWFV1_FSHL(w0, w1, z) | (w0 < 1u ? w0 : 1u);
    // the exponent word (kh holds the significand's leading bit); without Z
    // the sign bits add up to the result's along with it, modulo 2^32
    constexpr uint32_t mask = Z ? 0x7FF00000u : 0xFFF00000u;
    const uint32_t e = (ah & mask) + (bh & mask) - (1012u << 20) - (z << 20);
    uint32_t rl, rh;
#ifdef __CUDA_ARCH__
    asm("{.reg .u32 t; shl.b32 t, %2, 31; add.cc.u32 t, t, t; addc.cc.u32 t, %4, 0x7fffffff; addc.cc.u32 %0, %2, 0; "
        "addc.u32 %1, %3, %5;}"
        : "=&r"(rl), "=r"(rh) : "r"(kl), "r"(kh), "r"(f), "r"(e));   // (%0 is written before kh and e are read)
#else
    const uint64_t r = (uint64_t)f + 0x7FFFFFFFu + (kl & 1u);
    const uint64_t k = ((uint64_t)(kh + e) << 32 | kl) + (r >> 32);
    rl = (uint32_t)k;
    rh = (uint32_t)(k >> 32);
#endif
    if (Z) {
        // times 0 for a zero factor, as multiplications: the pipe they run on
        // has slots to spare, the one selections run on has not
        const uint32_t ea = ah & mask, eb = bh & mask;
        const uint32_t nz = (ea < 1u ? ea : 1u) * (eb < 1u ? eb : 1u);
        rl = rl * nz;
        rh = rh * nz + ((ah ^ bh) & 0x80000000u);
    }
    return (uint64_t)rh << 32 | rl;
}

// ---- scaling by a power of two -----------------------------------------------
// x 2^K, |K| <= 2, where x or the result is not normal: zeros and subnormals
// (rounded where bits are lost), overflow, infinities (NaN: x)
template <int K>
__host__ __device__ __forceinline__ uint64_t pow2_bits(uint64_t b) {
    const uint64_t s = b & 0x8000000000000000ull, a = b ^ s;
    const int e = (int)(a >> 52);
    if (e == 0x7FF) return b;
    if (K > 0) {
        if (e + K > 2046) return s | 0x7FF0000000000000ull;
        if (e != 0) return b + ((uint64_t)K << 52);
        uint64_t m = a;
        for (int k = 0; k < K; ++k) m = m >> 52 ? m + (1ull << 52) : m << 1;
        return s | m;
    }
    if (e > -K) return b - ((uint64_t)(-K) << 52);
    const uint64_t m = e == 0 ? a : (a & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    const int sh = e == 0 ? -K : 1 - K - e;
    const uint64_t r = m >> sh, rem = m & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    return s | (r + (rem > half || (rem == half && (r & 1ull)) ? 1ull : 0ull));
}

#ifdef __CUDACC__
// Device forms on doubles.  Operands outside an operation's range (next to
// no lane meets one) take the FP64 instruction in a function of its own: a
// call the compiler can neither predicate nor hoist, so that the common path
// leaves the FP64 pipe alone.
__device__ __forceinline__ void d_split(double x, uint32_t& lo, uint32_t& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(x));
}
__device__ __forceinline__ double d_join(uint64_t b) {
    double x;
    asm("mov.b64 %0, %1;" : "=d"(x) : "l"(b));
    return x;
}
static __device__ __noinline__ double sqrt_rare(double x) { return sqrt(x); }
static __device__ __noinline__ double mul_rare(double a, double b) { return __dmul_rn(a, b); }
static __device__ __noinline__ double rcp_rare(double x) { return 1.0 / x; }

// sqrt(x) and 1 / x
__device__ __forceinline__ double root(double x) {
    uint32_t lo, hi;
    d_split(x, lo, hi);
    if ((lo | hi) == 0u) return x;                    // a dry side
    if (!sqrt_in_range(hi)) return sqrt_rare(x);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(sqrt_seed_arg(lo, hi))));
    return d_join(sqrt_bits(lo, hi, __float_as_uint(y)));
}
__device__ __forceinline__ double recip(double x) {
    uint32_t lo, hi;
    d_split(x, lo, hi);
    if (!rcp_in_range(hi)) return rcp_rare(x);
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(rcp_seed_arg(lo, hi))));
    return d_join(rcp_bits(lo, hi, __float_as_uint(y)));
}
// a b.  prod: any operands.  prod_nz: operands known to be in range.
// prod_z: operands known to be in range or zero.
__device__ __forceinline__ double prod(double a, double b) {
    uint32_t al, ah, bl, bh;
    d_split(a, al, ah);
    d_split(b, bl, bh);
    if (!mul_in_range(ah, bh)) {
        const uint32_t xa = ah & 0x7FFFFFFFu, xb = bh & 0x7FFFFFFFu;
        if (((xa | al) == 0u || (xb | bl) == 0u) && xa < 0x7FF00000u && xb < 0x7FF00000u)
            return d_join((uint64_t)((ah ^ bh) & 0x80000000u) << 32);
        return mul_rare(a, b);
    }
    return d_join(mul_bits<false>(al, ah, bl, bh));
}
__device__ __forceinline__ double prod_nz(double a, double b) {
    uint32_t al, ah, bl, bh;
    d_split(a, al, ah);
    d_split(b, bl, bh);
    return d_join(mul_bits<false>(al, ah, bl, bh));
}
__device__ __forceinline__ double prod_z(double a, double b) {
    uint32_t al, ah, bl, bh;
    d_split(a, al, ah);
    d_split(b, bl, bh);
    return d_join(mul_bits<true>(al, ah, bl, bh));
}
__device__ __forceinline__ float prod(float a, float b) { return a * b; }
__device__ __forceinline__ float root(float x) { return sqrtf(x); }
__device__ __forceinline__ float recip(float x) { return 1.0f / x; }
#endif

}  // namespace hwfv1
