// FP64 add and multiplication on the integer pipes, correctly rounded (to nearest, ties to even): the bits of
// the hardware instruction for the operands that they take. GB300 has 2 FP64 lanes per SM and 128
// integer lanes, so an FP64 instruction holds its pipe for 16 cycles in which the SM issues 64
// others: a sweep that is bound by the FP64 pipe gets faster where some of its operations go this
// way (plain.cu has the figures). Method: IEEE 754 addition and multiplication by aligned
// significands with a sticky bit.
//
// Operands or results outside the range that the integer form takes set `bad`; the caller then
// computes with the hardware instruction instead.
#pragma once
#include <stdint.h>

namespace stg {

#ifdef __CUDACC__
#define SOFT64_FN __host__ __device__ __forceinline__
#else
#define SOFT64_FN inline
#endif

SOFT64_FN uint64_t s64_bits(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t r;
    __builtin_memcpy(&r, &x, 8);
    return r;
#endif
}
SOFT64_FN double s64_value(uint64_t b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double r;
    __builtin_memcpy(&r, &b, 8);
    return r;
#endif
}
SOFT64_FN int s64_clz(uint32_t x) {
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}

// Rounds the significand n (leading bit 63; bit 0 also stands for anything below it) to 53 bits and
// puts it together with the exponent field e (1 <= e <= 2046 before rounding) and the sign bit.
SOFT64_FN double s64_round(uint64_t n, int e, uint32_t sign) {
    const uint64_t q = n >> 11;  // leading bit at 52: adding it to the field e - 1 gives e
    const uint32_t low = ((uint32_t)n & 0x7ffu) + ((uint32_t)q & 1u);
    uint64_t r = q + ((uint64_t)(uint32_t)(e - 1) << 52) + (low > 0x400u ? 1u : 0u);
    return s64_value(r | (uint64_t)sign << 32);
}

// a + b. Taken: the larger magnitude is finite, below 2^1023 and at least 2^-959 (the smaller one may
// be anything, zeros included), and the sum keeps at least 31 of the bits above cancellation. A
// smaller operand with exponent field 0 is taken as 1.f x 2^-1023: as far as it can matter here it
// is only a sticky bit.
SOFT64_FN double soft_add(double a, double b, uint32_t& bad) {
    const uint64_t A0 = s64_bits(a), B0 = s64_bits(b);
    const bool sw = (B0 << 1) > (A0 << 1);
    const uint64_t A = sw ? B0 : A0, B = sw ? A0 : B0;
    const uint32_t ah = (uint32_t)(A >> 32), bh = (uint32_t)(B >> 32);
    const int ea = (int)(ah >> 20 & 0x7ffu), eb = (int)(bh >> 20 & 0x7ffu);
    const uint64_t ma = (A << 10 & 0x3fffffffffffffffull) | 0x4000000000000000ull;  // leading bit 62
    const uint64_t mb = (B << 10 & 0x3fffffffffffffffull) | 0x4000000000000000ull;
    const int d = ea - eb < 63 ? ea - eb : 63;
    uint64_t sh = mb >> d;
    sh |= (sh << d) != mb ? 1u : 0u;
    const uint64_t neg = (uint64_t)((int64_t)(A ^ B) >> 63);
    const uint64_t sum = ma + (sh ^ neg) - neg;
    const uint32_t top = (uint32_t)(sum >> 32);
    const int lz = s64_clz(top);
    bad |= (uint32_t)(ea - 64) >= 0x7feu - 64u || top == 0u ? 1u : 0u;
    return s64_round(sum << (lz & 31), ea + 1 - lz, ah & 0x80000000u);
}

// c * u with the factor c prepared once.
struct SoftFactor {
    uint32_t lo, hi;  // significand, leading bit 63
    int e;            // exponent field - 1023
    uint32_t sign, bad;
    SOFT64_FN explicit SoftFactor(double c) {
        const uint64_t b = s64_bits(c), m = (b << 11) | 0x8000000000000000ull;
        const int f = (int)(b >> 52 & 0x7ffu);
        lo = (uint32_t)m;
        hi = (uint32_t)(m >> 32);
        e = f - 1023;
        sign = (uint32_t)(b >> 32) & 0x80000000u;
        bad = (uint32_t)(f - 1) >= 0x7feu ? 1u : 0u;
    }
};
// Taken: c and u normal, the product's magnitude at least 2^-1022 and below 2^1022 before the carry.
SOFT64_FN double soft_mul(const SoftFactor& c, double u, uint32_t& bad) {
    const uint64_t b = s64_bits(u);
    const int eu = (int)(b >> 52 & 0x7ffu), e = eu + c.e;
    const uint64_t m = (b << 11) | 0x8000000000000000ull;
    const uint32_t ml = (uint32_t)m, mh = (uint32_t)(m >> 32);
    const uint64_t p0 = (uint64_t)ml * c.lo;
    const uint64_t p1 = (uint64_t)ml * c.hi + (p0 >> 32);
    const uint64_t p2 = (uint64_t)mh * c.lo + (uint32_t)p1;
    uint64_t h = (uint64_t)mh * c.hi + (p1 >> 32) + (p2 >> 32);  // the product's upper half
    h |= ((uint32_t)p2 | (uint32_t)p0) != 0u ? 1u : 0u;
    const int lz = (h >> 63) == 0 ? 1 : 0;  // the product of two significands is in [1, 4)
    bad |= c.bad | ((uint32_t)(eu - 1) >= 0x7feu || (uint32_t)(e - 1) >= 0x7fcu ? 1u : 0u);
    return s64_round(h << lz, e + 1 - lz, ((uint32_t)(b >> 32) & 0x80000000u) ^ c.sign);
}

}  // namespace stg
