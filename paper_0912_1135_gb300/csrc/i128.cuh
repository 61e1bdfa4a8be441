// Exact products of float64 numbers summed in 128-bit integers, on the integer pipes.
//
// GB300's FP64 pipe takes 64 cycles per warp instruction, so one double-double
// multiply-add (13 of them) holds an SM sub-partition for 832 cycles; the integer form
// below takes about 60 instructions of one or two cycles each. A sum is a 128-bit
// two's-complement integer w times 2^E. Every product of two 53-bit significands (106
// bits, exact) is shifted right onto the sum's unit 2^E and added; E follows the largest
// product seen: a product 2^9 times larger than the one that set E (or the first) moves E
// up, and the sum is shifted along. Bits lost in a shift lie below 2^-105 of that largest
// product, and each addition loses less than one unit 2^E, so a sum of N products is within
// N 2^-105 of the largest product's magnitude: the bound of a double-double sum, whose
// every addition rounds at 2^-105 of the partial sum. Capacity: products enter at most
// 2^115 units large, so 2^11 of them fit 127 bits (I128_MAX_TERMS).
#pragma once

#include <cstdint>

namespace rtp {

constexpr int I128_MAX_TERMS = 2048;
constexpr int I128_E_EMPTY = -(1 << 20);

struct i128acc {
    uint32_t w0, w1, w2, w3;   // two's complement, w0 the lowest word
    int E;                     // unit 2^E
};

// One operand decoded: |x| = (hi 2^32 + lo) 2^e, neg = all ones for a negative x.
struct i128op {
    uint32_t lo, hi;
    int e;
    uint32_t neg;
};

__device__ __forceinline__ i128acc i128_zero() { return {0u, 0u, 0u, 0u, I128_E_EMPTY}; }

__device__ __forceinline__ bool i128_finite(uint32_t xh) { return (xh & 0x7FF00000u) != 0x7FF00000u; }

// The bits (xl, xh) of a double as an operand; subnormals are exact, an infinity or NaN
// must be caught by the caller (i128_finite).
__device__ __forceinline__ i128op i128_decode(uint32_t xl, uint32_t xh) {
    const uint32_t ex = (xh >> 20) & 0x7FFu;
    i128op o;
    o.lo = xl;
    o.hi = (xh & 0xFFFFFu) | (ex ? 0x100000u : 0u);
    o.e = (int)(ex ? ex : 1u) - 1075;
    o.neg = (uint32_t)((int32_t)xh >> 31);
    return o;
}

// The same operand with its significand moved up by 9 bits (the left factor of i128_mac).
__device__ __forceinline__ i128op i128_left(i128op o) {
    o.hi = (o.hi << 9) | (o.lo >> 23);
    o.lo <<= 9;
    o.e -= 9;
    return o;
}

// Arithmetic right shift of the sum by r >= 0.
__device__ __forceinline__ void i128_sar(i128acc& a, int r) {
    if (r > 127) r = 127;
    const uint32_t s = (uint32_t)((int32_t)a.w3 >> 31);
    if (r & 64) { a.w0 = a.w2; a.w1 = a.w3; a.w2 = s; a.w3 = s; }
    if (r & 32) { a.w0 = a.w1; a.w1 = a.w2; a.w2 = a.w3; a.w3 = s; }
    const int b = r & 31;
    if (b) {
        a.w0 = (a.w0 >> b) | (a.w1 << (32 - b));
        a.w1 = (a.w1 >> b) | (a.w2 << (32 - b));
        a.w2 = (a.w2 >> b) | (a.w3 << (32 - b));
        a.w3 = (uint32_t)((int32_t)a.w3 >> b);
    }
}

__device__ __forceinline__ uint32_t i128_funnel(uint32_t lo, uint32_t hi, int r) {
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, r);       // shift by r mod 32
#else
    r &= 31;
    return r ? (lo >> r) | (hi << (32 - r)) : lo;
#endif
}

// a += (p3:p0 xor m) - m: adds the 128-bit integer p (m = 0) or subtracts it (m = ~0)
__device__ __forceinline__ void i128_add_signed(i128acc& a, uint32_t p0, uint32_t p1, uint32_t p2, uint32_t p3,
                                                uint32_t m) {
    p0 ^= m; p1 ^= m; p2 ^= m; p3 ^= m;
#ifdef __CUDA_ARCH__
    uint32_t t;
    asm("add.cc.u32 %4, %9, %9;\n\t"          // the carry in: 1 when m is all ones
        "addc.cc.u32 %0, %0, %5;\n\t"
        "addc.cc.u32 %1, %1, %6;\n\t"
        "addc.cc.u32 %2, %2, %7;\n\t"
        "addc.u32 %3, %3, %8;\n\t"
        : "+r"(a.w0), "+r"(a.w1), "+r"(a.w2), "+r"(a.w3), "=&r"(t)
        : "r"(p0), "r"(p1), "r"(p2), "r"(p3), "r"(m));
#else
    uint64_t c = (uint64_t)a.w0 + p0 + (m & 1u);
    a.w0 = (uint32_t)c;
    c = (uint64_t)a.w1 + p1 + (c >> 32);
    a.w1 = (uint32_t)c;
    c = (uint64_t)a.w2 + p2 + (c >> 32);
    a.w2 = (uint32_t)c;
    a.w3 = (uint32_t)((uint64_t)a.w3 + p3 + (c >> 32));
#endif
}

// a += x y for x from i128_left(i128_decode(.)) and y from i128_decode(.); flip = ~0 subtracts
__device__ __forceinline__ void i128_mac(i128acc& a, const i128op& x, const i128op& y, uint32_t flip = 0u) {
    const int e = x.e + y.e;
    int r = a.E - e;
    if (r < 0) {                             // a larger product: the unit moves up
        const int E = e + 9;
        i128_sar(a, E - a.E);
        a.E = E;
        r = 9;
    }
    const uint64_t t0 = (uint64_t)x.lo * y.lo;
    const uint64_t t1 = (uint64_t)x.hi * y.lo + (t0 >> 32);
    const uint64_t t2 = (uint64_t)x.lo * y.hi + (uint32_t)t1;
    const uint64_t t3 = (uint64_t)x.hi * y.hi + (t1 >> 32) + (t2 >> 32);
    uint32_t p0 = (uint32_t)t0, p1 = (uint32_t)t2, p2 = (uint32_t)t3, p3 = (uint32_t)(t3 >> 32);
    r = r > 127 ? 127 : r;                   // p < 2^115: a shift by 127 leaves zero
    const bool s64 = (r & 64) != 0, s32 = (r & 32) != 0;
    p0 = s64 ? p2 : p0;
    p1 = s64 ? p3 : p1;
    p2 = s64 ? 0u : p2;
    p3 = s64 ? 0u : p3;
    p0 = s32 ? p1 : p0;
    p1 = s32 ? p2 : p1;
    p2 = s32 ? p3 : p2;
    p3 = s32 ? 0u : p3;
    p0 = i128_funnel(p0, p1, r);
    p1 = i128_funnel(p1, p2, r);
    p2 = i128_funnel(p2, p3, r);
    p3 >>= (r & 31);
    i128_add_signed(a, p0, p1, p2, p3, x.neg ^ y.neg ^ flip);
}

// a += b for two sums
__device__ __forceinline__ void i128_merge(i128acc& a, i128acc b) {
    const int E = a.E > b.E ? a.E : b.E;
    i128_sar(a, E - a.E);
    i128_sar(b, E - b.E);
    a.E = E;
    i128_add_signed(a, b.w0, b.w1, b.w2, b.w3, 0u);
}

// V * 2^e for the 128-bit two's-complement integer V = (H:L), rounded to nearest even.
__device__ __forceinline__ double u128_to_double(unsigned long long H, unsigned long long L, int e) {
    // |V| by a masked negation (no branch: the lanes of a warp hold values of either sign)
    const unsigned long long sg = (unsigned long long)((long long)H >> 63);
    L ^= sg;
    H ^= sg;
    const unsigned long long one = sg & 1ull;
    const unsigned long long L1 = L + one;
    H += one & (L1 == 0 ? 1ull : 0ull);
    L = L1;
    if ((H | L) == 0) return 0.0;
    // normalise: shift left by the leading zeros so that the leading one is bit 127
    const int s = H != 0 ? __clzll((long long)H) : 64 + __clzll((long long)L);
    const int s1 = s & 63;
    const unsigned long long hl = s1 ? (H << s1) | (L >> (64 - s1)) : H;
    const unsigned long long Hn = s < 64 ? hl : (L << s1);
    const unsigned long long Ln = s < 64 ? (L << s1) : 0ull;
    // 53 bits, round to nearest even on the round bit and the sticky bits below it
    unsigned long long m = Hn >> 11;
    const unsigned long long rb = (Hn >> 10) & 1ull;
    const unsigned long long st = ((Hn & 0x3FFull) | Ln) != 0 ? 1ull : 0ull;
    m += rb & (st | (m & 1ull));
    const unsigned long long ovf = m >> 53;       // rounding carried into bit 53
    m >>= ovf;
    const int ex = 127 - s + (int)ovf;             // position of the leading bit of |V|
    const int biased = ex + e + 1023;
    if (biased <= 0 || biased >= 2047) {
        const double mag = ldexp((double)m, ex - 52 + e);
        return sg ? -mag : mag;
    }
    const unsigned long long bits =
        ((unsigned long long)biased << 52) | (m & 0xFFFFFFFFFFFFFull) | (sg & 0x8000000000000000ull);
    return __longlong_as_double((long long)bits);
}

__device__ __forceinline__ unsigned long long i128_high(const i128acc& a) { return ((unsigned long long)a.w3 << 32) | a.w2; }
__device__ __forceinline__ unsigned long long i128_low(const i128acc& a) { return ((unsigned long long)a.w1 << 32) | a.w0; }

// The sum rounded once to nearest.
__device__ __forceinline__ double i128_to_double(const i128acc& a) { return u128_to_double(i128_high(a), i128_low(a), a.E); }

// The sum as an unevaluated pair hi + lo (at least 106 bits): hi the leading 53 bits, lo the
// rest rounded.
__device__ __forceinline__ void i128_to_pair(const i128acc& a, double& hi, double& lo) {
    unsigned long long H = i128_high(a), L = i128_low(a);
    const unsigned long long sg = (unsigned long long)((long long)H >> 63);
    const unsigned long long aH = H ^ sg, aL = L ^ sg;            // |V|, or |V| - 1 for a negative V
    const int len = aH ? 128 - __clzll((long long)aH) : aL ? 64 - __clzll((long long)aL) : 0;
    const int cut = len - 52;                                     // V's low `cut` bits go to lo
    unsigned long long mH = 0ull, mL = 0ull;
    if (cut >= 64) { mL = ~0ull; mH = cut > 64 ? (1ull << (cut - 64)) - 1ull : 0ull; }
    else if (cut > 0) mL = (1ull << cut) - 1ull;
    hi = u128_to_double(H & ~mH, L & ~mL, a.E);
    lo = u128_to_double(H & mH, L & mL, a.E);
}

}  // namespace rtp
