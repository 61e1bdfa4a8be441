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
// every addition rounds at 2^-105 of the partial sum. A zero's product moves nothing; a subnormal
// factor counts as 2^-1022 in "largest" (its own last place is 2^52 times coarser). Capacity: products
// enter at most 2^115 units large, so 2^11 of them fit 127 bits (I128_MAX_TERMS); a longer sum is
// taken in parts of at most that many, which are added in double-double (i128_flush).
#pragma once

#include <cstdint>

namespace rtp {

constexpr int I128_MAX_TERMS = 2048;
constexpr int I128_E_EMPTY = -(1 << 20);

struct i128acc {
    uint32_t w0, w1, w2, w3;   // two's complement, w0 the lowest word
    int E;                     // unit 2^E
};

__device__ __forceinline__ double i128_from_words(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    return __longlong_as_double((long long)(((uint64_t)hi << 32) | lo));
#endif
}

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
    asm("{\n\t.reg .u32 t;\n\t"
        "add.cc.u32 t, %8, %8;\n\t"            // the carry in: 1 when m is all ones
        "addc.cc.u32 %0, %0, %4;\n\t"
        "addc.cc.u32 %1, %1, %5;\n\t"
        "addc.cc.u32 %2, %2, %6;\n\t"
        "addc.u32 %3, %3, %7;\n\t}\n"
        : "+r"(a.w0), "+r"(a.w1), "+r"(a.w2), "+r"(a.w3)
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
    if (r < 0) {                             // a larger product: the unit moves up, but not for a zero's
        const int E = (x.hi | x.lo) != 0u && (y.hi | y.lo) != 0u ? e + 9 : a.E;
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

// A result outside the normal range (rare): m 2^e for the 53-bit m, by ldexp.
static __device__ __noinline__ double i128_edge_result(unsigned long long m, int e, uint32_t neg) {
    const double mag = ldexp((double)m, e);
    return neg ? -mag : mag;
}

// The magnitude (w3:w0) 2^e, negative when neg = ~0, rounded to nearest (ties to even). All in
// 32-bit operations and without branches (the lanes of a warp hold values of every size): the
// three words from the leading nonzero one on are selected and normalised by one count of
// leading zeros and two funnel shifts, the rest joins the sticky bits; about 45 instructions.
// (Written with 64-bit shifts by variable amounts the conversion took about 290 cycles per warp,
// which bounded the sliced products with a short contraction.)
__device__ __forceinline__ double i128_round(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, int e, uint32_t neg) {
    const bool n3 = w3 != 0u, n2 = w2 != 0u, n1 = w1 != 0u;
    const uint32_t t2 = n3 ? w3 : n2 ? w2 : n1 ? w1 : w0;
    const uint32_t t1 = n3 ? w2 : n2 ? w1 : n1 ? w0 : 0u;
    const uint32_t t0 = n3 ? w1 : n2 ? w0 : 0u;
    const uint32_t rest = n3 ? w0 : 0u;
    const int top = n3 ? 127 : n2 ? 95 : n1 ? 63 : 31;          // bit of t2's most significant place
#ifdef __CUDA_ARCH__
    const int z = __clz((int)t2);
    const uint32_t a = __funnelshift_l(t1, t2, z), b = __funnelshift_l(t0, t1, z), c = t0 << (z & 31);
#else
    const int z = t2 ? __builtin_clz(t2) : 32;
    const int y = z & 31;
    const uint32_t a = y ? (t2 << y) | (t1 >> (32 - y)) : t2, b = y ? (t1 << y) | (t0 >> (32 - y)) : t1, c = t0 << y;
#endif
    const uint32_t mlo = (a << 21) | (b >> 11), mhi = a >> 11;  // 53 bits, the leading one at bit 20 of mhi
    const bool up = (b & 0x400u) && (((b & 0xBFFu) | c | rest) != 0u);   // round bit; sticky bits or the last bit
    const int biased = top - z + e + 1023;
    if (t2 == 0u) return 0.0;
    if (biased <= 0 || biased >= 2046)                          // 2046: the rounding could carry into 2047
        return i128_edge_result((((unsigned long long)mhi << 32) | mlo) + (up ? 1ull : 0ull), top - z - 52 + e, neg);
    const unsigned long long bits = ((((unsigned long long)(uint32_t)(biased - 1) << 20) + mhi) << 32 | mlo) + (up ? 1ull : 0ull);
    const uint32_t hi = (uint32_t)(bits >> 32) | (neg & 0x80000000u), lo = (uint32_t)bits;
    return i128_from_words(hi, lo);
}

// V * 2^e for the 128-bit two's-complement integer V = (v3:v0), rounded to nearest even.
__device__ __forceinline__ double i128_round_signed(uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3, int e) {
    const uint32_t neg = (uint32_t)((int32_t)v3 >> 31);
    i128acc a = {0u, 0u, 0u, 0u, 0};
    i128_add_signed(a, v0, v1, v2, v3, neg);                    // |V|: (V xor neg) - neg
    return i128_round(a.w0, a.w1, a.w2, a.w3, e, neg);
}

__device__ __forceinline__ double u128_to_double(unsigned long long H, unsigned long long L, int e) {
    return i128_round_signed((uint32_t)L, (uint32_t)(L >> 32), (uint32_t)H, (uint32_t)(H >> 32), e);
}

// 2^sh times the 128-bit integer (v3:v0), 0 <= sh < 32 (bits past the top are lost).
__device__ __forceinline__ void i128_shl(uint32_t& v0, uint32_t& v1, uint32_t& v2, uint32_t& v3, int sh) {
#ifdef __CUDA_ARCH__
    v3 = __funnelshift_l(v2, v3, sh);
    v2 = __funnelshift_l(v1, v2, sh);
    v1 = __funnelshift_l(v0, v1, sh);
#else
    if (sh) {
        v3 = (v3 << sh) | (v2 >> (32 - sh));
        v2 = (v2 << sh) | (v1 >> (32 - sh));
        v1 = (v1 << sh) | (v0 >> (32 - sh));
    }
#endif
    v0 <<= sh;
}

// x - V 2^e rounded once, for V = (v3:v0) two's complement and a double x given by its bits: the
// two are brought to a common unit (x's significand moves up by at most 63 bits, or V by at most
// 22) and subtracted exactly. false (out untouched) when their units lie further apart, V is not
// within 2^103, or x is not finite.
__device__ __forceinline__ bool i128_sub_from(uint32_t xl, uint32_t xh, uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3,
                                              int e, double& out) {
    const i128op o = i128_decode(xl, xh);
    const int sh = o.e - e;
    if (sh > 63 || sh < -22 || v3 + 0x80u >= 0x100u || !i128_finite(xh)) return false;
    const int sv = sh < 0 ? -sh : 0, sx = sh > 0 ? sh : 0;
    i128_shl(v0, v1, v2, v3, sv);
    // -V
    i128acc a = {0u, 0u, 0u, 0u, 0};
    i128_add_signed(a, v0, v1, v2, v3, ~0u);
    // the significand's two words at bit sx
    const bool w = sx >= 32;
    uint32_t x0 = w ? 0u : o.lo, x1 = w ? o.lo : o.hi, x2 = w ? o.hi : 0u, x3 = 0u;
    i128_shl(x0, x1, x2, x3, sx & 31);
    i128_add_signed(a, x0, x1, x2, x3, o.neg);
    out = i128_round_signed(a.w0, a.w1, a.w2, a.w3, e - sv);
    return true;
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

// ---- sums of more products than one integer holds: each full sum joins a double-double pair

__device__ __forceinline__ void two_sum_d(double a, double b, double& s, double& e) {   // Knuth's TwoSum
    s = a + b;
    const double bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ void dd_add(double& hi, double& lo, double bh, double bl) {
    double s, e;
    two_sum_d(hi, bh, s, e);
    e += lo + bl;
    hi = s + e;
    lo = e - (hi - s);
}

// The sum moves over to the pair hi + lo and starts anew.
__device__ __forceinline__ void i128_flush(i128acc& a, double& hi, double& lo) {
    double h, l;
    i128_to_pair(a, h, l);
    dd_add(hi, lo, h, l);
    a = i128_zero();
}

}  // namespace rtp
