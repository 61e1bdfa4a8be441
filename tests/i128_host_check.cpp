// Host build of the 128-bit sums of exact products (csrc/i128.cuh) for the CPU tests: reads
// "sum N" or "two N" and N pairs of doubles (hexadecimal), prints the rounded sum of their
// products and the pair form; "two" forms the sum from two halves merged, "long" takes a sum of any
// length in parts. "sub N" prints x - V 2^e and V 2^e, each rounded once, for 128-bit integers V.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#define __device__
#define __forceinline__ inline
#define __noinline__
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
static inline double __longlong_as_double(long long x) {
    double d;
    std::memcpy(&d, &x, 8);
    return d;
}
using std::ldexp;
#include "i128.cuh"

static rtp::i128op dec(double x) {
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return rtp::i128_decode((uint32_t)u, (uint32_t)(u >> 32));
}

int main() {
    char op[16];
    int n;
    while (std::scanf("%15s %d", op, &n) == 2) {
        if (!std::strcmp(op, "sub")) {       // n lines: x, the words of V (lowest first), e
            for (int i = 0; i < n; ++i) {
                double x, out = 0.0;
                unsigned w[4];
                int e;
                if (std::scanf("%la %x %x %x %x %d", &x, &w[0], &w[1], &w[2], &w[3], &e) != 6) return 1;
                uint64_t u;
                std::memcpy(&u, &x, 8);
                const bool ok = rtp::i128_sub_from((uint32_t)u, (uint32_t)(u >> 32), w[0], w[1], w[2], w[3], e, out);
                std::printf("%d %a %a\n", (int)ok, out, rtp::i128_round_signed(w[0], w[1], w[2], w[3], e));
            }
            continue;
        }
        rtp::i128acc a = rtp::i128_zero(), b = rtp::i128_zero();
        const bool two = op[0] == 't', longer = op[0] == 'l';
        int terms = 0;
        double hi = 0.0, lo = 0.0;
        for (int i = 0; i < n; ++i) {
            double x, y;
            if (std::scanf("%la %la", &x, &y) != 2) return 1;
            rtp::i128_mac(two && (i & 1) ? b : a, rtp::i128_left(dec(x)), dec(y), i % 3 == 2 ? ~0u : 0u);
            if (longer && ++terms == rtp::I128_MAX_TERMS) {
                rtp::i128_flush(a, hi, lo);
                terms = 0;
            }
        }
        if (longer) {
            rtp::i128_flush(a, hi, lo);
            std::printf("%a %a %a\n", hi + lo, hi, lo);
            continue;
        }
        rtp::i128_merge(a, b);
        rtp::i128_to_pair(a, hi, lo);
        std::printf("%a %a %a\n", rtp::i128_to_double(a), hi, lo);
    }
    return 0;
}
