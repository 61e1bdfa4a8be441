// Pivoted Householder QR of S^* (Section 4, Eq. 13): one cooperative launch, columns in registers,
// exchanges through self-validating packets; in float-float for the mixed form, in float64 for the
// others.
//
// The factorization is m strictly sequential steps, so a step's latency is its cost. CTA b keeps
// columns [b cpc, b cpc + cpc) of S^* (rows of S), WPC warps each, in registers: the warps take
// 64-row groups in turn, lane t rows 2 t and 2 t + 1 of a group. Float-float column arithmetic runs
// two rows at a time in packed float32 instructions (add/mul/fma.f32x2; ff2.cuh). Step j:
//  1. warp 0 polls the CTAs' candidate records of step j (one 16-byte word each) until all carry the
//     step's tag, and takes the largest key: the squared trailing norm to 44 mantissa bits, lowest
//     column on ties (Businger-Golub);
//  2. every CTA loads the pivot column's packets (two rows in 16 bytes, tagged with the step) and
//     its exact squared norm, and derives the same reflector; a packet whose tag is not yet the
//     step's is loaded again;
//  3. each active column's dot product with the reflector gives its row-j entry r, hence its next
//     trailing norm n - r^2 before the column is updated: the CTA's record for step j + 1 is
//     published here, and the exchange overlaps the update;
//  4. the update, which also sums the new norm afresh and writes the column's packets and norm for
//     step j + 1.
// A packet, record or norm is one 128-bit store and one 128-bit load, which are single-copy
// atomic, so a reader needs neither a fence nor a flag behind the data: the former kernel's
// release fence, arrival counter, winner word and column load were four L2 round trips in a row
// (3.7 us a step at 512 x 516). What remains is the exchange (about 2800 cycles from a record's store
// until every CTA has seen all of them, across both dies) and one column load (850). A retired
// column's packets are never rewritten, so late readers of a pivot column are safe; a record buffer is
// rewritten only after every CTA has published the step between. Every wait has a clock deadline;
// on expiry the kernel raises RTPROJ_ETIMEOUT and all CTAs leave.
// Measured: 512 x 516 1.89 -> 1.50 ms (2.9 us a step), 64 x 256 246 -> 172 us, 333 x 698 1.37 -> 1.15 ms,
// 256 x 1024 1.27 -> 1.02 ms, 1024 x 2080 7.6 -> 6.9 ms. Past what registers hold (LONG), against the
// kernels with the columns in shared memory or in L2: 700 x 1900 5.1 -> 4.3 ms, 1500 x 1504 10.0 -> 8.8,
// 1024 x 4096 23 -> 12, 2048 x 4128 52 -> 39; there the column arithmetic of the CTA with most columns left
// counts. Float64, against the persistent kernel: 1000 x 1004 10.4 -> 7.2 ms, 256 x 544 1.49 -> 1.12 ms;
// the FP64 pipe (64 cycles a warp instruction) bounds its columns. Not kept: one 16-CTA cluster with
// the same columns and a hardware barrier a step (5 to 8 us a step: distributed shared memory answers
// no sooner than L2 here), per-column records polled by every warp, scalars formed after the packets'
// barrier.
//
// The early norm n - r^2 is exact to 2^-47 of n (n is summed afresh every step). When the winner's
// has cancelled by more than 2^10 the candidates are exchanged once more with their fresh
// sums, so the choice never rests on fewer than 37 bits. The reflector always uses the fresh sum.
// Range: S^* is scaled by a power of two below 1 / sqrt(l) of its largest entry; columns whose largest
// entries span more than 2^40 (2^400 in float64), or a pivot whose squared norm falls below 2^-112
// (2^-900), send the factorization to the float64 kernel enqueued behind (*fallback), and S is not
// modified. Accuracy: R is the exact factor of S^* + E with ||E|| of order l 2^-48 ||S|| (l 2^-53).
#include "rtproj_internal.cuh"
#include "ff2.cuh"

#include <climits>
#include <algorithm>
#include <iterator>

namespace rtp {
namespace {

struct QrRegsDev {
    const double* S; int m, l; int64_t lds;
    double* R; int32_t* perm;
    int cpc;
    ulonglong2* slots;       // m x npk: the columns' packets
    int tg, ts;              // LONG: row pairs of a column kept in its packets only, and in shared memory
    ulonglong2* rec;         // 2 x G: candidate records by step parity
    ulonglong2* rec_exact;   // 2 x G: the same with fresh norms (only when a winner has cancelled)
    ulonglong2* nrm;         // 2 x m: fresh squared norms
    int* emax;               // 2 x G: exponents of the CTAs' largest entries, and smallest column maxima
    unsigned int* counter;   // arrivals of the scale exchange
    int* abort_flag;
    int* status;
    long long timeout;
    int* fallback;
};

constexpr int LB = 4;                                // packets of a column in flight per lane (LONG)
constexpr int MAX_SCALE = 1000;                      // largest scale's exponent that is taken here

// ---- 128-bit words in global memory, single-copy atomic at GPU scope
__device__ __forceinline__ ulonglong2 ld_word(const ulonglong2* p) {
    ulonglong2 v;
    asm volatile("{\n\t.reg .b128 r;\n\tld.relaxed.gpu.global.b128 r, [%2];\n\tmov.b128 {%0, %1}, r;\n\t}"
                 : "=l"(v.x), "=l"(v.y)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_word(ulonglong2* p, unsigned long long x, unsigned long long y) {
    asm volatile("{\n\t.reg .b128 r;\n\tmov.b128 r, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], r;\n\t}" ::"l"(p), "l"(x),
                 "l"(y)
                 : "memory");
}

struct Tag {
    f2 h, l;                 // the tag's bits in a packet's two words
};

// The arithmetic: a scalar S, and a pair of rows (2 q, 2 q + 1) as two 64-bit words. A packet is the
// pair's words as they are, with a tag of step j in exponent bits that are zero: S^* is scaled so that
// no column's norm exceeds 1, and reflections keep the norms, so every entry is below 2 in magnitude.
// A slot's previous content is the packet of the step before (or the zero written at the start),
// whose tag differs.

// Float-float: the words are both rows' high parts and both rows' low parts; 4 tag bits.
struct FfArith {
    using S = ff;
    static constexpr f2 TAG_BITS = 0x4000000040000000ull;
    static constexpr int RANGE = 40;                          // binades between the columns' largest entries
    static constexpr int ACCS = 3;                            // independent partial sums of a lane
    static constexpr bool SHARED_SCALARS = false;             // every thread forms the reflector's scalars
    static __device__ __forceinline__ bool too_small(S n) { return !(n.hi >= 0x1p-112f); }
    static __device__ __forceinline__ Tag tag(int j) {
        const uint32_t n = ((uint32_t)j & 7u) + 1u;
        return {((f2)((n & 1u) << 30)) | ((f2)((n & 2u) << 29) << 32), ((f2)((n & 4u) << 28)) | ((f2)((n & 8u) << 27) << 32)};
    }
    static __device__ __forceinline__ S zero() { return {0.f, 0.f}; }
    static __device__ __forceinline__ S add(S a, S b) { return ff_add(a, b); }
    static __device__ __forceinline__ S mul(S a, S b) { return ff_mul(a, b); }
    static __device__ __forceinline__ S neg(S a) { return ff_neg(a); }
    static __device__ __forceinline__ S sqrt(S a) { return ff_sqrt_newton(a); }
    static __device__ __forceinline__ S recip(S a) { return ff_recip_newton(a); }
    static __device__ __forceinline__ bool nonneg(S a) { return a.hi >= 0.f; }
    static __device__ __forceinline__ S clamp(S a) { return a.hi > 0.f ? a : zero(); }
    static __device__ __forceinline__ bool cancelled(S now, S before) { return now.hi < before.hi * 0x1p-10f; }
    static __device__ __forceinline__ f2 bits(S a) { return pack2(a.hi, a.lo); }
    static __device__ __forceinline__ S of(f2 w) { return {lo2(w), hi2(w)}; }
    static __device__ __forceinline__ double to_double(S a) { return ff_to_double(a); }
    static __device__ __forceinline__ unsigned long long key(S n, int c) { return norm_key(n, c); }
    static __device__ __forceinline__ S row(const ffp& x, bool odd) {
        return odd ? S{hi2(x.h), hi2(x.l)} : S{lo2(x.h), lo2(x.l)};
    }
    static __device__ __forceinline__ ffp pair(double a, double b) {
        const ff x = ff_from_double(a), y = ff_from_double(b);
        return {pack2(x.hi, y.hi), pack2(x.lo, y.lo)};
    }
    static __device__ __forceinline__ ffp both(S a) { return {pack2(a.hi, a.hi), pack2(a.lo, a.lo)}; }
    // the reflector's pair that holds row j (odd: its second row), whose entry there is v0
    static __device__ __forceinline__ ffp first(const ffp& v, bool odd, S v0) {
        if (odd) return {pack2(0.f, v0.hi), pack2(0.f, v0.lo)};
        return {pack2(v0.hi, hi2(v.h)), pack2(v0.lo, hi2(v.l))};
    }
    // the pair, its second row only, or nothing
    static __device__ __forceinline__ ffp keep(const ffp& x, bool all, bool second) {
        const f2 k = all ? ~0ull : second ? 0xFFFFFFFF00000000ull : 0ull;
        return {x.h & k, x.l & k};
    }
    static __device__ __forceinline__ void dot(ffp& acc, const ffp& x, const ffp& y) { dot_acc2(acc, x, y); }
    static __device__ __forceinline__ ffp update(const ffp& c, const ffp& w, const ffp& v) { return update2(c, w, v); }
    static __device__ __forceinline__ S total(const ffp (&a)[ACCS]) { return warp_total(sum3(a)); }
};

// Float64: the words are the two rows; 2 tag bits (1, 2, 3 in turn, 0 at the start). The FP64 pipe
// holds a sub-partition for 64 cycles a warp instruction, whatever depends on what and however many
// lanes count: one chain of partial sums, comparisons on the bits, and the reflector's scalars formed
// by one warp (by all 14 of a CTA, with three partial sums, 1000 x 1004 took 11.3 ms; the persistent
// kernel 10.4).
struct F64Arith {
    using S = double;
    static constexpr f2 TAG_BITS = 0x4000000000000000ull;
    static constexpr int RANGE = 400;
    static constexpr int ACCS = 1;
    static constexpr bool SHARED_SCALARS = true;
    // the order of non-negative doubles is that of their bits; a NaN counts as small
    static __device__ __forceinline__ bool too_small(S n) {
        return bits(n) - (123ull << 52) >= (2047ull - 123ull) << 52;      // below 2^-900
    }
    static __device__ __forceinline__ Tag tag(int j) {
        const uint32_t n = (uint32_t)j % 3u + 1u;
        return {(f2)(n & 1u) << 62, (f2)(n & 2u) << 61};
    }
    static __device__ __forceinline__ double d(f2 w) { return __longlong_as_double((long long)w); }
    static __device__ __forceinline__ f2 bits(S a) { return (f2)__double_as_longlong(a); }
    static __device__ __forceinline__ S of(f2 w) { return d(w); }
    static __device__ __forceinline__ S zero() { return 0.0; }
    static __device__ __forceinline__ S add(S a, S b) { return a + b; }
    static __device__ __forceinline__ S mul(S a, S b) { return a * b; }
    static __device__ __forceinline__ S neg(S a) { return d(bits(a) ^ (1ull << 63)); }
    // Newton's iterations from the approximate functions (20 bits): x r^2 = 1 twice, then s^2 = x with
    // the residual exact; 1 / a twice. Within a few units in the last place, far inside the QR's l 2^-53; a
    // third of the FP64 pipe's chain.
    static __device__ __forceinline__ S sqrt(S a) {
        double r;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
        r = fma(r * 0.5, fma(-a * r, r, 1.0), r);
        r = fma(r * 0.5, fma(-a * r, r, 1.0), r);
        const double s = a * r;
        return fma(fma(-s, s, a), 0.5 * r, s);
    }
    static __device__ __forceinline__ S recip(S a) {
        double q;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(q) : "d"(a));
        q = fma(fma(-a, q, 1.0), q, q);
        return fma(fma(-a, q, 1.0), q, q);
    }
    static __device__ __forceinline__ bool nonneg(S a) { return (long long)bits(a) >= 0; }
    static __device__ __forceinline__ S clamp(S a) { return (long long)bits(a) > 0 ? a : 0.0; }
    static __device__ __forceinline__ bool cancelled(S now, S before) {
        return (long long)bits(now) < (long long)bits(before) - (10ll << 52);
    }
    static __device__ __forceinline__ double to_double(S a) { return a; }
    // the bits of a norm below 2 (two leading zeros) without the 10 lowest, then 4095 - c
    static __device__ __forceinline__ unsigned long long key(S n, int c) {
        return ((bits(n) << 2) & ~4095ull) | (unsigned long long)(4095 - c);
    }
    static __device__ __forceinline__ S row(const ffp& x, bool odd) { return d(odd ? x.l : x.h); }
    static __device__ __forceinline__ ffp pair(double a, double b) { return {bits(a), bits(b)}; }
    static __device__ __forceinline__ ffp both(S a) { return {bits(a), bits(a)}; }
    static __device__ __forceinline__ ffp first(const ffp& v, bool odd, S v0) {
        if (odd) return {0ull, bits(v0)};
        return {bits(v0), v.l};
    }
    static __device__ __forceinline__ ffp keep(const ffp& x, bool all, bool second) {
        return {all ? x.h : 0ull, all || second ? x.l : 0ull};
    }
    static __device__ __forceinline__ void dot(ffp& acc, const ffp& x, const ffp& y) {
        acc.h = bits(fma(d(x.h), d(y.h), d(acc.h)));
        acc.l = bits(fma(d(x.l), d(y.l), d(acc.l)));
    }
    static __device__ __forceinline__ ffp update(const ffp& c, const ffp& w, const ffp& v) {
        return {bits(fma(d(w.h), d(v.h), d(c.h))), bits(fma(d(w.l), d(v.l), d(c.l)))};
    }
    static __device__ __forceinline__ S total(const ffp (&a)[ACCS]) {
        double s = d(a[0].h) + d(a[0].l);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    }
};

template <class A>
__device__ __forceinline__ bool has_tag(const ulonglong2& w, const Tag& t) {
    return (w.x & A::TAG_BITS) == t.h && (w.y & A::TAG_BITS) == t.l;
}
__device__ __forceinline__ void st_packet(ulonglong2* p, const ffp& x, const Tag& t) { st_word(p, x.h | t.h, x.l | t.l); }
template <class A>
__device__ __forceinline__ ffp unpack(const ulonglong2& w) { return {w.x & ~A::TAG_BITS, w.y & ~A::TAG_BITS}; }

// A wait's deadline: true while it may go on.
struct Deadline {
    long long t0 = 0;
    unsigned int it = 0;
    __device__ __forceinline__ bool more(const QrRegsDev& p) {
        if (it == 0u) t0 = clock64();
        if (clock64() - t0 >= p.timeout && it > 0u) {
            atomicExch(p.abort_flag, 1);
            set_status(p.status, RTPROJ_ETIMEOUT);
            return false;
        }
        return !((++it & 63u) == 0u && *(volatile int*)p.abort_flag);
    }
};

// Warp-wide: waits until the G records carry `tag`, returns the largest key and whether its norm
// has cancelled; false on expiry.
__device__ __forceinline__ bool poll_records(const QrRegsDev& p, const ulonglong2* rec, int G, uint32_t tag, int lane,
                                             unsigned long long& key, bool& cancelled) {
    Deadline d;
    while (true) {
        unsigned long long best = 0ull;
        bool flag = false, ready = true;
        for (int g = lane; g < G; g += 32) {
            const ulonglong2 w = ld_word(rec + g);
            ready &= (uint32_t)w.y == tag;
            if (w.x > best) { best = w.x; flag = (w.y >> 32) != 0ull; }
        }
        if (__all_sync(0xffffffffu, ready)) {
            key = warp_max_key(best);
            cancelled = __any_sync(0xffffffffu, best == key && flag);
            return true;
        }
        if (!__all_sync(0xffffffffu, d.more(p))) return false;
    }
}

// The warps of one column meet (WPC of them; barrier 0 is the CTA's).
template <int WPC>
__device__ __forceinline__ void column_barrier(int c) {
    if (WPC == 1) __syncwarp();
    else asm volatile("barrier.sync %0, %1;" ::"r"(c + 1), "n"(32 * WPC) : "memory");
}

// NP: row pairs per lane; WPC: warps per column; MAXW: most warps of a CTA. l <= 64 NP WPC, or with
// LONG any l: a column's first pairs p.tg live in its packets (read back from L2 in both passes), the
// next p.ts in shared memory, the rest in registers -- the rows that leave the factorization first
// are the ones whose reads cost most. tg and ts are multiples of 32 WPC. Few pairs in registers and
// few packets in flight, so that nothing spills: 12 and 6 of them took 51 ms at 2048 x 4128, 3 and 4
// take 39.
template <class A, int NP, int WPC, int MAXW, bool LONG>
__global__ void __launch_bounds__(32 * MAXW, 1) qr_regs_kernel(QrRegsDev p) {
    using S = typename A::S;
    constexpr int GR = 32 * WPC;                     // pairs of a column's group: one a lane
    extern __shared__ __align__(16) ulonglong2 qr_smem[];
    __shared__ ulonglong2 vs_short[LONG ? 1 : NP * GR];
    const int base = LONG ? p.tg + p.ts : 0;         // the first pair in registers
    ulonglong2* vs = LONG ? qr_smem : vs_short;      // the reflector, zero above row j
    __shared__ double col_mx[MAXW];
    __shared__ unsigned long long key_s[MAXW];       // the columns' keys (0: retired)
    __shared__ uint32_t flag_s[MAXW];                // whether a column's early norm has cancelled
    __shared__ unsigned long long win_s[2];          // the winner by round
    __shared__ int state_s[2];                       // 0: expired, 1: winner, 2: winner has cancelled
    __shared__ f2 dot_s[MAXW], nsq_s[MAXW], cj_s[MAXW];
    __shared__ f2 scal_s[3];                         // alpha, v0, beta where one warp forms them
    __shared__ int ok_s, e_s, range_s;
    const int l = p.l, m = p.m, cpc = p.cpc, npk = (l + 1) >> 1;
    const int b = blockIdx.x, G = gridDim.x, t = threadIdx.x, lane = t & 31, warp = t >> 5, NT = blockDim.x;
    const int c0 = b * cpc, nc = max(0, min(cpc, m - c0));
    const int cw = warp / WPC, part = warp % WPC, col = c0 + cw;      // the warp's column and its share of the rows
    const bool mine = cw < nc;
    // pair of the warp's i-th group in registers, and of the column's g-th group
    auto pair_of = [&](int i) { return base + 32 * (i * WPC + part) + lane; };
    auto pair_in = [&](int g) { return g * GR + 32 * part + lane; };
    ulonglong2* held = LONG ? qr_smem + base + NP * GR + (size_t)cw * p.ts - p.tg : nullptr;   // indexed by pair
    const int g_l2 = LONG ? p.tg / GR : 0, g_sm = LONG ? base / GR : 0;   // groups: [0, g_l2) L2, [g_l2, g_sm) shared

    // 0. tags cleared; the scale: exponents of the CTAs' largest entries, and of their columns'
    //    smallest largest entry, exchanged once (see the top)
    if (mine) {
        double cm = 0.0;
        for (int i = 32 * part + lane; i < l; i += 32 * WPC) {
            const double x = fabs(p.S[(int64_t)col * p.lds + i]);
            cm = fmax(cm, isfinite(x) ? x : INFINITY);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cm = fmax(cm, __shfl_xor_sync(0xffffffffu, cm, o));
        if (lane == 0) col_mx[warp] = cm;
        for (int q = 32 * part + lane; q < npk; q += 32 * WPC) {
            st_word(p.slots + (size_t)col * npk + q, 0ull, 0ull);
        }
    }
    for (int q = t; q < base + NP * GR; q += NT) vs[q] = make_ulonglong2(0ull, 0ull);
    __syncthreads();
    if (t == 0) {
        int e_hi = INT_MIN / 2, e_lo = INT_MAX / 2;
        for (int q = 0; q < nc; ++q) {
            double cm = col_mx[q * WPC];
            for (int u = 1; u < WPC; ++u) cm = fmax(cm, col_mx[q * WPC + u]);
            int e = INT_MIN / 2;
            if (isinf(cm)) e = 2 * MAX_SCALE;                // an entry that is not finite
            else if (cm > 0.0) frexp(cm, &e);                // cm < 2^e
            e_hi = max(e_hi, e);
            e_lo = min(e_lo, e);
        }
        p.emax[b] = e_hi;
        p.emax[G + b] = e_lo;
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;\n" ::"l"(p.counter), "r"(1u) : "memory");
        Deadline d;
        bool ok = true;
        while (true) {
            unsigned int v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p.counter) : "memory");
            if (v >= (unsigned int)G) break;
            if (!d.more(p)) { ok = false; break; }
        }
        int E = INT_MIN / 2, Elo = INT_MAX / 2;
        if (ok)
            for (int g = 0; g < G; ++g) {
                E = max(E, __ldcg(p.emax + g));
                Elo = min(Elo, __ldcg(p.emax + G + g));
            }
        int half = 0;                                       // 4^half >= l: every column's norm is below 1
        while ((1 << (2 * half)) < l) ++half;
        e_s = E == INT_MIN / 2 ? 0 : E + half;
        range_s = E - Elo;
        ok_s = ok;
    }
    __syncthreads();
    if (!ok_s) return;
    if (range_s > A::RANGE || abs(e_s) > MAX_SCALE) {            // the same decision in every CTA
        if (b == 0 && t == 0) *p.fallback = 1;
        return;
    }
    const int E = e_s;

    // the column, its norm and its packets for step 0
    f2 ch[NP], cl[NP];
    S nsq = A::zero();
    bool active = mine;
    int pos = -1;
    S alpha_mine = A::zero();
    // the column's sum over its warps of each warp's total (every lane receives it)
    auto column_sum = [&](S x, f2* buf) {
        if (WPC == 1) return x;
        if (lane == 0) buf[warp] = A::bits(x);
        column_barrier<WPC>(cw);
        S sum = A::of(buf[cw * WPC]);
#pragma unroll
        for (int u = 1; u < WPC; ++u) sum = A::add(sum, A::of(buf[cw * WPC + u]));
        return sum;
    };
    // the CTA's record of step s (warp 0, after a barrier): its largest key, and that column's flag
    auto publish = [&](ulonglong2* rec, int s, bool flags) {
        const unsigned long long k = lane < nc ? key_s[lane] : 0ull;
        const unsigned long long best = warp_max_key(k);
        const uint32_t f =
            flags && __any_sync(0xffffffffu, k == best && k != 0ull && flag_s[lane < nc ? lane : 0] != 0u) ? 1u : 0u;
        if (lane == 0)
            st_word(rec + (s & 1) * G + b, best, (unsigned long long)(uint32_t)(s + 1) | ((unsigned long long)f << 32));
    };
    if (t < MAXW) {
        key_s[t] = 0ull;
        flag_s[t] = 0u;
    }
    __syncthreads();
    if (mine) {
        const double sc = ldexp(1.0, -E);
        const double* src = p.S + (int64_t)col * p.lds;
        ffp a[A::ACCS] = {};
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int q = pair_of(i), r0 = 2 * q;
            const ffp x = A::pair(r0 < l ? src[r0] * sc : 0.0, r0 + 1 < l ? src[r0 + 1] * sc : 0.0);
            ch[i] = x.h;
            cl[i] = x.l;
            A::dot(a[i % A::ACCS], x, x);
            if (q < npk) st_packet(p.slots + (size_t)col * npk + q, x, A::tag(0));
        }
        if constexpr (LONG) {
            for (int g = 0; g < g_sm; ++g) {
                const int q = pair_in(g), r0 = 2 * q;
                const ffp x = A::pair(r0 < l ? src[r0] * sc : 0.0, r0 + 1 < l ? src[r0 + 1] * sc : 0.0);
                A::dot(a[0], x, x);
                if (q < npk) st_packet(p.slots + (size_t)col * npk + q, x, A::tag(0));
                if (g >= g_l2) held[q] = make_ulonglong2(x.h, x.l);
            }
        }
        nsq = column_sum(A::total(a), nsq_s);
        if (lane == 0 && part == 0) {
            st_word(p.nrm + col, A::bits(nsq), 1ull);
            key_s[cw] = A::key(nsq, col);
        }
    } else {
#pragma unroll
        for (int i = 0; i < NP; ++i) ch[i] = cl[i] = 0ull;
    }

    __syncthreads();
    if (warp == 0) publish(p.rec, 0, false);

    for (int j = 0; j < m; ++j) {
        const int par = j & 1;
        // 1. the winner; once more with fresh norms when its own has cancelled (the same decision in
        //    every CTA)
        int round = 0;
        for (; round < 2; ++round) {
            if (round == 1) {
                if (active && lane == 0 && part == 0) key_s[cw] = A::key(nsq, col);
                __syncthreads();
                if (warp == 0) publish(p.rec_exact, j, false);
            }
            if (warp == 0) {
                unsigned long long key = 0ull;
                bool cancelled = false;
                const bool ok = poll_records(p, (round == 0 ? p.rec : p.rec_exact) + par * G, G, (uint32_t)(j + 1), lane, key,
                                             cancelled);
                if (lane == 0) {
                    win_s[round] = key;
                    state_s[round] = !ok || key == 0ull ? 0 : cancelled ? 2 : 1;
                }
            }
            __syncthreads();
            if (state_s[round] == 0) return;
            if (state_s[round] == 1) break;
        }
        const unsigned long long win = win_s[round];
        const int piv = 4095 - (int)(win & 4095ull);
        if (piv < 0 || piv >= m) return;                      // cannot happen while columns remain
        // 2. the reflector: the pivot's packets of rows j .. l-1, the row-j packet and the norm
        const ulonglong2* slot = p.slots + (size_t)piv * npk;
        const Tag tag = A::tag(j);
        const int q0 = j >> 1;
        bool good = true;
        constexpr int VL = LONG ? 6 : (NP * GR + 127) / 128; // packets per thread (at 128 threads all of them)
        ulonglong2 w[VL];
#pragma unroll
        for (int k = 0; k < VL; ++k)
            if (q0 + t + k * NT < npk) w[k] = ld_word(slot + q0 + t + k * NT);
        const bool scalars = !A::SHARED_SCALARS || warp == 0;
        S alpha = A::zero(), v0 = A::zero(), beta = A::zero();
        bool small = false;                                  // the kernel enqueued behind takes over
        if (t == 0 && q0 > 0) vs[q0 - 1] = make_ulonglong2(0ull, 0ull);
        if (scalars) {
            ulonglong2 wj = ld_word(slot + q0), wn = ld_word(p.nrm + (size_t)par * m + piv);
            Deadline d;
            while (!has_tag<A>(wj, tag) && good) { good = d.more(p); wj = ld_word(slot + q0); }
            while ((uint32_t)wn.y != (uint32_t)(j + 1) && good) { good = d.more(p); wn = ld_word(p.nrm + (size_t)par * m + piv); }
            const S npiv = A::of(wn.x);
            small = A::too_small(npiv);
            const S x0 = A::row(unpack<A>(wj), (j & 1) != 0);
            const S nx = A::sqrt(npiv);
            alpha = A::nonneg(x0) ? A::neg(nx) : nx;
            v0 = A::add(x0, A::neg(alpha));
            beta = A::recip(A::mul(nx, A::add(nx, A::nonneg(x0) ? x0 : A::neg(x0))));
            if (A::SHARED_SCALARS && t == 0) {
                scal_s[0] = A::bits(alpha);
                scal_s[1] = A::bits(v0);
                scal_s[2] = A::bits(beta);
            }
        }
#pragma unroll
        for (int k = 0; k < VL; ++k) {
            const int q = q0 + t + k * NT;
            if (q < npk) {
                Deadline d;
                while (!has_tag<A>(w[k], tag) && good) { good = d.more(p); w[k] = ld_word(slot + q); }
                ffp v = unpack<A>(w[k]);
                if (q == q0) v = A::first(v, (j & 1) != 0, v0);   // rows above j stay out, row j: x0 - alpha
                vs[q] = make_ulonglong2(v.h, v.l);
            }
        }
        if constexpr (LONG)
            for (int q = q0 + t + VL * NT; q < npk; q += NT) {
                ulonglong2 x = ld_word(slot + q);
                Deadline d;
                while (!has_tag<A>(x, tag) && good) { good = d.more(p); x = ld_word(slot + q); }
                const ffp v = unpack<A>(x);
                vs[q] = make_ulonglong2(v.h, v.l);
            }
        good = __syncthreads_and(good && !small);
        if (A::SHARED_SCALARS) {
            alpha = A::of(scal_s[0]);
            v0 = A::of(scal_s[1]);
            beta = A::of(scal_s[2]);
        }
        if (!good) {
            if (small && b == 0 && t == 0) *p.fallback = 1;   // every thread of every CTA reads the same norm
            return;
        }
        if (active && col == piv) {
            active = false;
            pos = j;
            alpha_mine = alpha;
            if (lane == 0 && part == 0) {
                p.perm[j] = piv;
                key_s[cw] = 0ull;
            }
        }
        // 3. the dot product (v is zero outside rows j .. l - 1, so whole groups of rows go through;
        //    in float-float three at a time, to keep independent chains in flight) and the next trailing norm
        S nw = A::zero();
        if (active) {
            ffp a[A::ACCS] = {};
            f2 xh = 0ull, xl = 0ull;                          // the pair that holds row j
            if constexpr (LONG) {
                const ulonglong2* own = p.slots + (size_t)col * npk;
                int g = q0 / GR;                              // the first group with a row from j on
                for (; g < g_l2; g += LB) {
                    ulonglong2 x[LB];
#pragma unroll
                    for (int u = 0; u < LB; ++u)
                        if (g + u < g_l2) x[u] = ld_word(own + pair_in(g + u));
#pragma unroll
                    for (int u = 0; u < LB; ++u)
                        if (g + u < g_l2) {
                            const int q = pair_in(g + u);
                            const ulonglong2 v = vs[q];
                            const ffp c = unpack<A>(x[u]);
                            A::dot(a[0], {v.x, v.y}, c);
                            if (q == q0) { xh = c.h; xl = c.l; }
                        }
                }
                g = max(q0 / GR, g_l2);
#pragma unroll 2
                for (; g < g_sm; ++g) {
                    const int q = pair_in(g);
                    const ulonglong2 v = vs[q], c = held[q];
                    A::dot(a[0], {v.x, v.y}, {c.x, c.y});
                    if (q == q0) { xh = c.x; xl = c.y; }
                }
            }
#pragma unroll
            for (int i = 0; i < NP; i += A::ACCS)
                if (base + GR * (i + A::ACCS) > q0 && (A::ACCS > 1 || base + GR * i < npk)) {
#pragma unroll
                    for (int u = 0; u < A::ACCS; ++u) {
                        const ulonglong2 v = vs[pair_of(i + u)];
                        A::dot(a[u], {v.x, v.y}, {ch[i + u], cl[i + u]});
                    }
                    if (base + GR * i <= q0) {
#pragma unroll
                        for (int u = 0; u < A::ACCS; ++u)
                            if (pair_of(i + u) == q0) { xh = ch[i + u]; xl = cl[i + u]; }
                    }
                }
            S cj = A::row({xh, xl}, (j & 1) != 0);
            if (WPC == 1) cj = A::of(__shfl_sync(0xffffffffu, A::bits(cj), q0 & 31));
            else if ((q0 >> 5) % WPC == part && lane == (q0 & 31)) cj_s[cw] = A::bits(cj);
            nw = A::neg(A::mul(column_sum(A::total(a), dot_s), beta));
            if (WPC > 1) cj = A::of(cj_s[cw]);
            if (part == 0) {
                const S r = A::add(cj, A::mul(nw, v0));       // R's entry
                const S ne = A::add(nsq, A::neg(A::mul(r, r)));
                if (lane == 0) {
                    key_s[cw] = A::key(A::clamp(ne), col);
                    flag_s[cw] = A::cancelled(ne, nsq) ? 1u : 0u;
                }
            }
        }
        __syncthreads();
        if (warp == 0) publish(p.rec, j + 1, true);
        // 4. the update, the fresh norm, the packets of step j + 1
        if (active) {
            const ffp w2 = A::both(nw);
            ulonglong2* dst = p.slots + (size_t)col * npk;
            const Tag ntag = A::tag(j + 1);
            const int qn = (j + 1) >> 1;
            ffp a[A::ACCS] = {};
            // one pair: the updated rows, counted in the fresh norm from row j + 1 on (of the pair that holds
            // row j its second row, or none)
            auto step = [&](const ffp& c, int q, ffp& acc, bool st) {
                const ulonglong2 v = vs[q];
                const ffp x = A::update(c, w2, {v.x, v.y});
                if (st) st_packet(dst + q, x, ntag);
                const ffp y = A::keep(x, q > q0, q == q0 && !(j & 1));
                A::dot(acc, y, y);
                return x;
            };
            if constexpr (LONG) {
                int g = q0 / GR;
                for (; g < g_l2; g += LB) {
                    ulonglong2 x[LB];
#pragma unroll
                    for (int u = 0; u < LB; ++u)
                        if (g + u < g_l2) x[u] = ld_word(dst + pair_in(g + u));
#pragma unroll
                    for (int u = 0; u < LB; ++u)
                        if (g + u < g_l2) {
                            const int q = pair_in(g + u);
                            const ffp y = step(unpack<A>(x[u]), q, a[0], q >= q0);
                        }
                }
                g = max(q0 / GR, g_l2);
#pragma unroll 2
                for (; g < g_sm; ++g) {
                    const int q = pair_in(g);
                    const ulonglong2 c = held[q];
                    const ffp y = step({c.x, c.y}, q, a[0], q >= qn);
                    held[q] = make_ulonglong2(y.h, y.l);
                }
            }
#pragma unroll
            for (int i = 0; i < NP; i += A::ACCS)
                if (base + GR * (i + A::ACCS) > q0 && (A::ACCS > 1 || base + GR * i < npk)) {
#pragma unroll
                    for (int u = 0; u < A::ACCS; ++u) {
                        const int q = pair_of(i + u);
                        const ffp x = step({ch[i + u], cl[i + u]}, q, a[u], q >= qn && q < npk);
                        ch[i + u] = x.h;
                        cl[i + u] = x.l;
                    }
                }
            nsq = column_sum(A::total(a), nsq_s);
            if (lane == 0 && part == 0)
                st_word(p.nrm + (size_t)(par ^ 1) * m + col, A::bits(nsq), (unsigned long long)(uint32_t)(j + 2));
        }
    }
    // R[:, pos] = rows 0 .. pos of the retired column, scaled back by 2^E
    if (!mine || pos < 0) return;
    auto store_pair = [&](int q, const ffp& c) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int row = 2 * q + u;
            if (row >= m) continue;
            const S x = row == pos ? alpha_mine : A::row(c, u != 0);
            p.R[(int64_t)row * m + pos] = row <= pos ? ldexp(A::to_double(x), E) : 0.0;
        }
    };
#pragma unroll
    for (int i = 0; i < NP; ++i) store_pair(pair_of(i), {ch[i], cl[i]});
    if constexpr (LONG)
        for (int g = 0; g < g_sm; ++g) {
            const int q = pair_in(g);
            if (2 * q >= m) break;
            if (g >= g_l2) store_pair(q, {held[q].x, held[q].y});
            else store_pair(q, unpack<A>(ld_word(p.slots + (size_t)col * npk + q)));
        }
}

struct Shape {
    const void* kern;
    int np, wpc, maxw;
    bool longer;
};

}  // namespace

// Workspace: the packets, the records, the norms and the scale exchange.
size_t qr_regs_work_doubles(int m, int l) {
    const size_t npk = ((size_t)l + 1) / 2;
    return 2 * ((size_t)m * npk) + 2 * 6 * (size_t)m + (size_t)m + 64;
}

cudaError_t pivoted_qr_regs(const double* S, int m, int l, int64_t lds, double* R, int32_t* perm, double* work,
                            int* status, cudaStream_t s, long long spin_limit, int* fallback, bool f64, bool* launched) {
    *launched = false;
    int dev = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    const int sms = sm_count();
    if (!coop) return cudaSuccess;
    // Float64 with few columns: the steps saved are less than the launch of the kernel behind (QR phase, us,
    // persistent alone / this form: 1 x 5 14 / 21, 4 x 8 25 / 32, 8 x 12 39 / 44, 10 x 14 45 / 50, 12 x 16
    // 59 / 56, 16 x 20 74 / 71).
    if (f64 && m < 12) return cudaSuccess;
    // Warps per column, and row pairs a lane holds.
#define QR_SHAPE(A, NP, WPC, MAXW) {(const void*)qr_regs_kernel<A, NP, WPC, MAXW, false>, NP, WPC, MAXW, false}
#define QR_LONG(A, NP, WPC, MAXW) {(const void*)qr_regs_kernel<A, NP, WPC, MAXW, true>, NP, WPC, MAXW, true}
    const Shape ff_shapes[] = {QR_SHAPE(FfArith, 3, 1, 16),  QR_SHAPE(FfArith, 6, 1, 16),  QR_SHAPE(FfArith, 9, 1, 16),
                               QR_SHAPE(FfArith, 6, 2, 16),  QR_SHAPE(FfArith, 12, 1, 16), QR_SHAPE(FfArith, 9, 2, 16),
                               QR_SHAPE(FfArith, 12, 2, 16), QR_SHAPE(FfArith, 30, 1, 8),  QR_SHAPE(FfArith, 33, 1, 8),
                               QR_LONG(FfArith, 3, 4, 16),   QR_LONG(FfArith, 3, 2, 16),   QR_LONG(FfArith, 3, 1, 16)};
    const Shape f64_shapes[] = {QR_SHAPE(F64Arith, 3, 2, 16), QR_SHAPE(F64Arith, 6, 2, 16), QR_SHAPE(F64Arith, 9, 2, 16),
                                QR_SHAPE(F64Arith, 12, 2, 16), QR_SHAPE(F64Arith, 9, 4, 16)};
#undef QR_SHAPE
#undef QR_LONG
    // Four columns a CTA while that fits the chip (float64: two, whose arithmetic then has a sub-
    // partition each; 256 x 544 took 1.35 ms by fours, 1.17 by twos), more beyond.
    const int few = f64 ? 2 : 4;
    const int cpc = std::max((m + sms - 1) / sms, std::min(few, m));
    const int G = (m + cpc - 1) / cpc;
    const Shape* sh = nullptr;
    const Shape* first = f64 ? std::begin(f64_shapes) : std::begin(ff_shapes);
    const Shape* last = f64 ? std::end(f64_shapes) : std::end(ff_shapes);
    for (const Shape* x = first; x != last && !sh; ++x)
        if ((x->longer || l <= 64 * x->np * x->wpc) && cpc * x->wpc <= x->maxw) {
            // A warp with 30 or more pairs a lane pays from seven columns a CTA up (with fewer, two or four
            // warps a column are faster: 900 x 2100, six columns, 5.6 ms as LONG, 6.3 so) and when its rows fill
            // nine tenths of the registers (1000 x 1600 5.8 as LONG, 6.1 so; 1000 x 1900 6.6 and 6.2; 1024 x 2080
            // 7.2 and 6.9).
            if (x->np >= 30 && (cpc < 7 || 10 * l <= 9 * 64 * x->np)) continue;
            sh = x;
        }
    if (!sh) return cudaSuccess;
    const int nt = 32 * std::max(cpc * sh->wpc, 4);   // at least 128 threads load the pivot column's packets
    // LONG: as many groups of each column in shared memory as fit beside the reflector, the rest in L2
    const size_t npk = ((size_t)l + 1) / 2;
    const int gr = 32 * sh->wpc, in_regs = gr * sh->np;
    int tg = 0, ts = 0;
    size_t smem = 0;
    if (sh->longer) {
        const int rest = std::max(0, ((int)npk - in_regs + gr - 1) / gr * gr);
        constexpr size_t most = (size_t)220 << 10;
        const size_t room = most / sizeof(ulonglong2), reflector = (size_t)rest + in_regs;
        if (reflector + (size_t)cpc * gr > room) return cudaSuccess;
        ts = std::min(rest, (int)((room - reflector) / cpc) / gr * gr);
        tg = rest - ts;
        smem = (reflector + (size_t)cpc * ts) * sizeof(ulonglong2);
        if (allow_dynamic_shared(sh->kern, most) != cudaSuccess) {
            cudaGetLastError();
            return cudaSuccess;
        }
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sh->kern, nt, smem) != cudaSuccess || per_sm < 1 ||
        G > per_sm * sms) {
        cudaGetLastError();
        return cudaSuccess;
    }
    QrRegsDev p;
    p.S = S; p.m = m; p.l = l; p.lds = lds; p.R = R; p.perm = perm; p.cpc = cpc;
    p.tg = tg; p.ts = ts;
    ulonglong2* w = reinterpret_cast<ulonglong2*>(work);
    p.slots = w;      w += (size_t)m * npk;
    ulonglong2* cleared = w;                       // words whose tags must start at zero
    p.rec = w;        w += 2 * (size_t)G;
    p.rec_exact = w;  w += 2 * (size_t)G;
    p.nrm = w;        w += 2 * (size_t)m;
    p.counter = reinterpret_cast<unsigned int*>(w);
    p.abort_flag = reinterpret_cast<int*>(p.counter + 1);
    w += 1;
    const size_t cleared_bytes = (size_t)((char*)w - (char*)cleared);
    p.emax = reinterpret_cast<int*>(w);            // 2 G ints
    p.status = status;
    p.timeout = spin_limit;
    p.fallback = fallback;
    cudaError_t e = cudaMemsetAsync(cleared, 0, cleared_bytes, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(fallback, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    void* args[] = {&p};
    e = cudaLaunchCooperativeKernel(sh->kern, dim3((unsigned)G), dim3((unsigned)nt), args, smem, s);
    note_launch();
    if (e != cudaSuccess) {
        cudaGetLastError();   // clear; the caller's other kernels run
        return cudaSuccess;
    }
    *launched = true;
    return cudaSuccess;
}

}  // namespace rtp
