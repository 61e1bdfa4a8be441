// Exact fixed-point slicing of float64 operands into bfloat16 digit planes (mixed mode).
//
// For a row x of an operand (the products reduce along the row), with e the smallest
// integer such that max |x_c| < 2^e, every entry is written as
//     x_c ~= 2^e * sum_{p < s} d_p * 2^{-7-8p},     d_p integers in [-128, 128] (s <= 10),
// the balanced base-256 digits of F = round(|x_c| 2^{7+8(s-1)-e}), signed like x_c.
// Each d_p is exact in bfloat16, so the tensor cores multiply digits exactly and the
// float32 accumulator sums them exactly as long as a partial sum stays below 2^24.
// Truncation error per entry: at most 2^{e-8s} (half a unit of the last digit).
//
// The digits come from 32-bit integer operations on the float64 bit pattern (no FP64 pipe): with
// the significand left-aligned in a word of W x 32 bits, the entry's digits for any s are bytes
// of that word shifted right by 1023 - E + e, after one addition of 0x80 in each of the s bytes
// below the top one -- the carries of the balanced digits and the rounding at once (byte - 128
// is the digit; the byte below the last digit takes the rounding's half). A byte becomes a
// bfloat16 by one byte permutation and one float32 multiply-add that also takes off the 128 and
// sets the sign. About 16 + 3.5 s instructions an entry; with a carry chain and 64-bit shifts
// a digit it took 14 s, and slicing 4096 x 8192 into 9 planes took 187 us instead of 154 (the bytes
// need 128).
#include "rtproj_internal.cuh"

#include <algorithm>
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace rtp {
namespace {

constexpr int SR_THREADS = 256;        // contiguous rows, a cluster per row
constexpr int SL_THREADS = 512;        // spans of contiguous rows
constexpr int SC_THREADS = 256;        // columns of a row-major block
constexpr int SL_MAX_PARTS = 8;        // CTAs per row (one cluster)
constexpr uint32_t EXP_MASK = 0x7FF00000u;

struct SliceDev {
    const void* X; int64_t x_rs;
    int rows, cols, s;
    __nv_bfloat16* d; int64_t ld, ps;
    int32_t* e;
    int* status;
};

// What a pass over right-hand sides does besides the digits (each optional).
struct RowExtras {
    double* wide = nullptr; int64_t ldw = 0;        // the row as float64 (for a float32 source)
    double* norms = nullptr;                        // its 2-norm
    unsigned long long* clear = nullptr;            // two words to be zeroed
};

// What a pass over a correction's columns does besides the digits: h += dh, and the report's
// maxima of ||r_j|| and ||dh_j|| (see column_stats).
struct Correction {
    double* h; const double* r; const double* bnorm; const double* normA; unsigned long long* stats;
};

template <int W>
struct DigitWord { uint32_t w[W]; };   // w[W - 1] the highest

// One float64 given by its halves: left-aligned significand (H, L) and biased exponent E
// (a subnormal is normalised; zero and the non-finite values give H = L = 0).
__device__ __forceinline__ void split_double(uint32_t xl, uint32_t xh, uint32_t& H, uint32_t& L, int& E) {
    E = (int)((xh & EXP_MASK) >> 20);
    H = ((xh & 0xFFFFFu) << 11) | (xl >> 21) | (E ? 0x80000000u : 0u);
    L = xl << 11;
    if (E == 0x7FF) H = L = 0u;
    if (E == 0 && (H | L)) {
        const int z = H ? __clz((int)H) : 32 + __clz((int)L);
        if (z >= 32) { H = L << (z - 32); L = 0u; }
        else { H = __funnelshift_l(L, H, z); L <<= z; }
        E = 1 - z;
    }
}

// The digits' word: |x| scaled so that 2^e is the top byte's 128, plus the digits' biases
// (k: 0x80 in each of the s bytes below the top one). W = 2 holds s <= 7 (and a byte for the
// rounding), W = 3 s <= 11.
template <int W>
__device__ __forceinline__ DigitWord<W> digit_word(uint32_t xl, uint32_t xh, int e, const DigitWord<W>& k) {
    uint32_t H, L;
    int E;
    split_double(xl, xh, H, L, E);
    int r = 1023 - E + e;                      // >= 1 for a nonzero entry, since |x| < 2^e
    r = r > 32 * W - 1 ? 32 * W - 1 : r;
    DigitWord<W> a;
    if constexpr (W == 2) {
        const bool s32 = (r & 32) != 0;
        a.w[0] = s32 ? H : L;
        a.w[1] = s32 ? 0u : H;
        a.w[0] = __funnelshift_r(a.w[0], a.w[1], r);
        a.w[1] >>= (r & 31);
        asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+r"(a.w[0]), "+r"(a.w[1]) : "r"(k.w[0]), "r"(k.w[1]));
    } else {
        const bool s64 = (r & 64) != 0, s32 = (r & 32) != 0;
        uint32_t w2 = s64 ? 0u : H, w1 = s64 ? 0u : L, w0 = s64 ? H : 0u;
        w0 = s32 ? w1 : w0;
        w1 = s32 ? w2 : w1;
        w2 = s32 ? 0u : w2;
        a.w[0] = __funnelshift_r(w0, w1, r);
        a.w[1] = __funnelshift_r(w1, w2, r);
        a.w[2] = w2 >> (r & 31);
        asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
            : "+r"(a.w[0]), "+r"(a.w[1]), "+r"(a.w[2]) : "r"(k.w[0]), "r"(k.w[1]), "r"(k.w[2]));
    }
    return a;
}

template <int W>
__device__ __forceinline__ DigitWord<W> digit_bias(int s) {
    DigitWord<W> k;
#pragma unroll
    for (int w = 0; w < W; ++w) k.w[w] = 0u;
#pragma unroll
    for (int p = 1; p < 4 * W; ++p) {
        const int b = 4 * W - 1 - p;
        if (p <= s) k.w[b >> 2] |= 0x80u << (8 * (b & 3));
    }
    return k;
}

// Digit P of an entry as the float32 whose upper half is the bfloat16 (sg = 1 or -1): the byte
// under the exponent of 2^23 is 2^23 + byte, exact.
template <int W, int P>
__device__ __forceinline__ uint32_t digit_float(const DigitWord<W>& a, float sg) {
    constexpr int b = 4 * W - 1 - P;
    const float f = __uint_as_float(__byte_perm(a.w[b >> 2], 0x4B000000u, 0x7440 | (b & 3)));
    return __float_as_uint(fmaf(f, sg, sg * (P ? -8388736.0f : -8388608.0f)));
}

__device__ __forceinline__ float sign_of(uint32_t xh) { return __uint_as_float(0x3F800000u | (xh & 0x80000000u)); }

// Digits of eight entries (consecutive along the row) to planes P, P + 1, ..., s - 1: one 16-byte
// store a plane.
template <int W, int P>
__device__ __forceinline__ void store_digits(const DigitWord<W> (&a)[8], const float (&sg)[8], int s, __nv_bfloat16* d,
                                             int64_t ps) {
    if constexpr (P < (W == 2 ? 7 : 10)) {
        if (P >= s) return;
        uint32_t v[4];
#pragma unroll
        for (int h = 0; h < 4; ++h)
            v[h] = __byte_perm(digit_float<W, P>(a[2 * h], sg[2 * h]), digit_float<W, P>(a[2 * h + 1], sg[2 * h + 1]), 0x7632);
        *reinterpret_cast<uint4*>(d + (int64_t)P * ps) = make_uint4(v[0], v[1], v[2], v[3]);
        store_digits<W, P + 1>(a, sg, s, d, ps);
    }
}

__device__ __forceinline__ uint2 entry_bits(const double* p) { return __ldg(reinterpret_cast<const uint2*>(p)); }
__device__ __forceinline__ uint2 entry_bits(const float* p) { return widen_bits(__ldg(p)); }

// 32-byte accesses (a whole sector a lane: 16-byte ones at this 64-byte stride move every
// sector in two halves).
__device__ __forceinline__ void load_sector(const double* p, uint2& a, uint2& b, uint2& c, uint2& d) {
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(a.x), "=r"(a.y), "=r"(b.x), "=r"(b.y), "=r"(c.x), "=r"(c.y), "=r"(d.x), "=r"(d.y) : "l"(p));
}
__device__ __forceinline__ void store_sector(double* p, uint2 a, uint2 b, uint2 c, uint2 d) {
    asm volatile("st.global.v8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
                 :: "r"(a.x), "r"(a.y), "r"(b.x), "r"(b.y), "r"(c.x), "r"(c.y), "r"(d.x), "r"(d.y), "l"(p) : "memory");
}

// Eight entries from column c on (zeros past cols); vec: the row starts on a 32-byte boundary.
template <typename T>
__device__ __forceinline__ void load_eight(const T* row, int c, int cols, bool vec, uint2 (&x)[8]) {
    if (vec && c + 8 <= cols) {
        if constexpr (sizeof(T) == 8) {
            load_sector(row + c, x[0], x[1], x[2], x[3]);
            load_sector(row + c + 4, x[4], x[5], x[6], x[7]);
        } else {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(row + c) + q);
                x[4 * q] = widen_bits(v.x);
                x[4 * q + 1] = widen_bits(v.y);
                x[4 * q + 2] = widen_bits(v.z);
                x[4 * q + 3] = widen_bits(v.w);
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = c + q < cols ? entry_bits(row + c + q) : make_uint2(0u, 0u);
    }
}

// frexp exponent of the maximum of a row's columns [c0, c1) when all finite ones lie below the
// normal range (rare): every bit is looked at again. smax: a word per warp; all threads call it.
template <int THREADS, typename T>
__device__ __noinline__ int small_max_exponent(const T* row, int c0, int c1, unsigned long long* smax) {
    unsigned long long mx = 1;
    for (int c = c0 + (int)threadIdx.x; c < c1; c += THREADS) {
        const uint2 x = entry_bits(row + c);
        if ((x.y & EXP_MASK) == EXP_MASK) continue;
        const unsigned long long u = ((unsigned long long)(x.y & 0x7FFFFFFFu) << 32) | x.x;
        mx = u > mx ? u : mx;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = v > mx ? v : mx;
    }
    if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = mx;
    __syncthreads();
    for (int w = 0; w < THREADS / 32; ++w) mx = smax[w] > mx ? smax[w] : mx;
    return (64 - __clzll((long long)mx)) - 1074;
}

// The exponent for a running maximum of take_max: kZeroRowExp for zeros only, and SUBNORMAL where
// small_max_exponent has to look again.
constexpr int SUBNORMAL = kZeroRowExp + 1;
__device__ __forceinline__ int exponent_of_max(uint32_t mx) {
    return mx >= 0x00100000u ? (int)(mx >> 20) - 1022 : mx ? SUBNORMAL : kZeroRowExp;
}

// One entry into a running maximum of the upper halves (non-finite entries apart); a nonzero lower
// half counts as its last bit, so that a maximum of zero means zeros only.
__device__ __forceinline__ void take_max(uint2 x, uint32_t& mx, bool& bad) {
    const uint32_t u = (x.y & 0x7FFFFFFFu) | (x.x ? 1u : 0u);
    if (u >= EXP_MASK) bad = true;
    else mx = u > mx ? u : mx;
}

// Contiguous rows, a cluster of CTAs per row (slice_parts): a thread loads eight consecutive
// entries, takes the row's maximum and what RowExtras asks for, the parts are exchanged through
// distributed shared memory, then the digits follow from the entries still in registers (a span
// longer than one pass of the threads is read again, from L1 or L2).
// Bound by memory: a 4096 x 8192 float64 block into 9 planes reads 268 MB and writes 604, at 5.7
// TB/s. One launch takes the place of five for a float32 block of few rows (widening, norms,
// exponents filled, exponents, digits: 17 us at 16 x 2048, now 7) and of three for many (4096 x
// 8192 into 7 planes: 350 us, now 214).
template <int W, typename T>
__global__ void __launch_bounds__(SR_THREADS, 4) slice_rows_kernel(SliceDev a, RowExtras x) {
    __shared__ uint32_t smax[SR_THREADS / 32];
    __shared__ double ssum[SR_THREADS / 32];
    __shared__ unsigned long long slow[SR_THREADS / 32];
    __shared__ uint32_t part_max;
    __shared__ double part_sum;
    __shared__ int e_s;
    cg::cluster_group cl = cg::this_cluster();
    const int parts = (int)cl.num_blocks(), q = (int)cl.block_rank();
    const int r = blockIdx.x / parts, t = threadIdx.x;
    const T* row = reinterpret_cast<const T*>(a.X) + (int64_t)r * a.x_rs;
    const int per = (int)(((a.ld / parts) + 7) / 8 * 8);
    const int c0 = q * per, c1 = min((int)a.ld, c0 + per);
    const bool vec = ((uintptr_t)row & 31) == 0, once = per <= 8 * SR_THREADS;
    uint32_t mx = 0;
    bool bad = false;
    double s0 = 0.0, s1 = 0.0;
    uint2 v[8];
#pragma unroll 1
    for (int cc = c0 + 8 * t; cc < c1; cc += 8 * SR_THREADS) {
        load_eight(row, cc, a.cols, vec, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) take_max(v[i], mx, bad);
        if (x.norms) {
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                const double d0 = __hiloint2double((int)v[i].y, (int)v[i].x);
                const double d1 = __hiloint2double((int)v[i + 1].y, (int)v[i + 1].x);
                s0 = fma(d0, d0, s0);
                s1 = fma(d1, d1, s1);
            }
        }
        if (x.wide) {
            double* w = x.wide + (int64_t)r * x.ldw + cc;
            if (((uintptr_t)w & 31) == 0 && cc + 8 <= a.cols) {
                store_sector(w, v[0], v[1], v[2], v[3]);
                store_sector(w + 4, v[4], v[5], v[6], v[7]);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (cc + i < a.cols) w[i] = __hiloint2double((int)v[i].y, (int)v[i].x);
            }
        }
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (x.norms) {
        s0 += s1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    }
    if ((t & 31) == 0) { smax[t >> 5] = mx; ssum[t >> 5] = s0; }
    const int any_bad = __syncthreads_or(bad);
    if (t == 0) {
        uint32_t m2 = 0;
        double s2 = 0.0;
        for (int w = 0; w < SR_THREADS / 32; ++w) { m2 = max(m2, smax[w]); s2 += ssum[w]; }
        part_max = m2;
        part_sum = s2;
        if (any_bad) set_status(a.status, RTPROJ_ENONFINITE);
        if (x.clear && blockIdx.x == 0) { x.clear[0] = 0ull; x.clear[1] = 0ull; }
    }
    if (parts > 1) cl.sync(); else __syncthreads();
    if (t == 0) {
        uint32_t m2 = part_max;
        double s2 = 0.0;
        for (int w = 0; w < parts; ++w) {
            if (parts > 1) m2 = max(m2, *cl.map_shared_rank(&part_max, w));
            if (x.norms && q == 0) s2 += parts > 1 ? *cl.map_shared_rank(&part_sum, w) : part_sum;
        }
        if (x.norms && q == 0) x.norms[r] = sqrt(s2);
        e_s = exponent_of_max(m2);
    }
    if (parts > 1) cl.sync(); else __syncthreads();        // parts stay readable until every CTA has read them
    int e = e_s;
    if (e == SUBNORMAL) e = small_max_exponent<SR_THREADS>(row, 0, a.cols, slow);   // the same in every CTA of the row
    if (e == kZeroRowExp) e = 0;                           // an all-zero row: exponent 0
    if (t == 0 && q == 0) a.e[r] = e;
    const DigitWord<W> k = digit_bias<W>(a.s);
    __nv_bfloat16* drow = a.d + (int64_t)r * a.ld;
#pragma unroll 1
    for (int cc = c0 + 8 * t; cc < c1; cc += 8 * SR_THREADS) {
        if (!once) load_eight(row, cc, a.cols, vec, v);
        DigitWord<W> w[8];
        float sg[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) { w[i] = digit_word<W>(v[i].x, v[i].y, e, k); sg[i] = sign_of(v[i].y); }
        store_digits<W, 0>(w, sg, a.s, drow + cc, a.ps);
    }
}

// The maximum exponents of contiguous rows, gathered over spans of SL_SPAN columns by atomic
// maxima (e pre-filled with kZeroRowExp).
constexpr int SL_SPAN = 8 * SL_THREADS;

__global__ void __launch_bounds__(SL_THREADS) row_exponents_kernel(SliceDev a) {
    __shared__ uint32_t smax[SL_THREADS / 32];
    __shared__ unsigned long long slow[SL_THREADS / 32];
    const int r = blockIdx.y, c0 = blockIdx.x * SL_SPAN, c1 = min(a.cols, c0 + SL_SPAN), t = threadIdx.x;
    const double* row = reinterpret_cast<const double*>(a.X) + (int64_t)r * a.x_rs;
    uint32_t mx = 0;
    bool bad = false;
#pragma unroll 8
    for (int c = c0 + t; c < c1; c += SL_THREADS) take_max(entry_bits(row + c), mx, bad);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((t & 31) == 0) smax[t >> 5] = mx;
    const int any_bad = __syncthreads_or(bad);
    for (int w = 0; w < SL_THREADS / 32; ++w) mx = max(mx, smax[w]);
    int e = exponent_of_max(mx);
    if (e == SUBNORMAL) e = small_max_exponent<SL_THREADS>(row, c0, c1, slow);
    if (t == 0) {
        if (e != kZeroRowExp) atomicMax(a.e + r, e);
        if (any_bad) set_status(a.status, RTPROJ_ENONFINITE);
    }
}

// Digits of contiguous rows whose exponents are in e already, one CTA per (span, row).
template <int W>
__global__ void __launch_bounds__(SL_THREADS) slice_span_kernel(SliceDev a) {
    const int r = blockIdx.y, c0 = blockIdx.x * SL_SPAN;
    const double* row = reinterpret_cast<const double*>(a.X) + (int64_t)r * a.x_rs;
    int e = a.e[r];
    if (e == kZeroRowExp) e = 0;                           // an all-zero row: exponent 0
    __syncthreads();                                       // every thread has read e[r]
    if (blockIdx.x == 0 && threadIdx.x == 0) a.e[r] = e;
    const int cc = c0 + 8 * (int)threadIdx.x;
    if (cc >= a.ld) return;
    uint2 v[8];
    load_eight(row, cc, a.cols, ((uintptr_t)row & 31) == 0, v);
    const DigitWord<W> k = digit_bias<W>(a.s);
    DigitWord<W> w[8];
    float sg[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { w[i] = digit_word<W>(v[i].x, v[i].y, e, k); sg[i] = sign_of(v[i].y); }
    store_digits<W, 0>(w, sg, a.s, a.d + (int64_t)r * a.ld + cc, a.ps);
}

// Columns of a row-major block X (a.cols x a.rows, leading dimension a.x_rs): row j of the stack
// is column j of X, entry i scaled by 2^{cexp[i]} (cexp optional). A CTA takes JB = 2^lgjb adjacent
// columns (a 32-byte sector of each row of X for JB = 4): JB threads side by side read one row's
// entries, and each thread turns eight rows of one column into digits. FIN: X is a correction dh
// (see Correction). One CTA per column read a sector per entry and used an eighth to a quarter of it.
template <int W, bool FIN>
__global__ void __launch_bounds__(SC_THREADS) slice_columns_kernel(SliceDev a, const int32_t* __restrict__ cexp, int lgjb,
                                                                   Correction f) {
    constexpr int WARPS = SC_THREADS / 32;
    __shared__ int smax[WARPS][8];
    __shared__ double sums[3][WARPS][8];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, jb = 1 << lgjb;
    const int jl = t & (jb - 1), g = t >> lgjb, groups = SC_THREADS >> lgjb;
    const int j = blockIdx.x * jb + jl;
    const bool live = j < a.rows;
    const double* X = reinterpret_cast<const double*>(a.X) + j;
    int mx = kZeroRowExp;
    bool bad = false;
    double sr = 0.0, sh = 0.0, sd = 0.0;
    if (live) {
#pragma unroll 4
        for (int i = g; i < a.cols; i += groups) {
            const uint2 x = entry_bits(X + (int64_t)i * a.x_rs);
            const uint32_t xh = x.y & 0x7FFFFFFFu;
            int e = (int)(xh >> 20) - 1022;
            if (xh < 0x00100000u) {
                const unsigned long long u = ((unsigned long long)xh << 32) | x.x;
                e = u ? (64 - __clzll((long long)u)) - 1074 : kZeroRowExp;
            }
            if (xh >= EXP_MASK) bad = true;
            else if (e != kZeroRowExp) mx = max(mx, e + (cexp ? __ldg(cexp + i) : 0));
            if constexpr (FIN) {
                const int64_t at = (int64_t)i * a.x_rs + j;
                const double dh = __hiloint2double((int)x.y, (int)x.x), h = f.h[at] + dh, r = __ldg(f.r + at);
                f.h[at] = h;
                sr = fma(r, r, sr);
                sh = fma(h, h, sh);
                sd = fma(dh, dh, sd);
            }
        }
    }
    for (int o = jb; o < 32; o <<= 1) {
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if constexpr (FIN) {
            sr += __shfl_xor_sync(0xffffffffu, sr, o);
            sh += __shfl_xor_sync(0xffffffffu, sh, o);
            sd += __shfl_xor_sync(0xffffffffu, sd, o);
        }
    }
    if (lane < jb) {
        smax[warp][lane] = mx;
        if constexpr (FIN) { sums[0][warp][lane] = sr; sums[1][warp][lane] = sh; sums[2][warp][lane] = sd; }
    }
    const int any_bad = __syncthreads_or(bad);
    for (int w = 0; w < WARPS; ++w) mx = max(mx, smax[w][jl]);
    const int e = mx == kZeroRowExp ? 0 : mx;              // an all-zero column: exponent 0
    if (t == 0 && any_bad) set_status(a.status, RTPROJ_ENONFINITE);
    if (t < jb && live) {
        a.e[j] = e;
        if constexpr (FIN) {
            sr = sh = sd = 0.0;
            for (int w = 0; w < WARPS; ++w) { sr += sums[0][w][jl]; sh += sums[1][w][jl]; sd += sums[2][w][jl]; }
            report_residual(sr, f.bnorm[j], *f.normA, f.stats);
            report_change(sh, sd, f.bnorm[j], *f.normA, f.stats);
        }
    }
    if (!live) return;
    const DigitWord<W> k = digit_bias<W>(a.s);
    __nv_bfloat16* drow = a.d + (int64_t)j * a.ld;
    for (int i0 = 8 * g; i0 < a.ld; i0 += 8 * groups) {
        DigitWord<W> w[8];
        float sg[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = i0 + q;
            const uint2 x = i < a.cols ? entry_bits(X + (int64_t)i * a.x_rs) : make_uint2(0u, 0u);
            w[q] = digit_word<W>(x.x, x.y, e - (cexp && i < a.cols ? __ldg(cexp + i) : 0), k);
            sg[q] = sign_of(x.y);
        }
        store_digits<W, 0>(w, sg, a.s, drow + i0, a.ps);
    }
}

// G^* (l x n) as one digit plane: row j, column i holds the digit of G(i, j).
// uniform: d = 2u - 255 (exponent -1, value d / 256); rademacher: d = +-1 (exponent 7).
__global__ void omega_plane_kernel(uint32_t key0, uint32_t key1, int dist, int n, int l, __nv_bfloat16* d,
                                   int64_t ld, int64_t ps) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t blocks_per_row = ld / 16;
    if (gid >= blocks_per_row * l) return;
    const int j = (int)(gid / blocks_per_row);
    const int i0 = (int)(gid % blocks_per_row) * 16;
    alignas(16) __nv_bfloat16 out[16];
    if (dist == RTPROJ_OMEGA_GAUSSIAN) {
        // N = 4096 G = 256 d0 + d1 with d1 in [-128, 127]: two exact digit planes
        // (exponent 3: G = 2^3 (d0 2^-7 + d1 2^-15))
        alignas(16) __nv_bfloat16 lo[16];
#pragma unroll
        for (int qd = 0; qd < 4; ++qd) {
            int N[4];
            gauss_quad((uint32_t)((i0 >> 2) + qd), (uint32_t)j, key0, key1, N);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int v = (i0 + 4 * qd + b < n) ? N[b] : 0;
                const int d0 = (v + 128) >> 8;          // floor((v + 128) / 256)
                out[4 * qd + b] = __int2bfloat16_rn(d0);
                lo[4 * qd + b] = __int2bfloat16_rn(v - 256 * d0);
            }
        }
        uint4* dst1 = reinterpret_cast<uint4*>(d + ps + (int64_t)j * ld + i0);
        dst1[0] = reinterpret_cast<const uint4*>(lo)[0];
        dst1[1] = reinterpret_cast<const uint4*>(lo)[1];
    } else {
        const uint4 w = philox4x32_10(make_uint4((uint32_t)(i0 >> 4), (uint32_t)j, 0u, 0u), key0, key1);
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            const uint32_t u = block_byte(w, b);
            int dv = dist == RTPROJ_OMEGA_RADEMACHER ? (u >= 128u ? 1 : -1) : (2 * (int)u - 255);
            if (i0 + b >= n) dv = 0;
            out[b] = __int2bfloat16_rn(dv);
        }
    }
    uint4* dst = reinterpret_cast<uint4*>(d + (int64_t)j * ld + i0);
    dst[0] = reinterpret_cast<const uint4*>(out)[0];
    dst[1] = reinterpret_cast<const uint4*>(out)[1];
}

// G itself (n x l, float64, row-major): one thread per 16 rows of one column.
__global__ void omega_dense_kernel(uint32_t key0, uint32_t key1, int dist, int n, int l, double* G, int64_t ldg) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t blocks_per_col = (n + 15) / 16;
    if (gid >= blocks_per_col * l) return;
    const int j = (int)(gid % l);
    const int i0 = (int)(gid / l) * 16;
    double v[16];
    if (dist == RTPROJ_OMEGA_GAUSSIAN) {
#pragma unroll
        for (int qd = 0; qd < 4; ++qd) {
            int N[4];
            gauss_quad((uint32_t)((i0 >> 2) + qd), (uint32_t)j, key0, key1, N);
#pragma unroll
            for (int b = 0; b < 4; ++b) v[4 * qd + b] = (double)N[b] * (1.0 / 4096.0);
        }
    } else {
        const uint4 w = philox4x32_10(make_uint4((uint32_t)(i0 >> 4), (uint32_t)j, 0u, 0u), key0, key1);
#pragma unroll
        for (int b = 0; b < 16; ++b) v[b] = (double)omega_from_byte(block_byte(w, b), dist);
    }
#pragma unroll
    for (int b = 0; b < 16; ++b)
        if (i0 + b < n) G[(int64_t)(i0 + b) * ldg + j] = v[b];
}

__global__ void fill_int_kernel(int32_t* e, int n, int v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) e[i] = v;
}

// Both digit layouts of a long-row operand in one pass over it: with the row exponents
// already in e (row_exponents_kernel), CTA (bx, by) takes rows [64 by, 64 by + 64) and
// columns [64 bx, 64 bx + 64) of X, writes their digits to the row-major planes (a.d,
// rows < a.rows) and, through a shared-memory tile per plane, to the transposed planes
// t_d (row c holds column c of X, leading dimension t_ld, rows < t_rows). Tile rows at or
// past a.rows and columns at or past a.cols give zero digits (the padding of both
// layouts). Each thread turns two groups of eight consecutive entries of a row (one group
// per pass, the two in different rows) into digits: one 16-byte store per plane to the
// row-major planes; the transposed planes are written from shared memory as 16-byte
// stores of eight consecutive rows of X.
constexpr int SLD_TILE = 64;
constexpr int SLD_THREADS = 256;
constexpr int SLD_PAD = SLD_TILE + 2;   // bfloat16 per shared row: odd word stride, no bank conflicts on reads

// As store_digits, and each digit to its place in the tile of its plane ([plane][column][row]).
template <int W, int P>
__device__ __forceinline__ void store_digits_dual(const DigitWord<W> (&a)[8], const float (&sg)[8], int s, bool live,
                                                  __nv_bfloat16* d, int64_t ps, __nv_bfloat16* tile) {
    if constexpr (P < (W == 2 ? 7 : 10)) {
        if (P >= s) return;
        uint32_t v[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const uint32_t f0 = digit_float<W, P>(a[2 * h], sg[2 * h]), f1 = digit_float<W, P>(a[2 * h + 1], sg[2 * h + 1]);
            v[h] = __byte_perm(f0, f1, 0x7632);
            tile[(P * SLD_TILE + 2 * h) * SLD_PAD] = __ushort_as_bfloat16((unsigned short)(f0 >> 16));
            tile[(P * SLD_TILE + 2 * h + 1) * SLD_PAD] = __ushort_as_bfloat16((unsigned short)(f1 >> 16));
        }
        if (live) *reinterpret_cast<uint4*>(d + (int64_t)P * ps) = make_uint4(v[0], v[1], v[2], v[3]);
        store_digits_dual<W, P + 1>(a, sg, s, live, d, ps, tile);
    }
}

template <int W>
__global__ void __launch_bounds__(SLD_THREADS) slice_dual_kernel(SliceDev a, __nv_bfloat16* t_d, int64_t t_ld,
                                                                 int64_t t_ps, int t_rows) {
    extern __shared__ __align__(16) unsigned char sld_raw[];
    __nv_bfloat16* tile = reinterpret_cast<__nv_bfloat16*>(sld_raw);   // [plane][column][row], rows padded to SLD_PAD
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int r0 = blockIdx.y * SLD_TILE, c0 = blockIdx.x * SLD_TILE;
    const int g = lane & 7;                                  // group of eight columns
    const DigitWord<W> k = digit_bias<W>(a.s);
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
        const int rr = (warp * 2 + it) * 4 + (lane >> 3);    // tile row, 0 .. 63
        const int r = r0 + rr, cb = c0 + 8 * g;
        const bool live = r < a.rows;
        int e = live ? a.e[r] : 0;
        if (e == kZeroRowExp) e = 0;                         // an all-zero row: exponent 0
        const double* row = reinterpret_cast<const double*>(a.X) + (int64_t)r * a.x_rs;
        uint2 x[8];
        load_eight(row, cb, live ? a.cols : 0, ((uintptr_t)row & 31) == 0, x);
        DigitWord<W> w[8];
        float sg[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) { w[i] = digit_word<W>(x[i].x, x[i].y, e, k); sg[i] = sign_of(x[i].y); }
        store_digits_dual<W, 0>(w, sg, a.s, live, a.d + (int64_t)r * a.ld + cb, a.ps, tile + (8 * g) * SLD_PAD + rr);
    }
    __syncthreads();   // the tile is complete, and every thread has read its rows' exponents
    if (blockIdx.x == 0 && t < SLD_TILE && r0 + t < a.rows && a.e[r0 + t] == kZeroRowExp) a.e[r0 + t] = 0;
    // transposed planes: row c0 + cc, columns r0 + 8 q .. r0 + 8 q + 7 (eight lanes per row)
    for (int v = t; v < a.s * SLD_TILE * (SLD_TILE / 8); v += SLD_THREADS) {
        const int q = v & 7, cc = (v >> 3) & (SLD_TILE - 1), p = v / (SLD_TILE * (SLD_TILE / 8));
        const int c = c0 + cc;
        if (c >= t_rows) continue;
        const uint32_t* src = reinterpret_cast<const uint32_t*>(tile + (p * SLD_TILE + cc) * SLD_PAD + 8 * q);
        *reinterpret_cast<uint4*>(t_d + (int64_t)p * t_ps + (int64_t)c * t_ld + r0 + 8 * q) =
            make_uint4(src[0], src[1], src[2], src[3]);
    }
}

}  // namespace

namespace {

SliceDev slice_dev(const void* X, int64_t x_rs, const SliceStack& st, int* status) {
    SliceDev a;
    a.X = X; a.x_rs = x_rs;
    a.rows = st.rows; a.cols = st.cols; a.s = st.s;
    a.d = st.d; a.ld = st.ld; a.ps = st.plane_stride; a.e = st.e; a.status = status;
    return a;
}

// 16-byte stores need planes and rows of whole multiples of eight entries.
bool planes_ok(const SliceStack& st) {
    return st.s >= 1 && st.s <= 10 && st.ld >= st.cols && st.ld % 64 == 0 && st.plane_stride % 8 == 0 &&
           ((uintptr_t)st.d & 15) == 0;
}

// CTAs per row: one where the rows fill the chip (a cluster's two barriers hold up its CTAs: 4096 x
// 8192 into 7 planes took 377 us with four CTAs a row, 218 with one), else up to eight with at least
// one full pass of the threads each (64 x 65536: 72 us with one, 41 with eight; 7 x 12345: 29 and 13).
int slice_parts(int rows, int64_t ld) {
    int parts = 1;
    while (parts < SL_MAX_PARTS && (int64_t)rows * parts < 2 * sm_count() && ld > (int64_t)parts * 16 * SR_THREADS) parts *= 2;
    return parts;
}

template <typename T>
cudaError_t slice_rows_t(const T* X, int64_t x_rs, const RowExtras& x, const SliceStack& st, int* status, cudaStream_t s) {
    if (st.rows <= 0) return cudaSuccess;
    if (!planes_ok(st) || ((uintptr_t)X & (sizeof(T) - 1))) return cudaErrorInvalidValue;
    const int parts = slice_parts(st.rows, st.ld);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(st.rows * parts));
    cfg.blockDim = dim3(SR_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)parts;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const SliceDev a = slice_dev(X, x_rs, st, status);
    const cudaError_t e = st.s <= 7 ? cudaLaunchKernelEx(&cfg, slice_rows_kernel<2, T>, a, x)
                                    : cudaLaunchKernelEx(&cfg, slice_rows_kernel<3, T>, a, x);
    if (e != cudaSuccess) return e;
    note_launch();
    return cudaGetLastError();
}

cudaError_t slice_columns_t(const double* X, int64_t ldx, const int32_t* cexp, const Correction* f, const SliceStack& st,
                            int* status, cudaStream_t s) {
    if (st.rows <= 0) return cudaSuccess;
    if (!planes_ok(st)) return cudaErrorInvalidValue;
    // columns per CTA: two sectors of each row where that leaves two CTAs per SM, down to one
    // column (latency counts then, not the sectors: 512 x 64 took 10 us by fours, 6 by ones)
    int lgjb = 3;
    while (lgjb > 0 && (st.rows >> lgjb) < 2 * sm_count()) --lgjb;
    const unsigned grid = (unsigned)((st.rows + (1 << lgjb) - 1) >> lgjb);
    const SliceDev a = slice_dev(X, ldx, st, status);
    const Correction none = {};
    if (st.s <= 7) {
        if (f) slice_columns_kernel<2, true><<<grid, SC_THREADS, 0, s>>>(a, cexp, lgjb, *f);
        else slice_columns_kernel<2, false><<<grid, SC_THREADS, 0, s>>>(a, cexp, lgjb, none);
    } else {
        if (f) slice_columns_kernel<3, true><<<grid, SC_THREADS, 0, s>>>(a, cexp, lgjb, *f);
        else slice_columns_kernel<3, false><<<grid, SC_THREADS, 0, s>>>(a, cexp, lgjb, none);
    }
    note_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t slice_rows(const double* X, int64_t x_rs, const SliceStack& st, int* status, cudaStream_t s,
                       unsigned long long* clear) {
    RowExtras x;
    x.clear = clear;
    return slice_rows_t(X, x_rs, x, st, status, s);
}

cudaError_t slice_rhs(const void* B, int dt, int64_t ldb, double* wide, int64_t ldw, double* norms,
                      unsigned long long* clear, const SliceStack& st, int* status, cudaStream_t s) {
    RowExtras x;
    x.norms = norms;
    x.clear = clear;
    if (dt != RTPROJ_F32) return slice_rows_t((const double*)B, ldb, x, st, status, s);
    x.wide = wide;
    x.ldw = ldw;
    return slice_rows_t((const float*)B, ldb, x, st, status, s);
}

cudaError_t slice_columns(const double* X, int64_t ldx, const int32_t* cexp, const SliceStack& st, int* status,
                          cudaStream_t s) {
    return slice_columns_t(X, ldx, cexp, nullptr, st, status, s);
}

cudaError_t slice_correction(const double* dh, int64_t ldx, double* h, const double* r, const double* bnorm,
                             const double* normA, unsigned long long* stats, const int32_t* cexp, const SliceStack& st,
                             int* status, cudaStream_t s) {
    const Correction f = {h, r, bnorm, normA, stats};
    return slice_columns_t(dh, ldx, cexp, &f, st, status, s);
}

cudaError_t row_exponents(const double* X, int64_t x_rs, int rows, int cols, int32_t* e, int* status, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    if (((uintptr_t)X & 7) != 0) return cudaErrorInvalidValue;
    SliceDev a{};
    a.X = X; a.x_rs = x_rs; a.rows = rows; a.cols = cols; a.e = e; a.status = status;
    const dim3 grid((unsigned)((cols + SL_SPAN - 1) / SL_SPAN), (unsigned)rows);
    row_exponents_kernel<<<grid, SL_THREADS, 0, s>>>(a);
    note_launch();
    return cudaGetLastError();
}

cudaError_t slice_rows_given_exp(const double* X, int64_t x_rs, const SliceStack& st, int* status, cudaStream_t s) {
    if (st.rows <= 0) return cudaSuccess;
    if (!planes_ok(st) || ((uintptr_t)X & 7)) return cudaErrorInvalidValue;
    const SliceDev a = slice_dev(X, x_rs, st, status);
    const dim3 grid((unsigned)((st.ld + SL_SPAN - 1) / SL_SPAN), (unsigned)st.rows);
    if (st.s <= 7) slice_span_kernel<2><<<grid, SL_THREADS, 0, s>>>(a);
    else slice_span_kernel<3><<<grid, SL_THREADS, 0, s>>>(a);
    note_launch();
    return cudaGetLastError();
}

cudaError_t slice_rows_dual(const double* X, int64_t x_rs, const SliceStack& st, const SliceStack& tst, int* status,
                            cudaStream_t s) {
    if (st.rows <= 0) return cudaSuccess;
    if (!planes_ok(st) || !planes_ok(tst) || ((uintptr_t)X & 7) || tst.s != st.s || tst.rows != st.cols ||
        tst.cols != st.rows || tst.ld % SLD_TILE || st.ld % SLD_TILE)
        return cudaErrorInvalidValue;
    const SliceDev a = slice_dev(X, x_rs, st, status);
    cudaError_t e = fill_int(st.e, st.rows, kZeroRowExp, s);
    if (e != cudaSuccess) return e;
    e = row_exponents(X, x_rs, st.rows, st.cols, st.e, status, s);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(st.ld / SLD_TILE), (unsigned)(tst.ld / SLD_TILE));
    const size_t smem = (size_t)st.s * SLD_TILE * SLD_PAD * sizeof(__nv_bfloat16);
    auto launch = [&](auto kern, int most_planes) {
        allow_dynamic_shared((const void*)kern, (size_t)most_planes * SLD_TILE * SLD_PAD * sizeof(__nv_bfloat16));
        kern<<<grid, SLD_THREADS, smem, s>>>(a, tst.d, tst.ld, tst.plane_stride, tst.rows);
    };
    if (st.s <= 7) launch(slice_dual_kernel<2>, 7);
    else launch(slice_dual_kernel<3>, 10);
    note_launch();
    return cudaGetLastError();
}

cudaError_t omega_plane(uint64_t seed, int dist, int n, int l, const SliceStack& st, cudaStream_t s) {
    if (st.ld % 16 || st.ld < n || st.s < omega_planes(dist)) return cudaErrorInvalidValue;
    const int64_t total = (st.ld / 16) * (int64_t)l;
    omega_plane_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>((uint32_t)(seed & 0xFFFFFFFFull),
                                                                       (uint32_t)(seed >> 32), dist, n, l, st.d, st.ld,
                                                                       st.plane_stride);
    note_launch();
    const int e = dist == RTPROJ_OMEGA_RADEMACHER ? 7 : dist == RTPROJ_OMEGA_GAUSSIAN ? 3 : -1;
    fill_int_kernel<<<(l + 255) / 256, 256, 0, s>>>(st.e, l, e);
    note_launch();
    return cudaGetLastError();
}

cudaError_t omega_dense(uint64_t seed, int dist, int n, int l, double* G, int64_t ldg, cudaStream_t s) {
    const int64_t total = (int64_t)((n + 15) / 16) * l;
    if (total <= 0) return cudaSuccess;
    omega_dense_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>((uint32_t)(seed & 0xFFFFFFFFull),
                                                                       (uint32_t)(seed >> 32), dist, n, l, G, ldg);
    note_launch();
    return cudaGetLastError();
}

cudaError_t fill_int(int32_t* e, int n, int v, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    fill_int_kernel<<<(n + 255) / 256, 256, 0, s>>>(e, n, v);
    note_launch();
    return cudaGetLastError();
}

}  // namespace rtp
