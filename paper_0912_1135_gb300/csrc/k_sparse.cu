// A sparse A, optionally plus a low-rank term: A = S + U V with S m x n in compressed
// sparse row form, U m x r and V r x n dense (r small). This is the setting of the paper's
// Section 5: the sparse test matrix of Eq. 21 (five nonzeros per column) and its sum with
// a rank-10 term (Eq. 22), applied as operators at O(nnz + r(m + n)) per vector.
//
//   S_k = A G                 one CTA per (row, 64 columns of G); G generated a panel at a time
//                             (the same entries as the dense forms), Eq. 12
//   X column by column as in steps a-e that follow Eq. 15, all m columns at once:
//     D = A^* P^-             (n x m) a thread per column of P^-, a gather over the nonzeros of A's
//                             columns; the low-rank part, and V D after it, by limbs
//     E = A D                 (m x m) one CTA per row of A
//     X = R^{-*} Pi E         one float64 product with the triangular R^{-*}
//   apply (the seven steps) and its refinement (Remark 4.3) with every product with A or
//   A^* summed from exact products in 128-bit integers and rounded once: c = A b,
//   s = b - A^* h, r = A s, s <- s - A^* dh. The sparse part of each of these is exact to
//   about 2^-105 of its largest term, so the refinement converges to the projection of the
//   stored matrix; the low-rank part's inner products (V b, U^* h) are float64.
#include "rtproj_internal.cuh"
#include "i128.cuh"

#include <algorithm>
#include <climits>
#include <cstring>
#include <vector>

using namespace rtp;

namespace {

constexpr size_t kAlign = 256;
size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

#define SP_CHECK(expr)                                  \
    do {                                                \
        if ((expr) != cudaSuccess) return RTPROJ_ECUDA; \
    } while (0)

// Rows are cut into chunks of at most SP_CHUNK nonzeros (a table built at create), so that
// a few long rows still spread over many warps, and no sum exceeds the 128 bits' capacity.
constexpr int SP_CHUNK = 2048;
static_assert(SP_CHUNK <= I128_MAX_TERMS, "a chunk's sum must fit 128 bits");

// ---------------------------------------------------------------------------------
// The column-compressed copy: counting sort by column, then each column's entries put in
// (row, value) order, so that every sum over a column runs in one fixed order whatever the
// order in which the scatter's atomics landed.
// ---------------------------------------------------------------------------------
__global__ void count_cols_kernel(const int32_t* __restrict__ col, int64_t nnz, int n, int64_t* cnt, int* status) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        const int c = col[p];
        if (c < 0 || c >= n) { set_status(status, RTPROJ_EINVAL); continue; }
        atomicAdd((unsigned long long*)&cnt[c], 1ull);
    }
}

// Exclusive scan of cnt[0..n) into ptr[0..n] in blocks of SCAN_T: per-block totals, one CTA
// scanning those totals, then each block's scan plus its offset.
constexpr int SCAN_T = 1024;

__device__ __forceinline__ int64_t block_inclusive_scan(int64_t v, int64_t* buf) {
    buf[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < SCAN_T; o <<= 1) {
        const int64_t x = threadIdx.x >= (unsigned)o ? buf[threadIdx.x - o] : 0;
        __syncthreads();
        buf[threadIdx.x] += x;
        __syncthreads();
    }
    return buf[threadIdx.x];
}

// *longest (zeroed before) = the largest count.
__global__ void block_totals_kernel(const int64_t* cnt, int n, int64_t* tot, int* longest) {
    __shared__ int64_t buf[SCAN_T];
    __shared__ int most;
    const int64_t i = (int64_t)blockIdx.x * SCAN_T + threadIdx.x, v = i < n ? cnt[i] : 0;
    if (threadIdx.x == 0) most = 0;
    const int64_t incl = block_inclusive_scan(v, buf);        // and a barrier
    const unsigned mine = __reduce_max_sync(0xffffffffu, (unsigned)min(v, (int64_t)INT_MAX));
    if ((threadIdx.x & 31) == 0) atomicMax(&most, (int)mine);
    __syncthreads();
    if (threadIdx.x == SCAN_T - 1) {
        tot[blockIdx.x] = incl;
        atomicMax(longest, most);
    }
}

// fill[0 .. nfill) = kZeroRowExp on the way (row_tops_kernel's maxima start from it).
__global__ void scan_totals_kernel(int64_t* tot, int nb, int32_t* fill, int nfill) {
    __shared__ int64_t buf[SCAN_T];
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    for (int i = threadIdx.x; i < nfill; i += SCAN_T) fill[i] = kZeroRowExp;
    __syncthreads();
    for (int b0 = 0; b0 < nb; b0 += SCAN_T) {
        const int i = b0 + threadIdx.x;
        const int64_t v = i < nb ? tot[i] : 0;
        const int64_t incl = block_inclusive_scan(v, buf);
        const int64_t base = carry;
        __syncthreads();
        if (i < nb) tot[i] = base + incl - v;
        if (threadIdx.x == SCAN_T - 1) carry = base + incl;
        __syncthreads();
    }
}

__global__ void block_scan_kernel(const int64_t* cnt, int n, const int64_t* tot, int64_t* ptr) {
    __shared__ int64_t buf[SCAN_T];
    const int64_t i = (int64_t)blockIdx.x * SCAN_T + threadIdx.x;
    const int64_t v = i < n ? cnt[i] : 0;
    const int64_t incl = block_inclusive_scan(v, buf);
    if (i < n) ptr[i] = tot[blockIdx.x] + incl - v;
    if (i == n - 1) ptr[n] = tot[blockIdx.x] + incl;
}

__global__ void scatter_csc_kernel(const int64_t* __restrict__ rptr, const int32_t* __restrict__ col,
                                   const double* __restrict__ val, int m, int n, const int64_t* __restrict__ cptr,
                                   int64_t* cursor, int32_t* __restrict__ crow, double* __restrict__ cval) {
    for (int i = blockIdx.x; i < m; i += gridDim.x) {
        for (int64_t p = rptr[i] + threadIdx.x; p < rptr[i + 1]; p += blockDim.x) {
            const int c = col[p];
            if (c < 0 || c >= n) continue;   // counted nowhere; create fails on RTPROJ_EINVAL
            const int64_t at = cptr[c] + (int64_t)atomicAdd((unsigned long long*)&cursor[c], 1ull);
            crow[at] = i;
            cval[at] = val[p];
        }
    }
}

__device__ __forceinline__ bool entry_before(int32_t ra, double va, int32_t rb, double vb) {
    if (ra != rb) return ra < rb;
    return __double_as_longlong(va) < __double_as_longlong(vb);   // duplicates: a fixed order
}

__global__ void sort_columns_kernel(const int64_t* __restrict__ cptr, int n, int32_t* crow, double* cval) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        const int64_t b = cptr[c], e = cptr[c + 1];
        for (int64_t p = b + 1; p < e; ++p) {      // insertion sort
            const int32_t r = crow[p];
            const double v = cval[p];
            int64_t q = p - 1;
            while (q >= b && entry_before(r, v, crow[q], cval[q])) {
                crow[q + 1] = crow[q];
                cval[q + 1] = cval[q];
                --q;
            }
            crow[q + 1] = r;
            cval[q + 1] = v;
        }
    }
}

// ---------------------------------------------------------------------------------
// ||A||_F^2 = ||S||_F^2 + 2 <S, U V> + trace((U^* U)(V V^*)), each part summed in two
// deterministic levels (per-CTA partials, then one thread).
// ---------------------------------------------------------------------------------
__device__ __forceinline__ double block_sum(double s, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    return t;
}

__global__ void sumsq_vals_kernel(const double* __restrict__ val, int64_t nnz, double* part) {
    __shared__ double red[8];
    double s = 0.0;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x)
        s = fma(val[p], val[p], s);
    const double t = block_sum(s, red);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// part[b] = sum over the rows i = b, b + gridDim.x, ... of sum_p val (U V)(i, col)
__global__ void cross_term_kernel(const int64_t* __restrict__ rptr, const int32_t* __restrict__ col,
                                  const double* __restrict__ val, int m, int n, int r, const double* __restrict__ U,
                                  const double* __restrict__ V, double* part) {
    __shared__ double red[8];
    double s = 0.0;
    for (int i = blockIdx.x; i < m; i += gridDim.x)
        for (int64_t p = rptr[i] + threadIdx.x; p < rptr[i + 1]; p += blockDim.x) {
            const int c = col[p];
            if (c < 0 || c >= n) continue;       // create fails on RTPROJ_EINVAL
            double uv = 0.0;
            for (int q = 0; q < r; ++q) uv = fma(U[(int64_t)i * r + q], V[(int64_t)q * n + c], uv);
            s = fma(val[p], uv, s);
        }
    const double t = block_sum(s, red);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__device__ __forceinline__ void ldg_words(const double* p, uint32_t& lo, uint32_t& hi) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    lo = u.x;
    hi = u.y;
}

// ---------------------------------------------------------------------------------
// S = A G in panels of SK_COLS columns of G. A panel's entries are generated once, as the integers
// behind them (N = 4096 G, 256 G or G; 16 bits; the counter-based Philox words that the dense
// forms use: entries 16q .. 16q+15 of column j from the block at (q, j, 0, 0), Gaussian entries
// 4q .. 4q+3 from the block at (q, j, 1, 0)), into n x SK_COLS words that stay in L2, and every
// nonzero of a row reads SK_COLS consecutive ones. The products run on the integer pipes: a row's
// values are 61-bit multiples of 2^-61 of a power of two above its largest, in two limbs, and
// sums of limb times N are exact in 64 bits; each entry of S is rounded once. Its error is below
// nnz 2^-61 of the largest value times |N|, against about 2^-53 of every partial sum in float64.
// (Generated per nonzero and multiplied in float64 - 192 FP64 cycles a warp and nonzero with the
// conversions - the sketch at 1000 x 300,000, l = 1004, took 8.7 ms and V G of a rank-10 term 7.3;
// now 2.0 with the panels' generation, and 2.3.)
// ---------------------------------------------------------------------------------
constexpr int SK_COLS = 64;
constexpr int SK_T = 256;
constexpr int SK_WARPS = SK_T / 32;
constexpr int SK_LIMB = 30;                      // bits of the lower limb
constexpr int SK_FLUSH = 1 << 16;                // products whose lower-limb sums fit 62 bits

// A launch takes as many panels as stay in L2 together (their storage allowing), one on grid.y (grid.z
// for V G): at 1000 x 5000, l = 1004, the 16 panels one after the other took 241 us, launches mostly.
constexpr int64_t SK_L2_BYTES = (int64_t)32 << 20;
// G is generated in place for rows of at most SK_GEN_ROW nonzeros and at most SK_GEN nonzeros times
// panels: 64 x 512, two panels, 16 a row 41 us, by panels 46; 500 x 2000, eight panels, 2 a row 55 and 56,
// 16 a row 68 and 62; 2000 x 20,000, 32 panels, 16 a row 487 and 375.
constexpr int SK_GEN_ROW = 16, SK_GEN = 1 << 13;

// Panel entries (c, jj), jj < SK_COLS: N of G(c, j0 + jj), zero past column l. One warp per 4
// (Gaussian) or 16 rows, two columns a lane.
__global__ void __launch_bounds__(SK_T) omega_panel_kernel(int n, int l, int j0, int dist, uint32_t k0, uint32_t k1,
                                                           int16_t* __restrict__ P) {
    const int lane = threadIdx.x & 31;
    const int j = j0 + blockIdx.y * SK_COLS + 2 * lane;
    P += (int64_t)blockIdx.y * n * SK_COLS;
    const int per = dist == RTPROJ_OMEGA_GAUSSIAN ? 4 : 16;
    const int64_t groups = ((int64_t)n + per - 1) / per;
    for (int64_t q = (int64_t)blockIdx.x * SK_WARPS + (threadIdx.x >> 5); q < groups; q += (int64_t)gridDim.x * SK_WARPS) {
        if (dist == RTPROJ_OMEGA_GAUSSIAN) {
            int a[4], b[4];
            gauss_quad((uint32_t)q, (uint32_t)j, k0, k1, a);
            gauss_quad((uint32_t)q, (uint32_t)(j + 1), k0, k1, b);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t c = 4 * q + u;
                if (c < n)
                    *reinterpret_cast<short2*>(P + c * SK_COLS + 2 * lane) =
                        make_short2((short)(j < l ? a[u] : 0), (short)(j + 1 < l ? b[u] : 0));
            }
        } else {
            const uint4 wa = philox4x32_10(make_uint4((uint32_t)q, (uint32_t)j, 0u, 0u), k0, k1);
            const uint4 wb = philox4x32_10(make_uint4((uint32_t)q, (uint32_t)(j + 1), 0u, 0u), k0, k1);
            const float sc = dist == RTPROJ_OMEGA_RADEMACHER ? 1.0f : 256.0f;
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const int64_t c = 16 * q + u;
                const int a = (int)(omega_from_byte(block_byte(wa, u), dist) * sc);
                const int b = (int)(omega_from_byte(block_byte(wb, u), dist) * sc);
                if (c < n)
                    *reinterpret_cast<short2*>(P + c * SK_COLS + 2 * lane) =
                        make_short2((short)(j < l ? a : 0), (short)(j + 1 < l ? b : 0));
            }
        }
    }
}
// G = N 2^omega_exp
int omega_exp(int dist) { return dist == RTPROJ_OMEGA_GAUSSIAN ? -12 : dist == RTPROJ_OMEGA_RADEMACHER ? 0 : -8; }

// The exponents of the largest values in the rows of S and of V, and the check that they and U are
// finite: a CTA per chunk of S, then per TOPS_SPAN entries of a row of V, then of U. top[i]
// (pre-filled with kZeroRowExp, and left so for an empty or zero row) is the frexp exponent of row i's
// largest magnitude: S's m rows, then V's r. (A CTA a row took 165 us of 966 at create for 2 x 500,000.)
constexpr int TOPS_SPAN = 2048;
static_assert(TOPS_SPAN <= 8 * 256 && SP_CHUNK <= 8 * 256, "a CTA's values are loaded at once");
__global__ void __launch_bounds__(256) row_tops_kernel(const int32_t* __restrict__ crow_of, const int64_t* __restrict__ cbeg,
                                                       const int64_t* __restrict__ rptr, const double* __restrict__ val,
                                                       int nchunks, int m, int n, int r, const double* __restrict__ U,
                                                       const double* __restrict__ V, int32_t* __restrict__ top, int* status) {
    __shared__ uint32_t buf[8][2];
    const int spans = (n + TOPS_SPAN - 1) / TOPS_SPAN;
    const int64_t v = (int64_t)blockIdx.x - nchunks, u = v - (int64_t)spans * r;
    const double* x = val;
    int64_t b, e;
    int row = -1;
    if (v < 0) {
        row = crow_of[blockIdx.x];
        b = cbeg[blockIdx.x];
        e = min(b + (int64_t)SP_CHUNK, rptr[row + 1]);
    } else if (u < 0) {
        const int q = (int)(v / spans);
        row = m + q;
        x = V;
        b = (int64_t)q * n + (v % spans) * TOPS_SPAN;
        e = min(b + (int64_t)TOPS_SPAN, (int64_t)(q + 1) * n);
    } else {
        x = U;
        b = u * TOPS_SPAN;
        e = min(b + (int64_t)TOPS_SPAN, (int64_t)m * r);
    }
    uint32_t mxh = 0u, orl = 0u, lo[8], hi[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int64_t p = b + u * 256 + threadIdx.x;
        lo[u] = hi[u] = 0u;
        if (p < e) ldg_words(x + p, lo[u], hi[u]);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        mxh = max(mxh, hi[u] & 0x7FFFFFFFu);
        orl |= lo[u];
    }
    mxh = __reduce_max_sync(0xffffffffu, mxh);
    orl = __reduce_or_sync(0xffffffffu, orl);
    if ((threadIdx.x & 31) == 0) {
        buf[threadIdx.x >> 5][0] = mxh;
        buf[threadIdx.x >> 5][1] = orl;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < 8; ++w) {
        mxh = max(mxh, buf[w][0]);
        orl |= buf[w][1];
    }
    if (mxh >= 0x7FF00000u) set_status(status, RTPROJ_ENONFINITE);
    if (row < 0 || (mxh | orl) == 0u) return;
    atomicMax(top + row, mxh >> 20 ? (int)(mxh >> 20) - 1022
                         : mxh     ? 32 - __clz((int)mxh) + 32 - 1074
                                   : 32 - __clz((int)orl) - 1074);
}

// Whether V's row q is flat: its largest entry, rounded up to a power of two, at most 2^LR_FLAT times
// its root mean square (g: its squared norm).
constexpr int LR_FLAT = 4;
__device__ __forceinline__ bool row_is_flat(int top, double g, int n) {
    if (top == kZeroRowExp) return true;
    return isfinite(g) && g > 1e-280 && ldexp((double)n, 2 * (top - LR_FLAT)) <= g;
}

// ||A||_F from its parts; V's rows: *flat, and the exponent of a row of zeros made 0.
__global__ void frobenius_total_kernel(const double* part_s, int np, const double* part_x, int nx, const double* GU,
                                       const double* GV, int r, int n, int32_t* lr_top, int* flat, double* out) {
    bool ok = true;
    for (int q = threadIdx.x; q < r; q += blockDim.x) {
        ok &= row_is_flat(lr_top[q], GV[q * r + q], n);
        if (lr_top[q] == kZeroRowExp) lr_top[q] = 0;
    }
    ok = __all_sync(0xffffffffu, ok);
    if (threadIdx.x != 0) return;
    *flat = ok ? 1 : 0;
    double s = 0.0, x = 0.0, t = 0.0;
    for (int i = 0; i < np; ++i) s += part_s[i];
    for (int i = 0; i < nx; ++i) x += part_x[i];
    for (int a = 0; a < r; ++a)
        for (int b = 0; b < r; ++b) t = fma(GU[a * r + b], GV[b * r + a], t);
    *out = sqrt(fmax(s + 2.0 * x + t, 0.0));
}

// x 2^(bits - top) rounded to an integer (|x| < 2^top, bits <= 61), in a signed upper and a
// LIMB-bit lower limb.
template <int LIMB = SK_LIMB>
__device__ __forceinline__ int2 to_limbs(double x, int top, int bits) {
    const i128op o = i128_decode((uint32_t)__double2loint(x), (uint32_t)__double2hiint(x));
    long long v = (long long)(((unsigned long long)o.hi << 32) | o.lo);
    const int sh = o.e - top + bits;               // the significand's last place in units
    if (sh >= 0) v <<= sh;                         // at most bits - 53
    else if (sh > -62) v = (v + (1ll << (-sh - 1))) >> -sh;
    else v = 0;
    if (o.neg) v = -v;
    return make_int2((int)(v >> LIMB), (int)(v & ((1ll << LIMB) - 1)));
}
// acc += a N for a signed 32-bit a
__device__ __forceinline__ void mad_limb(long long& acc, int a, int N) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(N));
}
// (hi 2^SK_LIMB + lo) 2^e rounded once
__device__ __forceinline__ double limbs_to_double(__int128 hi, __int128 lo, int e) {
    const __int128 v = (hi << SK_LIMB) + lo;
    return u128_to_double((unsigned long long)(v >> 64), (unsigned long long)v, e);
}
// bits of a value in a sum of `count` products with N (16 bits): the upper limb's sum stays
// below 2^62
__host__ __device__ __forceinline__ int limb_bits(int64_t count) {
    int b = 61;
    while (b > 40 && count > ((int64_t)1 << (16 + 61 - b))) --b;
    return b;
}

// Rows of several chunks: which CTA sums what, and where the sums go.
struct SharedRows {
    const int32_t* chunk_row; const int64_t* chunk_beg; const int32_t* row_chunk;
    int group;               // chunks a CTA
    int slots;
    longlong2* part;         // [panel][slot][SK_COLS]
};
// The place of a row's share s among the partial sums (`first`: the row's first chunk): rows do not overlap.
__device__ __forceinline__ int sketch_slot(const SharedRows& a, int i, int first, int s) { return first / a.group + i + s; }

// Entries (c, j) and (c, j + 1) of G as integers, one in each half.
__device__ __forceinline__ int omega_pair(int c, int j, int l, int dist, uint32_t k0, uint32_t k1) {
    int a, b;
    if (dist == RTPROJ_OMEGA_GAUSSIAN) {           // as gauss_quad, the pair that holds row c only
        const uint4 u = philox4x32_10(make_uint4((uint32_t)c >> 2, (uint32_t)j, 1u, 0u), k0, k1);
        const uint4 v = philox4x32_10(make_uint4((uint32_t)c >> 2, (uint32_t)(j + 1), 1u, 0u), k0, k1);
        int a1, b1;
        gauss_pair(c & 2 ? u.z : u.x, c & 2 ? u.w : u.y, a, a1);
        gauss_pair(c & 2 ? v.z : v.x, c & 2 ? v.w : v.y, b, b1);
        if (c & 1) {
            a = a1;
            b = b1;
        }
    } else {
        const float sc = dist == RTPROJ_OMEGA_RADEMACHER ? 1.0f : 256.0f;
        const uint4 u = philox4x32_10(make_uint4((uint32_t)c >> 4, (uint32_t)j, 0u, 0u), k0, k1);
        const uint4 v = philox4x32_10(make_uint4((uint32_t)c >> 4, (uint32_t)(j + 1), 0u, 0u), k0, k1);
        a = (int)(omega_from_byte(block_byte(u, c & 15), dist) * sc);
        b = (int)(omega_from_byte(block_byte(v, c & 15), dist) * sc);
    }
    return (j < l ? a & 0xFFFF : 0) | (j + 1 < l ? b << 16 : 0);
}

// S(i, j0 .. j0 + SK_COLS - 1): a CTA takes `group` chunks of a row, its warps the nonzeros in turn, two
// columns a lane. A row of more chunks is summed by several CTAs and added by sketch_rows_kernel (one
// CTA a row, panel after panel, took 11.4 ms for 888 x 250,000 with a tenth of the nonzeros in one row;
// now 1.4). GEN: G's entries are generated where they are used, which for rows of a few nonzeros takes
// less than the panels' launch.
template <bool GEN, bool SHARED>
__global__ void __launch_bounds__(SK_T) sparse_sketch_kernel(const int64_t* __restrict__ rptr, const int32_t* __restrict__ col,
                                                             const double* __restrict__ val, const int32_t* __restrict__ top,
                                                             const int16_t* __restrict__ P, int n, int l, int j0, int gexp, int r,
                                                             const double* __restrict__ U, const double* __restrict__ VG,
                                                             int64_t ldvg, double* S, int64_t lds, int dist, uint32_t k0,
                                                             uint32_t k1, SharedRows a) {
    __shared__ int4 ent[SK_T];                     // upper limb, lower limb, column
    __shared__ unsigned long long sum[2][SK_COLS];
    const int i = SHARED ? a.chunk_row[blockIdx.x] : (int)blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int64_t b = rptr[i], e = rptr[i + 1];
    const int tp = max(top[i], -1073), bits = limb_bits(e - b);   // -1073: the smallest value's, or an empty row
    if (SHARED) {
        if (((int)blockIdx.x - a.row_chunk[i]) % a.group) return;
        b = a.chunk_beg[blockIdx.x];
        e = min(b + (int64_t)a.group * SP_CHUNK, e);
    }
    if (t < SK_COLS) sum[0][t] = sum[1][t] = 0ull;
    long long h0 = 0, h1 = 0, l0 = 0, l1 = 0;
    int held = 0;
    for (int64_t p0 = b; p0 < e; p0 += SK_T) {
        __syncthreads();
        if (p0 + t < e) {
            const int2 v = to_limbs(val[p0 + t], tp, bits);
            ent[t] = make_int4(v.x, v.y, col[p0 + t] + (GEN ? 0 : (int)blockIdx.y * n), 0);   // the panel's row
        } else {
            ent[t] = make_int4(0, 0, 0, 0);
        }
        __syncthreads();
        const int cnt = (int)min((int64_t)SK_T, e - p0);
        for (int q = warp; q < cnt; q += 4 * SK_WARPS) {
            int4 v[4];
            int N[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                v[u] = ent[(q + u * SK_WARPS) & (SK_T - 1)];
                if constexpr (GEN) N[u] = q + u * SK_WARPS < cnt ? omega_pair(v[u].z, j0 + (int)blockIdx.y * SK_COLS + 2 * lane,
                                                                              l, dist, k0, k1) : 0;
                else N[u] = __ldg(reinterpret_cast<const int*>(P + (int64_t)v[u].z * SK_COLS) + lane);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (q + u * SK_WARPS >= SK_T) break;
                const int n0 = (int)(short)(N[u] & 0xFFFF), n1 = N[u] >> 16;
                mad_limb(h0, v[u].x, n0);
                mad_limb(l0, v[u].y, n0);
                mad_limb(h1, v[u].x, n1);
                mad_limb(l1, v[u].y, n1);
            }
        }
        if ((held += SK_T) >= SK_FLUSH) {          // the lower sums' upper part moves over
            h0 += l0 >> SK_LIMB;
            l0 &= (1ll << SK_LIMB) - 1;
            h1 += l1 >> SK_LIMB;
            l1 &= (1ll << SK_LIMB) - 1;
            held = 0;
        }
    }
    h0 += l0 >> SK_LIMB;
    l0 &= (1ll << SK_LIMB) - 1;
    h1 += l1 >> SK_LIMB;
    l1 &= (1ll << SK_LIMB) - 1;
    __syncthreads();                               // integer sums: the order does not matter
    atomicAdd(&sum[0][2 * lane], (unsigned long long)h0);
    atomicAdd(&sum[1][2 * lane], (unsigned long long)l0);
    atomicAdd(&sum[0][2 * lane + 1], (unsigned long long)h1);
    atomicAdd(&sum[1][2 * lane + 1], (unsigned long long)l1);
    __syncthreads();
    const int j = j0 + (int)blockIdx.y * SK_COLS + t;
    if (t >= SK_COLS || j >= l) return;
    if (SHARED) {
        const int first = a.row_chunk[i];
        if (a.row_chunk[i + 1] - first > a.group) {
            const int slot = sketch_slot(a, i, first, ((int)blockIdx.x - first) / a.group);
            a.part[((int64_t)blockIdx.y * a.slots + slot) * SK_COLS + t] =
                make_longlong2((long long)sum[0][t], (long long)sum[1][t]);
            return;
        }
    }
    double s = limbs_to_double((long long)sum[0][t], (long long)sum[1][t], tp - bits + gexp);
    for (int q = 0; q < r; ++q) s = fma(U[(int64_t)i * r + q], VG[(int64_t)q * ldvg + j], s);
    S[(int64_t)i * lds + j] = s;
}

// The rows that several CTAs have summed.
__global__ void __launch_bounds__(SK_COLS) sketch_rows_kernel(const int64_t* __restrict__ rptr, const int32_t* __restrict__ top,
                                                              int l, int j0, int gexp, int r, const double* __restrict__ U,
                                                              const double* __restrict__ VG, int64_t ldvg, double* S, int64_t lds,
                                                              SharedRows a) {
    const int i = blockIdx.x, j = j0 + (int)blockIdx.y * SK_COLS + (int)threadIdx.x;
    const int first = a.row_chunk[i], chunks = a.row_chunk[i + 1] - first;
    if (chunks <= a.group || j >= l) return;
    const longlong2* p = a.part + ((int64_t)blockIdx.y * a.slots + sketch_slot(a, i, first, 0)) * SK_COLS + threadIdx.x;
    long long h = 0, lo = 0;                       // h: within 2^62 over the whole row (limb_bits)
    for (int s = 0; s < (chunks + a.group - 1) / a.group; ++s) {
        h += p[(int64_t)s * SK_COLS].x;
        lo += p[(int64_t)s * SK_COLS].y;
    }
    double s = limbs_to_double(h, lo, max(top[i], -1073) - limb_bits(rptr[i + 1] - rptr[i]) + gexp);
    for (int q = 0; q < r; ++q) s = fma(U[(int64_t)i * r + q], VG[(int64_t)q * ldvg + j], s);
    S[(int64_t)i * lds + j] = s;
}

// Partial sums of (V G)(q, j0 ..) over chunk blockIdx.x of the rows of G: rows q0 .. q0 + VG_ROWS - 1
// of V (blockIdx.y; as many as cover r in equal parts of at most 12), the warps take G's rows in
// turn, two columns a lane.
constexpr int VG_KC = 128;
template <int VG_ROWS>
__global__ void __launch_bounds__(SK_T) lowrank_panel_kernel(const double* __restrict__ V, const int32_t* __restrict__ top,
                                                             int r, int n, int chunk, int bits, const int16_t* __restrict__ P,
                                                             longlong2* __restrict__ part) {
    __shared__ int2 vs[VG_KC][VG_ROWS];
    __shared__ unsigned long long sum[2][VG_ROWS][SK_COLS];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, q0 = blockIdx.y * VG_ROWS;
    P += (int64_t)blockIdx.z * n * SK_COLS;
    part += (int64_t)blockIdx.z * gridDim.x * r * SK_COLS;
    const int64_t kb = (int64_t)blockIdx.x * chunk, ke = min((int64_t)n, kb + chunk);
    for (int e = t; e < 2 * VG_ROWS * SK_COLS; e += SK_T) (&sum[0][0][0])[e] = 0ull;
    long long h[VG_ROWS][2], lo[VG_ROWS][2];
#pragma unroll
    for (int q = 0; q < VG_ROWS; ++q) h[q][0] = h[q][1] = lo[q][0] = lo[q][1] = 0;
    int held = 0;
    for (int64_t k0 = kb; k0 < ke; k0 += VG_KC) {
        __syncthreads();
        for (int e = t; e < VG_KC * VG_ROWS; e += SK_T) {
            const int q = e / VG_KC, k = e % VG_KC;
            int2 v = make_int2(0, 0);
            if (q0 + q < r && k0 + k < ke) v = to_limbs(V[(int64_t)(q0 + q) * n + k0 + k], top[q0 + q], bits);
            vs[k][q] = v;
        }
        __syncthreads();
        const int cnt = (int)min((int64_t)VG_KC, ke - k0);
        for (int k = warp; k < cnt; k += SK_WARPS) {
            const int N = __ldg(reinterpret_cast<const int*>(P + (k0 + k) * SK_COLS) + lane);
            const int n0 = (int)(short)(N & 0xFFFF), n1 = N >> 16;
#pragma unroll
            for (int q = 0; q < VG_ROWS; ++q) {
                const int2 v = vs[k][q];
                mad_limb(h[q][0], v.x, n0);
                mad_limb(lo[q][0], v.y, n0);
                mad_limb(h[q][1], v.x, n1);
                mad_limb(lo[q][1], v.y, n1);
            }
        }
        if ((held += VG_KC) >= SK_FLUSH) {
#pragma unroll
            for (int q = 0; q < VG_ROWS; ++q)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    h[q][u] += lo[q][u] >> SK_LIMB;
                    lo[q][u] &= (1ll << SK_LIMB) - 1;
                }
            held = 0;
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < VG_ROWS; ++q)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            h[q][u] += lo[q][u] >> SK_LIMB;
            lo[q][u] &= (1ll << SK_LIMB) - 1;
            atomicAdd(&sum[0][q][2 * lane + u], (unsigned long long)h[q][u]);
            atomicAdd(&sum[1][q][2 * lane + u], (unsigned long long)lo[q][u]);
        }
    __syncthreads();
    for (int e = t; e < VG_ROWS * SK_COLS; e += SK_T) {
        const int q = e / SK_COLS, j = e % SK_COLS;
        if (q0 + q < r)
            part[((int64_t)blockIdx.x * r + q0 + q) * SK_COLS + j] =
                make_longlong2((long long)sum[0][q][j], (long long)sum[1][q][j]);
    }
}
// (V G)(q, j0 + j) from the chunks' partial sums: one warp per entry.
__global__ void lowrank_panel_sum_kernel(const longlong2* __restrict__ part, const int32_t* __restrict__ top, int chunks, int r,
                                         int l, int j0, int bits, int gexp, double* __restrict__ VG, int64_t ldvg) {
    const int idx = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    const int q = idx / SK_COLS, j = idx % SK_COLS;
    j0 += blockIdx.y * SK_COLS;
    part += (int64_t)blockIdx.y * chunks * r * SK_COLS;
    if (q >= r || j0 + j >= l) return;
    // the upper limbs' sums are below 2^62 a chunk: kept as a high and a low half
    long long hh = 0, hl = 0, lo = 0;
    for (int z = lane; z < chunks; z += 32) {
        const longlong2 v = part[((int64_t)z * r + q) * SK_COLS + j];
        hh += v.x >> 32;
        hl += v.x & 0xFFFFFFFFll;
        lo += v.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        hh += __shfl_xor_sync(0xffffffffu, hh, o);
        hl += __shfl_xor_sync(0xffffffffu, hl, o);
        lo += __shfl_xor_sync(0xffffffffu, lo, o);
    }
    if (lane != 0) return;
    const __int128 h = ((__int128)hh << 32) + hl;
    VG[(int64_t)q * ldvg + j0 + j] = limbs_to_double(h, lo, top[q] - bits + gexp);
}

// ---------------------------------------------------------------------------------
// The Gram matrix, in the paper's order (steps a-e that follow Eq. 15, for all k at once).
// ---------------------------------------------------------------------------------
// P^- = Pi^* R^{-1} (Eq. 15): P^-(perm[t], k) = R^{-1}(t, k) = RinvT(k, t)
__global__ void pminus_kernel(const double* __restrict__ RinvT, const int32_t* __restrict__ perm, int m,
                              double* Pm) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)m * m) return;
    const int t = (int)(idx / m), k = (int)(idx % m);
    Pm[(int64_t)perm[t] * m + k] = RinvT[(int64_t)k * m + t];
}

// D = A^* P^-: its sparse part on the FP64 pipe (the entries of P^- span too many binades for
// fixed point), the low-rank part V^* (U^* P^-) and then V D on the integer pipes where V's rows are
// flat, else on the FP64 pipe too. On the integer pipes V(q, :) is taken in units of 2^{lr_top[q]} and
// the other factor (times 2^{lr_top[q]} for U^* P^-) in units of its largest value in column k, each
// as LR_BITS = 57 bits in two limbs; a product is the three upper of the four limb products. An FP64
// multiply-add holds an SM sub-partition for 64 cycles, the three limb products for 12: with r = 10
// at 1000 x 300,000 D took 7.5 ms and V D 6.0 in float64, 4.5 and 2.9 so.
// The line (lr_flat, decided at create): fixed point rounds every entry of V(q, :) to 2^-58 of the
// largest, so over a column of D the term V(q, :)^* T(q, k) moves by 2^-58 2^{lr_top[q]} |T(q, k)| sqrt(n)
// at most: with the largest entry up to 2^LR_FLAT root mean squares that is 2^-54 of the term's own
// norm, float64's rounding of one product. Rows of normal variates stay below 13 for any n up to
// 2^30. Rows with few large entries or scaled columns do not: one entry a row 2^10
// times the others at 100 x 200,000 left a first correction of 2e-13 in fixed point, 6e-15 in float64.
constexpr int LR_LO = 28;
constexpr int LR_BITS = 57;            // 29 bits and the sign in the upper limb
constexpr int LR_TERMS = 16;           // products whose upper sums (2^58 each) stay below 2^62
constexpr int DC_STAGE_LG = 5;         // log2 of the columns of V staged at a time, at most
constexpr int DC_COLS_LG = 2, DC_COLS = 1 << DC_COLS_LG;   // columns c a thread works on at once,
constexpr int DC_TOGETHER = 16;                            // for their first entries
constexpr int DC_LONG = 256;           // entries of a column that others should not wait for

// An upper sum and the sum of the two middle products (2^-LR_LO of it).
struct LimbSum { long long h, m; };
__device__ __forceinline__ void mad_limbs(LimbSum& s, int2 a, int2 b) {
    mad_limb(s.h, a.x, b.x);
    mad_limb(s.m, a.x, b.y);
    mad_limb(s.m, a.y, b.x);
}
// The middle sum's upper part moves over.
__device__ __forceinline__ void fold(LimbSum& s) {
    s.h += s.m >> LR_LO;
    s.m &= (1ll << LR_LO) - 1;
}

// h 2^e rounded once
__device__ __forceinline__ double limb_value(long long h, int e) {
    const unsigned long long neg = (unsigned long long)(h >> 63), w = ((unsigned long long)h ^ neg) - neg;
    return i128_round((uint32_t)w, (uint32_t)(w >> 32), 0u, 0u, e, (uint32_t)neg);
}

__device__ __forceinline__ int top_of(double x) {          // |x| < 2^top, tight for a normal x
    const int e = (int)(((uint32_t)__double2hiint(x) & 0x7FF00000u) >> 20);
    return (e ? e : 1) - 1022;
}

// D(c, k): a thread per k (blockIdx.y picks blockDim of them), the CTA walks the columns c, 2^lgt at a
// time: 32, or fewer where that leaves less than eight CTAs an SM (a preconditioner of a 200 x 2000
// matrix with 60 nonzeros a column took 1,713 us by 32, 1,438 by 4), down to one where a column has
// more than DC_LONG entries, which then has several of them in flight (three of 3,000 among 27: 2,814
// and 683 us). The low-rank part by limbs or in float64 (the words of ts and vs are then doubles).
// dtop[k] (limbs; pre-filled with kZeroRowExp) gathers the frexp exponents of D(:, k)'s maxima.
enum LowRank { LR_NONE, LR_LIMBS, LR_FLOAT64 };
template <LowRank LR>
__global__ void __launch_bounds__(256) sparse_d_kernel(const int64_t* __restrict__ cptr, const int32_t* __restrict__ crow,
                                                       const double* __restrict__ cval, const double* __restrict__ Pm, int m,
                                                       int n, int r, const double* __restrict__ V,
                                                       const int32_t* __restrict__ vtop, const double* __restrict__ UtP,
                                                       double* __restrict__ D, int32_t* __restrict__ dtop, int lgt) {
    extern __shared__ __align__(16) int2 d_smem[];
    const int t = threadIdx.x, nt = blockDim.x, k = blockIdx.y * nt + t;
    const int turn = 1 << lgt, lgst = max(lgt, DC_COLS_LG), stage = 1 << lgst;   // V's columns: DC_COLS of them at least
    constexpr bool LOWRANK = LR != LR_NONE;
    int2* ts = d_smem;                                     // [r][nt]: (U^* P^-)(q, k) 2^{vtop[q]}
    int2* vs = d_smem + (LOWRANK ? r * nt : 0);            // [stage][r]
    double* ts_d = reinterpret_cast<double*>(ts);
    double* vs_d = reinterpret_cast<double*>(vs);
    int ek = 0, tmax = kZeroRowExp;
    bool bad = false;
    if (LR == LR_FLOAT64)
        for (int q = 0; q < r; ++q) ts_d[q * nt + t] = k < m ? UtP[(int64_t)q * m + k] : 0.0;
    if (LR == LR_LIMBS) {
        int e = kZeroRowExp;
        for (int q = 0; q < r; ++q) {
            const double x = k < m ? UtP[(int64_t)q * m + k] : 0.0;
            bad |= !isfinite(x);
            if (x != 0.0) e = max(e, top_of(x) + vtop[q]);
        }
        ek = e == kZeroRowExp ? 0 : e;
        for (int q = 0; q < r; ++q)
            ts[q * nt + t] = to_limbs<LR_LO>(k < m && !bad ? UtP[(int64_t)q * m + k] : 0.0, ek - vtop[q], LR_BITS);
    }
    for (int64_t c0 = (int64_t)blockIdx.x * turn; c0 < n; c0 += (int64_t)gridDim.x * turn) {
        if (LOWRANK) {
            __syncthreads();
            for (int e = t; e < stage * r; e += nt) {
                const int q = e >> lgst, cc = e & (stage - 1);
                const double v = c0 + cc < n ? V[(int64_t)q * n + c0 + cc] : 0.0;
                if (LR == LR_FLOAT64) vs_d[cc * r + q] = v;
                else vs[cc * r + q] = to_limbs<LR_LO>(v, vtop[q], LR_BITS);
            }
            __syncthreads();
        }
        if (k >= m) continue;
        const int cnt = (int)min((int64_t)turn, n - c0);
#pragma unroll 1
        for (int cc = 0; cc < cnt; cc += DC_COLS) {
            double s[DC_COLS];
            int64_t b[DC_COLS];
            int len[DC_COLS], most = 0;
#pragma unroll
            for (int u = 0; u < DC_COLS; ++u) {
                const bool live = cc + u < cnt;
                b[u] = live ? cptr[c0 + cc + u] : 0;
                len[u] = live ? (int)(cptr[c0 + cc + u + 1] - b[u]) : 0;
                most = max(most, len[u]);
                s[u] = 0.0;
            }
            for (int p = 0; p < min(most, DC_TOGETHER); ++p)
#pragma unroll
                for (int u = 0; u < DC_COLS; ++u)
                    if (p < len[u]) s[u] = fma(cval[b[u] + p], __ldg(Pm + (int64_t)crow[b[u] + p] * m + k), s[u]);
            if (most > DC_TOGETHER)              // long columns: each by itself, several of its entries in flight
#pragma unroll
                for (int u = 0; u < DC_COLS; ++u)
#pragma unroll 4
                    for (int p = DC_TOGETHER; p < len[u]; ++p)
                        s[u] = fma(cval[b[u] + p], __ldg(Pm + (int64_t)crow[b[u] + p] * m + k), s[u]);
            if (LR == LR_FLOAT64) {
#pragma unroll 2
                for (int q = 0; q < r; ++q) {
                    const double x = ts_d[q * nt + t];
#pragma unroll
                    for (int u = 0; u < DC_COLS; ++u) s[u] = fma(vs_d[(cc + u) * r + q], x, s[u]);
                }
            }
            if (LR == LR_LIMBS) {
                for (int q0 = 0; q0 < r; q0 += LR_TERMS) {
                    LimbSum w[DC_COLS];
#pragma unroll
                    for (int u = 0; u < DC_COLS; ++u) w[u].h = w[u].m = 0;
                    const int qe = min(r, q0 + LR_TERMS);
#pragma unroll 2
                    for (int q = q0; q < qe; ++q) {
                        const int2 x = ts[q * nt + t];
#pragma unroll
                        for (int u = 0; u < DC_COLS; ++u) mad_limbs(w[u], x, vs[(cc + u) * r + q]);
                    }
#pragma unroll
                    for (int u = 0; u < DC_COLS; ++u) {
                        fold(w[u]);
                        s[u] += limb_value(w[u].h, ek - 58);
                    }
                }
                if (bad)
#pragma unroll
                    for (int u = 0; u < DC_COLS; ++u) s[u] = __longlong_as_double(0x7FF8000000000000ll);
            }
#pragma unroll
            for (int u = 0; u < DC_COLS; ++u)
                if (cc + u < cnt) {
                    D[(c0 + cc + u) * m + k] = s[u];
                    if (LR == LR_LIMBS && s[u] != 0.0) tmax = max(tmax, top_of(s[u]));
                }
        }
    }
    if (LR == LR_LIMBS && k < m && tmax != kZeroRowExp) atomicMax(dtop + k, tmax);
}

// Partial sums of (V D)(q, k) over chunk blockIdx.x of D's rows: 32 columns k a CTA (a lane each),
// rows q0 .. q0 + ROWS - 1 of V (blockIdx.z), the warps take D's rows in turn. part[chunk][q][k].
constexpr int VD_KC = 128;
template <int ROWS>
__global__ void __launch_bounds__(SK_T) lowrank_d_kernel(const double* __restrict__ V, const int32_t* __restrict__ vtop, int r,
                                                         int n, int m, int chunk, const double* __restrict__ D,
                                                         const int32_t* __restrict__ dtop, double* __restrict__ part) {
    __shared__ int2 vs[VD_KC][ROWS];
    __shared__ unsigned long long sum[2][ROWS][32];
    __shared__ int bad_s[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, q0 = blockIdx.z * ROWS, k = blockIdx.y * 32 + lane;
    const int64_t kb = (int64_t)blockIdx.x * chunk, ke = min((int64_t)n, kb + chunk);
    for (int e = t; e < 2 * ROWS * 32; e += SK_T) (&sum[0][0][0])[e] = 0ull;
    if (t < 32) bad_s[t] = 0;
    const int top = k < m ? max(dtop[k], -1022) : 0;      // a column of zeros or subnormals: the smallest normal's
    LimbSum a[ROWS];
    long long up[ROWS];                                    // the upper sums' own upper words
#pragma unroll
    for (int q = 0; q < ROWS; ++q) a[q].h = a[q].m = up[q] = 0;
    bool bad = false;
    for (int64_t c0 = kb; c0 < ke; c0 += VD_KC) {
        __syncthreads();
        for (int e = t; e < VD_KC * ROWS; e += SK_T) {
            const int q = e / VD_KC, c = e % VD_KC;
            vs[c][q] = q0 + q < r && c0 + c < ke ? to_limbs<LR_LO>(V[(int64_t)(q0 + q) * n + c0 + c], vtop[q0 + q], LR_BITS)
                                                 : make_int2(0, 0);
        }
        __syncthreads();
        const int cnt = (int)min((int64_t)VD_KC, ke - c0);
        if (k < m) {
#pragma unroll 4
            for (int c = warp; c < cnt; c += SK_WARPS) {   // VD_KC / SK_WARPS = LR_TERMS rows a stage at most
                const double x = __ldg(D + (c0 + c) * m + k);
                bad |= !isfinite(x);
                const int2 d = to_limbs<LR_LO>(x, top, LR_BITS);
#pragma unroll
                for (int q = 0; q < ROWS; ++q) mad_limbs(a[q], d, vs[c][q]);
            }
        }
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
            fold(a[q]);
            up[q] += a[q].h >> 32;
            a[q].h &= 0xFFFFFFFFll;
        }
    }
    // integer sums: the order does not matter. Below 2^60 a warp: h and m; above: up
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
        atomicAdd(&sum[0][q][lane], (unsigned long long)up[q]);
        atomicAdd(&sum[1][q][lane], (unsigned long long)((a[q].h << LR_LO) + a[q].m));
    }
    if (bad) bad_s[lane] = 1;
    __syncthreads();
    for (int e = t; e < ROWS * 32; e += SK_T) {
        const int q = e >> 5, l = e & 31, kk = blockIdx.y * 32 + l;
        if (q0 + q >= r || kk >= m) continue;
        const __int128 v = ((__int128)(long long)sum[0][q][l] << (32 + LR_LO)) + (__int128)sum[1][q][l];
        const int e2 = vtop[q0 + q] + max(dtop[kk], -1022) - 58 - LR_LO;
        part[((int64_t)blockIdx.x * r + q0 + q) * m + kk] =
            bad_s[l] ? __longlong_as_double(0x7FF8000000000000ll)
                     : u128_to_double((unsigned long long)(v >> 64), (unsigned long long)v, e2);
    }
}
static_assert(VD_KC <= SK_WARPS * LR_TERMS, "a stage's upper sums must fit before they are folded");

// VD(q, k) from the chunks' partial sums, 32 entries a CTA, eight threads an entry.
__global__ void __launch_bounds__(256) lowrank_d_sum_kernel(const double* __restrict__ part, int chunks, int total,
                                                            double* __restrict__ VD) {
    __shared__ double s[8][32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, idx = blockIdx.x * 32 + lane;
    double a = 0.0;
    if (idx < total)
        for (int z = g; z < chunks; z += 8) a += part[(int64_t)z * total + idx];
    s[g][lane] = a;
    __syncthreads();
    if (g == 0 && idx < total) {
        for (int w = 1; w < 8; ++w) a += s[w][lane];
        VD[idx] = a;
    }
}

// E(i, :) = sum over row i's nonzeros of val D(col, :)  [+ sum_q U(i, q) (V D)(q, :)]
__global__ void sparse_e_kernel(const int64_t* __restrict__ rptr, const int32_t* __restrict__ col,
                                const double* __restrict__ val, const double* __restrict__ D, int m, int r,
                                const double* __restrict__ U, const double* __restrict__ VD, double* E) {
    const int i = blockIdx.x;
    const int64_t b = rptr[i], e = rptr[i + 1];
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        double s0 = 0.0, s1 = 0.0;
        int64_t p = b;
        for (; p + 1 < e; p += 2) {
            s0 = fma(val[p], D[(int64_t)col[p] * m + k], s0);
            s1 = fma(val[p + 1], D[(int64_t)col[p + 1] * m + k], s1);
        }
        if (p < e) s0 = fma(val[p], D[(int64_t)col[p] * m + k], s0);
        double s = s0 + s1;
        for (int q = 0; q < r; ++q) s = fma(U[(int64_t)i * r + q], VD[(int64_t)q * m + k], s);
        E[(int64_t)i * m + k] = s;
    }
}

// ---------------------------------------------------------------------------------
// Products of the apply: exact products summed in 128-bit integers (i128.cuh).
//
// The right-hand sides are kept as an n x k block (row c holds entry c of every vector), so
// that a nonzero's gather reads k consecutive doubles. A warp is cut into groups of
// 2^LG lanes, one lane per right-hand side: 32 lanes from k = 17 up, fewer below, when the
// groups take different nonzeros (A x) or columns (A^* h). Bound: the integer pipes, about 60
// instructions per nonzero and right-hand side; the double-double form on the FP64 pipe took
// 832 cycles per warp of them, and gathered one double per 32-byte sector. An apply of 100
// vectors with two refinement passes at 1000 x 300,000, 1.5e6 nonzeros: 40.6 -> 5.7 ms.
// ---------------------------------------------------------------------------------
constexpr int SP_PART = I128_MAX_TERMS - 1 - (int)kMaxLowRank;   // a column's part, beside y and the low-rank terms
constexpr int SP_WARPS = 8;

__device__ __forceinline__ i128acc i128_shfl_xor(const i128acc& a, int o) {
    return {__shfl_xor_sync(0xffffffffu, a.w0, o), __shfl_xor_sync(0xffffffffu, a.w1, o),
            __shfl_xor_sync(0xffffffffu, a.w2, o), __shfl_xor_sync(0xffffffffu, a.w3, o),
            __shfl_xor_sync(0xffffffffu, a.E, o)};
}

// part(c, j) = the sum over chunk c of val x_j[col], as an unevaluated pair of doubles: one
// warp per (chunk, 2^LG right-hand sides), X n x k (ld ldx). 32 nonzeros are decoded at a time
// (one per lane) into shared memory, from which every group reads the ones it takes; four
// gathers are in flight per lane.
template <int LG>
__global__ void __launch_bounds__(32 * SP_WARPS)
    spmv_chunk_kernel(const int32_t* __restrict__ crow_of, const int64_t* __restrict__ cbeg,
                      const int64_t* __restrict__ rptr, const int32_t* __restrict__ col,
                      const double* __restrict__ val, const double* __restrict__ X, int64_t ldx, int nchunks, int k,
                      double2* __restrict__ part) {
    constexpr int KL = 1 << LG, SUB = 32 / KL, UN = 4;
    __shared__ uint4 entries[SP_WARPS][32];      // left factor: low word, high word | sign, exponent, column
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int jb = (k + KL - 1) / KL;
    const int64_t wid = (int64_t)blockIdx.x * SP_WARPS + warp;
    if (wid >= (int64_t)nchunks * jb) return;
    const int c = (int)(wid / jb), j = (int)(wid % jb) * KL + (lane & (KL - 1)), g = lane >> LG;
    const bool live = j < k;
    const double* x = X + (live ? j : 0);
    const int64_t b = cbeg[c];
    const int64_t e = min(b + (int64_t)SP_CHUNK, rptr[crow_of[c] + 1]);
    uint4* ent = entries[warp];
    i128acc acc = i128_zero();
    bool bad = false;
    for (int64_t p0 = b; p0 < e; p0 += 32) {
        uint4 w = make_uint4(0u, 0u, (uint32_t)(I128_E_EMPTY / 2), 0u);   // past the end: a zero
        if (p0 + lane < e) {
            uint32_t lo, hi;
            ldg_words(val + p0 + lane, lo, hi);
            const i128op o = i128_left(i128_decode(lo, hi));
            w = make_uint4(o.lo, o.hi | (o.neg & 0x80000000u), (uint32_t)o.e, (uint32_t)col[p0 + lane]);
        }
        __syncwarp();
        ent[lane] = w;
        __syncwarp();
        const int steps = ((int)min((int64_t)32, e - p0) + SUB - 1) / SUB;
        for (int t0 = 0; t0 < steps; t0 += UN) {
            uint32_t xl[UN], xh[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                const int at = (t0 + u) * SUB + g;
                ldg_words(x + (int64_t)ent[at & 31].w * ldx, xl[u], xh[u]);
            }
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                const int at = (t0 + u) * SUB + g;
                if (at >= 32) break;             // the same for every group of the warp
                const uint4 v = ent[at];
                i128op a;
                a.lo = v.x;
                a.hi = v.y & 0x7FFFFFFFu;
                a.e = (int)v.z;
                a.neg = (uint32_t)((int32_t)v.y >> 31);
                bad |= !i128_finite(xh[u]) && v.z != (uint32_t)(I128_E_EMPTY / 2);
                i128_mac(acc, a, i128_decode(xl[u], xh[u]));
            }
        }
    }
    int any_bad = bad ? 1 : 0;
#pragma unroll
    for (int o = KL; o < 32; o <<= 1) {
        i128_merge(acc, i128_shfl_xor(acc, o));
        any_bad |= __shfl_xor_sync(0xffffffffu, any_bad, o);
    }
    if (g == 0 && live) {
        double hi, lo;
        i128_to_pair(acc, hi, lo);
        if (any_bad) hi = __longlong_as_double(0x7FF8000000000000ll);   // an infinity or NaN among the x
        part[(int64_t)c * k + j] = make_double2(hi, lo);
    }
}

// out(i, j) (m x k, ld k) = (A x_j)_i: the chunks of row i added in order in double-double,
// plus the low-rank part sum_q U(i, q) (V X^*)(q, j) (a float64 sum added once), rounded
// once. One thread per (i, j).
__global__ void spmv_rows_kernel(const int32_t* __restrict__ rchunk, const double2* __restrict__ part, int m, int k,
                                 int r, const double* __restrict__ U, const double* __restrict__ VX, double* out) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)m * k) return;
    const int i = (int)(idx / k), j = (int)(idx % k);
    double hi = 0.0, lo = 0.0;
    for (int c = rchunk[i]; c < rchunk[i + 1]; ++c) {
        const double2 v = part[(int64_t)c * k + j];
        dd_add(hi, lo, v.x, v.y);
    }
    if (r > 0) {
        double t = 0.0;
        for (int q = 0; q < r; ++q) t = fma(U[(int64_t)i * r + q], VX[(int64_t)q * k + j], t);
        dd_add(hi, lo, t, 0.0);
    }
    out[idx] = hi + lo;
}

// out(c, j) = Y(c, j) - (A^* h_j)_c for h (m x k, ld k), rounded once: a group of 2^LG lanes
// per column c, JB right-hand sides per lane. The low-rank part subtracts
// sum_q V(q, c) (U^* h)(q, j) the same way. out may be Y. Y and out: n x k (ld ldy, ldo).
template <int LG, int JB>
__global__ void __launch_bounds__(32 * SP_WARPS)
    spmvT_kernel(const int64_t* __restrict__ cptr, const int32_t* __restrict__ crow, const double* __restrict__ cval,
                 const double* __restrict__ H, int k, int n, int r, const double* __restrict__ V,
                 const double* __restrict__ UtH, const double* Y, int64_t ldy, double* out, int64_t ldo) {
    constexpr int KL = 1 << LG, SUB = 32 / KL;
    __shared__ double2 full[SP_WARPS][JB][32];   // full sums so far of a column with more terms than one sum holds
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j0 = blockIdx.y * (KL * JB) + (lane & (KL - 1));
    const int64_t step = (int64_t)gridDim.x * SP_WARPS * SUB;
    for (int64_t c = ((int64_t)blockIdx.x * SP_WARPS + warp) * SUB + (lane >> LG); c < n; c += step) {
        i128acc acc[JB];
        bool bad[JB];
        const i128op one = i128_left(i128_decode(0u, 0x3FF00000u));
#pragma unroll
        for (int q = 0; q < JB; ++q) {
            acc[q] = i128_zero();
            bad[q] = false;
            const int j = j0 + q * KL;
            uint32_t lo = 0u, hi = 0x3FF00000u;     // lanes past k: any value but zero
            if (j < k) {
                const double y = Y[c * ldy + j];
                lo = (uint32_t)__double2loint(y);
                hi = (uint32_t)__double2hiint(y);
            }
            bad[q] |= !i128_finite(hi);
            i128_mac(acc[q], one, i128_decode(lo, hi));
        }
        bool longer = false;
        auto flush = [&](int q) {
            double2 v = longer ? full[warp][q][lane] : make_double2(0.0, 0.0);
            i128_flush(acc[q], v.x, v.y);
            return v;
        };
        auto term = [&](double v, const double* h) {
            const i128op a = i128_left(i128_decode((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v)));
            uint32_t lo[JB], hi[JB];
#pragma unroll
            for (int q = 0; q < JB; ++q) {
                lo[q] = 0u;
                hi[q] = 0x3FF00000u;
                if (j0 + q * KL < k) ldg_words(h + j0 + q * KL, lo[q], hi[q]);
            }
#pragma unroll
            for (int q = 0; q < JB; ++q) {
                bad[q] |= !i128_finite(hi[q]);
                i128_mac(acc[q], a, i128_decode(lo[q], hi[q]), ~0u);
            }
        };
        const int64_t pe = cptr[c + 1];
        int64_t p = cptr[c];
        while (pe - p > SP_PART) {                // a very long column
            const int64_t part_end = p + SP_PART;
#pragma unroll 1
            for (; p < part_end; ++p) term(cval[p], H + (int64_t)crow[p] * k);
#pragma unroll
            for (int q = 0; q < JB; ++q) full[warp][q][lane] = flush(q);
            longer = true;
        }
        if (p < pe) {                             // the next entry is loaded ahead of this one's products
            double v = cval[p];
            int row = crow[p];
            while (++p < pe) {
                const double v1 = cval[p];
                const int row1 = crow[p];
                term(v, H + (int64_t)row * k);
                v = v1;
                row = row1;
            }
            term(v, H + (int64_t)row * k);
        }
        for (int q = 0; q < r; ++q) term(V[(int64_t)q * n + c], UtH + (int64_t)q * k);
#pragma unroll
        for (int q = 0; q < JB; ++q) {
            const int j = j0 + q * KL;
            double v;
            if (longer) {
                const double2 f = flush(q);
                v = f.x + f.y;
            } else {
                v = i128_to_double(acc[q]);
            }
            if (j < k) out[c * ldo + j] = bad[q] ? __longlong_as_double(0x7FF8000000000000ll) : v;
        }
    }
}

// dst (k x n, ld ldd) = B - X or X for X n x k (ld k): 32 x 32 tiles through shared memory.
__global__ void __launch_bounds__(256) finish_rows_kernel(const double* __restrict__ X, int n, int k,
                                                          const double* __restrict__ B, int64_t ldb, double* dst,
                                                          int64_t ldd) {
    __shared__ double tile[32][33];
    const int c0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int y = ty; y < 32; y += 8)
        tile[y][tx] = (c0 + y < n && j0 + tx < k) ? X[(int64_t)(c0 + y) * k + j0 + tx] : 0.0;
    __syncthreads();
    for (int y = ty; y < 32; y += 8) {
        const int j = j0 + y, c = c0 + tx;
        if (j < k && c < n) {
            const double v = tile[tx][y];
            dst[(int64_t)j * ldd + c] = B ? B[(int64_t)j * ldb + c] - v : v;
        }
    }
}

__global__ void add_kernel(double* y, const double* x, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] += x[i];
}

unsigned grid_of(int64_t total, int threads) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + threads - 1) / threads, (int64_t)sm_count() * 32));
}

int row_threads(int m) { return std::min(256, (m + 31) / 32 * 32); }

// Low-rank helpers on the float64 GEMM: C (r x cols, ld ldc) = U^* Y for Y m x cols
// (ld ldy), and C = V Y for Y n x k.
cudaError_t ut_times(const rtproj_ctx* h, const double* Y, int64_t ldy, int cols, double* C, int64_t ldc) {
    Gemm64 g;
    g.M = h->lr; g.N = cols; g.K = (int)h->m;
    g.A = h->lrU; g.a_rs = 1; g.a_cs = h->lr;
    g.B = Y; g.b_rs = ldy; g.b_cs = 1;
    g.C = C; g.c_rs = ldc; g.c_cs = 1;
    return gemm64(g, h->part, h->part_elems, h->stream);
}

// C (r x k, ld ldc) = V Y for Y n x k (ld k)
cudaError_t v_times(const rtproj_ctx* h, const double* Y, int k, double* C, int64_t ldc) {
    Narrow64 g;
    g.M = h->lr; g.N = k; g.K = (int)h->n;
    g.A = h->lrV; g.a_rs = h->n;
    g.B = Y; g.b_rs = k; g.b_cs = 1;
    g.C = C; g.c_rs = ldc;
    return gemm64_narrow(g, h->part, h->part_elems, h->stream);
}

}  // namespace

namespace rtp {

int64_t sparse_max_chunks(int64_t m, int64_t nnz) { return m + nnz / SP_CHUNK + 1; }

// G's panel lies in D's region, which is free during the sketch, when that holds it.
size_t panel_bytes(int64_t m, int64_t n) { return m * 8 >= SK_COLS * 2 ? 0 : (size_t)n * SK_COLS * 2; }

size_t sparse_bytes(int64_t m, int64_t n, int64_t nnz, int64_t r, int64_t l_max, int64_t k_max) {
    const int64_t nb = (n + SCAN_T - 1) / SCAN_T;
    const int64_t nz = std::max<int64_t>(nnz, 1);
    const int64_t nc = sparse_max_chunks(m, nnz);
    return align_up((size_t)(n + 1) * 8) + align_up((size_t)nz * 4) + align_up((size_t)nz * 8) +
           align_up((size_t)n * 8) + align_up((size_t)nb * 8) + 2 * align_up((size_t)m * m * 8) +
           align_up((size_t)r * std::max(l_max, m) * 8) + align_up((size_t)r * k_max * 8) +
           align_up((size_t)(2 * r * r + norm_parts()) * 8) + align_up((size_t)nc * 4) + align_up((size_t)nc * 8) +
           align_up((size_t)(m + 1) * 4) + align_up((size_t)nc * k_max * 16) + align_up((size_t)(m + r) * 4) +
           align_up((size_t)m * 4) + align_up(panel_bytes(m, n));
}

void sparse_bind(rtproj_ctx* h, char* base) {
    size_t off = 0;
    auto take = [&](size_t bytes) { char* p = base + off; off += align_up(bytes); return p; };
    const int64_t n = h->n, m = h->m, r = h->lr;
    const int64_t nz = std::max<int64_t>(h->nnz, 1);
    h->csc_ptr = (int64_t*)take((size_t)(n + 1) * 8);
    h->csc_row = (int32_t*)take((size_t)nz * 4);
    h->csc_val = (double*)take((size_t)nz * 8);
    h->csc_cursor = (int64_t*)take((size_t)n * 8);
    h->scan_tot = (int64_t*)take((size_t)((n + SCAN_T - 1) / SCAN_T) * 8);
    h->Pminus = (double*)take((size_t)m * m * 8);
    h->Esp = (double*)take((size_t)m * m * 8);
    h->lr_a = (double*)take((size_t)r * std::max(h->l_max, m) * 8);
    h->lr_b = (double*)take((size_t)r * h->k_max * 8);
    h->lr_small = (double*)take((size_t)(2 * r * r + norm_parts()) * 8);
    const int64_t nc = sparse_max_chunks(m, h->nnz);
    h->chunk_row = (int32_t*)take((size_t)nc * 4);
    h->chunk_beg = (int64_t*)take((size_t)nc * 8);
    h->row_chunk = (int32_t*)take((size_t)(m + 1) * 4);
    h->chunk_part = (double*)take((size_t)nc * h->k_max * 16);
    h->row_top = (int32_t*)take((size_t)(m + r) * 4);
    h->lr_top = h->row_top + m;
    h->d_top = (int32_t*)take((size_t)m * 4);
    int16_t* own = (int16_t*)take(panel_bytes(m, n));
    h->panel = panel_bytes(m, n) ? own : reinterpret_cast<int16_t*>(h->W);
}

// The chunk table from the row pointers (on the host): row i is cut into
// max(1, ceil(nnz_i / SP_CHUNK)) chunks. Copied to the device on the handle's stream.
rtproj_status sparse_chunks(rtproj_ctx* h, const int64_t* rp_host) {
    const int64_t m = h->m;
    std::vector<int32_t> crow, rch((size_t)m + 1);
    std::vector<int64_t> cbeg;
    h->longest_row = 0;
    for (int64_t i = 0; i < m; ++i) {
        rch[(size_t)i] = (int32_t)crow.size();
        const int64_t b = rp_host[i], e = rp_host[i + 1];
        h->longest_row = std::max(h->longest_row, e - b);
        int64_t p = b;
        do {
            crow.push_back((int32_t)i);
            cbeg.push_back(p);
            p += SP_CHUNK;
        } while (p < e);
    }
    rch[(size_t)m] = (int32_t)crow.size();
    h->nchunks = (int)crow.size();
    if ((int64_t)h->nchunks > sparse_max_chunks(m, h->nnz)) return RTPROJ_EINVAL;
    SP_CHECK(cudaMemcpyAsync(h->chunk_row, crow.data(), crow.size() * 4, cudaMemcpyHostToDevice, h->stream));
    SP_CHECK(cudaMemcpyAsync(h->chunk_beg, cbeg.data(), cbeg.size() * 8, cudaMemcpyHostToDevice, h->stream));
    SP_CHECK(cudaMemcpyAsync(h->row_chunk, rch.data(), rch.size() * 4, cudaMemcpyHostToDevice, h->stream));
    SP_CHECK(cudaStreamSynchronize(h->stream));   // the host vectors go out of scope
    return RTPROJ_OK;
}

// At create: the column-compressed copy, the value check and ||A||_F.
rtproj_status sparse_prepare(rtproj_ctx* h) {
    cudaStream_t s = h->stream;
    const int m = (int)h->m, n = (int)h->n, r = h->lr;
    const int64_t nnz = h->nnz;
    const int nb = (n + SCAN_T - 1) / SCAN_T;
    SP_CHECK(cudaMemsetAsync(h->csc_cursor, 0, (size_t)n * 8, s));
    if (nnz > 0) {
        count_cols_kernel<<<grid_of(nnz, 256), 256, 0, s>>>(h->csr_col, nnz, n, h->csc_cursor, h->status);
        note_launch();
    }
    block_totals_kernel<<<nb, SCAN_T, 0, s>>>(h->csc_cursor, n, h->scan_tot, h->longest_col_dev);
    scan_totals_kernel<<<1, SCAN_T, 0, s>>>(h->scan_tot, nb, h->row_top, m + r);
    const int64_t tops = h->nchunks + (int64_t)((n + TOPS_SPAN - 1) / TOPS_SPAN) * r + ((int64_t)m * r + TOPS_SPAN - 1) / TOPS_SPAN;
    row_tops_kernel<<<(unsigned)tops, 256, 0, s>>>(h->chunk_row, h->chunk_beg, h->csr_ptr, h->csr_val, h->nchunks, m, n, r,
                                                   h->lrU, h->lrV, h->row_top, h->status);
    note_launch();
    block_scan_kernel<<<nb, SCAN_T, 0, s>>>(h->csc_cursor, n, h->scan_tot, h->csc_ptr);
    note_launch(3);
    SP_CHECK(cudaMemsetAsync(h->csc_cursor, 0, (size_t)n * 8, s));
    scatter_csc_kernel<<<(unsigned)std::min(m, sm_count() * 32), 256, 0, s>>>(
        h->csr_ptr, h->csr_col, h->csr_val, m, n, h->csc_ptr, h->csc_cursor, h->csc_row, h->csc_val);
    sort_columns_kernel<<<grid_of(n, 256), 256, 0, s>>>(h->csc_ptr, n, h->csc_row, h->csc_val);
    note_launch(2);
    // ||A||_F
    const unsigned np = std::min<unsigned>(grid_of(std::max<int64_t>(nnz, 1), 256), (unsigned)norm_parts());
    sumsq_vals_kernel<<<np, 256, 0, s>>>(h->csr_val, nnz, h->norm_part);
    note_launch();
    double* GU = h->lr_small;
    double* GV = GU + (size_t)r * r;
    double* px = GV + (size_t)r * r;
    unsigned nx = 0;
    if (r > 0) {
        nx = (unsigned)std::min(m, norm_parts());
        cross_term_kernel<<<nx, 256, 0, s>>>(h->csr_ptr, h->csr_col, h->csr_val, m, n, r, h->lrU, h->lrV, px);
        note_launch();
        Gemm64 u;                                 // U^* U
        u.M = r; u.N = r; u.K = m;
        u.A = h->lrU; u.a_rs = 1; u.a_cs = r;
        u.B = h->lrU; u.b_rs = r; u.b_cs = 1;
        u.C = GU; u.c_rs = r; u.c_cs = 1;
        SP_CHECK(gemm64(u, h->part, h->part_elems, s));
        Gemm64 v;                                 // V V^*
        v.M = r; v.N = r; v.K = n;
        v.A = h->lrV; v.a_rs = n; v.a_cs = 1;
        v.B = h->lrV; v.b_rs = 1; v.b_cs = n;
        v.C = GV; v.c_rs = r; v.c_cs = 1;
        SP_CHECK(gemm64(v, h->part, h->part_elems, s));
    }
    frobenius_total_kernel<<<1, 32, 0, s>>>(h->norm_part, (int)np, px, (int)nx, GU, GV, r, n, h->lr_top, h->lr_flat_dev,
                                            h->normA);
    note_launch();
    SP_CHECK(cudaGetLastError());
    return RTPROJ_OK;
}

rtproj_status sparse_sketch(rtproj_ctx* h, uint64_t seed, int64_t l, double* S, int64_t lds) {
    const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFull), k1 = (uint32_t)(seed >> 32);
    const int m = (int)h->m, n = (int)h->n, r = h->lr, dist = h->opts.omega, gexp = omega_exp(dist);
    cudaStream_t s = h->stream;
    const int64_t panel = (int64_t)n * SK_COLS * 2, room = panel_bytes(m, n) ? panel : (int64_t)m * n * 8;
    const int total = (int)((l + SK_COLS - 1) / SK_COLS);
    const bool gen = r == 0 && h->longest_row <= SK_GEN_ROW && h->nnz * total <= SK_GEN;
    int panels = gen ? total : (int)std::max<int64_t>(1, std::min<int64_t>(total, std::min(room, SK_L2_BYTES) / panel));   // a launch
    panels = std::min(panels, 65535);
    // chunks a CTA: as many as keep the CTAs at some eight an SM, and their partial sums within the scratch
    SharedRows a = {h->chunk_row, h->chunk_beg, h->row_chunk, 1, 0, reinterpret_cast<longlong2*>(h->part)};
    const bool shared_rows = h->nchunks > m;
    const int64_t places = (int64_t)(h->part_elems / (2 * SK_COLS));
    while (shared_rows && (h->nnz / ((int64_t)a.group * SP_CHUNK) > 8 * sm_count() || h->nchunks / a.group + m + 1 > places)) a.group *= 2;
    a.slots = h->nchunks / a.group + m + 1;
    if (shared_rows) panels = (int)std::max<int64_t>(1, std::min<int64_t>(panels, places / a.slots));
    // the chunks of V G: up to four CTAs an SM, their partial sums within the scratch
    const int64_t cap = std::max<int64_t>(1, (int64_t)(h->part_elems / ((size_t)std::max(r, 1) * SK_COLS * 2 * panels)));
    int64_t chunks = std::min<int64_t>(cap, std::min<int64_t>(std::max(1, 4 * sm_count() / panels), ((int64_t)n + VG_KC - 1) / VG_KC));
    const int64_t chunk = (((int64_t)n + chunks - 1) / chunks + VG_KC - 1) / VG_KC * VG_KC;
    chunks = ((int64_t)n + chunk - 1) / chunk;
    const int vbits = limb_bits(chunk);
    const int per = dist == RTPROJ_OMEGA_GAUSSIAN ? 4 : 16;
    const unsigned pgrid = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>(((int64_t)n + per * SK_WARPS - 1) / (per * SK_WARPS), (int64_t)sm_count() * 32));
    for (int p0 = 0; p0 < total; p0 += panels) {
        const int j0 = p0 * SK_COLS;
        const unsigned np = (unsigned)std::min(panels, total - p0);
        if (!gen) {
            omega_panel_kernel<<<dim3(pgrid, np), SK_T, 0, s>>>(n, (int)l, j0, dist, k0, k1, h->panel);
            note_launch();
        }
        if (r > 0) {   // V G (r x l), this panel's columns
            longlong2* part = reinterpret_cast<longlong2*>(h->part);
            const int groups = (r + 11) / 12, rows = (r + groups - 1) / groups;   // 1 .. 12 rows a CTA
            const dim3 grid((unsigned)chunks, (unsigned)groups, np);
            auto run = [&](auto kern) {
                kern<<<grid, SK_T, 0, s>>>(h->lrV, h->lr_top, r, n, (int)chunk, vbits, h->panel, part);
            };
            if (rows <= 4) run(lowrank_panel_kernel<4>);
            else if (rows <= 8) run(lowrank_panel_kernel<8>);
            else if (rows <= 10) run(lowrank_panel_kernel<10>);
            else run(lowrank_panel_kernel<12>);
            lowrank_panel_sum_kernel<<<dim3((unsigned)((r * SK_COLS + 7) / 8), np), 256, 0, s>>>(
                part, h->lr_top, (int)chunks, r, (int)l, j0, vbits, gexp, h->lr_a, l);
            note_launch(2);
        }
        const dim3 grid((unsigned)h->nchunks, np);
        auto run = [&](auto kern) {
            kern<<<grid, SK_T, 0, s>>>(h->csr_ptr, h->csr_col, h->csr_val, h->row_top, h->panel, n, (int)l, j0, gexp, r, h->lrU,
                                       h->lr_a, l, S, lds, dist, k0, k1, a);
        };
        if (gen) run(sparse_sketch_kernel<true, false>);
        else if (shared_rows) run(sparse_sketch_kernel<false, true>);
        else run(sparse_sketch_kernel<false, false>);
        note_launch();
        if (shared_rows) {
            sketch_rows_kernel<<<dim3((unsigned)m, np), SK_COLS, 0, s>>>(h->csr_ptr, h->row_top, (int)l, j0, gexp, r, h->lrU,
                                                                         h->lr_a, l, S, lds, a);
            note_launch();
        }
    }
    SP_CHECK(cudaGetLastError());
    return RTPROJ_OK;
}

// X = R^{-*} Pi A A^* P^- (lower triangle) into Lc; D = A^* P^- lives in W's region (n x m)
rtproj_status sparse_gram(rtproj_ctx* h) {
    const int m = (int)h->m, n = (int)h->n, r = h->lr;
    cudaStream_t s = h->stream;
    const int64_t mm = (int64_t)m * m;
    double* D = h->W;
    pminus_kernel<<<(unsigned)((mm + 255) / 256), 256, 0, s>>>(h->RinvT, h->perm, m, h->Pminus);
    note_launch();
    if (r > 0) SP_CHECK(ut_times(h, h->Pminus, m, m, h->lr_a, m));                    // U^* P^-
    const int nt = row_threads(m), kgroups = (m + nt - 1) / nt;
    int lgt = DC_STAGE_LG;
    const int lgt_min = h->longest_col > DC_LONG ? 0 : DC_COLS_LG;
    while (lgt > lgt_min && (int64_t)((n + (1 << lgt) - 1) >> lgt) * kgroups < 8 * sm_count()) --lgt;
    const int turns = (n + (1 << lgt) - 1) >> lgt;
    const dim3 dgrid((unsigned)std::max(1, std::min(turns, sm_count() * 32 / kgroups)), (unsigned)kgroups);
    auto run_d = [&](auto kern, size_t smem) {
        const cudaError_t e = smem ? allow_dynamic_shared((const void*)kern, (size_t)kMaxLowRank * (256 + (1 << DC_STAGE_LG)) * sizeof(int2))
                                   : cudaSuccess;
        if (e != cudaSuccess) return e;
        kern<<<dgrid, nt, smem, s>>>(h->csc_ptr, h->csc_row, h->csc_val, h->Pminus, m, n, r, h->lrV, h->lr_top, h->lr_a, D,
                                     h->d_top, lgt);
        note_launch();
        return cudaGetLastError();
    };
    const size_t smem = (size_t)r * (nt + (1 << std::max(lgt, DC_COLS_LG))) * sizeof(int2);
    if (r == 0) {
        SP_CHECK(run_d(sparse_d_kernel<LR_NONE>, 0));
    } else if (!h->lr_flat) {
        SP_CHECK(run_d(sparse_d_kernel<LR_FLOAT64>, smem));
        Narrow64 g;                                                                     // V D
        g.M = r; g.N = m; g.K = n;
        g.A = h->lrV; g.a_rs = n;
        g.B = D; g.b_rs = m; g.b_cs = 1;
        g.C = h->lr_a; g.c_rs = m;
        SP_CHECK(gemm64_narrow(g, h->part, h->part_elems, s));
    } else {
        SP_CHECK(fill_int(h->d_top, m, kZeroRowExp, s));
        SP_CHECK(run_d(sparse_d_kernel<LR_LIMBS>, smem));
        // V D: about four CTAs an SM, their partial sums within the scratch
        const int groups = (r + 11) / 12, rows = (r + groups - 1) / groups, kg = (m + 31) / 32;
        const int64_t cap = std::max<int64_t>(1, (int64_t)(h->part_elems / ((size_t)r * m)));
        int64_t chunks = std::min<int64_t>(std::min<int64_t>(cap, 65535), std::max(1, 4 * sm_count() / (kg * groups)));
        const int64_t chunk = (((int64_t)n + chunks - 1) / chunks + VD_KC - 1) / VD_KC * VD_KC;
        chunks = ((int64_t)n + chunk - 1) / chunk;
        const dim3 grid((unsigned)chunks, (unsigned)kg, (unsigned)groups);
        auto run = [&](auto kern) {
            kern<<<grid, SK_T, 0, s>>>(h->lrV, h->lr_top, r, n, m, (int)chunk, D, h->d_top, h->part);
        };
        if (rows <= 4) run(lowrank_d_kernel<4>);
        else if (rows <= 8) run(lowrank_d_kernel<8>);
        else if (rows <= 10) run(lowrank_d_kernel<10>);
        else run(lowrank_d_kernel<12>);
        lowrank_d_sum_kernel<<<(unsigned)((r * m + 31) / 32), 256, 0, s>>>(h->part, (int)chunks, r * m, h->lr_a);
        note_launch(2);
    }
    sparse_e_kernel<<<m, row_threads(m), 0, s>>>(h->csr_ptr, h->csr_col, h->csr_val, D, m, r, h->lrU, h->lr_a,
                                                 h->Esp);
    note_launch();
    Gemm64 x;                                                                           // R^{-*} (Pi E)
    x.M = m; x.N = m; x.K = m;
    x.A = h->RinvT; x.a_rs = m; x.a_cs = 1; x.a_tri = 1;
    x.B = h->Esp; x.b_rs = m; x.b_cs = 1; x.bk = h->perm;
    x.C = h->Lc; x.c_rs = m; x.c_cs = 1;
    x.lower_only = true;
    SP_CHECK(gemm64(x, h->part, h->part_elems, s));
    SP_CHECK(cudaGetLastError());
    return RTPROJ_OK;
}

rtproj_status sparse_project(rtproj_ctx* h, const double* B, int64_t ldb, int k, void* Z, int64_t ldz, void* ROW,
                             int64_t ldr, void* X, int64_t ldx) {
    const rtproj_opts& o = h->opts;
    const int m = (int)h->m, n = (int)h->n, r = h->lr;
    cudaStream_t s = h->stream;
    const int64_t mk = (int64_t)m * k;
    double2* part = reinterpret_cast<double2*>(h->chunk_part);
    // lanes per right-hand side group: the smallest power of two that holds k, at most a warp
    int lg = 0;
    while (lg < 5 && (1 << lg) < k) ++lg;
    const int kl = 1 << lg;
    // A x: narrower groups, so that more of them share a chunk's nonzeros, while its warps would leave
    // sub-partitions without one (an apply of 17 vectors at 40 x 3000: 278 us by 32 lanes, 211 by this
    // rule; at 2 x 500,000 1,549 and 970)
    int lga = lg;
    while (lga > 0 && (int64_t)h->nchunks * ((k + (1 << lga) - 1) >> lga) < 4 * sm_count()) --lga;
    const int64_t warps_a = (int64_t)h->nchunks * ((k + (1 << lga) - 1) >> lga);
    const unsigned grid_a = (unsigned)((warps_a + SP_WARPS - 1) / SP_WARPS);
    const int jb = k > 64 ? 4 : k > 32 ? 2 : 1;          // right-hand sides per lane of A^* h
    const int per_cta = SP_WARPS * (32 / kl);
    const dim3 grid_t((unsigned)std::min<int64_t>((n + per_cta - 1) / per_cta, (int64_t)sm_count() * 32),
                      (unsigned)((k + kl * jb - 1) / (kl * jb)));
    SP_CHECK(row_norms(B, ldb, k, n, h->bnorm, s));
    SP_CHECK(cudaMemsetAsync(h->stats, 0, 16, s));
    // the vectors as an n x k block; one vector is already that
    const double* Bt = B;
    if (k > 1) {
        SP_CHECK(store_transposed(B, ldb, k, n, h->sbuf, k, RTPROJ_F64, s));
        Bt = h->sbuf;
    }
    auto apply_a = [&](const double* Xt, double* out) -> rtproj_status {   // out = A x
        phase_begin(h, RTPROJ_PHASE_APPLY_A);
        if (r > 0) SP_CHECK(v_times(h, Xt, k, h->lr_b, k));
        auto run = [&](auto kern) {
            kern<<<grid_a, 32 * SP_WARPS, 0, s>>>(h->chunk_row, h->chunk_beg, h->csr_ptr, h->csr_col, h->csr_val, Xt,
                                                  (int64_t)k, h->nchunks, k, part);
        };
        switch (lga) {
            case 0: run(spmv_chunk_kernel<0>); break;
            case 1: run(spmv_chunk_kernel<1>); break;
            case 2: run(spmv_chunk_kernel<2>); break;
            case 3: run(spmv_chunk_kernel<3>); break;
            case 4: run(spmv_chunk_kernel<4>); break;
            default: run(spmv_chunk_kernel<5>); break;
        }
        spmv_rows_kernel<<<(unsigned)((mk + 255) / 256), 256, 0, s>>>(h->row_chunk, part, m, k, r, h->lrU, h->lr_b,
                                                                      out);
        note_launch(2);
        phase_end(h, RTPROJ_PHASE_APPLY_A);
        return RTPROJ_OK;
    };
    auto apply_at = [&](const double* Hm, const double* Yt) -> rtproj_status {   // sbuf = Y - A^* h
        phase_begin(h, RTPROJ_PHASE_APPLY_AT);
        if (r > 0) SP_CHECK(ut_times(h, Hm, k, k, h->lr_b, k));
        auto run = [&](auto kern) {
            kern<<<grid_t, 32 * SP_WARPS, 0, s>>>(h->csc_ptr, h->csc_row, h->csc_val, Hm, k, n, r, h->lrV, h->lr_b,
                                                  Yt, (int64_t)k, h->sbuf, (int64_t)k);
        };
        switch (lg) {
            case 0: run(spmvT_kernel<0, 1>); break;
            case 1: run(spmvT_kernel<1, 1>); break;
            case 2: run(spmvT_kernel<2, 1>); break;
            case 3: run(spmvT_kernel<3, 1>); break;
            case 4: run(spmvT_kernel<4, 1>); break;
            default:
                if (jb == 1) run(spmvT_kernel<5, 1>);
                else if (jb == 2) run(spmvT_kernel<5, 2>);
                else run(spmvT_kernel<5, 4>);
                break;
        }
        note_launch();
        phase_end(h, RTPROJ_PHASE_APPLY_AT);
        return RTPROJ_OK;
    };
    // c = A b; h0 = Pi^* T1^* T1 Pi c; s = b - A^* h0
    rtproj_status st = apply_a(Bt, h->cbuf);
    if (st != RTPROJ_OK) return st;
    phase_begin(h, RTPROJ_PHASE_APPLY_M);
    st = middle_fp64(h, h->cbuf, h->hbuf, k);
    if (st != RTPROJ_OK) return st;
    phase_end(h, RTPROJ_PHASE_APPLY_M);
    st = apply_at(h->hbuf, Bt);
    if (st != RTPROJ_OK) return st;
    int passes = 0;
    for (int pass = 0; pass < o.refine_passes; ++pass) {
        // r = A s; dh = Pi^* T1^* T1 Pi r; h += dh; s <- s - A^* dh (Remark 4.3)
        st = apply_a(h->sbuf, h->cbuf);
        if (st != RTPROJ_OK) return st;
        phase_begin(h, RTPROJ_PHASE_APPLY_M);
        st = middle_fp64(h, h->cbuf, h->dhbuf, k);
        if (st != RTPROJ_OK) return st;
        add_kernel<<<(unsigned)((mk + 255) / 256), 256, 0, s>>>(h->hbuf, h->dhbuf, mk);
        note_launch();
        SP_CHECK(cudaMemsetAsync(h->stats, 0, 16, s));
        SP_CHECK(column_stats(h->cbuf, h->hbuf, h->dhbuf, m, k, h->bnorm, h->normA, h->stats, s));
        phase_end(h, RTPROJ_PHASE_APPLY_M);
        passes = pass + 1;
        bool last = passes == o.refine_passes;
        if (o.refine_tol > 0.0 && !last) {
            unsigned long long bits[2];
            SP_CHECK(cudaMemcpyAsync(bits, h->stats, 16, cudaMemcpyDeviceToHost, s));
            SP_CHECK(cudaStreamSynchronize(s));
            double v[2];
            std::memcpy(v, bits, 16);
            if (v[1] <= o.refine_tol) last = true;
        }
        st = apply_at(h->dhbuf, h->sbuf);   // in place: each entry reads its own s first
        if (st != RTPROJ_OK) return st;
        if (last) break;
    }
    h->last_passes = passes;
    const dim3 fgrid((unsigned)((n + 31) / 32), (unsigned)((k + 31) / 32));
    if (k == 1) {
        if (ROW) SP_CHECK(store_rows(h->sbuf, n, B, ldb, ROW, ldr, k, n, 1, RTPROJ_F64, s));
        if (Z) SP_CHECK(store_rows(h->sbuf, n, nullptr, 0, Z, ldz, k, n, 0, RTPROJ_F64, s));
    } else {   // ROW before Z, since Z may alias B
        if (ROW) finish_rows_kernel<<<fgrid, 256, 0, s>>>(h->sbuf, n, k, B, ldb, (double*)ROW, ldr);
        if (Z) finish_rows_kernel<<<fgrid, 256, 0, s>>>(h->sbuf, n, k, nullptr, 0, (double*)Z, ldz);
        note_launch((ROW ? 1 : 0) + (Z ? 1 : 0));
    }
    if (X) SP_CHECK(store_transposed(h->hbuf, k, m, k, X, ldx, RTPROJ_F64, s));
    SP_CHECK(cudaGetLastError());
    return RTPROJ_OK;
}

}  // namespace rtp
