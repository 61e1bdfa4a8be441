// The middle of the apply, h = Pi^* T1^* (T1 Pi c), taken straight from the float64 factor T1
// (lower triangular, m x m) when the problem is small: exact products summed in 128-bit
// integers (i128.cuh), each sum rounded once. Two launches in place of the four of the sliced
// form (digits of c, product, digits of u, product).
//
// What bounds it: at these sizes nothing but latency. The sliced product of a 64 x 64 factor
// occupies one or two tiles of the whole chip and takes 20 to 26 us (fetch of its unrolled
// code, TMA and TMEM set-up, the digit-pair chain), whatever the size; the sums below are
// spread over m k / LG blocks. A projection of one vector by a 64 x 2048 preconditioner took
// 201 us with the sliced middle and 144 us with this one, a step 800 and 626.
#include "i128.cuh"
#include "rtproj_internal.cuh"

#include <algorithm>

namespace rtp {
namespace {

constexpr int MD_MAX_WARPS = 8;
constexpr int MD_TERMS_PER_LANE = 8;   // products per lane that one more halving of the split would not repay
constexpr int MT = 32;                 // tile of the transposition

// T1's transpose (its lower triangle only; the rest of dst is never read), with the factor's
// entries checked as the digit slicing of the other form does.
__global__ void __launch_bounds__(256) middle_transpose_kernel(const double* T, int m, double* dst, int* status) {
    __shared__ double tile[MT][MT + 1];
    const int r0 = blockIdx.y * MT, c0 = blockIdx.x * MT;
    if (c0 > r0) return;
    bool bad = false;
    for (int y = threadIdx.y; y < MT; y += 8) {
        const int r = r0 + y, c = c0 + threadIdx.x;
        double v = 0.0;
        if (r < m && c <= r) v = T[(int64_t)r * m + c];
        bad |= !isfinite(v);
        tile[y][threadIdx.x] = v;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < MT; y += 8) {
        const int c = c0 + y, r = r0 + threadIdx.x;
        if (c < m && r < m) dst[(int64_t)c * m + r] = tile[threadIdx.x][y];
    }
    if (__any_sync(0xffffffffu, bad) && threadIdx.x == 0) set_status(status, RTPROJ_ENONFINITE);
}

__device__ __forceinline__ i128acc merge_lanes(i128acc a, int o) {
    const i128acc b = {__shfl_xor_sync(0xffffffffu, a.w0, o), __shfl_xor_sync(0xffffffffu, a.w1, o),
                       __shfl_xor_sync(0xffffffffu, a.w2, o), __shfl_xor_sync(0xffffffffu, a.w3, o),
                       __shfl_xor_sync(0xffffffffu, a.E, o)};
    i128_merge(a, b);
    return a;
}

// Block (g, r): row r of the product with T (row-major, leading dimension m; entries t of
// [r, m) when UPPER, of [0, r] otherwise) for the LG columns from g LG on. LG lanes of a warp
// take a column each and the 32 / LG lane groups of all warps split the sum over t (so that
// T's row is read coalesced where LG is small and once per warp where it is 32).
// gather: x's row of entry t; scatter: out's row of r (null: the same index).
template <int LG, bool UPPER>
__global__ void __launch_bounds__(32 * MD_MAX_WARPS) middle_rows_kernel(const double* __restrict__ T, int m,
                                                                        const double* __restrict__ x,
                                                                        const int32_t* __restrict__ gather,
                                                                        const int32_t* __restrict__ scatter, int k,
                                                                        double* __restrict__ out, int* status) {
    __shared__ i128acc part[MD_MAX_WARPS][LG];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int r = blockIdx.y, j = blockIdx.x * LG + (lane & (LG - 1));
    constexpr int GROUPS = 32 / LG;
    const int lo = UPPER ? r : 0, hi = UPPER ? m : r + 1;
    const unsigned long long* row = reinterpret_cast<const unsigned long long*>(T) + (int64_t)r * m;
    const unsigned long long* xb = reinterpret_cast<const unsigned long long*>(x);
    i128acc acc = i128_zero();
    bool bad = false;
    if (j < k) {
#pragma unroll 2
        for (int t = lo + warp * GROUPS + lane / LG; t < hi; t += warps * GROUPS) {
            const unsigned long long tb = __ldg(row + t);
            const unsigned long long vb = __ldg(xb + (int64_t)(gather ? __ldg(gather + t) : t) * k + j);
            const uint32_t th = (uint32_t)(tb >> 32), vh = (uint32_t)(vb >> 32);
            if (!i128_finite(th) || !i128_finite(vh)) { bad = true; continue; }
            i128_mac(acc, i128_left(i128_decode((uint32_t)tb, th)), i128_decode((uint32_t)vb, vh));
        }
    }
#pragma unroll
    for (int o = LG; o < 32; o <<= 1) acc = merge_lanes(acc, o);
    if (__any_sync(0xffffffffu, bad) && lane == 0) set_status(status, RTPROJ_ENONFINITE);
    if (warps > 1) {
        if (lane < LG) part[warp][lane] = acc;
        __syncthreads();
        if (warp) return;
        if (lane < LG)
            for (int w = 1; w < warps; ++w) i128_merge(acc, part[w][lane]);
    }
    if (lane < LG && j < k) out[(int64_t)(scatter ? scatter[r] : r) * k + j] = i128_to_double(acc);
}

template <bool UPPER>
void launch_rows(const double* T, int m, const double* x, const int32_t* gather, const int32_t* scatter, int k,
                 double* out, int* status, cudaStream_t s) {
    int lg = 1;
    while (lg < 32 && lg < k) lg <<= 1;
    int warps = 1;
    while (warps < MD_MAX_WARPS && (int64_t)m * lg > (int64_t)32 * MD_TERMS_PER_LANE * warps) warps <<= 1;
    const dim3 grid((unsigned)((k + lg - 1) / lg), (unsigned)m);   // m <= I128_MAX_TERMS; k may be any
    auto go = [&](auto kern) { kern<<<grid, 32 * warps, 0, s>>>(T, m, x, gather, scatter, k, out, status); };
    switch (lg) {
        case 1: go(middle_rows_kernel<1, UPPER>); break;
        case 2: go(middle_rows_kernel<2, UPPER>); break;
        case 4: go(middle_rows_kernel<4, UPPER>); break;
        case 8: go(middle_rows_kernel<8, UPPER>); break;
        case 16: go(middle_rows_kernel<16, UPPER>); break;
        default: go(middle_rows_kernel<32, UPPER>); break;
    }
    note_launch();
}

}  // namespace

// The columns that a block of k takes on the lanes: the next power of two, whole warps from 32 on.
static int64_t lane_columns(int64_t k) {
    int64_t lg = 1;
    while (lg < 32 && lg < k) lg <<= 1;
    return (k + lg - 1) / lg * lg;
}

// The sums cost 139 cycles a product and warp, the sliced form a fixed 50 us or so more than its
// work. A projection (us, direct / sliced): m = 256: k = 32 224 / 236, 64 224 / 236, 128 257 / 244;
// m = 384: 16 222 / 242, 32 266 / 244; m = 512: 8 210 / 251, 16 249 / 257, 32 302 / 257;
// m = 768: 4 234 / 285, 8 269 / 287, 16 341 / 287; m = 1024: 4 285 / 320, 8 335 / 320; m = 2048: 1 457 / 527,
// 4 556 / 537. The line lies at 2^22 products, counting the columns of idle lanes. It
// rises with k, so that a handle whose k_max lies below it needs no digits of T1.
bool middle_direct_ok(int64_t m, int64_t k) {
    return m <= I128_MAX_TERMS && m * m * lane_columns(k) <= MIDDLE_DIRECT_PRODUCTS;
}

cudaError_t middle_direct_prepare(const double* T1, int m, double* T1t, int* status, cudaStream_t s) {
    const unsigned tiles = (unsigned)((m + MT - 1) / MT);
    middle_transpose_kernel<<<dim3(tiles, tiles), dim3(32, 8), 0, s>>>(T1, m, T1t, status);
    note_launch();
    return cudaGetLastError();
}

cudaError_t middle_direct(const double* T1, const double* T1t, const int32_t* perm, int m, const double* c, int k, double* u,
                          double* out, int* status, cudaStream_t s) {
    launch_rows<false>(T1, m, c, perm, nullptr, k, u, status, s);      // u = T1 Pi c
    launch_rows<true>(T1t, m, u, nullptr, perm, k, out, status, s);    // out = Pi^* T1^* u
    return cudaGetLastError();
}

}  // namespace rtp
