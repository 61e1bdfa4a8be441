// Pivoted Householder QR of S^* (Section 4, Eq. 13) for the mixed form: float-float, one
// cooperative launch, columns in registers, exchanges through self-validating packets.
//
// The factorization is m strictly sequential steps, so a step's latency is its cost. CTA b keeps
// columns [b cpc, b cpc + cpc) of S^* (rows of S), WPC warps each, in registers: the warps take
// 64-row groups in turn, lane t rows 2 t and 2 t + 1 of a group. All column arithmetic runs two rows
// at a time in packed float32 instructions (add/mul/fma.f32x2; ff2.cuh). Step j:
//  1. warp 0 polls the CTAs' candidate records of step j (one 16-byte word each) until all carry the
//     step's tag, and takes the largest key: the squared trailing norm to 44 mantissa bits, lowest
//     column on ties (Businger-Golub);
//  2. every CTA loads the pivot column's packets (two rows in 16 bytes, tagged with the step) and
//     its exact squared norm, and derives the same reflector; a packet whose tag is not yet the
//     step's is loaded again;
//  3. each active column's dot product with the reflector gives its row-j entry r, hence its next
//     trailing norm n - r^2 before the column is updated: the CTA's record for step j + 1 is
//     published here, and the exchange overlaps the update;
//  4. the update, which also sums the new norm afresh and writes the column's packets (into
//     the other of two buffers) and norm for step j + 1.
// A packet, record or norm is one 128-bit store and one 128-bit load, which are single-copy
// atomic, so a reader needs neither a fence nor a flag behind the data: the former kernel's
// release fence, arrival counter, winner word and column load were four L2 round trips in a row
// (3.7 us a step at 512 x 516). What remains is the exchange (about 2800 cycles from a record's store
// until every CTA has seen all of them, across both dies) and one column load (850). A retired
// column's slot is never rewritten, so late readers of a pivot column are safe; a record buffer is
// rewritten only after every CTA has published the step between. Every wait has a clock deadline;
// on expiry the kernel raises RTPROJ_ETIMEOUT and all CTAs leave.
// Measured: 512 x 516 1.89 -> 1.50 ms (2.9 us a step), 64 x 256 246 -> 172 us, 333 x 698 1.37 -> 1.15 ms,
// 256 x 1024 1.27 -> 1.02 ms, 1024 x 2080 7.55 -> 7.09 ms (there the column arithmetic counts: seven
// columns of 2080 rows a CTA). Not kept: one 16-CTA cluster with the same columns and a hardware
// barrier a step (5 to 8 us a step: distributed shared memory answers no sooner than L2 here),
// per-column records polled by every warp, scalars formed after the packets' barrier.
//
// The early norm n - r^2 is exact to 2^-47 of n (n is summed afresh every step). When the winner's
// has cancelled by more than 2^10 the candidates are exchanged once more with their fresh
// sums, so the choice never rests on fewer than 37 bits. The reflector always uses the fresh sum.
// Range: S^* is scaled by a power of two below 1 / sqrt(l) of its largest entry; columns whose largest
// entries span more than 2^40, or a pivot whose squared norm falls below 2^-112, send the
// factorization to the float64 kernel enqueued behind (*fallback), and S is not modified. Accuracy: R
// is the exact factor of S^* + E with ||E|| of order l 2^-48 ||S||.
#include "rtproj_internal.cuh"
#include "ff2.cuh"

#include <climits>
#include <algorithm>

namespace rtp {
namespace {

struct QrFfDev {
    const double* S; int m, l; int64_t lds;
    double* R; int32_t* perm;
    int cpc;
    ulonglong2* slots;       // 2 x m x npk: packets by step parity
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

// A packet is the pair's high and low parts as they are, with a step's 4-bit tag in the top exponent
// bits of the four floats, which are zero: S^* is scaled so that no column's norm exceeds 1, and
// reflections keep the norms, so every part is below 2 in magnitude. A slot's previous content is
// the packet of two steps before (or the zero written at the start), whose tag differs.
constexpr f2 TAG_BITS = 0x4000000040000000ull;
struct Tag {
    f2 h, l;                 // the tag's bits in the two words
};
__device__ __forceinline__ Tag step_tag(int j) {
    const uint32_t n = ((uint32_t)(j >> 1) + 1u) & 15u;
    return {((f2)((n & 1u) << 30)) | ((f2)((n & 2u) << 29) << 32), ((f2)((n & 4u) << 28)) | ((f2)((n & 8u) << 27) << 32)};
}
__device__ __forceinline__ bool has_tag(const ulonglong2& w, const Tag& t) {
    return (w.x & TAG_BITS) == t.h && (w.y & TAG_BITS) == t.l;
}
__device__ __forceinline__ void st_packet(ulonglong2* p, const ffp& x, const Tag& t) { st_word(p, x.h | t.h, x.l | t.l); }
__device__ __forceinline__ ffp unpack(const ulonglong2& w) { return {w.x & ~TAG_BITS, w.y & ~TAG_BITS}; }

// A wait's deadline: true while it may go on.
struct Deadline {
    long long t0 = 0;
    unsigned int it = 0;
    __device__ __forceinline__ bool more(const QrFfDev& p) {
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
__device__ __forceinline__ bool poll_records(const QrFfDev& p, const ulonglong2* rec, int G, uint32_t tag, int lane,
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

// NP: row pairs per lane; WPC: warps per column (l <= 64 NP WPC); MAXW: most warps of a CTA.
template <int NP, int WPC, int MAXW>
__global__ void __launch_bounds__(32 * MAXW, 1) qr_ff_kernel(QrFfDev p) {
    __shared__ ulonglong2 vs[32 * NP * WPC];         // the reflector, zero above row j: high pairs, low pairs
    __shared__ double col_mx[MAXW];
    __shared__ unsigned long long key_s[MAXW];       // the columns' keys (0: retired)
    __shared__ uint32_t flag_s[MAXW];                // whether a column's early norm has cancelled
    __shared__ unsigned long long win_s[2];          // the winner by round
    __shared__ int state_s[2];                       // 0: expired, 1: winner, 2: winner has cancelled
    __shared__ float2 dot_s[MAXW], nsq_s[MAXW], cj_s[MAXW];
    __shared__ int ok_s, e_s, range_s;
    const int l = p.l, m = p.m, cpc = p.cpc, npk = (l + 1) >> 1;
    const int b = blockIdx.x, G = gridDim.x, t = threadIdx.x, lane = t & 31, warp = t >> 5, NT = blockDim.x;
    const int c0 = b * cpc, nc = max(0, min(cpc, m - c0));
    const int cw = warp / WPC, part = warp % WPC, col = c0 + cw;      // the warp's column and its share of the rows
    const bool mine = cw < nc;
    const size_t par_stride = (size_t)m * npk;
    // pair (u) of the warp's i-th group of rows
    auto pair_of = [&](int i) { return 32 * (i * WPC + part) + lane; };

    // 0. tags cleared; the scale: exponents of the CTAs' largest entries, and of their columns'
    //    smallest largest entry, exchanged once (see the top)
    if (mine) {
        double cm = 0.0;
        for (int i = 32 * part + lane; i < l; i += 32 * WPC) cm = fmax(cm, fabs(p.S[(int64_t)col * p.lds + i]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cm = fmax(cm, __shfl_xor_sync(0xffffffffu, cm, o));
        if (lane == 0) col_mx[warp] = cm;
        for (int q = 32 * part + lane; q < npk; q += 32 * WPC) {
            st_word(p.slots + (size_t)col * npk + q, 0ull, 0ull);
            st_word(p.slots + par_stride + (size_t)col * npk + q, 0ull, 0ull);
        }
    }
    for (int q = t; q < 32 * NP * WPC; q += NT) vs[q] = make_ulonglong2(0ull, 0ull);
    __syncthreads();
    if (t == 0) {
        int e_hi = INT_MIN / 2, e_lo = INT_MAX / 2;
        for (int q = 0; q < nc; ++q) {
            double cm = col_mx[q * WPC];
            for (int u = 1; u < WPC; ++u) cm = fmax(cm, col_mx[q * WPC + u]);
            int e = INT_MIN / 2;
            if (cm > 0.0) frexp(cm, &e);                     // cm < 2^e
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
    if (range_s > 40) {                                     // the same decision in every CTA
        if (b == 0 && t == 0) *p.fallback = 1;
        return;
    }
    const int E = e_s;

    // the column, its norm and its packets for step 0
    f2 ch[NP], cl[NP];
    ff nsq = {0.f, 0.f};
    bool active = mine;
    int pos = -1;
    ff alpha_mine = {0.f, 0.f};
    // the column's sum over its warps of each warp's total (every lane receives it)
    auto column_sum = [&](ff x, float2* buf) {
        if (WPC == 1) return x;
        if (lane == 0) buf[warp] = make_float2(x.hi, x.lo);
        column_barrier<WPC>(cw);
        ff sum = {buf[cw * WPC].x, buf[cw * WPC].y};
#pragma unroll
        for (int u = 1; u < WPC; ++u) sum = ff_add(sum, {buf[cw * WPC + u].x, buf[cw * WPC + u].y});
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
        ffp a = {0ull, 0ull};
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int q = pair_of(i), r0 = 2 * q;
            const ff x = r0 < l ? ff_from_double(src[r0] * sc) : ff{0.f, 0.f};
            const ff y = r0 + 1 < l ? ff_from_double(src[r0 + 1] * sc) : ff{0.f, 0.f};
            ch[i] = pack2(x.hi, y.hi);
            cl[i] = pack2(x.lo, y.lo);
            dot_acc2(a, {ch[i], cl[i]}, {ch[i], cl[i]});
            if (q < npk) st_packet(p.slots + (size_t)col * npk + q, {ch[i], cl[i]}, step_tag(0));
        }
        nsq = column_sum(warp_total(a), nsq_s);
        if (lane == 0 && part == 0) {
            st_word(p.nrm + col, pack2(nsq.hi, nsq.lo), 1ull);
            key_s[cw] = norm_key(nsq, col);
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
                if (active && lane == 0 && part == 0) key_s[cw] = norm_key(nsq, col);
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
        const ulonglong2* slot = p.slots + (size_t)par * par_stride + (size_t)piv * npk;
        const Tag tag = step_tag(j);
        const int q0 = j >> 1;
        bool good = true;
        constexpr int VL = (32 * NP * WPC + 127) / 128;      // packets per thread at 128 threads
        ulonglong2 w[VL];
#pragma unroll
        for (int k = 0; k < VL; ++k)
            if (q0 + t + k * NT < npk) w[k] = ld_word(slot + q0 + t + k * NT);
        ulonglong2 wj = ld_word(slot + q0), wn = ld_word(p.nrm + (size_t)par * m + piv);
        if (t == 0 && q0 > 0) vs[q0 - 1] = make_ulonglong2(0ull, 0ull);
        {
            Deadline d;
            while (!has_tag(wj, tag) && good) { good = d.more(p); wj = ld_word(slot + q0); }
            while ((uint32_t)wn.y != (uint32_t)(j + 1) && good) { good = d.more(p); wn = ld_word(p.nrm + (size_t)par * m + piv); }
        }
        const ff npiv = {lo2(wn.x), hi2(wn.x)};
        const bool small = !(npiv.hi >= 0x1p-112f);          // the float64 kernel takes over
        const ffp pj = unpack(wj);
        const ff x0 = (j & 1) ? ff{hi2(pj.h), hi2(pj.l)} : ff{lo2(pj.h), lo2(pj.l)};
        const ff nx = ff_sqrt_newton(npiv);
        const ff alpha = x0.hi >= 0.f ? ff_neg(nx) : nx;
        const ff v0 = ff_add(x0, ff_neg(alpha));
        const ff beta = ff_recip_newton(ff_mul(nx, ff_add(nx, x0.hi >= 0.f ? x0 : ff_neg(x0))));
#pragma unroll
        for (int k = 0; k < VL; ++k) {
            const int q = q0 + t + k * NT;
            if (q < npk) {
                Deadline d;
                while (!has_tag(w[k], tag) && good) { good = d.more(p); w[k] = ld_word(slot + q); }
                ffp v = unpack(w[k]);
                if (q == q0) {                               // rows above j stay out, row j: x0 - alpha
                    if (j & 1) v = {pack2(0.f, v0.hi), pack2(0.f, v0.lo)};
                    else v = {pack2(v0.hi, hi2(v.h)), pack2(v0.lo, hi2(v.l))};
                }
                vs[q] = make_ulonglong2(v.h, v.l);
            }
        }
        good = __syncthreads_and(good && !small);
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
        //    three at a time keep independent chains in flight) and the next trailing norm
        ff nw = {0.f, 0.f};
        if (active) {
            ffp a[3] = {{0ull, 0ull}, {0ull, 0ull}, {0ull, 0ull}};
            f2 xh = 0ull, xl = 0ull;                          // the pair that holds row j
#pragma unroll
            for (int i = 0; i < NP; i += 3)
                if (64 * WPC * (i + 3) > j) {
#pragma unroll
                    for (int u = 0; u < 3; ++u) {
                        const ulonglong2 v = vs[pair_of(i + u)];
                        dot_acc2(a[u], {v.x, v.y}, {ch[i + u], cl[i + u]});
                    }
                    if (64 * WPC * i <= j) {
#pragma unroll
                        for (int u = 0; u < 3; ++u)
                            if (pair_of(i + u) == q0) { xh = ch[i + u]; xl = cl[i + u]; }
                    }
                }
            ff cj;
            if (WPC == 1) {
                cj = {__shfl_sync(0xffffffffu, (j & 1) ? hi2(xh) : lo2(xh), q0 & 31),
                      __shfl_sync(0xffffffffu, (j & 1) ? hi2(xl) : lo2(xl), q0 & 31)};
            } else if ((q0 >> 5) % WPC == part && lane == (q0 & 31)) {
                cj_s[cw] = (j & 1) ? make_float2(hi2(xh), hi2(xl)) : make_float2(lo2(xh), lo2(xl));
            }
            nw = ff_neg(ff_mul(column_sum(warp_total(sum3(a)), dot_s), beta));
            if (WPC > 1) cj = {cj_s[cw].x, cj_s[cw].y};
            if (part == 0) {
                const ff r = ff_add(cj, ff_mul(nw, v0));      // R's entry
                const ff ne = ff_add(nsq, ff_neg(ff_mul(r, r)));
                if (lane == 0) {
                    key_s[cw] = norm_key(ne.hi > 0.f ? ne : ff{0.f, 0.f}, col);
                    flag_s[cw] = ne.hi < nsq.hi * 0x1p-10f ? 1u : 0u;
                }
            }
        }
        __syncthreads();
        if (warp == 0) publish(p.rec, j + 1, true);
        // 4. the update, the fresh norm, the packets of step j + 1
        if (active) {
            const ffp w2 = {pack2(nw.hi, nw.hi), pack2(nw.lo, nw.lo)};
            ulonglong2* dst = p.slots + (size_t)(par ^ 1) * par_stride + (size_t)col * npk;
            const Tag ntag = step_tag(j + 1);
            const int qn = (j + 1) >> 1;
            // rows j + 1 .. count in the fresh norm: of the pair that holds row j its second row, or none
            const f2 edge = (j & 1) ? 0ull : 0xFFFFFFFF00000000ull;
            ffp a[3] = {{0ull, 0ull}, {0ull, 0ull}, {0ull, 0ull}};
#pragma unroll
            for (int i = 0; i < NP; i += 3)
                if (64 * WPC * (i + 3) > j) {
#pragma unroll
                    for (int u = 0; u < 3; ++u) {
                        const int q = pair_of(i + u);
                        const ulonglong2 v = vs[q];
                        const ffp x = update2({ch[i + u], cl[i + u]}, w2, {v.x, v.y});
                        ch[i + u] = x.h;
                        cl[i + u] = x.l;
                        if (q >= qn && q < npk) st_packet(dst + q, x, ntag);
                        const f2 keep = q > q0 ? ~0ull : q == q0 ? edge : 0ull;
                        const ffp y = {x.h & keep, x.l & keep};
                        dot_acc2(a[u], y, y);
                    }
                }
            nsq = column_sum(warp_total(sum3(a)), nsq_s);
            if (lane == 0 && part == 0)
                st_word(p.nrm + (size_t)(par ^ 1) * m + col, pack2(nsq.hi, nsq.lo), (unsigned long long)(uint32_t)(j + 2));
        }
    }
    // R[:, pos] = rows 0 .. pos of the retired column, scaled back by 2^E
    if (!mine || pos < 0) return;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const int r0 = 2 * pair_of(i);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int row = r0 + u;
            if (row >= m) continue;
            const ff x = row == pos ? alpha_mine : u ? ff{hi2(ch[i]), hi2(cl[i])} : ff{lo2(ch[i]), lo2(cl[i])};
            p.R[(int64_t)row * m + pos] = row <= pos ? ldexp(ff_to_double(x), E) : 0.0;
        }
    }
}

struct Shape {
    const void* kern;
    int np, wpc, maxw;
};

}  // namespace

// Workspace: the packets, the records, the norms and the scale exchange.
size_t qr_ff_work_doubles(int m, int l) {
    const size_t npk = ((size_t)l + 1) / 2;
    return 2 * (2 * (size_t)m * npk) + 2 * 6 * (size_t)m + (size_t)m + 64;
}

cudaError_t pivoted_qr_ff_regs(const double* S, int m, int l, int64_t lds, double* R, int32_t* perm, double* work,
                               int* status, cudaStream_t s, long long spin_limit, int* fallback, bool* launched) {
    *launched = false;
    int dev = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    const int sms = sm_count();
    if (!coop) return cudaSuccess;
    // Warps per column, and rows a lane holds. Four columns a CTA while that fits the chip, more beyond.
    const Shape shapes[] = {{(const void*)qr_ff_kernel<3, 1, 16>, 3, 1, 16}, {(const void*)qr_ff_kernel<6, 1, 16>, 6, 1, 16},
                            {(const void*)qr_ff_kernel<9, 1, 16>, 9, 1, 16}, {(const void*)qr_ff_kernel<6, 2, 16>, 6, 2, 16},
                            {(const void*)qr_ff_kernel<12, 1, 16>, 12, 1, 16}, {(const void*)qr_ff_kernel<9, 2, 16>, 9, 2, 16},
                            {(const void*)qr_ff_kernel<12, 2, 16>, 12, 2, 16}, {(const void*)qr_ff_kernel<24, 1, 12>, 24, 1, 12},
                            {(const void*)qr_ff_kernel<9, 4, 16>, 9, 4, 16}, {(const void*)qr_ff_kernel<33, 1, 8>, 33, 1, 8}};
    const int cpc = std::max((m + sms - 1) / sms, std::min(4, m));
    const int G = (m + cpc - 1) / cpc;
    const Shape* sh = nullptr;
    for (const Shape& x : shapes)
        if (l <= 64 * x.np * x.wpc && cpc * x.wpc <= x.maxw) { sh = &x; break; }
    if (!sh) return cudaSuccess;
    const int nt = 32 * std::max(cpc * sh->wpc, 4);   // at least 128 threads load the pivot column's packets
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sh->kern, nt, 0) != cudaSuccess || per_sm < 1 ||
        G > per_sm * sms) {
        cudaGetLastError();
        return cudaSuccess;
    }
    QrFfDev p;
    p.S = S; p.m = m; p.l = l; p.lds = lds; p.R = R; p.perm = perm; p.cpc = cpc;
    const size_t npk = ((size_t)l + 1) / 2;
    ulonglong2* w = reinterpret_cast<ulonglong2*>(work);
    p.slots = w;      w += 2 * (size_t)m * npk;
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
    e = cudaLaunchCooperativeKernel(sh->kern, dim3((unsigned)G), dim3((unsigned)nt), args, 0, s);
    note_launch();
    if (e != cudaSuccess) {
        cudaGetLastError();   // clear; the caller's other kernels run
        return cudaSuccess;
    }
    *launched = true;
    return cudaSuccess;
}

}  // namespace rtp
