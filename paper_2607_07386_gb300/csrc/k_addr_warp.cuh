// K-ADDR, device code that several kernels share: list conventions, compensated and float64
// rescoring, band resolution, and the warp finalize of one token-side (k <= 32).
#pragma once
#include "sdm_internal.h"

#include <float.h>
#include <limits.h>

namespace sdm {

constexpr int FW_WARPS = 8;    // warps (= token-sides) per finalize CTA (k <= 32)

// Per-chunk top-L lists: entry p of token u, chunk `chunk` of (side, head) z is at
// ((z * 2 ncc + chunk) * BT + u) * L + p  (a token's L entries are contiguous).
__host__ __device__ __forceinline__ int64_t part_at(int z, int ncc, int chunk, int64_t BT, int64_t u, int L, int p) {
    return ((static_cast<int64_t>(z) * (2 * ncc) + chunk) * BT + u) * L + p;
}

// Sorted (value desc, index asc) list of the L best entries seen so far; empty = -inf.
template <int L>
struct TopList {
    float v[L];
    int i[L];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int p = 0; p < L; ++p) { v[p] = -INFINITY; i[p] = INT_MAX; }
    }
    __device__ __forceinline__ static bool beats(float a, int ia, float b, int ib) {
        return (a > b) || (a == b && ia < ib);
    }
    __device__ __forceinline__ bool admits(float x, int ix) const { return beats(x, ix, v[L - 1], i[L - 1]); }
    // General insertion (caller checked admits()).
    __device__ __forceinline__ void push(float x, int ix) {
#pragma unroll
        for (int p = 0; p < L; ++p) {
            const bool b = beats(x, ix, v[p], i[p]);
            const float tv = v[p];
            const int ti = i[p];
            v[p] = b ? x : tv; i[p] = b ? ix : ti;
            x = b ? tv : x;   ix = b ? ti : ix;
        }
    }
    // Insertion when every present entry has a smaller index than ix (scan order):
    // equal values never move, so a strict compare suffices.
    __device__ __forceinline__ void push_scan(float x, int ix) {
#pragma unroll
        for (int p = 0; p < L; ++p) {
            const bool b = x > v[p];
            const float tv = v[p];
            const int ti = i[p];
            v[p] = b ? x : tv; i[p] = b ? ix : ti;
            x = b ? tv : x;   ix = b ? ti : ix;
        }
    }
};

// ------------------------------------------------------------------------------------------
// Kernel B helpers
// ------------------------------------------------------------------------------------------
struct TokenCtx {
    int* err;           // device status word / counters
    unsigned* stat;     // per-warp event counters in shared memory (nullptr: count in err directly)
    bool count_band;    // count band events (false when an earlier pass counted them)
    const void* P;      // P of this side (nullptr = DIRECT)
    const void* X;
    int64_t xoff;       // element offset of the token's x row
    int64_t prow0;      // row of P for column 0 of half 0 (= h * 2S)
    int dk, S;
};

// Event counter (called by one lane): per-warp shared counters, flushed once per warp,
// keep the diagnostics off the global atomic unit.
__device__ __forceinline__ void tstat(const TokenCtx& c, int which, unsigned n = 1u) {
    if (c.stat) c.stat[which] += n;
    else stat_add(c.err, which, n);
}

// Column of a list entry to score: entries of lists short of numbers (inputs of infinities and NaN) can hold none.
__device__ __forceinline__ int in_half(int j, int S) { return static_cast<int>(min(static_cast<unsigned>(j), static_cast<unsigned>(S - 1))); }

// Float64 score of column j of half hf, summed over d in ascending order.  The loads of a row's pieces go out
// four at a time ahead of the sum (a rare pass of one near-tie, k = 16: 56 to 50 us; of 24 with k = 32: 71 to 61).
template <class D>
__device__ __noinline__ double score64(const TokenCtx& c, int hf, int j) {
    j = in_half(j, c.S);
    if (c.P == nullptr) return static_cast<double>(load_elem<D>(c.X, c.xoff + static_cast<int64_t>(hf) * c.S + j));
    const int64_t prow = (c.prow0 + static_cast<int64_t>(hf) * c.S + j) * c.dk;
    const char* const pr = static_cast<const char*>(c.P) + prow * D::BYTES;
    const char* const xr = static_cast<const char*>(c.X) + c.xoff * D::BYTES;
    const int nq = c.dk * D::BYTES / 16;
    double acc = 0.0;
    int d = 0;
    if (((reinterpret_cast<uintptr_t>(pr) | reinterpret_cast<uintptr_t>(xr)) & 15) == 0) {
        for (int q0 = 0; q0 + 4 <= nq; q0 += 4, d += 4 * D::E) {
            uint4 pq[4], xq[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                pq[u] = __ldg(reinterpret_cast<const uint4*>(pr) + q0 + u);
                xq[u] = __ldg(reinterpret_cast<const uint4*>(xr) + q0 + u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float fp[D::E], fx[D::E];
                unpack16<D>(pq[u], fp);
                unpack16<D>(xq[u], fx);
#pragma unroll
                for (int e = 0; e < D::E; ++e) acc = fma(static_cast<double>(fp[e]), static_cast<double>(fx[e]), acc);
            }
        }
    }
    for (; d < c.dk; ++d)
        acc = fma(static_cast<double>(load_elem<D>(c.P, prow + d)), static_cast<double>(load_elem<D>(c.X, c.xoff + d)), acc);
    return acc;
}

__device__ __forceinline__ bool beats64(double a, int ia, double b, int ib) { return (a > b) || (a == b && ia < ib); }

// Uncertified half boundary: decide the band in float64.  lv/li: top-L by fp32 (sorted).  A list ends in
// (-inf, none) where the half has fewer than L scores above -inf; a band that reaches these entries
// (fewer than k scores above -inf: masked ones are among the k best) is read off the whole half.
// Writes the exact top-k (ordered by fp32 value, desc) to Av/Ai with pitch F_THREADS.
template <class D, int L>
__device__ __noinline__ void resolve_half(const float* lv, const int* li, int k, double eps, const TokenCtx& c, int hf,
                                          float* Av, int* Ai, int pitch) {
    const double lo = static_cast<double>(lv[k - 1]) - 2.0 * eps;
    const double hi = static_cast<double>(lv[k]) + 2.0 * eps;
    if (static_cast<double>(lv[L - 1]) >= lo && (c.S > L || lv[L - 1] == -INFINITY)) {
        // Band may extend past the list: exact top-k of the whole half in float64.
        double bv[64 + 4];
        int bi[64 + 4];
        int n = 0;
        for (int j = 0; j < c.S; ++j) {
            const double s = score64<D>(c, hf, j);
            if (s != s || (n == k && !beats64(s, j, bv[k - 1], bi[k - 1]))) continue;      // (a NaN is never selected)
            int p = (n < k) ? n++ : k - 1;
            while (p > 0 && beats64(s, j, bv[p - 1], bi[p - 1])) { bv[p] = bv[p - 1]; bi[p] = bi[p - 1]; --p; }
            bv[p] = s; bi[p] = j;
        }
        for (int p = 0; p < k; ++p) {
            Av[p * pitch] = p < n ? static_cast<float>(bv[p]) : -INFINITY;
            Ai[p * pitch] = p < n ? bi[p] : 0;
        }
        return;
    }
    int cin = 0;
    while (cin < L && static_cast<double>(lv[cin]) > hi) ++cin;
    int pend = cin;
    while (pend < L && static_cast<double>(lv[pend]) >= lo) ++pend;
    double s64[L];
    bool used[L];
    for (int p = cin; p < pend; ++p) { s64[p] = score64<D>(c, hf, li[p]); used[p] = false; }
    for (int p = 0; p < cin; ++p) { Av[p * pitch] = lv[p]; Ai[p * pitch] = li[p]; }
    // choose k - cin entries of the band by (float64 desc, index asc) ...
    int chosen[L];
    const int need = k - cin;
    for (int r = 0; r < need; ++r) {
        int best = -1;
        for (int p = cin; p < pend; ++p)
            if (!used[p] && (best < 0 || beats64(s64[p], li[p], s64[best], li[best]))) best = p;
        if (best < 0) {                 // list not sorted by value: never for the lists built here
            flag_error(c.err, ERR_SELECT);
            chosen[r] = -1;
            continue;
        }
        used[best] = true;
        chosen[r] = best;
    }
    // ... and keep them in fp32-value order (they all lie below the certain entries)
    for (int r = 0; r < need; ++r) {
        int best = -1;
        for (int q = 0; q < need; ++q) {
            const int p = chosen[q];
            if (p >= 0 && (best < 0 || TopList<L>::beats(lv[p], li[p], lv[chosen[best]], li[chosen[best]]))) best = q;
        }
        if (best < 0) {
            Av[(cin + r) * pitch] = -INFINITY;
            Ai[(cin + r) * pitch] = 0;
            continue;
        }
        Av[(cin + r) * pitch] = lv[chosen[best]];
        Ai[(cin + r) * pitch] = li[chosen[best]];
        chosen[best] = -1;
    }
}

// Uncertified combined boundary.  cv/cf: top-L candidates by fp32 (sorted).  A1/A2: the two
// exact half lists.  Writes the exact top-k (fp32 score, slot) to Fv/Fi.
template <class D, int L>
__device__ __noinline__ void resolve_combined(const float* cv, const int* cf, int k, double epsc, const TokenCtx& c,
                                              const float* A1v, const int* A1i, const float* A2v, const int* A2i,
                                              float* Fv, int* Fi, int pitch) {
    const int S = c.S;
    const double lo = static_cast<double>(cv[k - 1]) - 2.0 * epsc;
    const double hi = static_cast<double>(cv[k]) + 2.0 * epsc;
    if (static_cast<double>(cv[L - 1]) >= lo) {
        // All k^2 candidates in float64 (also where sums of -inf are among the k best).
        double s1[64], s2[64];
        for (int p = 0; p < k; ++p) { s1[p] = score64<D>(c, 0, A1i[p * pitch]); s2[p] = score64<D>(c, 1, A2i[p * pitch]); }
        double bv[64];
        int bf[64], bp1[64], bp2[64];
        int n = 0;
        for (int p1 = 0; p1 < k; ++p1)
            for (int p2 = 0; p2 < k; ++p2) {
                const double s = s1[p1] + s2[p2];
                const int f = A1i[p1 * pitch] * S + A2i[p2 * pitch];
                if (n == k && !beats64(s, f, bv[k - 1], bf[k - 1])) continue;
                int p = (n < k) ? n++ : k - 1;
                while (p > 0 && beats64(s, f, bv[p - 1], bf[p - 1])) {
                    bv[p] = bv[p - 1]; bf[p] = bf[p - 1]; bp1[p] = bp1[p - 1]; bp2[p] = bp2[p - 1]; --p;
                }
                bv[p] = s; bf[p] = f; bp1[p] = p1; bp2[p] = p2;
            }
        for (int p = 0; p < k; ++p) {
            Fv[p * pitch] = A1v[bp1[p] * pitch] + A2v[bp2[p] * pitch];
            Fi[p * pitch] = bf[p];
        }
        return;
    }
    int cin = 0;
    while (cin < L && static_cast<double>(cv[cin]) > hi) ++cin;
    int pend = cin;
    while (pend < L && static_cast<double>(cv[pend]) >= lo) ++pend;
    double s64[L];
    bool used[L];
    for (int p = cin; p < pend; ++p) {
        s64[p] = score64<D>(c, 0, cf[p] / S) + score64<D>(c, 1, cf[p] % S);
        used[p] = false;
    }
    for (int p = 0; p < cin; ++p) { Fv[p * pitch] = cv[p]; Fi[p * pitch] = cf[p]; }
    for (int r = cin; r < k; ++r) {
        int best = -1;
        for (int p = cin; p < pend; ++p)
            if (!used[p] && (best < 0 || beats64(s64[p], cf[p], s64[best], cf[best]))) best = p;
        if (best < 0) {                 // candidate list not sorted by value: never here
            flag_error(c.err, ERR_SELECT);
            Fv[r * pitch] = -INFINITY;
            Fi[r * pitch] = 0;
            continue;
        }
        used[best] = true;
        Fv[r * pitch] = cv[best];
        Fi[r * pitch] = cf[best];
    }
}

// ------------------------------------------------------------------------------------------
// Kernel B (k <= 32): one warp per token-side.  Lane p holds entry p (and p + 32) of a list.
//   merge of chunk lists: output rank = own position + number of entries of the other list
//     that come first (binary search across lanes), scattered through shared memory;
//   combined top-(k+4): exact k-way merge of the k rows i of the outer sum (lane i owns row
//     i, its head s1[i] + s2[j_i]); each step takes the largest head by a warp max-reduce of
//     order-preserving integer keys, ties to the smallest slot by a min-reduce;
//   softmax by warp reductions; ascending slot order by a 32-lane bitonic shuffle network.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t f2key(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key2f(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
// entry idx (< 64) of a list held two entries per lane (v0: idx < 32, v1: idx >= 32)
__device__ __forceinline__ float lane_get(float v0, float v1, int idx) {
    const float a = __shfl_sync(0xffffffffu, v0, idx & 31);
    const float b = __shfl_sync(0xffffffffu, v1, idx & 31);
    return idx < 32 ? a : b;
}
// number of the first L entries of a descending list that are > x (strict) or >= x
__device__ __forceinline__ int lane_count_before(float v0, float v1, int L, float x, bool strict) {
    int pos = 0;
#pragma unroll
    for (int step = 32; step >= 1; step >>= 1) {
        const int idx = pos + step - 1;
        const float v = lane_get(v0, v1, idx);
        const bool before = strict ? (v > x) : (v >= x);
        if (idx < L && before) pos += step;
    }
    return pos;
}

__device__ __forceinline__ int lane_geti(int i0, int i1, int idx) {
    const int a = __shfl_sync(0xffffffffu, i0, idx & 31);
    const int b = __shfl_sync(0xffffffffu, i1, idx & 31);
    return idx < 32 ? a : b;
}

// All decisions of the warp finalize run in fp32 (GB300's float64 rate is a small
// fraction of its fp32 rate): error bounds are rounded up and differences rounded down
// (directed-rounding intrinsics), so every "certain" decision is also certain in exact
// arithmetic.  float64 remains only in the serial fallbacks.

// Float-float value h + l (|l| <= ulp(h)/2) with an error bound b on its distance to the
// float64 score of the definition.
struct FF {
    float h, l, b;
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// Compensated score of column j of half hf, computed by the whole warp (every lane gets
// the result).  Lane l owns the terms d = l + 32 r (its x values are in xr).  Every product
// is split exactly (p + pe = P x; pe = 0 for bf16 operands) and every addition of the main
// sum -- within a lane and across the butterfly -- exactly by TwoSum; only the error terms
// are summed in plain fp32.  With n = d_k terms and u = 2^-24 the result s + e differs
// from the exact dot product by at most 2 n (n + 1) u^2 (1.03) sum|P x| <= 2^-31 sum|P x|
// for n <= 256, whatever the order of the additions.  The float64 sequential sum of the
// definition lies within (n - 1) 2^-53 sum|P x| of the exact value, so b = 2^-28 sum|P x|
// covers the distance to it with margin (also for the rounding of sum|P x| itself).
// DIRECT addressing: the score is x itself, exact.
template <class D>
__device__ FF ff_score_warp(const TokenCtx& c, const float (&xr)[8], int hf, int j, int lane) {
    j = in_half(j, c.S);
    if (c.P == nullptr) return FF{load_elem<D>(c.X, c.xoff + static_cast<int64_t>(hf) * c.S + j), 0.f, 0.f};
    const int64_t prow = (c.prow0 + static_cast<int64_t>(hf) * c.S + j) * c.dk;
    float pv[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int d = lane + 32 * r;
        pv[r] = (r * 32 < c.dk && d < c.dk) ? load_elem<D>(c.P, prow + d) : 0.f;
    }
    float sum = 0.f, err = 0.f, mag = 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        if (r * 32 < c.dk) {
            const float p = __fmul_rn(pv[r], xr[r]);
            const float pe = __fmaf_rn(pv[r], xr[r], -p);
            float t, e2;
            two_sum(sum, p, t, e2);
            sum = t;
            err = __fadd_rn(err, __fadd_rn(e2, pe));
            mag = __fadd_rn(mag, fabsf(p));
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float so = __shfl_xor_sync(0xffffffffu, sum, off);
        const float eo = __shfl_xor_sync(0xffffffffu, err, off);
        const float mo = __shfl_xor_sync(0xffffffffu, mag, off);
        float t, e2;
        two_sum(sum, so, t, e2);                   // same t and e2 in both lanes of the pair
        sum = t;
        err = __fadd_rn(__fadd_rn(err, eo), e2);   // (err + eo) is the same in both lanes
        mag = __fadd_rn(mag, mo);
    }
    FF r;
    r.h = __fadd_rn(sum, err);                      // FastTwoSum: |err| << |sum|
    r.l = __fsub_rn(err, __fsub_rn(r.h, sum));
    r.b = __fmul_ru(0x1p-28f, mag);
    return r;
}

// a + b for two compensated half scores (the float64 definition adds its two half scores
// with one more rounding of at most 2^-53 of the sum; 2^-44 |sum| covers that and ours).
__device__ __forceinline__ FF ff_add(const FF& a, const FF& b, bool direct) {
    float h, r;
    two_sum(a.h, b.h, h, r);
    const float l = __fadd_rn(__fadd_rn(a.l, b.l), r);
    FF o;
    o.h = __fadd_rn(h, l);
    o.l = __fsub_rn(l, __fsub_rn(o.h, h));
    const float slack = direct ? __fmul_ru(0x1p-52f, fabsf(o.h)) : __fmul_ru(0x1p-44f, fabsf(o.h));
    o.b = __fadd_ru(__fadd_ru(a.b, b.b), slack);
    return o;
}

// Band entries (lane e < m holds entry e: compensated score v, index id) are ranked under
// (score desc, index asc).  Returns false when two entries are closer than their bounds
// (the float64 definition must decide); otherwise the ranks are those of the float64
// definition.  The difference (hf + lf) - (h + l) is formed with TwoSum on the leading
// parts; the roundings of the rest are covered by `slack`.
__device__ __forceinline__ bool rank_band(const FF& v, int id, int m, int lane, int& rank) {
    rank = 0;
    bool unsure = false;
    for (int f = 0; f < m; ++f) {
        const float hf = __shfl_sync(0xffffffffu, v.h, f);
        const float lf = __shfl_sync(0xffffffffu, v.l, f);
        const float bf = __shfl_sync(0xffffffffu, v.b, f);
        const int jf = __shfl_sync(0xffffffffu, id, f);
        if (lane < m && f != lane) {
            float t, r;
            two_sum(hf, -v.h, t, r);
            const float w = __fadd_rn(__fsub_rn(lf, v.l), r);
            const float diff = __fadd_rn(t, w);
            const float slack = __fmul_ru(0x1p-21f, __fadd_ru(__fadd_ru(fabsf(t), fabsf(r)), __fadd_ru(fabsf(lf), fabsf(v.l))));
            const float tol = __fadd_ru(__fadd_ru(bf, v.b), slack);
            if (tol > 0.f && fabsf(diff) <= tol) unsure = true;
            else rank += (diff > 0.f || (diff == 0.f && jf < id)) ? 1 : 0;
        }
    }
    return !__any_sync(0xffffffffu, unsure);
}

// Band of an uncertified top-k boundary in a list of `len` (<= 64) entries sorted by fp32
// value (lane p: entry p in v0/i0, entry p + 32 in v1/i1): entries [cin, cin + m) lie
// within e2 (twice the error bound, rounded up) of the boundary.  False if the band may
// continue past the list, reaches its padding (-inf) or holds more than 32 entries.
__device__ __forceinline__ bool band_of(float v0, float v1, int len, int k, float e2, bool list_is_all, int lane,
                                        int& cin, int& m) {
    const float lo = __fsub_rd(lane_get(v0, v1, k - 1), e2);
    const float hi = __fadd_ru(lane_get(v0, v1, k), e2);
    const float vl = lane_get(v0, v1, len - 1);
    if (vl >= lo && (!list_is_all || vl == -INFINITY)) return false;
    cin = __popc(__ballot_sync(0xffffffffu, lane < len && v0 > hi)) +
          __popc(__ballot_sync(0xffffffffu, lane + 32 < len && v1 > hi));
    m = __popc(__ballot_sync(0xffffffffu, lane < len && v0 >= lo && v0 <= hi)) +
        __popc(__ballot_sync(0xffffffffu, lane + 32 < len && v1 >= lo && v1 <= hi));
    return m <= 32;
}

// Writes the certain entries [0, cin) and the chosen band entries (in list order) to ov/oi.
__device__ __forceinline__ void emit_band(float v0, int i0, float bv, int bi, bool chosen, int cin, float* ov, int* oi,
                                          int lane) {
    const unsigned ch = __ballot_sync(0xffffffffu, chosen);
    __syncwarp();
    if (lane < cin) { ov[lane] = v0; oi[lane] = i0; }
    if (chosen) {
        const int q = cin + __popc(ch & ((1u << lane) - 1u));
        ov[q] = bv;
        oi[q] = bi;
    }
    __syncwarp();
}

// Warp-cooperative resolution of an uncertified half boundary (e2 = twice the fp32 error
// bound of the scores).  On success writes the exact top-k, in fp32-list order, to
// ov/oi[0, k) and returns true; false when the serial float64 path must decide (band past
// the list, more than 32 band entries, or a near-tie).
enum : int { BAND_DONE = 0, BAND_NEAR_TIE = 1, BAND_OUTSIDE = 2 };

// x[lane + 32 r] of the token (projected mode) for the warp-cooperative rescoring
template <class D>
__device__ __forceinline__ void load_xr(const TokenCtx& c, int lane, float (&xr)[8]) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int d = lane + 32 * r;
        xr[r] = (c.P != nullptr && r * 32 < c.dk && d < c.dk) ? load_elem<D>(c.X, c.xoff + d) : 0.f;
    }
}

// Band resolvers.  The common-path kernel (MODE 0) does not contain them.
template <class D, int L>
__device__ __forceinline__ int warp_band_half(float v0, int i0, float v1, int i1, int k, float e2, const TokenCtx& c,
                                           int hf, float* ov, int* oi, int lane) {
    float xr[8];
    load_xr<D>(c, lane, xr);
    int cin, m;
    if (!band_of(v0, v1, L, k, e2, c.S <= L, lane, cin, m)) return BAND_OUTSIDE;
    if (lane == 0 && c.count_band) tstat(c, STAT_HALF_BAND_ENTRIES, static_cast<unsigned>(m));
    const int p = min(cin + lane, L - 1);
    const float bv = lane_get(v0, v1, p);
    const int bi = lane_geti(i0, i1, p);
    FF mine{0.f, 0.f, 0.f};
    for (int e = 0; e < m; ++e) {
        const FF sc = ff_score_warp<D>(c, xr, hf, __shfl_sync(0xffffffffu, bi, e), lane);
        if (lane == e) mine = sc;
    }
    int rank;
    if (!rank_band(mine, bi, m, lane, rank)) return BAND_NEAR_TIE;
    emit_band(v0, i0, bv, bi, lane < m && rank < k - cin, cin, ov, oi, lane);
    return BAND_DONE;
}

// Near-tie in the band: float64 scores of the definition (sequential d order, so equal to
// it bit for bit), one lane per band entry; the ranking is then exact.
template <class D>
__device__ __noinline__ void warp_band64(float v0, int i0, float v1, int i1, int len, int k, float e2, bool all,
                                         bool comb, const TokenCtx& c, int hf, float* ov, int* oi, int lane) {
    int cin, m;
    band_of(v0, v1, len, k, e2, all, lane, cin, m);       // succeeded before with the same arguments
    const int p = min(cin + lane, len - 1);
    const float bv = lane_get(v0, v1, p);
    const int bi = lane_geti(i0, i1, p);
    double s64 = 0.0;
    if (lane < m) s64 = comb ? score64<D>(c, 0, bi / c.S) + score64<D>(c, 1, bi % c.S) : score64<D>(c, hf, bi);
    int rank = 0;
    for (int f = 0; f < m; ++f) {
        const double sf = __shfl_sync(0xffffffffu, s64, f);
        const int jf = __shfl_sync(0xffffffffu, bi, f);
        if (lane < m && f != lane && beats64(sf, jf, s64, bi)) ++rank;
    }
    emit_band(v0, i0, bv, bi, lane < m && rank < k - cin, cin, ov, oi, lane);
}

// Descending bitonic sort of 64 floats held two per lane (element lane in a, lane + 32 in b).
__device__ __forceinline__ void warp_sort64_desc(float& a, float& b, int lane) {
#pragma unroll
    for (int size = 2; size <= 64; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride == 32) {                                 // elements lane and lane + 32
                const float hi = fmaxf(a, b), lo = fminf(a, b);
                a = hi; b = lo;                                 // size == 64: descending
            } else {
                const float pa = __shfl_xor_sync(0xffffffffu, a, stride);
                const float pb = __shfl_xor_sync(0xffffffffu, b, stride);
                const bool lower = (lane & stride) == 0;
                // element e = lane (+ 32): its block of `size` sorts descending iff (e & size) == 0
                const bool desc_a = (lane & size) == 0;
                const bool desc_b = ((lane + 32) & size) == 0;
                a = (lower == desc_a) ? fmaxf(a, pa) : fminf(a, pa);
                b = (lower == desc_b) ? fmaxf(b, pb) : fminf(b, pb);
            }
        }
    }
}

// Compensated score of column j of half hf by one thread (16-byte loads when aligned); the
// same error-free splitting and the same 2^-28 sum|P x| bound as ff_score_warp.
template <class D>
__device__ FF ff_score_thread(const void* P, const void* X, int64_t xoff, int64_t prow0, int dk, int S, int hf, int j) {
    j = in_half(j, S);
    if (P == nullptr) return FF{load_elem<D>(X, xoff + static_cast<int64_t>(hf) * S + j), 0.f, 0.f};
    const int64_t prow = (prow0 + static_cast<int64_t>(hf) * S + j) * dk;
    float sum = 0.f, err = 0.f, mag = 0.f;
    auto term = [&](float pv, float xv) {
        const float p = __fmul_rn(pv, xv);
        const float pe = __fmaf_rn(pv, xv, -p);
        float t, e2;
        two_sum(sum, p, t, e2);
        sum = t;
        err = __fadd_rn(err, __fadd_rn(e2, pe));
        mag = __fadd_rn(mag, fabsf(p));
    };
    const char* pr = static_cast<const char*>(P) + prow * D::BYTES;
    const char* xr = static_cast<const char*>(X) + xoff * D::BYTES;
    if (((reinterpret_cast<uintptr_t>(pr) | reinterpret_cast<uintptr_t>(xr)) & 15) == 0 && (dk * D::BYTES) % 16 == 0) {
        const int nq = dk * D::BYTES / 16;
        for (int q0 = 0; q0 < nq; q0 += 4) {            // four 16-byte loads in flight per operand
            uint4 pq[4], xq[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q0 + u < nq) {
                    pq[u] = __ldg(reinterpret_cast<const uint4*>(pr) + q0 + u);
                    xq[u] = __ldg(reinterpret_cast<const uint4*>(xr) + q0 + u);
                }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q0 + u < nq) {
                    float fp[D::E], fx[D::E];
                    unpack16<D>(pq[u], fp);
                    unpack16<D>(xq[u], fx);
#pragma unroll
                    for (int e = 0; e < D::E; ++e) term(fp[e], fx[e]);
                }
        }
    } else {
        for (int d = 0; d < dk; ++d) term(load_elem<D>(P, prow + d), load_elem<D>(X, xoff + d));
    }
    FF r;
    r.h = __fadd_rn(sum, err);
    r.l = __fsub_rn(err, __fsub_rn(r.h, sum));
    r.b = __fmul_ru(0x1p-28f, mag);
    return r;
}

// The band of a half boundary reaches past the kept list: exact top-k over the whole half,
// one column per lane at a time.
//   pass 1: fp32 scores (sequential FMA, error <= eps), each lane keeps the top 2 of its
//           columns j = lane (mod 32); theta = k-th largest of those 64 values (>= k columns
//           reach it, so the k-th largest exact score is >= theta - eps);
//   pass 2: columns with fp32 score >= theta - 2 eps (a superset of the exact top-k) are
//           collected (at most 64, else false), rescored compensated and ranked.
// Writes the top-k in order (value fl32 of the compensated score, index) to ov/oi.
template <class D>
__device__ __noinline__ bool warp_full_half(int k, float e2, const TokenCtx& c, int hf, float* ov, int* oi,
                                            int* scratch, int lane) {
    const int S = c.S;
    const char* xr = static_cast<const char*>(c.X) + c.xoff * D::BYTES;
    const bool vec = ((reinterpret_cast<uintptr_t>(c.P) | reinterpret_cast<uintptr_t>(xr)) & 15) == 0 &&
                     (c.dk * D::BYTES) % 16 == 0;
    auto fp32_score = [&](int j) -> float {             // sequential FMA over d (error <= eps)
        const int64_t prow = (c.prow0 + static_cast<int64_t>(hf) * S + j) * c.dk;
        float acc = 0.f;
        if (vec) {
            const uint4* pr = reinterpret_cast<const uint4*>(static_cast<const char*>(c.P) + prow * D::BYTES);
            for (int q = 0; q < c.dk * D::BYTES / 16; ++q) {
                float fp[D::E], fx[D::E];
                unpack16<D>(__ldg(pr + q), fp);
                unpack16<D>(__ldg(reinterpret_cast<const uint4*>(xr) + q), fx);
#pragma unroll
                for (int e = 0; e < D::E; ++e) acc = fmaf(fp[e], fx[e], acc);
            }
        } else {
            for (int d = 0; d < c.dk; ++d) acc = fmaf(load_elem<D>(c.P, prow + d), load_elem<D>(c.X, c.xoff + d), acc);
        }
        return acc;
    };
    float t1 = -INFINITY, t2 = -INFINITY;
    for (int j0 = 0; j0 < S; j0 += 32) {
        const int j = j0 + lane;
        const float sc = j < S ? fmaxf(fp32_score(j), -INFINITY) : -INFINITY;      // (NaN: -inf)
        t2 = fmaxf(t2, fminf(t1, sc));
        t1 = fmaxf(t1, sc);
    }
    warp_sort64_desc(t1, t2, lane);
    const float theta = lane_get(t1, t2, k - 1);
    const float lo = __fsub_rd(theta, e2);
    int m = 0;
    for (int j0 = 0; j0 < S; j0 += 32) {
        const int j = j0 + lane;
        const bool keep = j < S && fp32_score(j) >= lo;
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        const int pos = m + __popc(mask & ((1u << lane) - 1u));
        if (keep && pos < 64) scratch[pos] = j;
        m += __popc(mask);
    }
    if (m > 64 || m < k) return false;
    __syncwarp();
    const int j0 = lane < m ? scratch[lane] : 0;
    const int j1 = lane + 32 < m ? scratch[lane + 32] : 0;
    __syncwarp();
    FF f0{0.f, 0.f, 0.f}, f1{0.f, 0.f, 0.f};
    if (lane < m) f0 = ff_score_thread<D>(c.P, c.X, c.xoff, c.prow0, c.dk, S, hf, j0);
    if (lane + 32 < m) f1 = ff_score_thread<D>(c.P, c.X, c.xoff, c.prow0, c.dk, S, hf, j1);
    // rank both own entries against all m (pairs closer than their bounds: give up)
    int r0 = 0, r1 = 0;
    bool unsure = false;
    for (int f = 0; f < m; ++f) {
        const int src = f & 31;
        const bool hi = f >= 32;
        const float hA = __shfl_sync(0xffffffffu, f0.h, src), hB = __shfl_sync(0xffffffffu, f1.h, src);
        const float lA = __shfl_sync(0xffffffffu, f0.l, src), lB = __shfl_sync(0xffffffffu, f1.l, src);
        const float bA = __shfl_sync(0xffffffffu, f0.b, src), bB = __shfl_sync(0xffffffffu, f1.b, src);
        const FF ff{hi ? hB : hA, hi ? lB : lA, hi ? bB : bA};
        const int jf = lane_geti(j0, j1, f);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = lane + 32 * q;
            const FF& mine = q ? f1 : f0;
            const int je = q ? j1 : j0;
            if (e < m && e != f) {
                float t, r;
                two_sum(ff.h, -mine.h, t, r);
                const float w = __fadd_rn(__fsub_rn(ff.l, mine.l), r);
                const float diff = __fadd_rn(t, w);
                const float slack = __fmul_ru(0x1p-21f, __fadd_ru(__fadd_ru(fabsf(t), fabsf(r)), __fadd_ru(fabsf(ff.l), fabsf(mine.l))));
                const float tol = __fadd_ru(__fadd_ru(ff.b, mine.b), slack);
                if (tol > 0.f && fabsf(diff) <= tol) unsure = true;
                else if (diff > 0.f || (diff == 0.f && jf < je)) { if (q) ++r1; else ++r0; }
            }
        }
    }
    if (__any_sync(0xffffffffu, unsure)) return false;
    __syncwarp();
    if (lane < m && r0 < k) { ov[r0] = f0.h; oi[r0] = j0; }
    if (lane + 32 < m && r1 < k) { ov[r1] = f1.h; oi[r1] = j1; }
    __syncwarp();
    return true;
}

// Same for the outer-sum boundary over a candidate list of `len` (<= 64) entries: slot
// f = i S + j is rescored as the sum of the compensated half scores of column i (half 0)
// and column j (half 1).
template <class D>
__device__ __forceinline__ int warp_band_comb(float v0, int f0, float v1, int f1, int len, int k, float e2c,
                                           const TokenCtx& c, bool all, float* ov, int* oi, int lane) {
    float xr[8];
    load_xr<D>(c, lane, xr);
    int cin, m;
    if (!band_of(v0, v1, len, k, e2c, all, lane, cin, m)) return BAND_OUTSIDE;
    if (lane == 0 && c.count_band) tstat(c, STAT_COMB_BAND_ENTRIES, static_cast<unsigned>(m));
    const int p = min(cin + lane, len - 1);
    const float bv = lane_get(v0, v1, p);
    const int bf = lane_geti(f0, f1, p);
    FF mine{0.f, 0.f, 0.f};
    for (int e = 0; e < m; ++e) {
        const int fe = __shfl_sync(0xffffffffu, bf, e);
        const FF s1 = ff_score_warp<D>(c, xr, 0, fe / c.S, lane);
        const FF s2 = ff_score_warp<D>(c, xr, 1, fe % c.S, lane);
        const FF sum = ff_add(s1, s2, c.P == nullptr);
        if (lane == e) mine = sum;
    }
    int rank;
    if (!rank_band(mine, bf, m, lane, rank)) return BAND_NEAR_TIE;
    emit_band(v0, f0, bv, bf, lane < m && rank < k - cin, cin, ov, oi, lane);
    return BAND_DONE;
}

// Passes of the warp finalize (see k_addr_finalize).
enum : int { FIN_FAST = 0, FIN_BAND = 1, FIN_FULL = 2 };

// One token-side by one warp: certifies both halves' lists (load(hf, v0, i0, v1, i1): lane p gets
// entries p and p + 32), enumerates the outer sum, certifies its boundary, writes the slots in
// ascending order and their softmax.  e2: twice the fp32 score error bound.  sv*/si*: 64 words of the
// warp's shared memory each.  False (nothing written) when MODE leaves the item to a later pass.
template <class D, int L, int MODE, class Load>
__device__ __forceinline__ bool finalize_warp(const TokenCtx& c, int k, float e2, int32_t* idx_out, float* w_out,
                                              float* sv0, int* si0, float* sv1, int* si1, float* sv2, int* si2, int lane,
                                              Load load) {
    const int S = c.S;
    const double eps = 0.5 * static_cast<double>(e2);      // for the serial float64 fallbacks
    float av[2], bv[2];      // A1 and A2 after certification: lane p holds entry p (p < k)
    int ai[2], bi[2];
    float amax[2];
#pragma unroll 1
    for (int hf = 0; hf < 2; ++hf) {
        float v0, v1;
        int i0, i1;
        load(hf, v0, i0, v1, i1);
        // certify the boundary between entries k-1 and k (warp-uniform decision)
        const float vk = lane_get(v0, v1, k - 1);
        bool certified = S <= k && vk != -INFINITY;
        if (!certified) certified = __fsub_rd(vk, lane_get(v0, v1, k)) > e2;
        if (MODE == FIN_FAST && !certified) {
            return false;
        }
        if (!certified) {
            if (lane == 0 && c.count_band) tstat(c, STAT_HALF_BAND);
            const int res = warp_band_half<D, L>(v0, i0, v1, i1, k, e2, c, hf, sv0, si0, lane);
            bool done = res == BAND_DONE;
            if (MODE == FIN_BAND && !done) {
                return false;
            }
            if (res == BAND_NEAR_TIE) {
                if (lane == 0) tstat(c, STAT_BAND_F64);
                warp_band64<D>(v0, i0, v1, i1, L, k, e2, S <= L, false, c, hf, sv0, si0, lane);
                done = true;
            } else if (res == BAND_OUTSIDE) {
                if (lane == 0) tstat(c, STAT_HALF_FULL);
                done = c.P != nullptr && warp_full_half<D>(k, e2, c, hf, sv0, si0, si2, lane);
            }
            if (!done) {
                if (lane == 0) tstat(c, STAT_SERIAL);
                __syncwarp();
                if (lane < L) { sv0[lane] = v0; si0[lane] = i0; }
                if (lane + 32 < L) { sv0[lane + 32] = v1; si0[lane + 32] = i1; }
                __syncwarp();
                if (lane == 0) {
                    float lv[L];
                    int li[L];
                    for (int p = 0; p < L; ++p) { lv[p] = sv0[p]; li[p] = si0[p]; }
                    resolve_half<D, L>(lv, li, k, eps, c, hf, sv0, si0, 1);
                }
            }
            __syncwarp();
            v0 = lane < k ? sv0[lane] : -INFINITY;
            i0 = lane < k ? si0[lane] : INT_MAX;
        }
        if (hf == 0) { av[0] = lane < k ? v0 : -INFINITY; ai[0] = i0; }
        else { bv[0] = lane < k ? v0 : -INFINITY; bi[0] = i0; }
        amax[hf] = fmaxf(fabsf(lane_get(v0, v1, 0)), fabsf(lane_get(v0, v1, k - 1)));
    }
    // combined: k-way merge of the rows (lane i: row i; head = A1[i] + A2[j])
    // outer-sum bound: both half errors plus the fp32 rounding of A1 + A2 (rounded up, x2)
    const float e2c = __fadd_ru(__fmul_ru(2.f, e2), __fmul_ru(0x1p-21f, __fadd_ru(amax[0], amax[1])));
    const double epsc = 0.5 * static_cast<double>(e2c);  // for the serial float64 fallback
    int j = 0;
    const float b0v = __shfl_sync(0xffffffffu, bv[0], 0);
    const int b0i = __shfl_sync(0xffffffffu, bi[0], 0);
    float head = lane < k ? av[0] + b0v : -INFINITY;
    int flat = ai[0] * S + b0i;
    float nv = __shfl_sync(0xffffffffu, bv[0], 1);           // column j + 1 of A2, fetched beside the step before
    int ni = __shfl_sync(0xffffffffu, bi[0], 1);
    float cv0 = -INFINITY, cv1 = -INFINITY;    // candidate r in lane r (r < 32) / lane r-32
    int cf0 = INT_MAX, cf1 = INT_MAX;
    auto merge_steps = [&](int r0, int r1) {
        for (int r = r0; r < r1; ++r) {
            const uint32_t key = f2key(head);
            const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
            const bool tie = key == kmax;
            const uint32_t fmin = __reduce_min_sync(0xffffffffu, tie ? static_cast<uint32_t>(flat) : 0xffffffffu);
            const bool win = tie && static_cast<uint32_t>(flat) == fmin;
            const float val = key2f(kmax);
            const bool here = lane == (r & 31);
            cv0 = here && r < 32 ? val : cv0;
            cf0 = here && r < 32 ? static_cast<int>(fmin) : cf0;
            cv1 = here && r >= 32 ? val : cv1;
            cf1 = here && r >= 32 ? static_cast<int>(fmin) : cf1;
            j += win ? 1 : 0;
            const float nh = (j < k && lane < k) ? av[0] + nv : -INFINITY;
            const int nf = ai[0] * S + ni;
            head = win ? nh : head;
            flat = win ? nf : flat;
            nv = __shfl_sync(0xffffffffu, bv[0], (j + 1) & 31);
            ni = __shfl_sync(0xffffffffu, bi[0], (j + 1) & 31);
        }
    };
    merge_steps(0, k + 1);                                  // certification needs entries k-1 and k
    bool certified = (k == 1);
    if (!certified) {
        const float ck = lane_get(cv0, cv1, k - 1), ck1 = lane_get(cv0, cv1, k);
        // (k sums of numbers and no other; a NaN bound is that of a NaN input, whose order nothing decides)
        certified = (ck1 == -INFINITY && (ck != -INFINITY || e2c != e2c)) || (__fsub_rd(ck, ck1) > e2c);
    }
    float fv = cv0;
    int fi = cf0;
    if (MODE == FIN_FAST && !certified) {
        return false;
    }
    if (!certified) {
        if (lane == 0 && c.count_band) tstat(c, STAT_COMB_BAND);
        merge_steps(k + 1, L);
        // band may continue past the L candidates: extend the merge to 64 (or all k^2)
        int len = L;
        const float vl = lane_get(cv0, cv1, L - 1);
        if (k * k > L && vl != -INFINITY &&
            vl >= __fsub_rd(lane_get(cv0, cv1, k - 1), e2c)) {
            if (lane == 0) tstat(c, STAT_COMB_MERGE);
            len = min(64, k * k);
            merge_steps(L, len);
        }
        const int res = warp_band_comb<D>(cv0, cf0, cv1, cf1, len, k, e2c, c, len >= k * k, sv2, si2, lane);
        if (MODE == FIN_BAND && res != BAND_DONE) {
            return false;
        }
        if (res == BAND_NEAR_TIE) {
            if (lane == 0) tstat(c, STAT_BAND_F64);
            warp_band64<D>(cv0, cf0, cv1, cf1, len, k, e2c, len >= k * k, true, c, 0, sv2, si2, lane);
        } else if (res == BAND_OUTSIDE) {
            if (lane == 0) { tstat(c, STAT_COMB_FULL); tstat(c, STAT_SERIAL); }
            __syncwarp();
            sv0[lane] = av[0]; si0[lane] = ai[0];            // A1
            sv1[lane] = bv[0]; si1[lane] = bi[0];            // A2
            sv2[lane] = cv0; si2[lane] = cf0;                // candidates 0..31
            if (lane + 32 < L) { sv2[lane + 32] = cv1; si2[lane + 32] = cf1; }
            __syncwarp();
            if (lane == 0) {
                float cvl[L];
                int cfl[L];
                for (int p = 0; p < L; ++p) { cvl[p] = sv2[p]; cfl[p] = si2[p]; }
                resolve_combined<D, L>(cvl, cfl, k, epsc, c, sv0, si0, sv1, si1, sv2, si2, 1);
            }
        }
        __syncwarp();
        fv = lane < k ? sv2[lane] : -INFINITY;
        fi = lane < k ? si2[lane] : INT_MAX;
    }
    // softmax over the k selected scores
    if (lane >= k) { fv = -INFINITY; fi = INT_MAX; }
    const float m = key2f(__reduce_max_sync(0xffffffffu, f2key(fv)));
    float e = lane < k ? expf(fv - m) : 0.f;
    // ascending slot order: bitonic network across the 32 lanes
    int key = fi;
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const int pk = __shfl_xor_sync(0xffffffffu, key, stride);
            const float pe = __shfl_xor_sync(0xffffffffu, e, stride);
            const bool up = (lane & size) == 0;
            const bool lower = (lane & stride) == 0;
            const bool take_min = (up == lower);
            const bool mine = take_min ? (key <= pk) : (key >= pk);
            key = mine ? key : pk;
            e = mine ? e : pe;
        }
    }
    // summed in slot order by every pass, so that a token's weights do not depend on the pass that wrote them
    float zsum = 0.f;
#pragma unroll
    for (int r = 0; r < 32; ++r) zsum += __shfl_sync(0xffffffffu, e, r);   // (0 beyond k)
    if (lane < k) {
        idx_out[lane] = key;
        w_out[lane] = e / zsum;
    }
    return true;
}

}  // namespace sdm
