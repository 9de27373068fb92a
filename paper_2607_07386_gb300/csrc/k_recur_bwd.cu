// Backward of the sparse gated delta recurrence with in-place undo (App. A.3,
// "Memory-Efficient Backward").
//
// The forward (the recurrence kernels with an undo log) updates the memory in place and records, for every
// token t and write slot n, the row M_{t-1}[I^w_t[n]] its write overwrote.  The backward walks
// the tokens in reverse with the memory at M_t and an fp32 adjoint G = dL/dM_t of the rows
// touched so far (dense [N, d_v] per chain, zero elsewhere).  For L = sum_t <dy_t, y_t>:
//
//   read   y_t = sum_n rho_n M_t[r_n]:   d rho_n = <dy_t, M_t[r_n]>,  G[r_n] += rho_n dy_t
//   write  M_t[i] = r_i + beta w_i delta,  r_i = alpha M_{t-1}[i],  delta = v_t - sum_m w_m r_m:
//          d delta = beta sum_i w_i G_i,  d beta = sum_i w_i <G_i, delta>,
//          d w_i = beta <G_i, delta> - <r_i, d delta>,  d v_t = d delta,
//          d r_i = G_i - w_i d delta,  d alpha = sum_i <d r_i, M_{t-1}[i]>,
//          G[i] <- alpha d r_i,  M[i] <- M_{t-1}[i] (the undo)
//
// Storage rounding of the forward is not differentiated (the rows are the stored values).
//
// The log can also come back from a quantised snapshot (App. A.3: fp8 or int4 snapshots of
// the log for long sequences): k_undo_quantize codes every logged row with one float32 scale
// s = max|row| / top (448 for e4m3, 7 for int4) and codes round(row / s), all in float32 with
// correctly rounded operations; the backward then takes the logged row as the stored value of
// q * s (rounded to the storage type), for the chain rule and for the undo alike.
//
// Layout of the work: a conflict pass over all tokens at once, then one CTA per chain whose warps
// take (token, 32-element slice of d_v) pairs in reverse order (see k_recur_bwd below).  No waits
// on other CTAs.
#include "sdm_internal.h"

#include <cuda_fp8.h>

namespace sdm {

// The undo log as the backward reads it: Q = 0 the stored rows themselves; Q = 1 fp8 (e4m3)
// codes, one byte per element; Q = 2 int4 codes, two per byte (element 2i in the low nibble),
// two's complement; one float32 scale per row for Q > 0.
struct UndoLog {
    const void* rows;          // Q = 0: [rows][d_v] storage elements
    const uint8_t* codes;      // Q > 0: [rows][d_v] (fp8) or [rows][d_v / 2] (int4) bytes
    const float* scales;       // Q > 0: [rows]
};

template <class D> __device__ __forceinline__ float to_storage(float x);
template <> __device__ __forceinline__ float to_storage<F32>(float x) { return x; }
template <> __device__ __forceinline__ float to_storage<BF16>(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Quantised snapshot of the log.  A row is read as 16-byte vectors by `lpr` neighbouring lanes
// (the largest power of two that divides its vectors, at most 32), CPL vectors each, so a warp
// covers 32 / lpr rows and a thread keeps RPT of them in flight; the codes of a vector leave in one
// store of 2 to 8 bytes.  A row in, its codes and scale out is all the traffic (0.05 ms of HBM for
// 1 M rows of 128 bf16 to int4), but it is bound by instructions, which is why the arithmetic below
// is packed and divides once per row: 0.090 ms, 0.27 ms with an element per load and a division per
// element.
//
// Codes are round(fl32(x / s)) of a correctly rounded division.  The division is only carried out
// where it can decide: with r = fl32(x * fl32(1 / s)) the quotient lies within 2^-22 |r| of r, so
// when r (1 - 2^-20) and r (1 + 2^-20) round to the same code, that is the code (rounding is
// monotone); both roundings of a whole vector are formed as words, and their differences name
// the elements to divide.  (About half of the warps hold an element at half of its row's maximum,
// where bf16 values quotients in int4 meet 3.5.)  int4 rounds by adding M = 1.5 * 2^23 + 8 in one
// fused multiply-add, which leaves q + 8 (q the integer, ties to even) in the low bits; the sums of
// a vector are added up with weights 16^e and the offsets taken out of the total.  Rows whose
// scale is outside [2^-100, 2^100] (where 1 / s or r could leave the normal range) and rows with a
// NaN always divide.
constexpr float UQ_LO = 1.f - 0x1p-20f, UQ_HI = 1.f + 0x1p-20f;

// Largest magnitude of a vector's elements; NaN when one of them is NaN.
__device__ __forceinline__ float uq_max_nan(float a, float b) {
    float m;
    asm("max.NaN.f32 %0, %1, %2;\n" : "=f"(m) : "f"(a), "f"(b));
    return m;
}
__device__ __forceinline__ float uq_absmax(const uint4& u, F32) {
    return uq_max_nan(uq_max_nan(fabsf(__uint_as_float(u.x)), fabsf(__uint_as_float(u.y))),
                      uq_max_nan(fabsf(__uint_as_float(u.z)), fabsf(__uint_as_float(u.w))));
}
__device__ __forceinline__ float uq_absmax(const uint4& u, BF16) {
    auto ab = [](uint32_t w) {
        const uint32_t m = w & 0x7fff7fffu;
        return *reinterpret_cast<const __nv_bfloat162*>(&m);
    };
    const __nv_bfloat162 m = __hmax2_nan(__hmax2_nan(ab(u.x), ab(u.y)), __hmax2_nan(ab(u.z), ab(u.w)));
    return uq_max_nan(__low2float(m), __high2float(m));
}

// Element e of a vector.
template <class D> __device__ __forceinline__ float uq_elem(const uint4& u, int e);
template <> __device__ __forceinline__ float uq_elem<F32>(const uint4& u, int e) {
    return __uint_as_float(e == 0 ? u.x : e == 1 ? u.y : e == 2 ? u.z : u.w);
}
template <> __device__ __forceinline__ float uq_elem<BF16>(const uint4& u, int e) {
    const uint32_t w = e < 2 ? u.x : e < 4 ? u.y : e < 6 ? u.z : u.w;
    return __uint_as_float(e & 1 ? w & 0xffff0000u : w << 16);
}

// Codes of the E elements of a vector, low element first (w[1] only for 8 one-byte codes).
template <class D, int Q>
__device__ __forceinline__ void quant_vec(const uint4& raw, float s, float inv, bool divide, uint32_t (&w)[2]) {
    constexpr int E = D::E;
    constexpr int BITS = Q == 1 ? 8 : 4, PER = 32 / BITS;      // bits of a code, codes per word
    constexpr int NW = (E + PER - 1) / PER;
    float2 x[E / 2];
    unpack16x2<D>(raw, x);
    const float2 inv2 = make_float2(inv, inv), lo2 = make_float2(UQ_LO, UQ_LO), hi2 = make_float2(UQ_HI, UQ_HI);
    uint32_t lo[2] = {0u, 0u}, hi[2] = {0u, 0u};
    if constexpr (Q == 1) {
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            const float2 r = __fmul2_rn(x[e], inv2);
            lo[e >> 1] |= static_cast<uint32_t>(__nv_cvt_float2_to_fp8x2(__fmul2_rn(r, lo2), __NV_SATFINITE, __NV_E4M3)) << (16 * (e & 1));
            hi[e >> 1] |= static_cast<uint32_t>(__nv_cvt_float2_to_fp8x2(__fmul2_rn(r, hi2), __NV_SATFINITE, __NV_E4M3)) << (16 * (e & 1));
        }
    } else {
        constexpr float M = 12582912.f + 8.f;
        const float2 M2 = make_float2(M, M);
        uint32_t off = 0u;
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            const float2 r = __fmul2_rn(x[e], inv2);
            const float2 a = __ffma2_rn(r, lo2, M2), b = __ffma2_rn(r, hi2, M2);
            lo[0] += (__float_as_uint(a.x) << (8 * e)) + (__float_as_uint(a.y) << (8 * e + 4));
            hi[0] += (__float_as_uint(b.x) << (8 * e)) + (__float_as_uint(b.y) << (8 * e + 4));
            off += (0x4b400000u << (8 * e)) + (0x4b400000u << (8 * e + 4));
        }
        lo[0] = (lo[0] - off) ^ (E == 8 ? 0x88888888u : 0x8888u);
        hi[0] = (hi[0] - off) ^ (E == 8 ? 0x88888888u : 0x8888u);
    }
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        uint32_t open = divide ? 0xffffffffu >> (32 - BITS * (E < PER ? E : PER)) : lo[k] ^ hi[k];
        while (open != 0u) {
            const int e = (__ffs(open) - 1) / BITS;
            const uint32_t field = ((1u << BITS) - 1u) << (BITS * e);
            open &= ~field;
            const float y = __fdiv_rn(uq_elem<D>(raw, k * PER + e), s);
            uint32_t code;
            if constexpr (Q == 1) code = __nv_cvt_float_to_fp8(y, __NV_SATFINITE, __NV_E4M3);
            else code = static_cast<uint32_t>(min(max(__float2int_rn(y), -7), 7)) & 15u;
            lo[k] = (lo[k] & ~field) | (code << (BITS * e));
        }
        w[k] = lo[k];
    }
}

constexpr int UQ_THREADS = 256;

template <class D, int Q, int CPL, int RPT>
__global__ void __launch_bounds__(UQ_THREADS) k_undo_quantize(const uint4* __restrict__ undo, int64_t rows, int lpr_log2,
                                                              uint8_t* __restrict__ codes, float* __restrict__ scales) {
    constexpr int E = D::E;
    constexpr int CB = Q == 1 ? E : E / 2;                     // code bytes per vector
    const int lpr = 1 << lpr_log2, l = threadIdx.x & (lpr - 1);
    const int nvec = lpr * CPL;                                // vectors per row
    const int64_t stride = static_cast<int64_t>(gridDim.x) * (UQ_THREADS >> lpr_log2);
    const int64_t vstride = stride * nvec;
    const int64_t first = (static_cast<int64_t>(blockIdx.x) * UQ_THREADS + threadIdx.x) >> lpr_log2;
    // rows r, r + stride, ...: every lane of a warp makes the same number of passes (the shuffles
    // need them all), rows past the end are read as zeros and not stored
    const int64_t wfirst = (static_cast<int64_t>(blockIdx.x) * UQ_THREADS + (threadIdx.x & ~31)) >> lpr_log2;
    for (int64_t base = 0; wfirst + base < rows; base += stride * RPT) {
        uint4 raw[RPT][CPL];
        float am[RPT];
        const uint4* src0 = undo + (first + base) * nvec + l;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
#pragma unroll
            for (int c = 0; c < CPL; ++c)
                raw[q][c] = first + base + q * stride < rows ? __ldcs(src0 + q * vstride + c * lpr) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            am[q] = 0.f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) am[q] = uq_max_nan(am[q], uq_absmax(raw[q][c], D{}));
        }
        for (int off = lpr >> 1; off > 0; off >>= 1)
#pragma unroll
            for (int q = 0; q < RPT; ++q) am[q] = uq_max_nan(am[q], __shfl_xor_sync(0xffffffffu, am[q], off));
        // a NaN in a row: its maximum is that of the other entries
        bool nan = false;
#pragma unroll
        for (int q = 0; q < RPT; ++q) nan |= am[q] != am[q];
        if (__any_sync(0xffffffffu, nan)) {
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                float m = 0.f;
#pragma unroll
                for (int c = 0; c < CPL; ++c)
                    for (int e = 0; e < E; ++e) m = fmaxf(m, fabsf(uq_elem<D>(raw[q][c], e)));
                for (int off = lpr >> 1; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
                am[q] = m;
            }
        }
        nan = __any_sync(0xffffffffu, nan);
        // the scale of row q by the lanes l = q mod RPT of the row (one division per thread for all of
        // its rows), then handed round; lpr >= RPT (a row has at least four vectors, or CPL > 1)
        float mine = am[0];
#pragma unroll
        for (int q = 1; q < RPT; ++q) mine = (l & (RPT - 1)) == q ? am[q] : mine;
        const float s_m = mine > 0.f ? __fdiv_rn(mine, Q == 1 ? 448.f : 7.f) : 1.f;
        const float inv_m = __frcp_rn(s_m);
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int src = (threadIdx.x & 31 & ~(lpr - 1)) + q;
            const float s = __shfl_sync(0xffffffffu, s_m, src), inv = __shfl_sync(0xffffffffu, inv_m, src);
            const bool divide = nan || !(s >= 0x1p-100f && s <= 0x1p100f);
            const int64_t r = first + base + q * stride;
            if (r < rows) {
                if (l == 0) scales[r] = s;
                uint8_t* dst = codes + ((first + base) * nvec + q * vstride + l) * CB;
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    uint32_t w[2];
                    quant_vec<D, Q>(raw[q][c], s, inv, divide, w);
                    if constexpr (CB == 8) *reinterpret_cast<uint2*>(dst + c * lpr * CB) = make_uint2(w[0], w[1]);
                    else if constexpr (CB == 4) *reinterpret_cast<uint32_t*>(dst + c * lpr * CB) = w[0];
                    else *reinterpret_cast<unsigned short*>(dst + c * lpr * CB) = static_cast<unsigned short>(w[0]);
                }
            }
        }
    }
}

template <class D, int Q, int CPL>
static cudaError_t launch_uq_cpl(const void* undo, int64_t rows, int lpr_log2, uint8_t* codes, float* scales, int sms,
                                 cudaStream_t stream) {
    constexpr int RPT = CPL == 1 ? 4 : CPL == 2 ? 2 : 1;       // 16-byte loads in flight per thread
    const int64_t per_cta = (UQ_THREADS >> lpr_log2) * RPT;
    const int64_t want = (rows + per_cta - 1) / per_cta, cap = static_cast<int64_t>(sms) * 8;
    const unsigned grid = static_cast<unsigned>(want < cap ? (want > 0 ? want : 1) : cap);
    k_undo_quantize<D, Q, CPL, RPT><<<grid, UQ_THREADS, 0, stream>>>(static_cast<const uint4*>(undo), rows, lpr_log2, codes, scales);
    return cudaGetLastError();
}

template <class D, int Q>
static cudaError_t launch_uq(const void* undo, int64_t rows, int dv, uint8_t* codes, float* scales, int sms, cudaStream_t stream) {
    const int nvec = dv / D::E;                                // 4 .. 32 (bf16), 8 .. 64 (fp32)
    int lg = 0;
    while (lg < 5 && nvec % (2 << lg) == 0) ++lg;
    switch (nvec >> lg) {
        case 1: return launch_uq_cpl<D, Q, 1>(undo, rows, lg, codes, scales, sms, stream);
        case 2: return launch_uq_cpl<D, Q, 2>(undo, rows, lg, codes, scales, sms, stream);
        case 3: return launch_uq_cpl<D, Q, 3>(undo, rows, lg, codes, scales, sms, stream);
        case 5: return launch_uq_cpl<D, Q, 5>(undo, rows, lg, codes, scales, sms, stream);
        case 7: return launch_uq_cpl<D, Q, 7>(undo, rows, lg, codes, scales, sms, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_undo_quantize(int dtype, int kind, const void* undo, int64_t rows, int dv, void* codes,
                                 float* scales, cudaStream_t stream) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    uint8_t* c = static_cast<uint8_t*>(codes);
    if (dtype == 0)
        return kind == 1 ? launch_uq<F32, 1>(undo, rows, dv, c, scales, sms, stream)
                         : launch_uq<F32, 2>(undo, rows, dv, c, scales, sms, stream);
    return kind == 1 ? launch_uq<BF16, 1>(undo, rows, dv, c, scales, sms, stream)
                     : launch_uq<BF16, 2>(undo, rows, dv, c, scales, sms, stream);
}

// ------------------------------------------------------------------------------------------
// Conflict pass of the backward.  Several warps walk the tokens of a chain at once (below), so
// every token needs to know which of the tokens processed shortly before it (t + 1 .. t + LA)
// touch one of its slots: any shared slot, read or written, orders the two (the adjoint row of
// a slot is read and rewritten by every token that uses it).  The pass also matches the write
// slots of a token with its read slots.  Its results live in gradient outputs until the main
// pass, which needs them before it writes those gradients:
//   dalpha[t]     bit d - 1 set: token t + d shares a slot with token t;
//   dw_w[t][m]    1 + n when write slot m of the token is its read slot n, else 0;
//   dw_r[t][n]    1 when read slot n is also written by the token, else 0 (as int bits).
// One CTA per (chain, 32 tokens) with the lists of the LA tokens after them staged in shared
// memory; bitmaps of hash buckets seen once and twice leave only entries of buckets met twice
// to be searched (a few percent at random addressing), one lane per (later token, side).
// ------------------------------------------------------------------------------------------
constexpr int BW_K = 32;           // slots per list (k <= 32)
constexpr int BW_LA = 16;          // conflict window: tokens processed before that may be in flight
constexpr int BC_TILE = 32;
constexpr int BC_THREADS = 256;
constexpr int BC_PITCH = BW_K + 1;
constexpr int BC_BITS = 15;        // hash buckets of the bitmaps
constexpr int BC_WORDS = (1 << BC_BITS) / 32;

__device__ __forceinline__ uint32_t bc_bucket(int32_t s) {
    const uint32_t u = static_cast<uint32_t>(s);
    return ((u ^ (u >> 15)) * 0x85EBCA6Bu) >> (32 - BC_BITS);
}
// position of s in the ascending list l[0..k), or -1
__device__ __forceinline__ int bc_find(const int32_t* l, int k, int32_t s) {
    int lo = 0, hi = k;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (l[mid] < s) lo = mid + 1; else hi = mid;
    }
    return (lo < k && l[lo] == s) ? lo : -1;
}

__global__ void __launch_bounds__(BC_THREADS) k_bwd_conflicts(const RecArgs a, int* __restrict__ mask_o,
                                                              int* __restrict__ match_w, int* __restrict__ match_r) {
    // list pitch BC_PITCH: 16 lanes search 16 tokens' lists at the same position, which an even pitch
    // would put into one bank (0.33 ms against 0.10 ms for 65,536 tokens of 32 + 32 slots)
    __shared__ int32_t sw[(BC_TILE + BW_LA) * BC_PITCH], sr[(BC_TILE + BW_LA) * BC_PITCH];
    __shared__ uint32_t seen[BC_WORDS], dup[BC_WORDS];
    const int kw = a.kw, kr = a.kr, T = a.T;
    const int ntiles = (T + BC_TILE - 1) / BC_TILE;
    const int64_t chain = blockIdx.x / ntiles;
    const int t0 = static_cast<int>(blockIdx.x - chain * ntiles) * BC_TILE;
    const int t1 = min(T, t0 + BC_TILE), nu = min(T, t0 + BC_TILE + BW_LA) - t0;
    const int64_t tok0 = chain * T + t0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t N = static_cast<uint32_t>(a.N);
    for (int i = threadIdx.x; i < BC_WORDS; i += BC_THREADS) { seen[i] = 0u; dup[i] = 0u; }
    __syncthreads();
    for (int u = warp; u < nu; u += BC_THREADS / 32) {           // a warp per token, a lane per slot
        const int32_t s0 = lane < kw ? __ldg(a.idx_w + (tok0 + u) * kw + lane) : 0;
        const int32_t s1 = lane < kr ? __ldg(a.idx_r + (tok0 + u) * kr + lane) : 0;
        auto put = [&](int32_t s, int32_t* dst) {
            dst[lane] = s;
            const uint32_t h = bc_bucket(s), bit = 1u << (h & 31);
            if (atomicOr(seen + (h >> 5), bit) & bit) atomicOr(dup + (h >> 5), bit);
        };
        if (lane < kw) put(s0, sw + u * BC_PITCH);
        if (lane < kr) put(s1, sr + u * BC_PITCH);
    }
    __syncthreads();
    bool bad = false, unsorted = false;
    for (int t = t0 + warp; t < t1; t += BC_THREADS / 32) {
        const int32_t* lw = sw + (t - t0) * BC_PITCH;
        const int32_t* lr = sr + (t - t0) * BC_PITCH;
        const int64_t tok = chain * T + t;
        const int nd = min(BW_LA, T - 1 - t);              // later tokens in the window
        uint32_t mask = 0u;
#pragma unroll
        for (int side = 0; side < 2; ++side) {              // 0: write slots, 1: read slots
            const int k = side ? kr : kw;
            const int32_t* l = side ? lr : lw;
            const int32_t s = lane < k ? l[lane] : 0;
            const bool oks = lane < k && static_cast<uint32_t>(s) < N;
            bad |= lane < k && !oks;
            unsorted |= lane > 0 && lane < k && l[lane - 1] >= s;
            const uint32_t h = bc_bucket(s);
            const bool maybe = oks && ((dup[h >> 5] >> (h & 31)) & 1u);
            if (lane < k) {
                const int at = maybe ? bc_find(side ? lw : lr, side ? kw : kr, s) : -1;
                if (side) match_r[tok * kr + lane] = at >= 0 ? 1 : 0;
                else match_w[tok * kw + lane] = at + 1;
            }
            // lanes 0-15: write list of token t + 1 + lane, lanes 16-31: its read list
            const int d = lane & 15;
            const int32_t* other = (lane < 16 ? lw : lr) + (d + 1) * BC_PITCH;
            uint32_t todo = __ballot_sync(0xffffffffu, maybe);
            while (todo) {                                   // warp-uniform
                const int32_t q = __shfl_sync(0xffffffffu, s, __ffs(todo) - 1);
                todo &= todo - 1;
                const bool hit = d < nd && bc_find(other, lane < 16 ? kw : kr, q) >= 0;
                const uint32_t hits = __ballot_sync(0xffffffffu, hit);
                mask |= (hits & 0xffffu) | (hits >> 16);
            }
        }
        if (lane == 0) mask_o[tok] = static_cast<int>(mask);
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) flag_error(a.err, ERR_BAD_INDEX);
    if (__any_sync(0xffffffffu, unsorted) && lane == 0) flag_error(a.err, ERR_UNSORTED);
}

// ------------------------------------------------------------------------------------------
// The backward.  One CTA per (b, h) chain; warp (p, r) takes 32-element slice r of d_v of the
// tokens p, p + W, p + 2W, ... counted from the last one.  Every per-element quantity of the
// chain rule (the rows of M, of G and of the log, pred, delta, d delta, d r) stays within a slice, so
// slices of a token never wait for one another's rows; W tokens are in flight per chain.  Lane
// (g, c) of a warp moves the E elements (16 bytes of storage) of chunk c of the slots
// g * SPT .. g * SPT + SPT - 1, so rows move as 16-byte vectors and a warp has all its rows of a
// token in flight at once.
//
// Order.  Tokens depend on each other only through the rows of shared slots.  Before it loads
// its rows, a warp waits until the same slice of every earlier-processed token the conflict
// pass marked is stored, and until no token more than LA before it is in flight; progress words
// in shared memory, each published after a block-scope fence.  The waits are bounded: on timeout the CTA
// sets an abort flag, and its warps go through their remaining tokens without touching rows, so
// that the barriers below stay whole.  A read slot the token also writes gets its update inside
// the token (the read adds rho dy to the row the write then takes).
//
// The dot products over d_v (d rho, <G_i, delta>, <r_i, d delta>, d alpha) are reduced within
// a warp, then over the slices in slice order by one warp per token after a named barrier of
// the slices of a phase; the shares are double-buffered, so that is one barrier per token.
//
// What bounds it: each token's chain of list loads, waits, row loads and reductions (16 warps per
// SM wait on memory and shared memory for half of their time); the rows, (2 k_r + 2 k_w) loads and
// (k_r + 2 k_w) stores per token with the adjoint's in fp32, would take 0.9 ms of HBM in the case below.
// 64 chains x 1024 tokens, N = 2^18, k = 32, d_v = 128, bf16: 1.81 ms, conflict pass 0.10 ms; one warp
// per slice walking all tokens by itself, an element per lane, took 36.6 ms.  Logged rows, dy and v
// prefetched a token ahead through shared memory and fp32 pairs in the packed units: 2.42 -> 1.81 ms.
// ------------------------------------------------------------------------------------------
constexpr int BW_WARPS = 16;
constexpr int BW_SHARES = 3 * BW_K + 4;           // d rho, <G, delta>, <r, dd>, d alpha (padded)
constexpr int BW_LIST = 6 * BW_K;                 // idx_r, w_r, idx_w, w_w, match_r, match_w
constexpr long long BW_WAIT_CYCLES = 4000000000LL;

struct BwdArgs {
    UndoLog undo;
    const void* dy;
    float *dv, *dalpha, *dbeta, *dw_w, *dw_r, *dM;
    int lw;                                       // log2 of the token phases W; d_v / 32 slices
    bool vec_in;                                  // v and dy 16-byte aligned
    bool vec_g;                                   // dM 16-byte aligned
};

__device__ __forceinline__ void bw_cp4(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
// 16 bytes through L2 only; src_bytes = 0 writes zeros.
__device__ __forceinline__ void bw_cp16(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ uint4 bw_ldcg(const void* p) {
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void bw_bar(int id, int threads) {
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}
template <int N>
__device__ __forceinline__ void bw_lds(const int* p, int (&o)[N]) {
    if constexpr (N == 1) {
        o[0] = p[0];
    } else if constexpr (N == 2) {
        const int2 v = *reinterpret_cast<const int2*>(p);
        o[0] = v.x; o[1] = v.y;
    } else {
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const int4 v = *reinterpret_cast<const int4*>(p + 4 * q);
            o[4 * q] = v.x; o[4 * q + 1] = v.y; o[4 * q + 2] = v.z; o[4 * q + 3] = v.w;
        }
    }
}

// E consecutive floats of an adjoint row (zeros without `on`).
template <int E>
__device__ __forceinline__ void bw_load_g(const float* p, bool on, bool vec, float2 (&o)[E / 2]) {
#pragma unroll
    for (int e = 0; e < E / 2; ++e) o[e] = make_float2(0.f, 0.f);
    if (on && vec) {
#pragma unroll
        for (int q = 0; q < E / 4; ++q) {
            const uint4 v = bw_ldcg(p + 4 * q);
            o[2 * q] = make_float2(__uint_as_float(v.x), __uint_as_float(v.y));
            o[2 * q + 1] = make_float2(__uint_as_float(v.z), __uint_as_float(v.w));
        }
    } else if (on) {
#pragma unroll
        for (int e = 0; e < E / 2; ++e) o[e] = make_float2(__ldcg(p + 2 * e), __ldcg(p + 2 * e + 1));
    }
}
template <int E>
__device__ __forceinline__ void bw_store_g(float* p, bool vec, const float2 (&o)[E / 2]) {
    if (vec) {
#pragma unroll
        for (int q = 0; q < E / 4; ++q)
            *reinterpret_cast<float4*>(p + 4 * q) = make_float4(o[2 * q].x, o[2 * q].y, o[2 * q + 1].x, o[2 * q + 1].y);
    } else {
#pragma unroll
        for (int e = 0; e < E / 2; ++e) { p[2 * e] = o[e].x; p[2 * e + 1] = o[e].y; }
    }
}
// Storage element i in shared memory.
template <class D> __device__ __forceinline__ float bw_elem(const unsigned char* p, int i);
template <> __device__ __forceinline__ float bw_elem<F32>(const unsigned char* p, int i) { return reinterpret_cast<const float*>(p)[i]; }
template <> __device__ __forceinline__ float bw_elem<BF16>(const unsigned char* p, int i) {
    return __uint_as_float(static_cast<uint32_t>(reinterpret_cast<const unsigned short*>(p)[i]) << 16);
}
// Codes and scale of elements e0 .. e0 + E - 1 of logged row r (quantised log), and their stored values.
template <class D, int Q>
__device__ __forceinline__ void bw_load_undo(const UndoLog& u, int64_t r, int dv, int e0, uint4& raw, float& scale) {
    constexpr int E = D::E;
    scale = __ldg(u.scales + r);
    if constexpr (Q == 1) {
        const uint8_t* p = u.codes + r * dv + e0;
        if constexpr (E == 8) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
            raw.x = v.x; raw.y = v.y;
        } else {
            raw.x = __ldg(reinterpret_cast<const unsigned int*>(p));
        }
    } else {
        const uint8_t* p = u.codes + r * (dv / 2) + e0 / 2;
        if constexpr (E == 8) raw.x = __ldg(reinterpret_cast<const unsigned int*>(p));
        else raw.x = __ldg(reinterpret_cast<const unsigned short*>(p));
    }
}
template <class D, int Q>
__device__ __forceinline__ void bw_unpack_undo(const uint4& raw, float scale, float2 (&o)[D::E / 2]) {
    float f[D::E];
#pragma unroll
    for (int e = 0; e < D::E; ++e) {
        float q;
        if constexpr (Q == 1) {
            const uint32_t w = e < 4 ? raw.x : raw.y;
            const __half_raw hr = __nv_cvt_fp8_to_halfraw(static_cast<__nv_fp8_storage_t>((w >> (8 * (e & 3))) & 255u), __NV_E4M3);
            q = __half2float(__half(hr));
        } else {
            q = static_cast<float>(static_cast<int>(raw.x << (28 - 4 * e)) >> 28);
        }
        f[e] = to_storage<D>(q * scale);
    }
#pragma unroll
    for (int e = 0; e < D::E / 2; ++e) o[e] = make_float2(f[2 * e], f[2 * e + 1]);
}

// Sums of SPT per-lane values over the DCH lanes of a row (c = lane % DCH); lane c returns the
// sum of value c / (DCH / SPT).
template <int SPT, int DCH>
__device__ __forceinline__ float bw_sum_row(float (&x)[SPT], int c) {
    int n = SPT;
#pragma unroll
    for (int off = DCH / 2; off > 0; off >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = (c & off) != 0;
#pragma unroll
            for (int i = 0; i < SPT / 2; ++i) {
                if (i < n) {
                    const float send = up ? x[i] : x[i + n], keep = up ? x[i + n] : x[i];
                    x[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                }
            }
        } else {
            x[0] += __shfl_xor_sync(0xffffffffu, x[0], off);
        }
    }
    return x[0];
}
// Sums of E per-lane values over the G = E slot groups (g = lane / DCH); lane g returns the sum
// of value g.
template <int E, int DCH>
__device__ __forceinline__ float bw_sum_groups(const float2 (&v)[E / 2], int g) {
    float x[E];
#pragma unroll
    for (int e = 0; e < E / 2; ++e) { x[2 * e] = v[e].x; x[2 * e + 1] = v[e].y; }
#pragma unroll
    for (int n = E / 2; n > 0; n >>= 1) {
        const bool up = (g & n) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = up ? x[i] : x[i + n], keep = up ? x[i + n] : x[i];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, send, n * DCH);
        }
    }
    return x[0];
}

// Shared bytes of a warp: two tokens' lists, then (exact log) two tokens' logged rows, then two
// tokens' dy and v chunks, the dot products' shares and delta / d delta.
template <int Q, int SPT>
__host__ __device__ constexpr int bw_warp_bytes() {
    return 2 * BW_LIST * 4 + (Q == 0 ? 2 * SPT * 512 : 0) + 2 * 256 + 2 * BW_SHARES * 4 + 2 * 32 * 4;
}

template <class D, int Q, int SPT>
__global__ void __launch_bounds__(32 * BW_WARPS, 1) k_recur_bwd(const RecArgs a, const BwdArgs b) {
    constexpr int E = D::E, E2 = E / 2;
    constexpr int DCH = 32 / E;                    // lanes per row of a slice
    constexpr int G = 32 / DCH;                    // slot groups (= E)
    static_assert(G == E && SPT <= DCH, "lane layout");
    extern __shared__ __align__(16) unsigned char smB[];
    __shared__ int prog_s[BW_WARPS];               // [phase][slice]: own tokens stored so far
    __shared__ int abort_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nsl = a.dv >> 5, W = 1 << b.lw;
    const int p = warp / nsl, sl = warp - p * nsl;
    const int c = lane % DCH, g = lane / DCH;
    const int dv = a.dv, T = a.T, kw = a.kw, kr = a.kr;
    const int64_t chain = blockIdx.x, tok_last = chain * T + T - 1;
    const uint32_t N = static_cast<uint32_t>(a.N);
    const int e0 = sl * 32 + c * E;                // first element of this lane
    const int64_t mbase = chain * a.N * dv + e0;
    char* Mc = static_cast<char*>(a.mem) + mbase * D::BYTES;
    float* Gc = b.dM + mbase;
    const uint32_t mrow = static_cast<uint32_t>(dv) * D::BYTES;
    unsigned char* sm = smB + warp * bw_warp_bytes<Q, SPT>();
    int* const s_list = reinterpret_cast<int*>(sm);                              // [2][BW_LIST]
    unsigned char* const s_undo = sm + 2 * BW_LIST * 4;                          // [2][SPT][32] x 16 B
    unsigned char* const s_in = s_undo + (Q == 0 ? 2 * SPT * 512 : 0);           // [2][dy 128 B, v 128 B]
    float* const s_sh = reinterpret_cast<float*>(s_in + 2 * 256);                // [2][BW_SHARES]
    float* const s_pd = s_sh + 2 * BW_SHARES;                                    // delta [32], d delta [32]
    const uint32_t sm_u32 = static_cast<uint32_t>(__cvta_generic_to_shared(sm));
    volatile int* prog = prog_s;
    volatile int* abort_flag = &abort_s;
    if (threadIdx.x < BW_WARPS) prog_s[threadIdx.x] = 0;
    if (threadIdx.x == 0) abort_s = 0;
    __syncthreads();

    // everything of own token i that no other token touches, into ring slot i & 1: the lists (lane n:
    // entry n), the logged rows, dy and v; its gates and mask in registers
    float al_n = 0.f, be_n = 0.f;
    int mask_n = 0;
    auto fetch = [&](int i) {
        const int q = p + (i << b.lw);
        if (q < T) {
            const int64_t tok = tok_last - q;
            const uint32_t dst = sm_u32 + (i & 1) * (BW_LIST * 4) + lane * 4;
            if (lane < kr) {
                const int64_t o = tok * kr + lane;
                bw_cp4(dst, a.idx_r + o);
                bw_cp4(dst + 4 * BW_K, a.w_r + o);
                bw_cp4(dst + 16 * BW_K, b.dw_r + o);
            }
            if (lane < kw) {
                const int64_t o = tok * kw + lane;
                bw_cp4(dst + 8 * BW_K, a.idx_w + o);
                bw_cp4(dst + 12 * BW_K, a.w_w + o);
                bw_cp4(dst + 20 * BW_K, b.dw_w + o);
            }
            if constexpr (Q == 0) {                 // each lane copies what it will use: zeros past the list
                const char* src = static_cast<const char*>(b.undo.rows) + (tok * kw + g * SPT) * static_cast<int64_t>(mrow) + e0 * D::BYTES;
                const uint32_t ud = sm_u32 + 2 * BW_LIST * 4 + (i & 1) * (SPT * 512) + lane * 16;
#pragma unroll
                for (int j = 0; j < SPT; ++j) {
                    const bool in = g * SPT + j < kw;
                    bw_cp16(ud + j * 512, in ? src + j * mrow : static_cast<const char*>(b.undo.rows), in ? 16 : 0);
                }
            }
            if (b.vec_in && lane < 2 * DCH) {
                const char* src = static_cast<const char*>(lane < DCH ? b.dy : a.v) + (tok * dv + sl * 32 + c * E) * D::BYTES;
                bw_cp16(static_cast<uint32_t>(__cvta_generic_to_shared(s_in)) + (i & 1) * 256 + (lane < DCH ? 0 : 128) + c * 16, src, 16);
            }
            al_n = load_elem<D>(a.alpha, tok);
            be_n = load_elem<D>(a.beta, tok);
            mask_n = __float_as_int(__ldcg(b.dalpha + tok));
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    const int nown = T > p ? (T - p + W - 1) >> b.lw : 0;
    if (nown > 0) fetch(0);
    bool timed_out = false;
    for (int i = 0; i < nown; ++i) {
        const int q = p + (i << b.lw);
        const int64_t tok = tok_last - q;
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncwarp();
        const float alpha = al_n, beta = be_n;
        const uint32_t mask = static_cast<uint32_t>(mask_n);
        const int* L = s_list + (i & 1) * BW_LIST;
        int iw[SPT], ir[SPT];
        bw_lds<SPT>(L + 2 * BW_K + g * SPT, iw);
        bw_lds<SPT>(L + g * SPT, ir);
        bool okw[SPT], okr[SPT];
#pragma unroll
        for (int j = 0; j < SPT; ++j) {
            okw[j] = g * SPT + j < kw && static_cast<uint32_t>(iw[j]) < N;
            okr[j] = g * SPT + j < kr && static_cast<uint32_t>(ir[j]) < N;
        }
        if (i + 1 < nown) fetch(i + 1);
        uint4 uraw[SPT];                                // (quantised log: codes and scales in registers)
        float us[SPT];
        if constexpr (Q != 0) {
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                uraw[j] = make_uint4(0u, 0u, 0u, 0u);
                us[j] = 0.f;
                if (okw[j]) bw_load_undo<D, Q>(b.undo, tok * kw + g * SPT + j, dv, e0, uraw[j], us[j]);
            }
        }
        // ---- wait for the tokens that share a slot, and for the window
        {
            bool need = false;
            int wv = 0, at = 0;                         // warp (phase, this slice) and its count needed
            if (lane < BW_LA) {
                const int u = q - 1 - lane;             // processed d = lane + 1 tokens before
                if (u >= 0 && ((mask >> lane) & 1u)) { need = true; wv = u & (W - 1); at = (u >> b.lw) + 1; }
            } else if (lane - BW_LA < W) {
                wv = lane - BW_LA;                      // tokens <= q - 1 - LA of phase wv
                const int u = q - 1 - BW_LA;
                if (u >= wv) { need = true; at = ((u - wv) >> b.lw) + 1; }
            }
            const int at_w = wv * nsl + sl;
            if (__any_sync(0xffffffffu, need && prog[at_w] < at)) {
                const long long start = clock64();
                while (__any_sync(0xffffffffu, need && prog[at_w] < at)) {
                    const bool stop = *abort_flag != 0 || clock64() - start > BW_WAIT_CYCLES;
                    if (__any_sync(0xffffffffu, stop)) { timed_out = true; break; }     // warp-uniform
                    __nanosleep(32);
                }
                if (timed_out) *abort_flag = 1;
            }
            __threadfence_block();
            if (timed_out) {
#pragma unroll
                for (int j = 0; j < SPT; ++j) { okw[j] = false; okr[j] = false; }
            }
        }
        // ---- rows
        float2 gv[SPT][E2], gr[SPT][E2];
        uint4 mraw[SPT];
#pragma unroll
        for (int j = 0; j < SPT; ++j) {
            mraw[j] = make_uint4(0u, 0u, 0u, 0u);
            if (okr[j]) mraw[j] = bw_ldcg(Mc + static_cast<uint64_t>(static_cast<uint32_t>(ir[j])) * mrow);
        }
#pragma unroll
        for (int j = 0; j < SPT; ++j)
            bw_load_g<E>(Gc + static_cast<uint64_t>(okr[j] ? ir[j] : 0) * dv, okr[j], b.vec_g, gr[j]);
#pragma unroll
        for (int j = 0; j < SPT; ++j)
            bw_load_g<E>(Gc + static_cast<uint64_t>(okw[j] ? iw[j] : 0) * dv, okw[j], b.vec_g, gv[j]);
        float2 gy[E2];
        float vt;                                       // the element this lane owns after the group sums: c * E + g
        {
            const unsigned char* in = s_in + (i & 1) * 256;
            if (b.vec_in) {
                unpack16x2<D>(*reinterpret_cast<const uint4*>(in + c * 16), gy);
                vt = bw_elem<D>(in + 128, c * E + g);
            } else {
                float f[E];
#pragma unroll
                for (int e = 0; e < E; ++e) f[e] = load_elem<D>(b.dy, tok * dv + e0 + e);
#pragma unroll
                for (int e = 0; e < E2; ++e) gy[e] = make_float2(f[2 * e], f[2 * e + 1]);
                vt = load_elem<D>(a.v, tok * dv + e0 + g);
            }
        }
        float* sh = s_sh + (i & 1) * BW_SHARES;
        // ---- read of the post-write memory M_t: d rho_n = <dy, M_t[r_n]>, G[r_n] += rho_n dy
        {
            float x[SPT];
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                float2 m[E2], acc = make_float2(0.f, 0.f);
                unpack16x2<D>(mraw[j], m);
#pragma unroll
                for (int e = 0; e < E2; ++e) acc = __ffma2_rn(gy[e], m[e], acc);
                x[j] = acc.x + acc.y;
            }
            const float s = bw_sum_row<SPT, DCH>(x, c);
            if (c % (DCH / SPT) == 0) sh[g * SPT + c / (DCH / SPT)] = s;
        }
        __syncwarp();                                   // every lane's rows of M are read
        {
            int wr[SPT], mr[SPT];
            bw_lds<SPT>(L + BW_K + g * SPT, wr);
            bw_lds<SPT>(L + 4 * BW_K + g * SPT, mr);
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                const float2 rho = make_float2(__int_as_float(wr[j]), __int_as_float(wr[j]));
                float2 o[E2];
#pragma unroll
                for (int e = 0; e < E2; ++e) o[e] = __ffma2_rn(rho, gy[e], gr[j][e]);
                if (okr[j] && mr[j] == 0) bw_store_g<E>(Gc + static_cast<uint64_t>(static_cast<uint32_t>(ir[j])) * dv, b.vec_g, o);
            }
        }
        // ---- the write: prediction and delta from the logged rows, d delta from the adjoint
        float wm[SPT];
        {
            int ww[SPT], mw[SPT];
            bw_lds<SPT>(L + 3 * BW_K + g * SPT, ww);
            bw_lds<SPT>(L + 5 * BW_K + g * SPT, mw);
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                wm[j] = okw[j] ? __int_as_float(ww[j]) : 0.f;
                if (okw[j] && mw[j] != 0) {             // the read of this slot by the same token
                    const float rho = __int_as_float(L[BW_K + mw[j] - 1]);
#pragma unroll
                    for (int e = 0; e < E2; ++e) gv[j][e] = __ffma2_rn(make_float2(rho, rho), gy[e], gv[j][e]);
                }
            }
        }
        const unsigned char* ub = s_undo + (i & 1) * (SPT * 512) + lane * 16;
        auto logged = [&](int j, float2 (&o)[E2]) {     // M_{t-1} of slot j (zeros where there is none)
            if constexpr (Q == 0) {
                uint4 u = make_uint4(0u, 0u, 0u, 0u);   // (a slot out of range has no logged row)
                if (okw[j]) u = *reinterpret_cast<const uint4*>(ub + j * 512);
                unpack16x2<D>(u, o);
            } else {
                bw_unpack_undo<D, Q>(uraw[j], us[j], o);
            }
        };
        const float2 alpha2 = make_float2(alpha, alpha);
        {
            float2 pr[E2], dd[E2];
#pragma unroll
            for (int e = 0; e < E2; ++e) { pr[e] = make_float2(0.f, 0.f); dd[e] = make_float2(0.f, 0.f); }
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                float2 pv[E2];
                logged(j, pv);
                const float2 wm2 = make_float2(wm[j], wm[j]);
#pragma unroll
                for (int e = 0; e < E2; ++e) {
                    pr[e] = __ffma2_rn(wm2, __fmul2_rn(alpha2, pv[e]), pr[e]);
                    dd[e] = __ffma2_rn(wm2, gv[j][e], dd[e]);
                }
            }
            const float pe = bw_sum_groups<E, DCH>(pr, g), de = beta * bw_sum_groups<E, DCH>(dd, g);
            b.dv[tok * dv + e0 + g] = de;
            s_pd[c * E + g] = vt - pe;                  // delta
            s_pd[32 + c * E + g] = de;                  // d delta
        }
        __syncwarp();
        float2 delta[E2], dd[E2];
#pragma unroll
        for (int v4 = 0; v4 < E / 4; ++v4) {
            const float4 x = *reinterpret_cast<const float4*>(s_pd + c * E + 4 * v4);
            delta[2 * v4] = make_float2(x.x, x.y); delta[2 * v4 + 1] = make_float2(x.z, x.w);
            const float4 y = *reinterpret_cast<const float4*>(s_pd + 32 + c * E + 4 * v4);
            dd[2 * v4] = make_float2(y.x, y.y); dd[2 * v4 + 1] = make_float2(y.z, y.w);
        }
        float gd[SPT], rd[SPT];
        float2 da2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < SPT; ++j) {
            float2 pv[E2], o[E2], g2 = make_float2(0.f, 0.f), r2 = make_float2(0.f, 0.f);
            logged(j, pv);
            const float2 mwm = make_float2(-wm[j], -wm[j]);
#pragma unroll
            for (int e = 0; e < E2; ++e) {
                g2 = __ffma2_rn(gv[j][e], delta[e], g2);
                r2 = __ffma2_rn(__fmul2_rn(alpha2, pv[e]), dd[e], r2);
                const float2 dr = __ffma2_rn(mwm, dd[e], gv[j][e]);
                da2 = __ffma2_rn(dr, pv[e], da2);
                o[e] = __fmul2_rn(alpha2, dr);
            }
            gd[j] = g2.x + g2.y;
            rd[j] = r2.x + r2.y;
            if (okw[j]) {
                bw_store_g<E>(Gc + static_cast<uint64_t>(static_cast<uint32_t>(iw[j])) * dv, b.vec_g, o);
                uint4 st;
                if constexpr (Q == 0) st = *reinterpret_cast<const uint4*>(ub + j * 512);
                else st = pack16x2<D>(pv);
                *reinterpret_cast<uint4*>(Mc + static_cast<uint64_t>(static_cast<uint32_t>(iw[j])) * mrow) = st;   // the undo
            }
        }
        // ---- publish: the rows of this slice of the token are stored
        __syncwarp();
        if (lane == 0) {
            __threadfence_block();
            prog[warp] = i + 1;
        }
        // ---- this slice's shares of the dot products
        {
            const float s1 = bw_sum_row<SPT, DCH>(gd, c), s2 = bw_sum_row<SPT, DCH>(rd, c);
            float da = da2.x + da2.y;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) da += __shfl_xor_sync(0xffffffffu, da, off);
            if (c % (DCH / SPT) == 0) {
                sh[BW_K + g * SPT + c / (DCH / SPT)] = s1;
                sh[2 * BW_K + g * SPT + c / (DCH / SPT)] = s2;
            }
            if (lane == 0) sh[3 * BW_K] = da;
        }
        if (nsl > 1) bw_bar(1 + p, 32 * nsl);
        else __syncwarp();
        if (i % nsl == sl) {                            // the slices take turns
            float r = 0.f, gq = 0.f, rq = 0.f, al = 0.f;
            for (int s2 = 0; s2 < nsl; ++s2) {          // slices in order
                const float* o = sh + (s2 - sl) * (bw_warp_bytes<Q, SPT>() / 4);
                if (lane < G * SPT) {
                    r += o[lane];
                    gq += o[BW_K + lane];
                    rq += o[2 * BW_K + lane];
                }
                al += o[3 * BW_K];
            }
            const bool in_w = lane < kw;
            const int iwl = in_w ? L[2 * BW_K + lane] : 0;
            const bool okl = in_w && static_cast<uint32_t>(iwl) < N;
            if (lane < kr) b.dw_r[tok * kr + lane] = r;
            if (in_w) b.dw_w[tok * kw + lane] = okl ? beta * gq - rq : 0.f;
            float db = okl ? __int_as_float(L[3 * BW_K + lane]) * gq : 0.f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) db += __shfl_xor_sync(0xffffffffu, db, off);
            if (lane == 0) { b.dalpha[tok] = al; b.dbeta[tok] = db; }
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (timed_out && lane == 0) flag_error(a.err, ERR_TIMEOUT);
}

template <class D, int Q, int SPT>
static cudaError_t launch_bwd_spt(const RecArgs& a, const BwdArgs& b, cudaStream_t stream) {
    const unsigned grid = static_cast<unsigned>(static_cast<int64_t>(a.B) * a.H);
    const int threads = a.dv << b.lw;                    // 32 lanes x (d_v / 32) slices x W phases
    const int smem = threads / 32 * bw_warp_bytes<Q, SPT>();
    cudaError_t e = cudaFuncSetAttribute(k_recur_bwd<D, Q, SPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_ALLOWED);
    if (e != cudaSuccess) return e;
    k_recur_bwd<D, Q, SPT><<<grid, threads, smem, stream>>>(a, b);
    return cudaGetLastError();
}

template <class D, int Q>
static cudaError_t launch_bwd(const RecArgs& a, const BwdArgs& b, cudaStream_t stream) {
    constexpr int G = D::E;                              // slot groups of a warp
    const int k = a.kw > a.kr ? a.kw : a.kr;
    const int spt = (k + G - 1) / G;
    if (spt <= 1) return launch_bwd_spt<D, Q, 1>(a, b, stream);
    if (spt <= 2) return launch_bwd_spt<D, Q, 2>(a, b, stream);
    if (spt <= 4) return launch_bwd_spt<D, Q, 4>(a, b, stream);
    if constexpr (G == 4) return launch_bwd_spt<D, Q, 8>(a, b, stream);
    return cudaErrorInvalidValue;
}

cudaError_t launch_recur_backward(int dtype, const RecArgs& a, int kind, const void* undo, const void* codes,
                                  const float* scales, const void* dy, float* dv, float* dalpha, float* dbeta,
                                  float* dw_w, float* dw_r, float* dM, cudaStream_t stream) {
    if (a.kw > BW_K || a.kr > BW_K || a.dv % 32 != 0 || a.dv > 256) return cudaErrorInvalidValue;
    const int64_t chains = static_cast<int64_t>(a.B) * a.H;
    const int64_t tiles = chains * ((a.T + BC_TILE - 1) / BC_TILE);
    k_bwd_conflicts<<<static_cast<unsigned>(tiles), BC_THREADS, 0, stream>>>(a, reinterpret_cast<int*>(dalpha),
                                                                             reinterpret_cast<int*>(dw_w),
                                                                             reinterpret_cast<int*>(dw_r));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
    BwdArgs b{};
    b.undo = UndoLog{undo, static_cast<const uint8_t*>(codes), scales};
    b.dy = dy;
    b.dv = dv; b.dalpha = dalpha; b.dbeta = dbeta; b.dw_w = dw_w; b.dw_r = dw_r; b.dM = dM;
    // as many token phases as 16 warps (a full register file at 128 registers) allow, a power of
    // two, at most 8 (the conflict window holds two rounds of them)
    const int nsl = a.dv / 32;
    b.lw = 3;
    while ((nsl << b.lw) > BW_WARPS) --b.lw;
    b.vec_in = al16(a.v) && al16(dy);
    b.vec_g = al16(dM);
    if (dtype == 0)
        return kind == 0 ? launch_bwd<F32, 0>(a, b, stream) : kind == 1 ? launch_bwd<F32, 1>(a, b, stream)
                                                                        : launch_bwd<F32, 2>(a, b, stream);
    return kind == 0 ? launch_bwd<BF16, 0>(a, b, stream) : kind == 1 ? launch_bwd<BF16, 1>(a, b, stream)
                                                                     : launch_bwd<BF16, 2>(a, b, stream);
}

}  // namespace sdm
