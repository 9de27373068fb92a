// Chunkwise (WY) form of the recurrence (App. A.1 "Intra-Chunk Parallel vs. Chunkwise
// Recurrent", A.2 "Sparse Inner Product").
//
// One CTA per ((b, h) chain, d-range) walks the chain's chunks of C <= 32 tokens in order; the chain's
// rows split along d_v because everything but the slot matching is element-wise along it.
// Per chunk, with la_t = log(alpha_t) and lam the decay a slot has accumulated in the chunk up to
// and including a token:
//   matching    which tokens of the chunk write a slot.  Bitmaps of hash buckets met once and twice
//               leave a few percent of the entries; for those a warp looks the slot up in all
//               C write lists at once (lane u: token u), which gives the slot's writers as a mask, lam by a warp
//               scan, and the entry's terms of the gated inner products
//                 A[t][u]  += w_t w_u e^(lam_t - lam_u)      (u < t, write-write)
//                 QK[t][u] += rho_t w_u e^(lam_t - lam_u)    (u <= t, read-write)
//               lane by lane.  An entry met once has lam = la_t (write) or 0 (read) and no terms;
//   gather      R_t = sum_n w e^lam M[idx_w], I_t = sum_n rho e^lam M[idx_r] from the chunk-initial
//               memory: a warp per token, all its rows in flight;
//   solve       u_t = beta_t (v_t - R_t - sum_{u<t} A[t][u] u_u): forward substitution with the unit
//               lower-triangular I + diag(beta) A, whose rows are mostly empty (a mask per row says
//               where they are not), so most tokens need none of it;
//   output      y_t = I_t + sum_{u<=t} QK[t][u] u_u (stored, rounded);
//   scatter     the last writer of each slot forms its new row, e^lam M + sum over the slot's
//               writers of e^(lam - lam_u) w_u u_u, rounded.
// The memory is rounded at chunk boundaries only, like the chunkwise oracle.  The next chunk's lists and
// v come in by asynchronous copies under the memory phases; no waits on other CTAs.
//
// Bound by each chunk's chain of phases (9 us per chunk and CTA, of which the row traffic would take
// about 4 at the bandwidth of an SM).  A warp per token and 16 warps per CTA: 64 chains x 2048
// tokens, C = 16, k = 32, N = 2^18, bf16 take 1.20 ms; 8 warps, smaller bitmaps (four times the
// look-ups) and a scatter over flat entry numbers 2.47 ms; the first kernel (element-wise merges, a
// barrier per token) 17.6 ms.
#include "sdm_internal.h"

namespace sdm {

constexpr int CK_MAX_THREADS = 512;               // a warp per token up to C = 16
constexpr int CK_MAXC = 32;
constexpr int CK_BITS = 16;                       // hash buckets of the bitmaps
constexpr int CK_WORDS = (1 << CK_BITS) / 32;
constexpr int CK_ROWS = 8;                        // row loads in flight per lane and list

__device__ __forceinline__ uint32_t ck_bucket(int32_t s) {
    const uint32_t u = static_cast<uint32_t>(s);
    return ((u ^ (u >> 15)) * 0x85EBCA6Bu) >> (32 - CK_BITS);
}
// position of slot s in the ascending list l[0..k), or -1
__device__ __forceinline__ int find_slot(const int* l, int k, int s) {
    int lo = 0, hi = k;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (l[mid] < s) lo = mid + 1;
        else hi = mid;
    }
    return (lo < k && l[lo] == s) ? lo : -1;
}
__device__ __forceinline__ void ck_cp4(void* dst, const void* src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void ck_cp16(void* dst, const void* src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ uint4 ck_ldcg(const void* p) {     // rows are rewritten by this kernel: L2 only
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}

// Shared memory.  Lists have an odd pitch: the look-up reads the same position of C lists at once.
struct ChunkSmem {
    int pw, pr, dr;                               // list pitches; elements of the d-range
    size_t iw, ww, ir, wr, v, set, lam, cfw, cfr, link, A, QK, R, I, U, bits, tok, total;
};
__host__ __device__ inline ChunkSmem chunk_smem(int C, int kw, int kr, int dr, int bytes) {
    ChunkSmem s;
    s.pw = kw | 1;
    s.pr = kr | 1;
    s.dr = dr;
    size_t o = 0;
    // staged per chunk, two sets: lists, weights, v
    s.v = o;   o += static_cast<size_t>(C) * dr * bytes;
    s.iw = o;  o += static_cast<size_t>(C) * s.pw * 4;
    s.ww = o;  o += static_cast<size_t>(C) * s.pw * 4;
    s.ir = o;  o += static_cast<size_t>(C) * s.pr * 4;
    s.wr = o;  o += static_cast<size_t>(C) * s.pr * 4;
    s.set = (o + 15) / 16 * 16;
    o = 2 * s.set;
    s.R = o;   o += static_cast<size_t>(C) * dr * 4;          // R of the tokens that need the solve
    s.I = o;   o += static_cast<size_t>(C) * dr * 4;
    s.U = o;   o += static_cast<size_t>(C) * dr * 4;
    s.bits = (o + 15) / 16 * 16; o = s.bits + 2 * CK_WORDS * 4;
    s.lam = o; o += static_cast<size_t>(C) * s.pw * 4;
    s.cfw = o; o += static_cast<size_t>(C) * s.pw * 4;        // w e^lam
    s.cfr = o; o += static_cast<size_t>(C) * s.pr * 4;        // rho e^lam
    s.link = o; o += static_cast<size_t>(C) * s.pw * 4;       // previous writer of the slot, see below
    s.A = o;   o += static_cast<size_t>(C) * (C + 1) * 4;
    s.QK = o;  o += static_cast<size_t>(C) * (C + 1) * 4;
    s.tok = o; o += static_cast<size_t>(CK_MAXC) * 5 * 4;     // la, alpha, beta, masks of A and QK
    s.total = o;
    return s;
}
// link word of a write entry: bit 31 set unless it is the slot's last writer in the chunk (a
// valid slot's), bits 0-15: 0, or 1 + token * 64 + position of the writer before it
constexpr uint32_t CK_NOT_LAST = 0x80000000u;

template <class D, int DCH>
__global__ void __launch_bounds__(CK_MAX_THREADS, 1) k_recur_chunk(const RecArgs a, int C, int nsplit) {
    extern __shared__ __align__(16) unsigned char smC[];
    constexpr int E = D::E;
    constexpr int RG = 32 / DCH;                              // rows a warp moves at once
    const int kw = a.kw, kr = a.kr, dv = a.dv, T = a.T;
    const uint32_t N = static_cast<uint32_t>(a.N);
    const ChunkSmem S = chunk_smem(C, kw, kr, DCH * E, D::BYTES);
    const int pw = S.pw, pr = S.pr, dr = S.dr;
    float* const s_R = reinterpret_cast<float*>(smC + S.R);
    float* const s_I = reinterpret_cast<float*>(smC + S.I);
    float* const s_U = reinterpret_cast<float*>(smC + S.U);
    uint32_t* const seen = reinterpret_cast<uint32_t*>(smC + S.bits);
    uint32_t* const dup = seen + CK_WORDS;
    float* const s_lam = reinterpret_cast<float*>(smC + S.lam);
    float* const s_cfw = reinterpret_cast<float*>(smC + S.cfw);
    float* const s_cfr = reinterpret_cast<float*>(smC + S.cfr);
    uint32_t* const s_link = reinterpret_cast<uint32_t*>(smC + S.link);
    float* const s_A = reinterpret_cast<float*>(smC + S.A);
    float* const s_QK = reinterpret_cast<float*>(smC + S.QK);
    float* const s_la = reinterpret_cast<float*>(smC + S.tok);
    float* const s_al = s_la + CK_MAXC;
    float* const s_be = s_al + CK_MAXC;
    uint32_t* const s_mA = reinterpret_cast<uint32_t*>(s_be + CK_MAXC);
    uint32_t* const s_mQ = s_mA + CK_MAXC;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int threads = blockDim.x, warps = threads >> 5;
    const int c = lane % DCH, rg = lane / DCH;
    const int64_t chain = blockIdx.x / nsplit;
    const int split = static_cast<int>(blockIdx.x - chain * nsplit);
    const int nch = dv / E;                                   // 16-byte pieces of a row
    const int ch = split * DCH + c;                           // this lane's piece
    const bool on = ch < nch;
    const uint32_t rowbytes = static_cast<uint32_t>(dv) * D::BYTES;
    char* const mrow = static_cast<char*>(a.mem) + chain * a.N * static_cast<int64_t>(rowbytes) + (on ? ch : 0) * 16;
    bool bad = false, unsorted = false;

    // lists, weights and v of the chunk at token c0 into set b
    auto stage = [&](int c0, int b) {
        if (c0 < T) {
            const int n = min(C, T - c0);
            const int64_t tok0 = chain * T + c0;
            unsigned char* const set = smC + b * S.set;
            for (int t = warp; t < n; t += warps) {
                for (int e = lane; e < kw; e += 32) {
                    ck_cp4(set + S.iw + (t * pw + e) * 4, a.idx_w + (tok0 + t) * kw + e);
                    ck_cp4(set + S.ww + (t * pw + e) * 4, a.w_w + (tok0 + t) * kw + e);
                }
                for (int e = lane; e < kr; e += 32) {
                    ck_cp4(set + S.ir + (t * pr + e) * 4, a.idx_r + (tok0 + t) * kr + e);
                    ck_cp4(set + S.wr + (t * pr + e) * 4, a.w_r + (tok0 + t) * kr + e);
                }
            }
            for (int x = tid; x < n * DCH; x += threads) {
                const int t = x / DCH, q = x % DCH;
                if (split * DCH + q < nch)
                    ck_cp16(set + S.v + x * 16, static_cast<const char*>(a.v) + (tok0 + t) * rowbytes + (split * DCH + q) * 16);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    stage(0, 0);
    for (int c0 = 0, b = 0; c0 < T; c0 += C, b ^= 1) {
        const int n = min(C, T - c0);
        const int64_t tok0 = chain * T + c0;
        unsigned char* const set = smC + b * S.set;
        const int* const s_iw = reinterpret_cast<const int*>(set + S.iw);
        const float* const s_ww = reinterpret_cast<const float*>(set + S.ww);
        const int* const s_ir = reinterpret_cast<const int*>(set + S.ir);
        const float* const s_wr = reinterpret_cast<const float*>(set + S.wr);
        const unsigned char* const s_v = set + S.v;
        // ---- gates, cleared bitmaps
        for (int t = tid; t < n; t += threads) {
            const float al = load_elem<D>(a.alpha, tok0 + t);
            // log(alpha) floored at -80 (e^-80 < 2^-115): a gate of exactly 0, which the fp32
            // gate formula reaches for large A softplus(.), then decays to below fp32 precision
            // of any stored value instead of making lam = -inf and exp(-inf - -inf) = NaN
            const float la = al > 0.f ? fmaxf(logf(al), -80.f) : -80.f;
            s_la[t] = la;
            s_al[t] = la > -80.f ? al : __expf(-80.f);
            s_be[t] = load_elem<D>(a.beta, tok0 + t);
        }
        for (int i = tid; i < 2 * CK_WORDS / 4; i += threads) reinterpret_cast<uint4*>(seen)[i] = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
        // ---- matching: buckets met once, then twice
        for (int t = warp; t < n; t += warps) {
            auto mark = [&](const int* l, int k) {
                for (int e = lane; e < k; e += 32) {
                    const int s = l[e];
                    bad |= static_cast<uint32_t>(s) >= N;
                    unsorted |= e > 0 && l[e - 1] >= s;       // the look-ups need strictly ascending lists
                    const uint32_t h = ck_bucket(s), bit = 1u << (h & 31);
                    if (atomicOr(seen + (h >> 5), bit) & bit) atomicOr(dup + (h >> 5), bit);
                }
            };
            mark(s_iw + t * pw, kw);
            mark(s_ir + t * pr, kr);
        }
        __syncthreads();
        // a warp per token: coefficients, links and the token's rows of A and QK (lane u: column u)
        for (int t = warp; t < n; t += warps) {
            const float la_u = lane < n ? s_la[lane] : 0.f, la_t = s_la[t], al_t = s_al[t];
            const uint32_t upto = 0xffffffffu >> (31 - t);    // tokens u <= t
            float accA = 0.f, accQ = 0.f;
#pragma unroll
            for (int side = 0; side < 2; ++side) {            // 0: write entries, 1: read entries
                const int k = side ? kr : kw;
                const int* l = side ? s_ir + t * pr : s_iw + t * pw;
                const float* wl = side ? s_wr + t * pr : s_ww + t * pw;
                for (int e0 = 0; e0 < k; e0 += 32) {
                    const int e = e0 + lane;
                    const int s = e < k ? l[e] : 0;
                    const bool ok = e < k && static_cast<uint32_t>(s) < N;
                    const float w = ok ? wl[e] : 0.f;
                    const uint32_t h = ck_bucket(s);
                    const bool maybe = ok && ((dup[h >> 5] >> (h & 31)) & 1u);
                    if (e < k) {
                        if (side) {
                            s_cfr[t * pr + e] = w;
                        } else {
                            s_cfw[t * pw + e] = w * al_t;
                            s_lam[t * pw + e] = la_t;
                            s_link[t * pw + e] = ok ? 0u : CK_NOT_LAST;   // (a bad slot is never written)
                        }
                    }
                    uint32_t todo = __ballot_sync(0xffffffffu, maybe);
                    __syncwarp();
                    while (todo) {                            // warp-uniform
                        const int src = __ffs(todo) - 1;
                        todo &= todo - 1;
                        const int sq = __shfl_sync(0xffffffffu, s, src);
                        const float wq = __shfl_sync(0xffffffffu, w, src);
                        const int pos = lane < n ? find_slot(s_iw + lane * pw, kw, sq) : -1;
                        const uint32_t occ = __ballot_sync(0xffffffffu, pos >= 0);
                        const bool mine = pos >= 0 && lane <= t;
                        float pref = mine ? la_u : 0.f;       // inclusive scan of the slot's log-decays
#pragma unroll
                        for (int off = 1; off < 32; off <<= 1) {
                            const float x = __shfl_up_sync(0xffffffffu, pref, off);
                            if (lane >= off) pref += x;
                        }
                        const float lam = __shfl_sync(0xffffffffu, pref, 31);
                        const bool term = mine && (side != 0 || lane < t);
                        if (term) {
                            const float x = wq * s_ww[lane * pw + pos];
                            const float g = __expf(lam - pref);
                            if (side) accQ = fmaf(x, g, accQ); else accA = fmaf(x, g, accA);
                        }
                        const uint32_t before = occ & upto & ~(1u << t);
                        const int up = 31 - __clz(before | 1u);       // latest earlier writer (if any)
                        const int ppos = __shfl_sync(0xffffffffu, pos, up);
                        if (lane == 0) {
                            const int q = e0 + src;
                            if (side) {
                                s_cfr[t * pr + q] = (occ & upto) ? wq * __expf(lam) : wq;
                            } else if (occ & ~(1u << t)) {
                                if (before) s_cfw[t * pw + q] = wq * __expf(lam);
                                s_lam[t * pw + q] = lam;
                                s_link[t * pw + q] = ((occ & ~upto) ? CK_NOT_LAST : 0u) |
                                                     (before ? 1u + static_cast<uint32_t>(up * 64 + ppos) : 0u);
                            }
                        }
                    }
                }
            }
            const uint32_t mA = __ballot_sync(0xffffffffu, accA != 0.f), mQ = __ballot_sync(0xffffffffu, accQ != 0.f);
            if (lane < n) { s_A[t * (C + 1) + lane] = accA; s_QK[t * (C + 1) + lane] = accQ; }
            if (lane == 0) { s_mA[t] = mA; s_mQ[t] = mQ; }
        }
        stage(c0 + C, b ^ 1);                                 // under the memory phases
        __syncwarp();
        // ---- gather (the warp's own tokens: their coefficients are its own)
        bool solve = false;
        for (int t = warp; t < n; t += warps) {
            float2 R2[E / 2], I2[E / 2];
#pragma unroll
            for (int j = 0; j < E / 2; ++j) { R2[j] = make_float2(0.f, 0.f); I2[j] = make_float2(0.f, 0.f); }
            const int kmax = kw > kr ? kw : kr;
            for (int m0 = 0; m0 < kmax; m0 += CK_ROWS * RG) {
                uint4 xw[CK_ROWS], xr[CK_ROWS];
#pragma unroll
                for (int q = 0; q < CK_ROWS; ++q) {
                    const int m = m0 + q * RG + rg;
                    const int s = m < kw ? s_iw[t * pw + m] : -1;
                    xw[q] = make_uint4(0u, 0u, 0u, 0u);
                    if (on && static_cast<uint32_t>(s) < N) xw[q] = ck_ldcg(mrow + static_cast<uint64_t>(static_cast<uint32_t>(s)) * rowbytes);
                }
#pragma unroll
                for (int q = 0; q < CK_ROWS; ++q) {
                    const int m = m0 + q * RG + rg;
                    const int s = m < kr ? s_ir[t * pr + m] : -1;
                    xr[q] = make_uint4(0u, 0u, 0u, 0u);
                    if (on && static_cast<uint32_t>(s) < N) xr[q] = ck_ldcg(mrow + static_cast<uint64_t>(static_cast<uint32_t>(s)) * rowbytes);
                }
#pragma unroll
                for (int q = 0; q < CK_ROWS; ++q) {
                    const int m = m0 + q * RG + rg;
                    const float cf = m < kw ? s_cfw[t * pw + m] : 0.f;
                    float2 f[E / 2];
                    unpack16x2<D>(xw[q], f);
#pragma unroll
                    for (int j = 0; j < E / 2; ++j) R2[j] = __ffma2_rn(make_float2(cf, cf), f[j], R2[j]);
                }
#pragma unroll
                for (int q = 0; q < CK_ROWS; ++q) {
                    const int m = m0 + q * RG + rg;
                    const float cf = m < kr ? s_cfr[t * pr + m] : 0.f;
                    float2 f[E / 2];
                    unpack16x2<D>(xr[q], f);
#pragma unroll
                    for (int j = 0; j < E / 2; ++j) I2[j] = __ffma2_rn(make_float2(cf, cf), f[j], I2[j]);
                }
            }
            float R[E], I[E];
#pragma unroll
            for (int j = 0; j < E / 2; ++j) {
                R[2 * j] = R2[j].x; R[2 * j + 1] = R2[j].y;
                I[2 * j] = I2[j].x; I[2 * j + 1] = I2[j].y;
            }
#pragma unroll
            for (int off = DCH; off < 32; off <<= 1) {
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    R[j] += __shfl_xor_sync(0xffffffffu, R[j], off);
                    I[j] += __shfl_xor_sync(0xffffffffu, I[j], off);
                }
            }
            const bool dep = s_mA[t] != 0u;
            solve |= dep;
            if (rg == 0) {
                const float bt = s_be[t];
                float x[E];
                unpack16<D>(*reinterpret_cast<const uint4*>(s_v + (t * DCH + c) * 16), x);
#pragma unroll
                for (int j = 0; j < E; ++j) x[j] -= R[j];                 // v_t - R_t
                if (!dep) {
#pragma unroll
                    for (int j = 0; j < E; ++j) x[j] *= bt;
                }
                float* dst = (dep ? s_R : s_U) + t * dr + c * E;
#pragma unroll
                for (int q = 0; q < E / 4; ++q) {
                    *reinterpret_cast<float4*>(dst + 4 * q) = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
                    *reinterpret_cast<float4*>(s_I + t * dr + c * E + 4 * q) = make_float4(I[4 * q], I[4 * q + 1], I[4 * q + 2], I[4 * q + 3]);
                }
            }
        }
        // ---- solve: the tokens whose row of A is not empty, in order, a thread per element
        if (__syncthreads_or(solve)) {
            for (int d = tid; d < dr; d += threads) {
                for (int t = 0; t < n; ++t) {
                    uint32_t mask = s_mA[t];
                    if (mask == 0u) continue;
                    float acc = s_R[t * dr + d];
                    while (mask) {
                        const int u = __ffs(mask) - 1;
                        mask &= mask - 1;
                        acc = fmaf(-s_A[t * (C + 1) + u], s_U[u * dr + d], acc);
                    }
                    s_U[t * dr + d] = s_be[t] * acc;
                }
            }
            __syncthreads();
        }
        // ---- output
        for (int x = tid; x < n * DCH; x += threads) {
            const int t = x / DCH, q0 = x % DCH;
            if (split * DCH + q0 >= nch) continue;
            float o[E];
#pragma unroll
            for (int j = 0; j < E; ++j) o[j] = s_I[t * dr + q0 * E + j];
            uint32_t mask = s_mQ[t];
            while (mask) {
                const int u = __ffs(mask) - 1;
                mask &= mask - 1;
                const float qk = s_QK[t * (C + 1) + u];
#pragma unroll
                for (int j = 0; j < E; ++j) o[j] = fmaf(qk, s_U[u * dr + q0 * E + j], o[j]);
            }
            *reinterpret_cast<uint4*>(static_cast<char*>(a.y) + (tok0 + t) * rowbytes + (split * DCH + q0) * 16) = pack16<D>(o);
        }
        // ---- scatter: the last writer of each slot (a warp per token, all its rows in flight)
        for (int t = warp; t < n && on; t += warps) {
            const int* const it = s_iw + t * pw;
            const float al = s_al[t];
            float2 u[E / 2];
#pragma unroll
            for (int j = 0; j < E / 2; ++j) u[j] = *reinterpret_cast<const float2*>(s_U + t * dr + c * E + 2 * j);
            for (int m0 = rg; m0 < kw; m0 += CK_ROWS * RG) {
                uint4 x[CK_ROWS];
                uint32_t link[CK_ROWS];
#pragma unroll
                for (int q = 0; q < CK_ROWS; ++q) {
                    const int m = m0 + q * RG;
                    link[q] = m < kw ? s_link[t * pw + m] : CK_NOT_LAST;
                    x[q] = make_uint4(0u, 0u, 0u, 0u);
                    if (!(link[q] & CK_NOT_LAST)) x[q] = ck_ldcg(mrow + static_cast<uint64_t>(static_cast<uint32_t>(it[m])) * rowbytes);
                }
#pragma unroll
                for (int q = 0; q < CK_ROWS; ++q) {
                    if (link[q] & CK_NOT_LAST) continue;
                    const int m = m0 + q * RG;
                    const float w = s_ww[t * pw + m];
                    float2 f[E / 2];
                    unpack16x2<D>(x[q], f);
                    uint32_t prev = link[q];
                    if (prev == 0u) {
#pragma unroll
                        for (int j = 0; j < E / 2; ++j)
                            f[j] = __ffma2_rn(make_float2(w, w), u[j], __fmul2_rn(make_float2(al, al), f[j]));
                    } else {                                  // with the slot's earlier writers
                        const float lam = s_lam[t * pw + m], dec = __expf(lam);
#pragma unroll
                        for (int j = 0; j < E / 2; ++j)
                            f[j] = __ffma2_rn(make_float2(w, w), u[j], __fmul2_rn(make_float2(dec, dec), f[j]));
                        while (prev) {
                            const int pt = (prev - 1) >> 6, pe = pt * pw + static_cast<int>((prev - 1) & 63u);
                            const float cf = __expf(lam - s_lam[pe]) * s_ww[pe];
#pragma unroll
                            for (int j = 0; j < E / 2; ++j)
                                f[j] = __ffma2_rn(make_float2(cf, cf), *reinterpret_cast<const float2*>(s_U + pt * dr + c * E + 2 * j), f[j]);
                            prev = s_link[pe] & 0xffffu;
                        }
                    }
                    *reinterpret_cast<uint4*>(mrow + static_cast<uint64_t>(static_cast<uint32_t>(it[m])) * rowbytes) = pack16x2<D>(f);
                }
            }
        }
        __syncthreads();                                      // rows stored before the next chunk's gathers
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (bad) flag_error(a.err, ERR_BAD_INDEX);
    if (unsorted) flag_error(a.err, ERR_UNSORTED);
}

template <class D, int DCH>
static cudaError_t launch_chunk(const RecArgs& a, int C, int nsplit, cudaStream_t stream) {
    const size_t smem = chunk_smem(C, a.kw, a.kr, DCH * D::E, D::BYTES).total;
    cudaError_t e = cudaFuncSetAttribute(k_recur_chunk<D, DCH>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_ALLOWED);
    if (e != cudaSuccess) return e;
    const int64_t ctas = static_cast<int64_t>(a.B) * a.H * nsplit;
    const int threads = C <= 4 ? 128 : C <= 8 ? 256 : CK_MAX_THREADS;
    k_recur_chunk<D, DCH><<<static_cast<unsigned>(ctas), threads, smem, stream>>>(a, C, nsplit);
    return cudaGetLastError();
}

// The d-range of a CTA: 256-byte rows whole (16 pieces) when the chains alone fill the SMs, else
// split down to 64-byte pieces until they do, but no further: every d-range repeats the matching,
// and a second CTA waits for a first.  64 chains, d_v = 128 bf16: 1.60 ms whole, 1.20 ms in two
// d-ranges, 2.20 ms in four.
template <class D>
static cudaError_t launch_chunk_dtype(const RecArgs& a, int C, cudaStream_t stream) {
    const int64_t chains = static_cast<int64_t>(a.B) * a.H;
    const int nch = a.dv / D::E;
    int dch = 16;
    while (dch > 1 && dch / 2 >= nch) dch /= 2;
    while (dch > 4 && chains * ((nch + dch - 1) / dch) < 128) dch /= 2;
    const int nsplit = (nch + dch - 1) / dch;
    switch (dch) {
        case 16: return launch_chunk<D, 16>(a, C, nsplit, stream);
        case 8: return launch_chunk<D, 8>(a, C, nsplit, stream);
        case 4: return launch_chunk<D, 4>(a, C, nsplit, stream);
        case 2: return launch_chunk<D, 2>(a, C, nsplit, stream);
        default: return launch_chunk<D, 1>(a, C, nsplit, stream);
    }
}

cudaError_t launch_recur_chunkwise(int dtype, const RecArgs& a, int C, cudaStream_t stream) {
    return dtype == 0 ? launch_chunk_dtype<F32>(a, C, stream) : launch_chunk_dtype<BF16>(a, C, stream);
}

}  // namespace sdm
