// K-ADDR: sparse key selection (Sec. 3.1 item 1; Sec. 2 "Product Key Memory"; Sec. 4 softmax).
//
// For every token x (k for the write side, q for the read side) of head h:
//   s = P_h x in R^{2S} (PROJECTED) or s = x (DIRECT, d_k = 2S); s1 = s[0:S], s2 = s[S:2S];
//   T1 = top_k(s1), T2 = top_k(s2) under (score desc, index asc);
//   slots = top_k over (i, j) in T1 x T2 of s1[i] + s2[j] under (score desc, slot asc),
//           slot = i*S + j  (the PKM identity of Sec. 2 makes this the top-k of all N);
//   w = softmax of the selected scores; output sorted ascending by slot (App. A.2).
//
// Exactness.  The selected SETS must equal those of the float64 definition.  Scores are
// computed in fp32 with a rigorous error bound eps = cbound * max_j ||P_j|| * ||x||
// (Cauchy-Schwarz on the accumulation error bound gamma_dk * sum |P_jd x_d|).  A top-k
// boundary is certified when the gap between the k-th and (k+1)-th fp32 values exceeds
// 2 eps; otherwise the entries inside the uncertainty band are re-scored with compensated fp32
// sums, and those closer than that bound in float64 with the sequential ascending-d order
// (bit-identical to the float64 definition: products of two storage numbers are exact in
// float64).  Each chunk keeps the top L = k + margin entries so the band is normally inside the
// list; if it is not, the whole half (or all k^2 candidates) is looked through.  A NaN score (a
// row of P that holds one) is never selected; scores of -inf (masked ones of DIRECT
// addressing) rank last, by index.
//
// Scores and lists: k_addr_mma.cu (tensor cores, one list per half) or k_addr_scores here (FFMA,
//   fixed d order; one CTA = 128 tokens of one head x one column chunk, a thread per token).
// Certified pass, over every token-side: k_addr_finalize_stair (k <= 32) or
//   k_addr_finalize_thread (k > 32), a thread each, with one list per half;
//   k_addr_finalize<FIN_FAST>, a warp each, for several (k <= 32), or slots past the sort keys.
// Band pass, over those not certified (queue A): k_addr_band_thread, or k_addr_finalize<FIN_BAND>
//   for short queues and several lists per half.
// Rare pass, over what that leaves (queue B): k_addr_finalize<FIN_FULL> or k_addr_rare_wide, a
//   warp each.
// k_addr_finalize_wide does all three for k > 32 with several lists per half, or without queues.
// Small problems (a decode step) take one launch for all of it: k_addr_small.cu.
#include "k_addr_warp.cuh"

namespace sdm {

constexpr int A_TOK = 128;     // tokens per score CTA (one per thread)
constexpr int A_SUB = 32;      // columns accumulated per pass
constexpr int A_PPITCH = 36;   // fp32 pitch of the staged P sub-chunk (16-byte aligned, fewer bank conflicts)
constexpr int F_THREADS = 64;  // tokens per finalize CTA (wide lists)
template <int L>
__device__ __forceinline__ float pick(const float (&a)[L], int p) {
    float r = a[0];
#pragma unroll
    for (int q = 1; q < L; ++q) r = (q == p) ? a[q] : r;
    return r;
}

// ------------------------------------------------------------------------------------------
// Kernel A: fp32 half-scores + per-chunk top-L
// ------------------------------------------------------------------------------------------
template <class D, int L>
__global__ void __launch_bounds__(A_TOK) k_addr_scores(const AddrArgs a) {
    extern __shared__ __align__(16) float smA[];
    float* xs = smA;                               // [dk][A_TOK]  x of the CTA's tokens, transposed
    float* ps = smA + a.dk * A_TOK;                // [dk][A_PPITCH] staged P rows of one sub-chunk
    const int tid = threadIdx.x;
    const int which = blockIdx.z / a.H, h = blockIdx.z % a.H;
    const int chunk = blockIdx.y;
    const int hf = chunk / a.ncc, cc = chunk % a.ncc;
    const int c0 = cc * a.cw, c1 = min(a.S, c0 + a.cw);
    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    const int64_t u0 = static_cast<int64_t>(blockIdx.x) * A_TOK;
    const void* X = a.X[which];
    const void* P = a.P[which];

    for (int e = tid; e < A_TOK * a.dk; e += A_TOK) {
        const int ul = e / a.dk, d = e - ul * a.dk;
        const int64_t u = u0 + ul;
        float val = 0.f;
        if (u < BT) {
            const int64_t b = u / a.T, t = u - b * a.T;
            val = load_elem<D>(X, ((b * a.H + h) * a.T + t) * a.dk + d);
        }
        xs[d * A_TOK + ul] = val;
    }

    TopList<L> top;
    top.clear();
    const int64_t prow0 = static_cast<int64_t>(h) * 2 * a.S + static_cast<int64_t>(hf) * a.S;
    for (int s0 = c0; s0 < c1; s0 += A_SUB) {
        __syncthreads();   // xs staged / previous sub-chunk consumed
        float acc[A_SUB];
        if (P == nullptr) {
#pragma unroll
            for (int jj = 0; jj < A_SUB; ++jj) {
                const int col = s0 + jj;
                acc[jj] = (col < c1) ? xs[(hf * a.S + col) * A_TOK + tid] : -INFINITY;
            }
        } else {
            for (int e = tid; e < A_SUB * a.dk; e += A_TOK) {
                const int jj = e / a.dk, d = e - jj * a.dk;
                const int col = s0 + jj;
                ps[d * A_PPITCH + jj] = (col < c1) ? load_elem<D>(P, (prow0 + col) * a.dk + d) : 0.f;
            }
            __syncthreads();
#pragma unroll
            for (int jj = 0; jj < A_SUB; ++jj) acc[jj] = 0.f;
            for (int d = 0; d < a.dk; ++d) {            // ascending d, one rounding per step
                const float xv = xs[d * A_TOK + tid];
                const float4* pr = reinterpret_cast<const float4*>(ps + d * A_PPITCH);
#pragma unroll
                for (int q = 0; q < A_SUB / 4; ++q) {
                    const float4 p4 = pr[q];
                    acc[4 * q + 0] = fmaf(xv, p4.x, acc[4 * q + 0]);
                    acc[4 * q + 1] = fmaf(xv, p4.y, acc[4 * q + 1]);
                    acc[4 * q + 2] = fmaf(xv, p4.z, acc[4 * q + 2]);
                    acc[4 * q + 3] = fmaf(xv, p4.w, acc[4 * q + 3]);
                }
            }
        }
#pragma unroll
        for (int jj = 0; jj < A_SUB; ++jj) {
            const int col = s0 + jj;
            if (col < c1 && acc[jj] > top.v[L - 1]) top.push_scan(acc[jj], col);
        }
    }

    const int64_t u = u0 + tid;
    if (u < BT) {
        const int64_t base = part_at(blockIdx.z, a.ncc, chunk, BT, u, L, 0);
#pragma unroll
        for (int p = 0; p < L; ++p) {
            a.part_v[base + p] = top.v[p];
            a.part_i[base + p] = top.i[p];
        }
    }
}

// Twice the fp32 score error bound of a token-side, rounded up; sum of squares in d order, so that the passes of
// one token-side decide alike.
template <class D>
__device__ __forceinline__ float twice_error_bound(const AddrArgs& a, int side, int h, int64_t b, int64_t t) {
    if (a.P[side] == nullptr) return 0.f;
    const void* X = a.X[side];
    const int64_t xoff = ((b * a.H + h) * a.T + t) * a.dk;
    float ss = 0.f;
    const char* xr = static_cast<const char*>(X) + xoff * D::BYTES;
    if ((reinterpret_cast<uintptr_t>(xr) & 15) == 0 && (a.dk * D::BYTES) % 16 == 0) {
        const int nq = a.dk * D::BYTES / 16;
        for (int q0 = 0; q0 < nq; q0 += 4) {
            uint4 xq[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q0 + u < nq) xq[u] = __ldg(reinterpret_cast<const uint4*>(xr) + q0 + u);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (q0 + u < nq) {
                    float f[D::E];
                    unpack16<D>(xq[u], f);
#pragma unroll
                    for (int e = 0; e < D::E; ++e) ss = fmaf(f[e], f[e], ss);
                }
        }
    } else {
        for (int d = 0; d < a.dk; ++d) {
            const float xv = load_elem<D>(X, xoff + d);
            ss = fmaf(xv, xv, ss);
        }
    }
    // (1 + 2^-12) covers the roundings of ||x||^2, its square root and the products
    return __fmul_ru(__fmul_ru(__fmul_ru(2.f * a.cbound, a.pnorm[side * a.H + h]), sqrtf(ss)), 1.f + 0x1p-12f);
}

// Three passes over token-sides, each kernel holding only the code its cases need (the
// band code's registers and instruction footprint would otherwise slow the common path):
//   MODE 0: every token-side; those whose two half boundaries and outer-sum boundary are
//           all certified are finished, the others go to queue A (nothing written);
//   MODE 1: queue A, with band resolution by compensated rescoring; near-ties and bands
//           that leave the kept lists go to queue B;
//   MODE 2: queue B (or every token-side when there is no queue) with every path.

template <class D, int L, int MODE>
__global__ void __launch_bounds__(FW_WARPS * 32, 4) k_addr_finalize(const AddrArgs a) {
    static_assert(L <= 36, "warp finalize handles k <= 32");
    __shared__ float wv[FW_WARPS][3][64];
    __shared__ int wi[FW_WARPS][3][64];
    __shared__ unsigned wstat[FW_WARPS][STAT_COUNT];
    const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
    if (lane < STAT_COUNT) wstat[wq][lane] = 0u;
    __syncwarp();
    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    const int64_t all = 2 * a.H * BT;
    const bool queued = a.queue != nullptr;               // then all < 2^31
    int* const qa = queued ? a.queue + 2 : nullptr;        // queue A items
    int* const qb = queued ? a.queue + 2 + all : nullptr;  // queue B items
    const int64_t items = MODE == FIN_FAST || !queued ? all
                        : static_cast<int64_t>(reinterpret_cast<volatile int*>(a.queue)[MODE == FIN_BAND ? 0 : 1]);
    // persistent warps: a warp takes token-sides it, it + (all warps), ...
    for (int64_t it = static_cast<int64_t>(blockIdx.x) * FW_WARPS + wq; it < items;
         it += static_cast<int64_t>(gridDim.x) * FW_WARPS) {
    int64_t item, u, b, t;
    int z;
    if (queued) {                                          // 32-bit index arithmetic
        const uint32_t it32 = MODE == FIN_FAST ? static_cast<uint32_t>(it)
                            : static_cast<uint32_t>((MODE == FIN_BAND ? qa : qb)[it]);
        const uint32_t z32 = it32 / static_cast<uint32_t>(BT);
        const uint32_t u32 = it32 - z32 * static_cast<uint32_t>(BT);
        const uint32_t b32 = u32 / static_cast<uint32_t>(a.T);
        item = it32; z = static_cast<int>(z32); u = u32; b = b32; t = u32 - b32 * static_cast<uint32_t>(a.T);
    } else {
        item = it;
        z = static_cast<int>(item / BT);
        u = item - z * BT;
        b = u / a.T;
        t = u - b * a.T;
    }
    const int side = z / a.H, h = z % a.H;
    const int k = a.kk[side];
    const int S = a.S;
    TokenCtx c;
    c.err = a.err;
    c.stat = wstat[wq];
    c.count_band = MODE != FIN_FULL || !queued;
    c.P = a.P[side];
    c.X = a.X[side];
    c.xoff = ((b * a.H + h) * a.T + t) * a.dk;
    c.prow0 = static_cast<int64_t>(h) * 2 * S;
    c.dk = a.dk;
    c.S = S;
    float* sv0 = wv[wq][0]; int* si0 = wi[wq][0];          // staging / merge output / A1
    float* sv1 = wv[wq][1]; int* si1 = wi[wq][1];          // A2
    float* sv2 = wv[wq][2]; int* si2 = wi[wq][2];          // candidates / final

    float e2 = 0.f;                                        // 2 x the fp32 score error bound, rounded up
    if (c.P != nullptr) {
        float ss = 0.f;
        for (int d = lane; d < a.dk; d += 32) {
            const float xv = load_elem<D>(c.X, c.xoff + d);
            ss = fmaf(xv, xv, ss);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
        // (1 + 2^-12) covers the roundings of ||x||^2, its square root and the products
        e2 = __fmul_ru(__fmul_ru(__fmul_ru(2.f * a.cbound, a.pnorm[side * a.H + h]), sqrtf(ss)), 1.f + 0x1p-12f);
    }
    const int64_t tokoff = ((b * a.H + h) * a.T + t) * k;  // [B, H, T, k] layout
    auto load = [&](int hf, float& v0, int& i0, float& v1, int& i1) {
        // chunk 0 of this half
        int64_t base = part_at(z, a.ncc, hf * a.ncc, BT, u, L, 0);
        v0 = lane < L ? a.part_v[base + lane] : -INFINITY;
        v1 = lane + 32 < L ? a.part_v[base + lane + 32] : -INFINITY;
        i0 = lane < L ? a.part_i[base + lane] : INT_MAX;
        i1 = lane + 32 < L ? a.part_i[base + lane + 32] : INT_MAX;
        for (int cc = 1; cc < a.ncc; ++cc) {                  // merge later chunks (larger columns)
            base = part_at(z, a.ncc, hf * a.ncc + cc, BT, u, L, 0);
            const float w0 = lane < L ? a.part_v[base + lane] : -INFINITY;
            const float w1 = lane + 32 < L ? a.part_v[base + lane + 32] : -INFINITY;
            const int j0 = lane < L ? a.part_i[base + lane] : INT_MAX;
            const int j1 = lane + 32 < L ? a.part_i[base + lane + 32] : INT_MAX;
            // ties: the earlier chunk first
            const int ra0 = lane + lane_count_before(w0, w1, L, v0, true);
            const int ra1 = lane + 32 + lane_count_before(w0, w1, L, v1, true);
            const int rb0 = lane + lane_count_before(v0, v1, L, w0, false);
            const int rb1 = lane + 32 + lane_count_before(v0, v1, L, w1, false);
            __syncwarp();
            if (lane < L && ra0 < L) { sv0[ra0] = v0; si0[ra0] = i0; }
            if (lane + 32 < L && ra1 < L) { sv0[ra1] = v1; si0[ra1] = i1; }
            if (lane < L && rb0 < L) { sv0[rb0] = w0; si0[rb0] = j0; }
            if (lane + 32 < L && rb1 < L) { sv0[rb1] = w1; si0[rb1] = j1; }
            __syncwarp();
            v0 = lane < L ? sv0[lane] : -INFINITY;       i0 = lane < L ? si0[lane] : INT_MAX;
            v1 = lane + 32 < L ? sv0[lane + 32] : -INFINITY; i1 = lane + 32 < L ? si0[lane + 32] : INT_MAX;
        }
    };
    if (!finalize_warp<D, L, MODE>(c, k, e2, a.idx[side] + tokoff, a.w[side] + tokoff, sv0, si0, sv1, si1, sv2, si2, lane, load)) {
        if (lane == 0) {
            if (MODE == FIN_FAST) qa[atomicAdd(a.queue, 1)] = static_cast<int>(item);
            else qb[atomicAdd(a.queue + 1, 1)] = static_cast<int>(item);
        }
    }
    __syncwarp();                                           // per-warp staging is reused
    }
    __syncwarp();
    if (lane > 0 && lane < STAT_COUNT && wstat[wq][lane] != 0u) stat_add(a.err, lane, wstat[wq][lane]);
}
// ------------------------------------------------------------------------------------------
// Kernel B, wide lists (k > 32) in several chunks per half: insertion-based merge and candidate
// selection, one thread per token-side with every path
// ------------------------------------------------------------------------------------------
template <class D, int L>
__global__ void __launch_bounds__(F_THREADS) k_addr_finalize_wide(const AddrArgs a) {
    extern __shared__ __align__(16) float smB[];
    const int tid = threadIdx.x;
    float* A1v = smB + tid;                       // exact top-k of half 1 (fp32 value, column), pitch F_THREADS
    int* A1i = reinterpret_cast<int*>(smB + 1 * L * F_THREADS) + tid;
    float* A2v = smB + 2 * L * F_THREADS + tid;   // exact top-k of half 2
    int* A2i = reinterpret_cast<int*>(smB + 3 * L * F_THREADS) + tid;
    float* Fv = smB + 4 * L * F_THREADS + tid;    // final selection (fp32 score, slot)
    int* Fi = reinterpret_cast<int*>(smB + 5 * L * F_THREADS) + tid;

    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    const int z = blockIdx.y;
    const int side = z / a.H, h = z % a.H;
    const int64_t u = static_cast<int64_t>(blockIdx.x) * F_THREADS + tid;
    if (u >= BT) return;   // no block-level synchronisation below
    const int k = a.kk[side];
    const int S = a.S;
    const int64_t b = u / a.T, t = u - b * a.T;
    TokenCtx c;
    c.err = a.err;
    c.stat = nullptr;
    c.count_band = true;
    c.P = a.P[side];
    c.X = a.X[side];
    c.xoff = ((b * a.H + h) * a.T + t) * a.dk;
    c.prow0 = static_cast<int64_t>(h) * 2 * S;
    c.dk = a.dk;
    c.S = S;

    const double eps = 0.5 * static_cast<double>(twice_error_bound<D>(a, side, h, b, t));

    float amax[2];
#pragma unroll 1
    for (int hf = 0; hf < 2; ++hf) {
        TopList<L> top;
        top.clear();
        for (int cc = 0; cc < a.ncc; ++cc) {
            const int64_t base = part_at(z, a.ncc, hf * a.ncc + cc, BT, u, L, 0);
            for (int p = 0; p < L; ++p) {
                const float v = a.part_v[base + p];
                const int i = a.part_i[base + p];
                if (!top.admits(v, i)) break;
                top.push(v, i);
            }
        }
        float* Av = hf ? A2v : A1v;
        int* Ai = hf ? A2i : A1i;
        bool certified = S <= k && pick(top.v, k - 1) != -INFINITY;
        if (!certified) certified = static_cast<double>(pick(top.v, k - 1)) - static_cast<double>(pick(top.v, k)) > 2.0 * eps;
        if (certified) {
#pragma unroll
            for (int p = 0; p < L; ++p)
                if (p < k) { Av[p * F_THREADS] = top.v[p]; Ai[p * F_THREADS] = top.i[p]; }
        } else {
            float lv[L];
            int li[L];
#pragma unroll
            for (int p = 0; p < L; ++p) { lv[p] = top.v[p]; li[p] = top.i[p]; }
            stat_add(c.err, STAT_HALF_BAND);
            resolve_half<D, L>(lv, li, k, eps, c, hf, Av, Ai, F_THREADS);
        }
        amax[hf] = fmaxf(fabsf(Av[0]), fabsf(Av[(k - 1) * F_THREADS]));
    }

    // Candidates of the outer sum.  theta = a provable lower bound on the k-th best fp32 sum:
    // the first a entries of T1 times the first ceil(k/a) of T2 give >= k sums >= it.
    const double epsc = 2.0 * eps + 0x1p-22 * (static_cast<double>(amax[0]) + static_cast<double>(amax[1]));
    float theta = -INFINITY;
    for (int aa = 1;; aa *= 2) {
        if (aa > k) aa = k;
        const int bb = (k + aa - 1) / aa;
        theta = fmaxf(theta, A1v[(aa - 1) * F_THREADS] + A2v[(bb - 1) * F_THREADS]);
        if (aa == k) break;
    }
    const float lo = __double2float_rd(static_cast<double>(theta) - 2.0 * epsc);
    TopList<L> cand;
    cand.clear();
    for (int p1 = 0; p1 < k; ++p1) {
        const float a1 = A1v[p1 * F_THREADS];
        const int i1 = A1i[p1 * F_THREADS];
        if (a1 + A2v[0] < lo) break;
        for (int p2 = 0; p2 < k; ++p2) {
            const float cs = a1 + A2v[p2 * F_THREADS];
            if (cs < lo) break;
            const int f = i1 * S + A2i[p2 * F_THREADS];
            if (cand.admits(cs, f)) cand.push(cs, f);
        }
    }
    bool certified = (k == 1);
    if (!certified) certified = static_cast<double>(pick(cand.v, k - 1)) - static_cast<double>(pick(cand.v, k)) > 2.0 * epsc;
    if (certified) {
#pragma unroll
        for (int p = 0; p < L; ++p)
            if (p < k) { Fv[p * F_THREADS] = cand.v[p]; Fi[p * F_THREADS] = cand.i[p]; }
    } else {
        float cv[L];
        int cf[L];
#pragma unroll
        for (int p = 0; p < L; ++p) { cv[p] = cand.v[p]; cf[p] = cand.i[p]; }
        stat_add(c.err, STAT_COMB_BAND);
        resolve_combined<D, L>(cv, cf, k, epsc, c, A1v, A1i, A2v, A2i, Fv, Fi, F_THREADS);
    }

    // softmax over the selected scores, then ascending slot order
    float m = -INFINITY;
    for (int p = 0; p < k; ++p) m = fmaxf(m, Fv[p * F_THREADS]);
    float zsum = 0.f;                             // (in slot order, as the other passes)
    const int64_t tokoff = ((b * a.H + h) * a.T + t) * k;     // [B, H, T, k] layout
    int32_t* oi = a.idx[side] + tokoff;
    float* ow = a.w[side] + tokoff;
    // selection sort by slot (k <= 64; slots are distinct)
    int last = -1;
    for (int r = 0; r < k; ++r) {
        int best = INT_MAX, bp = 0;
        for (int p = 0; p < k; ++p) {
            const int f = Fi[p * F_THREADS];
            if (f > last && f < best) { best = f; bp = p; }
        }
        oi[r] = best;
        ow[r] = expf(Fv[bp * F_THREADS] - m);
        zsum += ow[r];
        last = best;
    }
    for (int r = 0; r < k; ++r) ow[r] /= zsum;
}

// ------------------------------------------------------------------------------------------
// Rare pass for k > 32 with one list per half: a warp per token-side of queue B (near-ties, bands that
// leave the lists).  Every float64 score of the definition (sequential d order) is one lane's, so
// the lanes of a band run side by side; one thread per token-side deciding them one after another took
// 6 ms for a handful.  A band past the kept list: the (at most RW_CAND) columns of the half whose fp32 scores reach
// the band are ranked in float64.  More of them (tied or masked scores, a token of zeros) make the warp go through all
// columns, or all k * k sums, 32 at a time.
// ------------------------------------------------------------------------------------------
constexpr int RW_WARPS = 4;
constexpr int RW_CAND = 128;

// The k (<= 64) best of n scored entries by (float64 score desc, id asc), sorted, into bv/bi (shared memory of
// the warp); score(j, id) gives entry j's score and sets its id.  A NaN is never taken.  Returns the number found.  Each
// lane scores an entry; those that beat the k-th so far go in one after another, few of them where scores
// tie.  4800 token-sides of zeros (S = 256, k = 64): 3.4 ms for the addressing, 73 ms with one lane doing all of it.
template <class Score>
__device__ __forceinline__ int warp_best64(int n, int k, double* bv, int* bi, int lane, Score score) {
    int cnt = 0;
    for (int j0 = 0; j0 < n; j0 += 32) {
        int id = 0;
        double s = 0.0;
        bool open = j0 + lane < n;
        if (open) s = score(j0 + lane, id);
        open = open && s == s;
        while (true) {
            const unsigned mk = __ballot_sync(0xffffffffu, open && (cnt < k || beats64(s, id, bv[k - 1], bi[k - 1])));
            if (mk == 0u) break;                              // (warp-uniform)
            const int src = __ffs(mk) - 1;
            const double sq = __shfl_sync(0xffffffffu, s, src);
            const int iq = __shfl_sync(0xffffffffu, id, src);
            open = open && lane != src;
            const double e0 = lane < cnt ? bv[lane] : 0.0, e1 = lane + 32 < cnt ? bv[lane + 32] : 0.0;
            const int f0 = lane < cnt ? bi[lane] : 0, f1 = lane + 32 < cnt ? bi[lane + 32] : 0;
            const int at = __popc(__ballot_sync(0xffffffffu, lane < cnt && beats64(e0, f0, sq, iq))) +
                           __popc(__ballot_sync(0xffffffffu, lane + 32 < cnt && beats64(e1, f1, sq, iq)));
            const int end = min(cnt + 1, k);
            __syncwarp();                                     // every lane has read its entries
            if (lane >= at && lane < cnt && lane + 1 < end) { bv[lane + 1] = e0; bi[lane + 1] = f0; }
            if (lane + 32 >= at && lane + 32 < cnt && lane + 33 < end) { bv[lane + 33] = e1; bi[lane + 33] = f1; }
            if (lane == 0) { bv[at] = sq; bi[at] = iq; }
            cnt = end;
            __syncwarp();
        }
    }
    return cnt;
}

template <class D, int L>
__global__ void __launch_bounds__(RW_WARPS * 32) k_addr_rare_wide(const AddrArgs a) {
    __shared__ float s_av[RW_WARPS][2][L], s_cv[RW_WARPS][RW_CAND], s_ov[RW_WARPS][L];
    __shared__ int s_ai[RW_WARPS][2][L], s_ci[RW_WARPS][RW_CAND], s_oi[RW_WARPS][L];
    __shared__ double s_s64[RW_WARPS][RW_CAND + 64];          // (192: a list of 64 and the scores of two)
    const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
    float *const cv = s_cv[wq], *const ov = s_ov[wq];
    int *const ci = s_ci[wq], *const oi = s_oi[wq];
    double* const s64 = s_s64[wq];
    const int64_t BT = static_cast<int64_t>(a.B) * a.T, all = 2 * a.H * BT;
    const int items = reinterpret_cast<volatile int*>(a.queue)[1];
    for (int it = blockIdx.x * RW_WARPS + wq; it < items; it += gridDim.x * RW_WARPS) {
        const int64_t item = a.queue[2 + all + it];
        const int z = static_cast<int>(item / BT);
        const int64_t u = item - z * BT, b = u / a.T, t = u - b * a.T;
        const int side = z / a.H, h = z % a.H, k = a.kk[side], S = a.S;
        TokenCtx c;
        c.err = a.err;
        c.stat = nullptr;
        c.count_band = false;
        c.P = a.P[side];
        c.X = a.X[side];
        c.xoff = ((b * a.H + h) * a.T + t) * a.dk;
        c.prow0 = static_cast<int64_t>(h) * 2 * S;
        c.dk = a.dk;
        c.S = S;
        const float e2 = twice_error_bound<D>(a, side, h, b, t);
        // entries [cin, cin + m) of a list (v, id) with float64 scores in s64[0, m): the `need` best by
        // (score desc, id asc) follow the certain entries [0, cin) into ov/oi, in list order
        auto choose = [&](const float* v, const int* id, int cin, int m, int need) {
            for (int e = lane; e < cin; e += 32) { ov[e] = v[e]; oi[e] = id[e]; }
            int base = cin;
            for (int e0 = 0; e0 < m; e0 += 32) {
                const int e = e0 + lane;
                int rank = 0;
                if (e < m)
                    for (int f = 0; f < m; ++f) rank += (f != e && beats64(s64[f], id[cin + f], s64[e], id[cin + e])) ? 1 : 0;
                const bool take = e < m && rank < need;
                const unsigned mk = __ballot_sync(0xffffffffu, take);
                if (take) {
                    const int q = base + __popc(mk & ((1u << lane) - 1u));
                    ov[q] = v[cin + e];
                    oi[q] = id[cin + e];
                }
                base += __popc(mk);
            }
            __syncwarp();
        };
        auto count_above = [&](const float* v, int n, float x, bool strict) {
            int cnt = 0;
            for (int e0 = 0; e0 < n; e0 += 32) {
                const int e = e0 + lane;
                const float q = e < n ? v[e] : -INFINITY;
                cnt += __popc(__ballot_sync(0xffffffffu, e < n && q != -INFINITY && (strict ? q > x : q >= x)));
            }
            return cnt;
        };
        float amax[2];
        for (int hf = 0; hf < 2; ++hf) {
            float* const av = s_av[wq][hf];
            int* const ai = s_ai[wq][hf];
            const int64_t base = part_at(z, 1, hf, BT, u, L, 0);
            for (int p = lane; p < L; p += 32) { av[p] = a.part_v[base + p]; ai[p] = a.part_i[base + p]; }
            __syncwarp();
            const float vk = av[k - 1], vk1 = av[k];
            if (!((S <= k && vk != -INFINITY) || __fsub_rd(vk, vk1) > e2)) {
                const float lo = __fsub_rd(vk, e2), hi = __fadd_ru(vk1, e2);
                const int cin = count_above(av, L, hi, true), pend = count_above(av, L, lo, false);
                bool done = true;
                // (the same test as resolve_half's: the values that a rescan writes go into the weights)
                if (!(static_cast<double>(av[L - 1]) >= static_cast<double>(vk) - static_cast<double>(e2) && (S > L || av[L - 1] == -INFINITY))) {
                    if (lane == 0) stat_add(c.err, STAT_BAND_F64);
                    for (int e = lane; e < pend - cin; e += 32) s64[e] = score64<D>(c, hf, ai[cin + e]);
                    __syncwarp();
                    choose(av, ai, cin, pend - cin, k - cin);
                } else {
                    // the whole half: k columns of the list have exact scores of at least vk - e2 / 2, so the k
                    // best have them too, and fp32 scores (whose bound is no larger here) of at least vk - e2
                    if (lane == 0) stat_add(c.err, STAT_HALF_FULL);
                    auto fp32_score = [&](int j) {
                        if (c.P == nullptr) return load_elem<D>(c.X, c.xoff + static_cast<int64_t>(hf) * S + j);
                        const int64_t prow = (c.prow0 + static_cast<int64_t>(hf) * S + j) * c.dk;
                        float acc = 0.f;
                        for (int d = 0; d < c.dk; ++d) acc = fmaf(load_elem<D>(c.P, prow + d), load_elem<D>(c.X, c.xoff + d), acc);
                        return acc;
                    };
                    int m = 0;
                    for (int j0 = 0; j0 < S; j0 += 32) {
                        const int j = j0 + lane;
                        const bool keep = j < S && fp32_score(j) >= lo;
                        const unsigned mk = __ballot_sync(0xffffffffu, keep);
                        const int q = m + __popc(mk & ((1u << lane) - 1u));
                        if (keep && q < RW_CAND) ci[q] = j;
                        m += __popc(mk);
                    }
                    __syncwarp();
                    done = m <= RW_CAND && m >= k;
                    if (done) {
                        for (int e = lane; e < m; e += 32) s64[e] = score64<D>(c, hf, ci[e]);
                        __syncwarp();
                        for (int e = lane; e < m; e += 32) {
                            int rank = 0;
                            for (int f = 0; f < m; ++f) rank += (f != e && beats64(s64[f], ci[f], s64[e], ci[e])) ? 1 : 0;
                            if (rank < k) { ov[rank] = static_cast<float>(s64[e]); oi[rank] = ci[e]; }
                        }
                    }
                    __syncwarp();
                }
                if (!done) {
                    if (lane == 0) stat_add(c.err, STAT_SERIAL);
                    const int n = warp_best64(S, k, s64, ci, lane, [&](int j, int& id) { id = j; return score64<D>(c, hf, j); });
                    for (int p = lane; p < k; p += 32) {
                        ov[p] = p < n ? static_cast<float>(s64[p]) : -INFINITY;
                        oi[p] = p < n ? ci[p] : 0;
                    }
                    __syncwarp();
                }
                for (int p = lane; p < k; p += 32) { av[p] = ov[p]; ai[p] = oi[p]; }
                __syncwarp();
            }
            amax[hf] = fmaxf(fabsf(av[0]), fabsf(av[k - 1]));
        }
        // outer sums in descending order: lane l owns rows l and l + 32
        const float *const A1v = s_av[wq][0], *const A2v = s_av[wq][1];
        const int *const A1i = s_ai[wq][0], *const A2i = s_ai[wq][1];
        const float e2c = __fadd_ru(__fmul_ru(2.f, e2), __fmul_ru(0x1p-21f, __fadd_ru(amax[0], amax[1])));
        int j0 = 0, j1 = 0, len = 0;
        auto head = [&](int i, int j) { return i < k && j < k ? A1v[i] + A2v[j] : -INFINITY; };
        float h0 = head(lane, 0), h1 = head(lane + 32, 0);
        auto merge_to = [&](int n) {
            for (; len < n; ++len) {
                const bool first = h0 >= h1;
                const uint32_t key = f2key(first ? h0 : h1), best = __reduce_max_sync(0xffffffffu, key);
                const int win = __ffs(__ballot_sync(0xffffffffu, key == best)) - 1;
                if (lane == win) {
                    const int i = first ? lane : lane + 32, j = first ? j0 : j1;
                    cv[len] = key2f(best);
                    ci[len] = A1i[i] * S + A2i[j < k ? j : 0];
                    if (first) h0 = head(lane, ++j0); else h1 = head(lane + 32, ++j1);
                }
            }
            __syncwarp();
        };
        merge_to(min(k * k, L));
        const float ck = cv[k - 1], ck1 = len > k ? cv[k] : -INFINITY;
        if ((ck1 == -INFINITY && ck != -INFINITY) || __fsub_rd(ck, ck1) > e2c) {
            for (int p = lane; p < k; p += 32) { ov[p] = cv[p]; oi[p] = ci[p]; }
        } else {
            const float lo = __fsub_rd(ck, e2c), hi = __fadd_ru(ck1, e2c);
            if (len < k * k && cv[len - 1] >= lo) {
                if (lane == 0) stat_add(c.err, STAT_COMB_MERGE);
                merge_to(min(k * k, RW_CAND));
            }
            if ((len < k * k || cv[len - 1] == -INFINITY) && cv[len - 1] >= lo) {
                if (lane == 0) {
                    stat_add(c.err, STAT_COMB_FULL);
                    stat_add(c.err, STAT_SERIAL);
                }
                double *const s1 = s64 + 64, *const s2 = s64 + 128;
                for (int p = lane; p < k; p += 32) { s1[p] = score64<D>(c, 0, A1i[p]); s2[p] = score64<D>(c, 1, A2i[p]); }
                __syncwarp();
                const int n = warp_best64(k * k, k, s64, ci, lane, [&](int e, int& id) {
                    const int p1 = e / k, p2 = e - p1 * k;
                    id = A1i[p1] * S + A2i[p2];
                    return s1[p1] + s2[p2];
                });
                for (int p = lane; p < k; p += 32) {
                    const int f = p < n ? ci[p] : 0;
                    int p1 = 0, p2 = 0;
                    while (p1 < k - 1 && A1i[p1] != f / S) ++p1;
                    while (p2 < k - 1 && A2i[p2] != f % S) ++p2;
                    ov[p] = p < n ? A1v[p1] + A2v[p2] : -INFINITY;
                    oi[p] = f;
                }
            } else {
                const int cin = count_above(cv, len, hi, true), pend = count_above(cv, len, lo, false);
                if (lane == 0) stat_add(c.err, STAT_BAND_F64);
                for (int e = lane; e < pend - cin; e += 32)
                    s64[e] = score64<D>(c, 0, ci[cin + e] / S) + score64<D>(c, 1, ci[cin + e] % S);
                __syncwarp();
                choose(cv, ci, cin, pend - cin, k - cin);
            }
        }
        __syncwarp();
        // softmax, ascending slot order by rank
        float m = -INFINITY, zsum = 0.f;
        for (int p = 0; p < k; ++p) m = fmaxf(m, ov[p]);
        const int64_t tokoff = ((b * a.H + h) * a.T + t) * k;
        for (int p = lane; p < k; p += 32) {
            int rank = 0;
            for (int q = 0; q < k; ++q) rank += oi[q] < oi[p] ? 1 : 0;
            a.idx[side][tokoff + rank] = oi[p];
            cv[rank] = expf(ov[p] - m);
        }
        __syncwarp();
        for (int p = 0; p < k; ++p) zsum += cv[p];         // (in slot order, as the other passes)
        for (int p = lane; p < k; p += 32) a.w[side][tokoff + p] = cv[p] / zsum;
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------
// max_j ||P_j|| per (side, head)
// ------------------------------------------------------------------------------------------
template <class D>
__global__ void __launch_bounds__(256) k_pnorm(const AddrArgs a) {
    // one warp per row of P (lanes split d), four consecutive rows per warp; the row norms are
    // folded into pnorm[side * H + h] (zeroed before) by an integer atomicMax, which orders
    // non-negative floats correctly.  (1 + 2^-12) covers the roundings of the norm.
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = 2 * a.S;
    const int64_t total = static_cast<int64_t>(2) * a.H * rows;
    const int64_t r0 = (static_cast<int64_t>(blockIdx.x) * 8 + warp) * 4;
    int zcur = -1;
    float mx = 0.f;
    for (int q = 0; q < 4; ++q) {
        const int64_t r = r0 + q;
        if (r >= total) break;                       // warp-uniform
        const int zs = static_cast<int>(r / rows);
        const int64_t jrow = r - static_cast<int64_t>(zs) * rows;
        const int side = zs / a.H, h = zs % a.H;
        const int64_t row = (static_cast<int64_t>(h) * rows + jrow) * a.dk;
        float ss = 0.f;
        for (int d = lane; d < a.dk; d += 32) {
            const float p = load_elem<D>(a.P[side], row + d);
            ss = fmaf(p, p, ss);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
        const float nrm = sqrtf(ss) * (1.f + 0x1p-12f);
        if (zs != zcur) {
            if (zcur >= 0 && lane == 0) atomicMax(reinterpret_cast<int*>(a.pnorm) + zcur, __float_as_int(mx));
            zcur = zs;
            mx = 0.f;
        }
        mx = fmaxf(mx, nrm);
    }
    if (zcur >= 0 && lane == 0) atomicMax(reinterpret_cast<int*>(a.pnorm) + zcur, __float_as_int(mx));
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
AddrPlan addr_plan(int dtype, int direct, int B, int H, int T, int dk, int S, int kmax) {
    AddrPlan p;
    p.L = (kmax <= 8 ? 8 : kmax <= 16 ? 16 : kmax <= 32 ? 32 : 64) + 4;
    p.mma = mma_path_supported(dtype, direct, dk, S, kmax);
    p.small = addr_small(dtype, direct, p.mma, B, H, T, dk, S, kmax);
    const int64_t tiles = (static_cast<int64_t>(B) * T + A_TOK - 1) / A_TOK;
    const int64_t base = 2LL * H * tiles * 2;   // sides x heads x token tiles x halves
    int ncc = 1;
    // The tensor-core path always leaves one list per half, which the one-thread passes finish.
    // FFMA path: chunks of <= 512 columns, more of them when the token tiles alone give too few CTAs.
    if (!p.mma) {
        while ((S + ncc - 1) / ncc > 512) ncc *= 2;
        while (base * ncc < 512 && (S / (2 * ncc)) >= 64) ncc *= 2;  // enough CTAs, chunks >= 64 columns
    }
    p.ncc = ncc;
    p.cw = (S + ncc - 1) / ncc;
    return p;
}

// Queues of the three-pass warp finalize (0 when the item ids would not fit in int32: a
// single full pass is used then).
size_t addr_queue_bytes(int B, int H, int T) {
    const int64_t items = static_cast<int64_t>(2) * H * B * T;
    if (2 * items >= (static_cast<int64_t>(1) << 31) - 2) return 0;
    return static_cast<size_t>(2 + 2 * items) * sizeof(int);       // two counts, queues A and B
}

size_t addr_partial_bytes(const AddrPlan& plan, int B, int H, int T) {
    return static_cast<size_t>(2) * H * (2 * plan.ncc) * plan.L * static_cast<size_t>(B) * T * (sizeof(float) + sizeof(int));
}

// ------------------------------------------------------------------------------------------
// Certified passes, one thread per token-side (one list per half).  Same decisions as the warp
// pass (MODE 0): a token-side whose half and outer-sum boundaries are certified is finished, the
// others go to queue A.  Once both half boundaries are certified only the cells A1[i] + A2[j]
// (i, j < k) can be among the k largest, and exact tie order is irrelevant: a certified boundary
// has a positive gap, so equal values never straddle it.
// ------------------------------------------------------------------------------------------
constexpr int FT_THREADS = 64;

// Coordinates of a token-side.
struct TokenSide {
    int side, h, k;
    uint32_t b, t, u, z;
};
__device__ __forceinline__ TokenSide token_side(const AddrArgs& a, uint32_t item) {
    const uint32_t BT = static_cast<uint32_t>(a.B) * static_cast<uint32_t>(a.T);
    TokenSide s;
    s.z = item / BT;
    s.u = item - s.z * BT;
    s.side = static_cast<int>(s.z) / a.H;
    s.h = static_cast<int>(s.z) % a.H;
    s.k = a.kk[s.side];
    s.b = s.u / static_cast<uint32_t>(a.T);
    s.t = s.u - s.b * static_cast<uint32_t>(a.T);
    return s;
}
// ---- k <= 32.  With both lists descending, cell (i, j) has (i + 1)(j + 1) - 1 cells above it, so
// only the cells with (i + 1)(j + 1) <= KM + 1 can be among the KM + 1 largest: 121 of 1024 at KM = 32, in
// sorted runs along the rows and columns of the staircase.  Merging the runs (Batcher's odd-even
// merge, everything in registers with static indexes, exchanges below the cut dropped by the
// compiler) gives the k-th and (k+1)-th sums; the selected cells are those >= the k-th, written to the
// thread's shared-memory column with predicated stores, and their slots are sorted as 32-bit keys.
// No data-dependent branch and about 3,000 instructions per token-side; a walk that took the largest
// outer corner k + 1 times (the pass for k > 32 below) 7,000.  1,048,576 token-sides, k = 32: 0.38 ms
// (0.43 beside the M0 copy), the walk 0.80 (0.87).
template <int NA, int NB>
__device__ __forceinline__ void merge_desc(const float (&a)[NA], const float (&b)[NB], float (&o)[NA + NB]) {
    if constexpr (NA == 1) {
        float x = a[0];
#pragma unroll
        for (int i = 0; i < NB; ++i) { o[i] = fmaxf(x, b[i]); x = fminf(x, b[i]); }
        o[NB] = x;
    } else if constexpr (NB == 1) {
        merge_desc<1, NA>(b, a, o);
    } else {
        constexpr int AE = (NA + 1) / 2, BE = (NB + 1) / 2, AO = NA / 2, BO = NB / 2, E = AE + BE, O = AO + BO;
        float ae[AE], be[BE], ao[AO], bo[BO], ev[E], od[O];
#pragma unroll
        for (int i = 0; i < AE; ++i) ae[i] = a[2 * i];
#pragma unroll
        for (int i = 0; i < BE; ++i) be[i] = b[2 * i];
#pragma unroll
        for (int i = 0; i < AO; ++i) ao[i] = a[2 * i + 1];
#pragma unroll
        for (int i = 0; i < BO; ++i) bo[i] = b[2 * i + 1];
        merge_desc<AE, BE>(ae, be, ev);
        merge_desc<AO, BO>(ao, bo, od);
        o[0] = ev[0];
#pragma unroll
        for (int i = 0; i < O && i + 1 < E; ++i) {
            o[2 * i + 1] = fmaxf(od[i], ev[i + 1]);
            o[2 * i + 2] = fminf(od[i], ev[i + 1]);
        }
        if constexpr (O == E) o[NA + NB - 1] = od[O - 1];
        if constexpr (E == O + 2) o[NA + NB - 1] = ev[E - 1];
    }
}
// cells of column s from row s on, and of row s from column s + 1 on, that are inside the staircase
__host__ __device__ constexpr int stair_end(int km, int s) { return (km + 1) / (s + 1) < km ? (km + 1) / (s + 1) : km; }
__host__ __device__ constexpr int col_cells(int km, int s) { return stair_end(km, s) > s ? stair_end(km, s) - s : 0; }
__host__ __device__ constexpr int row_cells(int km, int s) { return stair_end(km, s) > s + 1 ? stair_end(km, s) - s - 1 : 0; }
__host__ __device__ constexpr int stair_cells(int km, int s) {        // kept of shells s, s + 1, ...
    int n = 0;
    for (int q = s; col_cells(km, q) > 0; ++q) n += col_cells(km, q) + row_cells(km, q);
    return n < km + 1 ? n : km + 1;
}
// The largest cells of shells s, s + 1, ... of the staircase, descending (at most KM + 1 of them).
template <int KM, int S>
__device__ __forceinline__ void stair_top(const float (&A1)[KM], const float (&A2)[KM], float (&o)[stair_cells(KM, S)]) {
    constexpr int C = col_cells(KM, S), R = row_cells(KM, S), KEEP = stair_cells(KM, S);
    float shell[C + R];
    {
        float col[C];
#pragma unroll
        for (int i = 0; i < C; ++i) col[i] = A1[S + i] + A2[S];
        if constexpr (R > 0) {
            float row[R > 0 ? R : 1];
#pragma unroll
            for (int j = 0; j < R; ++j) row[j] = A1[S] + A2[S + 1 + j];
            merge_desc<C, R>(col, row, shell);
        } else {
#pragma unroll
            for (int i = 0; i < C; ++i) shell[i] = col[i];
        }
    }
    if constexpr (col_cells(KM, S + 1) > 0) {
        constexpr int IN = stair_cells(KM, S + 1), OUT = C + R < KM + 1 ? C + R : KM + 1;
        float inner[IN], outer[OUT], all[IN + OUT];
        stair_top<KM, S + 1>(A1, A2, inner);
#pragma unroll
        for (int i = 0; i < OUT; ++i) outer[i] = shell[i];
        merge_desc<OUT, IN>(outer, inner, all);
#pragma unroll
        for (int i = 0; i < KEEP; ++i) o[i] = all[i];
    } else {
#pragma unroll
        for (int i = 0; i < KEEP; ++i) o[i] = shell[i];
    }
}
// 32-bit keys ascending (merge exchange, as in the score kernel).
template <int N, int P, int K>
__device__ __forceinline__ void sort_keys_step(uint32_t (&v)[N]) {
#pragma unroll
    for (int j = K % P; j + K < N; j += 2 * K) {
#pragma unroll
        for (int i = 0; i < K; ++i) {
            if (i + j + K < N && (i + j) / (2 * P) == (i + j + K) / (2 * P)) {
                const uint32_t x = v[i + j], y = v[i + j + K];
                v[i + j] = min(x, y);
                v[i + j + K] = max(x, y);
            }
        }
    }
    if constexpr (K > 1) sort_keys_step<N, P, K / 2>(v);
}
template <int N, int P = 1>
__device__ __forceinline__ void sort_keys(uint32_t (&v)[N]) {
    sort_keys_step<N, P, P>(v);
    if constexpr (2 * P < N) sort_keys<N, 2 * P>(v);
}

// Shared bytes per thread: the selected cells' scores (later their exponentials) and codes, the
// first KM indices of each list (16-bit: S < 2^16).
__host__ __device__ constexpr int fs_bytes(int km) { return 4 * km + 2 * km + 2 * 2 * km; }

// Slots must fit 27 bits beside a 5-bit position (S * S <= 2^27).
template <class D, int L>
__global__ void __launch_bounds__(FT_THREADS, 6) k_addr_finalize_stair(const AddrArgs a) {
    constexpr int KM = L - 4;                     // largest k served
    static_assert(KM <= 32, "codes and keys hold five bits per index");
    extern __shared__ float fss[];
    const int tid = threadIdx.x;
    constexpr int W = FT_THREADS;
    // per-thread columns [element][FT_THREADS]: conflict-free for any element index
    float* const sv = fss + tid;                                              // [KM]
    unsigned short* const h16 = reinterpret_cast<unsigned short*>(fss + KM * W) + tid;
    unsigned short* const sc = h16;                                           // [KM]
    unsigned short* const A1i = h16 + KM * W;                                 // [KM]
    unsigned short* const A2i = h16 + 2 * KM * W;                             // [KM]

    const uint32_t BT = static_cast<uint32_t>(a.B) * static_cast<uint32_t>(a.T);
    const uint32_t item = blockIdx.x * FT_THREADS + tid;
    if (item >= 2u * static_cast<uint32_t>(a.H) * BT) return;      // (< 2^31: a queue exists) no barrier in this kernel
    const TokenSide ts = token_side(a, item);
    const int k = ts.k, S = a.S;
    auto defer = [&]() { a.queue[2 + atomicAdd(a.queue, 1)] = static_cast<int>(item); };

    // the two half lists: first k + 1 scores, first k indices
    float A1[KM], A2[KM], amax[2], vk1[2];
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
        const int64_t base = part_at(static_cast<int>(ts.z), 1, hf, BT, ts.u, L, 0);
        const float4* pv = reinterpret_cast<const float4*>(a.part_v + base);
        const int4* pi = reinterpret_cast<const int4*>(a.part_i + base);
        float (&Av)[KM] = hf ? A2 : A1;
        unsigned short* Ai = hf ? A2i : A1i;
        float after = -INFINITY;                  // entry KM of the list
#pragma unroll
        for (int q = 0; q <= KM / 4; ++q) {
            if (4 * q <= k) {
                const float4 v4 = __ldg(pv + q);
                const float vv[4] = {v4.x, v4.y, v4.z, v4.w};
                if (q == KM / 4) {
                    after = vv[0];
                } else {
                    const int4 i4 = __ldg(pi + q);
                    const int ii[4] = {i4.x, i4.y, i4.z, i4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        Av[4 * q + e] = vv[e];
                        Ai[(4 * q + e) * W] = static_cast<unsigned short>(ii[e]);
                    }
                }
            } else if (q < KM / 4) {
#pragma unroll
                for (int e = 0; e < 4; ++e) Av[4 * q + e] = -INFINITY;
            }
        }
        float vk = Av[KM - 1];
        vk1[hf] = after;
        if (k < KM) {                             // (uniform within a side)
#pragma unroll
            for (int p = 0; p < KM; ++p) {
                vk = p == k - 1 ? Av[p] : vk;
                vk1[hf] = p == k ? Av[p] : vk1[hf];
            }
#pragma unroll
            for (int p = 0; p < KM; ++p) Av[p] = p < k ? Av[p] : -INFINITY;
        }
        amax[hf] = fmaxf(fabsf(Av[0]), fabsf(vk));
        vk1[hf] = __fsub_rd(vk, vk1[hf]);         // the gap
    }
    const float e2 = twice_error_bound<D>(a, ts.side, ts.h, ts.b, ts.t);
    if (!((S <= k && amax[0] < INFINITY && amax[1] < INFINITY) || (vk1[0] > e2 && vk1[1] > e2))) { defer(); return; }
    const float e2c = __fadd_ru(__fmul_ru(2.f, e2), __fmul_ru(0x1p-21f, __fadd_ru(amax[0], amax[1])));
    float ck, ck1;
    {
        float top[KM + 1];
        stair_top<KM, 0>(A1, A2, top);
        ck = top[KM - 1];
        ck1 = top[KM];
        if (k < KM) {
#pragma unroll
            for (int p = 0; p < KM; ++p) {
                ck = p == k - 1 ? top[p] : ck;
                ck1 = p == k ? top[p] : ck1;
            }
        }
    }
    // (-inf cells are padding past a short half list; they only ever supply the (k+1)-th value)
    if (!(__fsub_rd(ck, ck1) > e2c)) { defer(); return; }
    // the selected cells (exactly k: the gap is positive)
    {
        int n = 0;
#pragma unroll
        for (int i = 0; i < KM; ++i)
#pragma unroll
            for (int j = 0; j < KM; ++j) {
                if ((i + 1) * (j + 1) <= KM) {
                    const float v = A1[i] + A2[j];
                    if (v >= ck) {
                        sv[n * W] = v;
                        sc[n * W] = static_cast<unsigned short>(i * 32 + j);
                        ++n;
                    }
                }
            }
    }
    // softmax over them, then ascending slot order
    const float vmax = A1[0] + A2[0];
    uint32_t key[KM];
#pragma unroll
    for (int r = 0; r < KM; ++r) {
        key[r] = 0xffffffffu;
        if (r < k) {
            const int c = sc[r * W];
            sv[r * W] = expf(sv[r * W] - vmax);
            const uint32_t slot = static_cast<uint32_t>(A1i[(c >> 5) * W]) * static_cast<uint32_t>(S) + A2i[(c & 31) * W];
            key[r] = slot * 32u + r;
        }
    }
    sort_keys<KM>(key);
    float zsum = 0.f;                             // (in slot order, as the other passes)
#pragma unroll
    for (int r = 0; r < KM; ++r)
        if (r < k) zsum += sv[(key[r] & 31) * W];
    const int64_t tokoff = ((static_cast<int64_t>(ts.b) * a.H + ts.h) * a.T + ts.t) * k;
    int32_t* oi = a.idx[ts.side] + tokoff;
    float* ow = a.w[ts.side] + tokoff;
    if (k % 4 == 0 && ((reinterpret_cast<uintptr_t>(oi) | reinterpret_cast<uintptr_t>(ow)) & 15) == 0) {
#pragma unroll
        for (int r = 0; r < KM; r += 4)
            if (r < k) {
                *reinterpret_cast<int4*>(oi + r) = make_int4(key[r] >> 5, key[r + 1] >> 5, key[r + 2] >> 5, key[r + 3] >> 5);
                *reinterpret_cast<float4*>(ow + r) = make_float4(sv[(key[r] & 31) * W] / zsum, sv[(key[r + 1] & 31) * W] / zsum,
                                                                 sv[(key[r + 2] & 31) * W] / zsum, sv[(key[r + 3] & 31) * W] / zsum);
            }
    } else {
#pragma unroll
        for (int r = 0; r < KM; ++r)
            if (r < k) { oi[r] = static_cast<int32_t>(key[r] >> 5); ow[r] = sv[(key[r] & 31) * W] / zsum; }
    }
}

// ---- k > 32.  The cells taken so far always form a staircase (row i holds the cells j < m_i, m
// non-increasing) and the next largest sum is one of its outer corners, at most 12 of them while at
// most 77 cells are taken; the frontier lives in registers.  k + 1 steps give the k-th and
// (k+1)-th values; the selected cells are the staircase after k steps.
constexpr int FT_FRONT = 12;      // frontier cells (outer corners of a staircase of <= 77 cells)

// Shared bytes per thread: the first k + 1 values of each half list (32-bit), the first k list
// indices (16-bit: S < 2^16) and the staircase row counts (bytes, k + 1 of them, padded to a word).
__host__ __device__ constexpr int ft_bytes(int km) { return 2 * 4 * (km + 1) + 2 * 2 * km + ((km + 4) & ~3); }

template <class D, int L>
__global__ void __launch_bounds__(FT_THREADS) k_addr_finalize_thread(const AddrArgs a) {
    constexpr int KM = L - 4;                     // largest k served
    static_assert(KM <= 64, "frontier bound holds for k <= 64");
    extern __shared__ float fts[];
    const int tid = threadIdx.x;
    constexpr int W = FT_THREADS;
    // per-thread columns [element][FT_THREADS]: conflict-free for any element index
    float* const A1v = fts + tid;                                             // [KM + 1]
    float* const A2v = fts + (KM + 1) * W + tid;                              // [KM + 1]
    unsigned short* const h16 = reinterpret_cast<unsigned short*>(fts + 2 * (KM + 1) * W);
    unsigned short* const A1i = h16 + tid;                                    // [KM]
    unsigned short* const A2i = h16 + KM * W + tid;                           // [KM]
    unsigned char* const m8 = reinterpret_cast<unsigned char*>(h16 + 2 * KM * W) + tid;   // [KM + 1]

    const uint32_t BT = static_cast<uint32_t>(a.B) * static_cast<uint32_t>(a.T);
    const uint32_t item = blockIdx.x * FT_THREADS + tid;
    if (item >= 2u * static_cast<uint32_t>(a.H) * BT) return;      // (< 2^31: a queue exists) no barrier in this kernel
    const TokenSide ts = token_side(a, item);
    const int k = ts.k, S = a.S, side = ts.side, h = ts.h;
    const uint32_t z = ts.z, u = ts.u, b = ts.b, t = ts.t;
    const float e2 = twice_error_bound<D>(a, ts.side, ts.h, ts.b, ts.t);
    auto defer = [&]() { a.queue[2 + atomicAdd(a.queue, 1)] = static_cast<int>(item); };

    // the two half lists (chunk 0 of each half), first k + 1 entries
    float amax[2];
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
        const int64_t base = part_at(static_cast<int>(z), 1, hf, BT, u, L, 0);
        const float4* pv = reinterpret_cast<const float4*>(a.part_v + base);
        const int4* pi = reinterpret_cast<const int4*>(a.part_i + base);
        float* Av = hf ? A2v : A1v;
        unsigned short* Ai = hf ? A2i : A1i;
#pragma unroll
        for (int q = 0; q < L / 4; ++q) {
            if (4 * q <= k) {
                const float4 v4 = __ldg(pv + q);
                const int4 i4 = __ldg(pi + q);
                const float vv[4] = {v4.x, v4.y, v4.z, v4.w};
                const int ii[4] = {i4.x, i4.y, i4.z, i4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int p = 4 * q + e;
                    if (p <= k && p <= KM) Av[p * W] = vv[e];
                    if (p < k && p < KM) Ai[p * W] = static_cast<unsigned short>(ii[e]);
                }
            }
        }
        const float vk = Av[(k - 1) * W], vk1 = Av[k * W];
        if (!((S <= k && vk != -INFINITY) || __fsub_rd(vk, vk1) > e2)) { defer(); return; }
        amax[hf] = fmaxf(fabsf(Av[0]), fabsf(vk));
    }
    const float e2c = __fadd_ru(__fmul_ru(2.f, e2), __fmul_ru(0x1p-21f, __fadd_ru(amax[0], amax[1])));

    // staircase walk: k + 1 steps, each taking the largest frontier cell
#pragma unroll
    for (int i = 0; i <= KM; ++i)
        if (i <= k) m8[i * W] = 0;
    float fv[FT_FRONT];
    int fij[FT_FRONT];                            // i | j << 8
#pragma unroll
    for (int f = 0; f < FT_FRONT; ++f) { fv[f] = -INFINITY; fij[f] = 0; }
    const float vmax = A1v[0] + A2v[0];
    fv[0] = vmax;
    float ck = -INFINITY, ck1 = -INFINITY;
    bool full = false;
    for (int r = 0; r <= k; ++r) {
        float bv = fv[0];
        int bf = 0;
#pragma unroll
        for (int f = 1; f < FT_FRONT; ++f) {
            const bool gt = fv[f] > bv;
            bv = gt ? fv[f] : bv;
            bf = gt ? f : bf;
        }
        if (r == k) { ck1 = bv; break; }
        ck = bv;                                   // the k-th value after the last step
        int bij = 0;
#pragma unroll
        for (int f = 0; f < FT_FRONT; ++f) bij = f == bf ? fij[f] : bij;
        const int i = bij & 255, j = bij >> 8;
        m8[i * W] = static_cast<unsigned char>(j + 1);
        // (i, j + 1) becomes a corner once row i - 1 holds more than j + 1 cells
        const bool right = j + 1 < k && (i == 0 || m8[(i - 1) * W] > j + 1);
        // (i + 1, j) becomes a corner when row i + 1 holds exactly j cells
        const bool down = i + 1 < k && m8[(i + 1) * W] == j;
        const float rv = right ? A1v[i * W] + A2v[(j + 1) * W] : -INFINITY;
        const float dv = down ? A1v[(i + 1) * W] + A2v[j * W] : -INFINITY;
#pragma unroll
        for (int f = 0; f < FT_FRONT; ++f)
            if (f == bf) { fv[f] = rv; fij[f] = i | ((j + 1) << 8); }
        bool placed = !down || dv == -INFINITY;
#pragma unroll
        for (int f = 0; f < FT_FRONT; ++f) {
            const bool here = !placed && fv[f] == -INFINITY;
            fv[f] = here ? dv : fv[f];
            fij[f] = here ? ((i + 1) | (j << 8)) : fij[f];
            placed |= here;
        }
        full |= !placed;
    }
    // (-inf cells are padding past a short half list; they only ever supply the (k+1)-th value)
    if (full || !(__fsub_rd(ck, ck1) > e2c)) { defer(); return; }
    // softmax over the k selected scores (the staircase, row by row), then ascending slot order
    // (bitonic network)
    float ew[KM];
    int sl[KM];
    int ci = 0, cj = 0, mi = m8[0];
#pragma unroll
    for (int r = 0; r < KM; ++r) {
        if (r < k) {
            ew[r] = expf((A1v[ci * W] + A2v[cj * W]) - vmax);
            sl[r] = static_cast<int>(A1i[ci * W]) * S + static_cast<int>(A2i[cj * W]);
            if (++cj == mi) { ++ci; cj = 0; mi = m8[ci * W]; }
        } else {
            ew[r] = 0.f;
            sl[r] = INT_MAX;
        }
    }
#pragma unroll
    for (int size = 2; size <= KM; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1)
#pragma unroll
            for (int i = 0; i < KM; ++i) {
                const int jx = i ^ stride;
                if (jx > i) {
                    const bool up = (i & size) == 0;
                    const bool sw = up ? (sl[i] > sl[jx]) : (sl[i] < sl[jx]);
                    const int si = sl[i];
                    const float ei = ew[i];
                    sl[i] = sw ? sl[jx] : si;  ew[i] = sw ? ew[jx] : ei;
                    sl[jx] = sw ? si : sl[jx]; ew[jx] = sw ? ei : ew[jx];
                }
            }
    float zsum = 0.f;                             // (in slot order, as the other passes)
#pragma unroll
    for (int r = 0; r < KM; ++r) zsum += ew[r];
    const int64_t tokoff = ((static_cast<int64_t>(b) * a.H + h) * a.T + t) * k;
    int32_t* oi = a.idx[side] + tokoff;
    float* ow = a.w[side] + tokoff;
#pragma unroll
    for (int r = 0; r < KM; ++r)
        if (r < k) { oi[r] = sl[r]; ow[r] = ew[r] / zsum; }
}

// ------------------------------------------------------------------------------------------
// Band pass, one thread per token-side of queue A (one list per half): the
// band of an uncertified boundary (entries within twice the error bound of it) is re-ranked
// by compensated scores, one thread computing each score sequentially.  A band that leaves
// the kept candidates, holds more than BT_BAND entries, or has two entries closer than their
// compensated bounds goes to queue B (float64 and whole-half paths).
// ------------------------------------------------------------------------------------------
constexpr int BT_THREADS = 32;
constexpr int BT_BAND = 8;        // band entries re-ranked here; wider bands go to queue B
// Shared bytes per thread: values, candidates and band scratch as 32-bit words, the half
// lists' column indices and the heap positions as 16-bit (one list per half, S < 2^16).
__host__ __device__ constexpr int bt_bytes(int L) { return 4 * (4 * L + (L - 4) + 4 * BT_BAND) + 2 * (2 * L + (L - 4)); }

// f versus e (compensated values): +1 if f is certainly larger, -1 if certainly smaller, 0 if
// equal with zero bounds (exact values: the caller breaks the tie); sets unsure when the two
// are closer than their bounds.
__device__ __forceinline__ int ff_cmp(const FF& f, const FF& e, bool& unsure) {
    float t, r;
    two_sum(f.h, -e.h, t, r);
    const float w = __fadd_rn(__fsub_rn(f.l, e.l), r);
    const float diff = __fadd_rn(t, w);
    const float slack = __fmul_ru(0x1p-21f, __fadd_ru(__fadd_ru(fabsf(t), fabsf(r)), __fadd_ru(fabsf(f.l), fabsf(e.l))));
    const float tol = __fadd_ru(__fadd_ru(f.b, e.b), slack);
    if (tol > 0.f && fabsf(diff) <= tol) { unsure = true; return 0; }
    return diff > 0.f ? 1 : diff < 0.f ? -1 : 0;
}

template <class D, int L>
__global__ void __launch_bounds__(BT_THREADS) k_addr_band_thread(const AddrArgs a) {
    constexpr int KM = L - 4;
    constexpr int LOG = KM <= 8 ? 3 : KM <= 16 ? 4 : KM <= 32 ? 5 : 6;
    constexpr int W = BT_THREADS;
    extern __shared__ float bts[];
    const int tid = threadIdx.x;
    float* const A1v = bts + tid;                                              // [L]
    float* const A2v = bts + L * W + tid;                                      // [L]
    float* const hv = bts + 2 * L * W + tid;                                   // [KM]
    float* const ov = bts + (2 * L + KM) * W + tid;                            // [L] candidates
    int* const os = reinterpret_cast<int*>(bts) + (3 * L + KM) * W + tid;      // [L]
    float* const bh = bts + (4 * L + KM) * W + tid;                            // [BT_BAND] band: h
    float* const bl = bts + (4 * L + KM + BT_BAND) * W + tid;                  //                 l
    float* const bb = bts + (4 * L + KM + 2 * BT_BAND) * W + tid;              //                 bound
    int* const bc = reinterpret_cast<int*>(bts) + (4 * L + KM + 3 * BT_BAND) * W + tid;   // chosen
    unsigned short* const h16 = reinterpret_cast<unsigned short*>(bts + (4 * L + KM + 4 * BT_BAND) * W);
    unsigned short* const A1i = h16 + tid;                                     // [L]
    unsigned short* const A2i = h16 + L * W + tid;                             // [L]
    unsigned short* const hp = h16 + 2 * L * W + tid;                          // [KM] row | col << 8

    const uint32_t BT = static_cast<uint32_t>(a.B) * static_cast<uint32_t>(a.T);
    const uint32_t nq = static_cast<uint32_t>(*reinterpret_cast<volatile int*>(a.queue));
    const uint32_t all = 2u * static_cast<uint32_t>(a.H) * BT;
    uint32_t stat_hb = 0, stat_he = 0, stat_cb = 0, stat_ce = 0;
    // grid-stride over queue A (the grid is sized to the SMs, not to the longest queue)
    for (uint32_t q = blockIdx.x * BT_THREADS + tid; q < nq; q += gridDim.x * BT_THREADS) {
        const uint32_t item = static_cast<uint32_t>(a.queue[2 + q]);
        int* const qb = a.queue + 2 + all;
        auto defer = [&]() { qb[atomicAdd(a.queue + 1, 1)] = static_cast<int>(item); };
        const uint32_t z = item / BT, u = item - z * BT;
        const int side = static_cast<int>(z) / a.H, h = static_cast<int>(z) % a.H;
        const int k = a.kk[side];
        const int S = a.S;
        const uint32_t b = u / static_cast<uint32_t>(a.T), t = u - b * static_cast<uint32_t>(a.T);
        const void* X = a.X[side];
        const void* P = a.P[side];
        const int64_t xoff = ((static_cast<int64_t>(b) * a.H + h) * a.T + t) * a.dk;
        const int64_t prow0 = static_cast<int64_t>(h) * 2 * S;

        float e2 = 0.f;
        if (P != nullptr) {
            float ss = 0.f;
            const char* xr = static_cast<const char*>(X) + xoff * D::BYTES;
            if ((reinterpret_cast<uintptr_t>(xr) & 15) == 0 && (a.dk * D::BYTES) % 16 == 0) {
                const int nq = a.dk * D::BYTES / 16;
                for (int q0 = 0; q0 < nq; q0 += 4) {
                    uint4 xq[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (q0 + u < nq) xq[u] = __ldg(reinterpret_cast<const uint4*>(xr) + q0 + u);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (q0 + u < nq) {
                            float f[D::E];
                            unpack16<D>(xq[u], f);
#pragma unroll
                            for (int e = 0; e < D::E; ++e) ss = fmaf(f[e], f[e], ss);
                        }
                }
            } else {
                for (int d = 0; d < a.dk; ++d) {
                    const float xv = load_elem<D>(X, xoff + d);
                    ss = fmaf(xv, xv, ss);
                }
            }
            e2 = __fmul_ru(__fmul_ru(__fmul_ru(2.f * a.cbound, a.pnorm[side * a.H + h]), sqrtf(ss)), 1.f + 0x1p-12f);
        }

        float amax[2];
        for (int hf = 0; hf < 2; ++hf) {
            const int64_t base = part_at(static_cast<int>(z), 1, hf, BT, u, L, 0);
            float* Av = hf ? A2v : A1v;
            unsigned short* Ai = hf ? A2i : A1i;
            const float4* pv = reinterpret_cast<const float4*>(a.part_v + base);   // L % 4 == 0, 16-byte aligned
            const int4* pi = reinterpret_cast<const int4*>(a.part_i + base);
#pragma unroll
            for (int q4 = 0; q4 < L / 4; ++q4) {
                const float4 v4 = __ldg(pv + q4);
                const int4 i4 = __ldg(pi + q4);
                Av[(4 * q4) * W] = v4.x; Av[(4 * q4 + 1) * W] = v4.y; Av[(4 * q4 + 2) * W] = v4.z; Av[(4 * q4 + 3) * W] = v4.w;
                Ai[(4 * q4) * W] = static_cast<unsigned short>(i4.x); Ai[(4 * q4 + 1) * W] = static_cast<unsigned short>(i4.y);
                Ai[(4 * q4 + 2) * W] = static_cast<unsigned short>(i4.z); Ai[(4 * q4 + 3) * W] = static_cast<unsigned short>(i4.w);
            }
            const float vk = Av[(k - 1) * W], vk1 = Av[k * W];
            if (!((S <= k && vk != -INFINITY) || __fsub_rd(vk, vk1) > e2)) {
                // band of the half boundary
                ++stat_hb;
                const float lo = __fsub_rd(vk, e2), hi = __fadd_ru(vk1, e2);
                if (Av[(L - 1) * W] >= lo && (S > L || Av[(L - 1) * W] == -INFINITY)) { defer(); goto next; }
                int cin = 0, m = 0;
                for (int p = 0; p < L; ++p) {        // (-inf padding never enters a band)
                    const float v = Av[p * W];
                    cin += v > hi ? 1 : 0;
                    m += (v >= lo && v <= hi && v != -INFINITY) ? 1 : 0;
                }
                if (m > BT_BAND) { defer(); goto next; }
                stat_he += m;
                for (int e = 0; e < m; ++e) {
                    const FF f = ff_score_thread<D>(P, X, xoff, prow0, a.dk, S, hf, Ai[(cin + e) * W]);
                    bh[e * W] = f.h; bl[e * W] = f.l; bb[e * W] = f.b;
                }
                bool unsure = false;
                for (int e = 0; e < m; ++e) {
                    const FF fe{bh[e * W], bl[e * W], bb[e * W]};
                    const int ie = Ai[(cin + e) * W];
                    int rank = 0;
                    for (int f = 0; f < m; ++f) {
                        if (f == e) continue;
                        const FF ff{bh[f * W], bl[f * W], bb[f * W]};
                        const int c = ff_cmp(ff, fe, unsure);
                        rank += (c > 0 || (c == 0 && Ai[(cin + f) * W] < ie)) ? 1 : 0;
                    }
                    bc[e * W] = rank < k - cin ? 1 : 0;
                }
                if (unsure) { defer(); goto next; }
                // chosen band entries, in list order, after the certain prefix
                int q2 = cin;
                for (int e = 0; e < m; ++e) {
                    if (bc[e * W]) {
                        const float v = Av[(cin + e) * W];
                        const int ix = Ai[(cin + e) * W];
                        Av[q2 * W] = v; Ai[q2 * W] = static_cast<unsigned short>(ix);   // q2 <= cin + e: in place
                        ++q2;
                    }
                }
            }
            amax[hf] = fmaxf(fabsf(Av[0]), fabsf(Av[(k - 1) * W]));
        }
        {
            const float e2c = __fadd_ru(__fmul_ru(2.f, e2), __fmul_ru(0x1p-21f, __fadd_ru(amax[0], amax[1])));
            // outer-sum candidates by a max-heap of the row heads (k+4 of them, 64 if the band needs)
            const float a20 = A2v[0];
            for (int i = 0; i < k; ++i) { hv[i * W] = A1v[i * W] + a20; hp[i * W] = static_cast<unsigned short>(i); }
            const int kk2 = k * k;
            int npop = 0;
            auto pops = [&](int upto) {
                for (; npop < upto; ++npop) {
                    const float v = hv[0];
                    const int pk = hp[0];
                    const int i = pk & 255, j = pk >> 8;
                    ov[npop * W] = v;
                    os[npop * W] = (j < k) ? A1i[i * W] * S + A2i[j * W] : INT_MAX;
                    const int j1 = j + 1;
                    const float nv = j1 < k ? A1v[i * W] + A2v[j1 * W] : -INFINITY;
                    const int np = i | (j1 << 8);
                    int pos = 0;
                    bool stop = false;
#pragma unroll
                    for (int lvl = 0; lvl < LOG; ++lvl) {
                        const int c = 2 * pos + 1;
                        const float v1 = c < k ? hv[c * W] : -INFINITY;
                        const float v2 = c + 1 < k ? hv[(c + 1) * W] : -INFINITY;
                        const int cm = v2 > v1 ? c + 1 : c;
                        const float vm = fmaxf(v1, v2);
                        if (!stop && vm > nv) { hv[pos * W] = vm; hp[pos * W] = hp[cm * W]; pos = cm; }
                        else stop = true;
                    }
                    hv[pos * W] = nv;
                    hp[pos * W] = static_cast<unsigned short>(np);
                }
            };
            const int len0 = kk2 < L ? kk2 : L;
            pops(len0 > k + 1 ? len0 : k + 1);
            int len = npop;
            const float ck = ov[(k - 1) * W], ck1 = k < npop ? ov[k * W] : -INFINITY;
            int nsel = k;                              // selected: candidates [0, k) unless a band is resolved
            // (ck = -inf: sums of -inf are among the k best, unless the bound is that of a NaN input)
            if (!((ck1 == -INFINITY && (ck != -INFINITY || e2c != e2c)) || __fsub_rd(ck, ck1) > e2c)) {
                ++stat_cb;
                const float lo = __fsub_rd(ck, e2c), hi = __fadd_ru(ck1, e2c);
                // a band reaching the last kept candidate (merge to be extended): queue B
                const bool all_cands = len >= kk2;
                if (ov[(len - 1) * W] >= lo && (!all_cands || ov[(len - 1) * W] == -INFINITY)) { defer(); goto next; }
                int cin = 0, m = 0;
                for (int p = 0; p < len; ++p) {      // (exhausted rows, -inf, never enter a band)
                    const float v = ov[p * W];
                    cin += v > hi ? 1 : 0;
                    m += (v >= lo && v <= hi && v != -INFINITY) ? 1 : 0;
                }
                if (m > BT_BAND) { defer(); goto next; }
                stat_ce += m;
                for (int e = 0; e < m; ++e) {
                    const int f = os[(cin + e) * W];
                    const FF s1 = ff_score_thread<D>(P, X, xoff, prow0, a.dk, S, 0, f / S);
                    const FF s2 = ff_score_thread<D>(P, X, xoff, prow0, a.dk, S, 1, f % S);
                    const FF sm = ff_add(s1, s2, P == nullptr);
                    bh[e * W] = sm.h; bl[e * W] = sm.l; bb[e * W] = sm.b;
                }
                bool unsure = false;
                for (int e = 0; e < m; ++e) {
                    const FF fe{bh[e * W], bl[e * W], bb[e * W]};
                    const int ie = os[(cin + e) * W];
                    int rank = 0;
                    for (int f = 0; f < m; ++f) {
                        if (f == e) continue;
                        const FF ff{bh[f * W], bl[f * W], bb[f * W]};
                        const int c = ff_cmp(ff, fe, unsure);
                        rank += (c > 0 || (c == 0 && os[(cin + f) * W] < ie)) ? 1 : 0;
                    }
                    bc[e * W] = rank < k - cin ? 1 : 0;
                }
                if (unsure) { defer(); goto next; }
                int q2 = cin;
                for (int e = 0; e < m; ++e) {
                    if (bc[e * W]) {
                        const float v = ov[(cin + e) * W];
                        const int f = os[(cin + e) * W];
                        ov[q2 * W] = v; os[q2 * W] = f;
                        ++q2;
                    }
                }
                nsel = q2;                             // = k
            }
            // softmax over the k selected scores, then ascending slot order
            float vmax = -INFINITY;
            for (int r = 0; r < nsel; ++r) vmax = fmaxf(vmax, ov[r * W]);
            float ew[KM];
            int sl[KM];
#pragma unroll
            for (int r = 0; r < KM; ++r) {
                if (r < k) { ew[r] = expf(ov[r * W] - vmax); sl[r] = os[r * W]; }
                else { ew[r] = 0.f; sl[r] = INT_MAX; }
            }
#pragma unroll
            for (int size = 2; size <= KM; size <<= 1)
#pragma unroll
                for (int stride = size >> 1; stride > 0; stride >>= 1)
#pragma unroll
                    for (int i = 0; i < KM; ++i) {
                        const int jx = i ^ stride;
                        if (jx > i) {
                            const bool up = (i & size) == 0;
                            const bool sw = up ? (sl[i] > sl[jx]) : (sl[i] < sl[jx]);
                            const int si = sl[i];
                            const float ei = ew[i];
                            sl[i] = sw ? sl[jx] : si;  ew[i] = sw ? ew[jx] : ei;
                            sl[jx] = sw ? si : sl[jx]; ew[jx] = sw ? ei : ew[jx];
                        }
                    }
            float zsum = 0.f;                          // (in slot order, as the other passes)
#pragma unroll
            for (int r = 0; r < KM; ++r) zsum += ew[r];
            const int64_t tokoff = ((static_cast<int64_t>(b) * a.H + h) * a.T + t) * k;
            int32_t* oi = a.idx[side] + tokoff;
            float* ow = a.w[side] + tokoff;
#pragma unroll
            for (int r = 0; r < KM; ++r)
                if (r < k) { oi[r] = sl[r]; ow[r] = ew[r] / zsum; }
        }
    next:;
    }
    if (stat_hb) stat_add(a.err, STAT_HALF_BAND, stat_hb);
    if (stat_he) stat_add(a.err, STAT_HALF_BAND_ENTRIES, stat_he);
    if (stat_cb) stat_add(a.err, STAT_COMB_BAND, stat_cb);
    if (stat_ce) stat_add(a.err, STAT_COMB_BAND_ENTRIES, stat_ce);
}

// Certified pass and band pass of one list per half, a thread per token-side.
template <class D, int L>
static cudaError_t launch_thread_certified(const AddrArgs& a, int64_t items, cudaStream_t stream) {
    const unsigned grid = static_cast<unsigned>((items + FT_THREADS - 1) / FT_THREADS);
    if constexpr (L <= 36) {
        const size_t sm = static_cast<size_t>(fs_bytes(L - 4)) * FT_THREADS;
        k_addr_finalize_stair<D, L><<<grid, FT_THREADS, sm, stream>>>(a);
    } else {
        const size_t sm = static_cast<size_t>(ft_bytes(L - 4)) * FT_THREADS;
        cudaError_t e = cudaFuncSetAttribute(k_addr_finalize_thread<D, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sm));
        if (e != cudaSuccess) return e;
        k_addr_finalize_thread<D, L><<<grid, FT_THREADS, sm, stream>>>(a);
    }
    return cudaGetLastError();
}
template <class D, int L>
static cudaError_t launch_thread_band(const AddrArgs& a, int64_t items, int sms, cudaStream_t stream) {
    const size_t smb = static_cast<size_t>(bt_bytes(L)) * BT_THREADS;
    cudaError_t e = cudaFuncSetAttribute(k_addr_band_thread<D, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smb));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_addr_band_thread<D, L>, BT_THREADS, smb);
    if (e != cudaSuccess) return e;
    const int64_t need = (items + BT_THREADS - 1) / BT_THREADS;       // `items`: upper bound of the queue's length
    const int64_t full = static_cast<int64_t>(sms) * (per_sm > 0 ? per_sm : 1);
    k_addr_band_thread<D, L><<<static_cast<unsigned>(need < full ? need : full), BT_THREADS, smb, stream>>>(a);
    return cudaGetLastError();
}

template <class D, int L>
static cudaError_t launch_finalize(const AddrArgs& a, bool mma, cudaStream_t stream) {
    const int64_t BT = static_cast<int64_t>(a.B) * a.T, items = 2 * a.H * BT;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (a.queue != nullptr && !mma) {            // (the tensor-core score kernel has emptied them)
        e = cudaMemsetAsync(a.queue, 0, 2 * sizeof(int), stream);
        if (e != cudaSuccess) return e;
    }
    if constexpr (L <= 36) {
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_addr_finalize<D, L, FIN_FAST>, FW_WARPS * 32, 0);
        if (e != cudaSuccess) return e;
        const int64_t need = (items + FW_WARPS - 1) / FW_WARPS;
        const int64_t full = static_cast<int64_t>(sms) * (per_sm > 0 ? per_sm : 1);
        const unsigned grid = static_cast<unsigned>(need < full ? need : full);
        // same carveout as the tensor-core kernel and the M0 copy: they share SMs
        for (auto fn : {k_addr_finalize<D, L, FIN_FAST>, k_addr_finalize<D, L, FIN_BAND>, k_addr_finalize<D, L, FIN_FULL>}) {
            e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
            if (e != cudaSuccess) return e;
        }
        if (a.queue != nullptr) {
            // one thread per token-side with one list per half and slots that fit the sort keys
            // (S * S <= 2^27); a warp per token-side otherwise
            if (a.ncc == 1 && static_cast<int64_t>(a.S) * a.S <= (1ll << 27)) {
                e = launch_thread_certified<D, L>(a, items, stream);
                if (e != cudaSuccess) return e;
            } else {
                k_addr_finalize<D, L, FIN_FAST><<<grid, FW_WARPS * 32, 0, stream>>>(a);
            }
            // band pass: one thread per queued token-side on large problems; a warp per item when
            // the problem is small (decode): there the queue is short and each item's serial
            // rescoring, not the item count, sets the pass's length
            if (a.ncc == 1 && items >= 32768) {
                e = launch_thread_band<D, L>(a, items, sms, stream);
                if (e != cudaSuccess) return e;
            } else {
                k_addr_finalize<D, L, FIN_BAND><<<grid, FW_WARPS * 32, 0, stream>>>(a);
            }
        }
        k_addr_finalize<D, L, FIN_FULL><<<grid, FW_WARPS * 32, 0, stream>>>(a);
    } else {
        // one list per half: the thread passes, then a warp per token-side they left (65,536 token-sides,
        // k = 64: 0.21 + 0.17 + 0.07 ms; one thread per token-side for all of it 3.1 ms)
        if (a.queue != nullptr && a.ncc == 1) {
            e = launch_thread_certified<D, L>(a, items, stream);
            if (e == cudaSuccess) e = launch_thread_band<D, L>(a, items, sms, stream);
            if (e != cudaSuccess) return e;
            const int64_t need = (items + RW_WARPS - 1) / RW_WARPS, cap = 4ll * sms;
            k_addr_rare_wide<D, L><<<static_cast<unsigned>(need < cap ? need : cap), RW_WARPS * 32, 0, stream>>>(a);
        } else {
            const size_t smB = static_cast<size_t>(6) * L * F_THREADS * sizeof(float);
            e = cudaFuncSetAttribute(k_addr_finalize_wide<D, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smB));
            if (e != cudaSuccess) return e;
            const dim3 gB(static_cast<unsigned>((BT + F_THREADS - 1) / F_THREADS), 2 * a.H);
            k_addr_finalize_wide<D, L><<<gB, F_THREADS, smB, stream>>>(a);
        }
    }
    return cudaGetLastError();
}

template <class D, int L>
static cudaError_t launch_typed(const AddrPlan& plan, const AddrArgs& a, cudaStream_t stream) {
    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    if (plan.mma) {                              // scores, row norms and empty queues in one launch
        cudaError_t e = launch_address_mma(plan, a, stream);
        if (e != cudaSuccess) return e;
        return launch_finalize<D, L>(a, true, stream);
    }
    if (a.P[0] != nullptr) {
        cudaError_t e = cudaMemsetAsync(a.pnorm, 0, static_cast<size_t>(2) * a.H * sizeof(float), stream);
        if (e != cudaSuccess) return e;
        const int64_t rows = static_cast<int64_t>(2) * a.H * 2 * a.S;
        k_pnorm<D><<<static_cast<unsigned>((rows + 31) / 32), 256, 0, stream>>>(a);
    }
    const size_t smA = (static_cast<size_t>(a.dk) * A_TOK + (a.P[0] ? static_cast<size_t>(a.dk) * A_PPITCH : 0)) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(k_addr_scores<D, L>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_ALLOWED);
    if (e != cudaSuccess) return e;
    dim3 gA(static_cast<unsigned>((BT + A_TOK - 1) / A_TOK), 2 * plan.ncc, 2 * a.H);
    k_addr_scores<D, L><<<gA, A_TOK, smA, stream>>>(a);
    return launch_finalize<D, L>(a, false, stream);
}

template <class D>
static cudaError_t launch_dtype(const AddrPlan& plan, const AddrArgs& a, cudaStream_t stream) {
    switch (plan.L) {
        case 12: return launch_typed<D, 12>(plan, a, stream);
        case 20: return launch_typed<D, 20>(plan, a, stream);
        case 36: return launch_typed<D, 36>(plan, a, stream);
        case 68: return launch_typed<D, 68>(plan, a, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_address(int dtype, const AddrPlan& plan, const AddrArgs& a, cudaStream_t stream) {
    if (plan.small) return launch_address_small(dtype, plan, a, stream);
    return dtype == 0 ? launch_dtype<F32>(plan, a, stream) : launch_dtype<BF16>(plan, a, stream);
}

}  // namespace sdm
