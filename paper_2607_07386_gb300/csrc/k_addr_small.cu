// K-ADDR for small problems (k <= 32): a decode step, short extensions.  One launch does what the score
// kernel, the row norms and the three finalize passes do on large ones: a CTA takes a few tokens of one
// (side, head) through all of it.
//   1. scores, bit for bit those of the kernels for large problems (so a sequence may be cut anywhere):
//      k_addr_small: fp32 FMAs in d order, a lane per row of P, rows staged by each warp for itself in
//      shared memory, two 128-byte pieces of 32 rows in flight;
//      k_addr_small_tc: tcgen05.mma (M = 128, N <= 256, K = 16 per step) on 256-row blocks of P that TMA
//      brings in a ring of four 32 KB units; the tokens' rows sit at the head of each of the four TMEM lane
//      quadrants, so that eight warps read a block's 256 columns, 32 each.  Row norms on the way.  Clusters of
//      two or four CTAs share the blocks and write the scores into the first one's shared memory;
//   2. selection: a warp per (token, half): the top two of each lane's columns, sorted, give a lower
//      bound of the L-th largest score; the columns that reach it (about L + 5) are ranked by
//      counting.  More than 64 of them (heavy ties): L rounds of a warp maximum instead;
//   3. a warp per token: finalize_warp with every path.
//
// What bounds it: latency.  One sequence's decode step (16 heads, S = 512, d_k = 128, k = 32) takes 14.6 us where
// the four passes for large problems took 45 (score kernel 19, stair 15, band 10, rest 2), each waiting for a few
// tokens' serial work; in cycles: start 2,700, scores 3,400 (15,400 on one CTA a head), hand-over 1,300,
// selection 3,500, lists and certificates 2,200, outer sum 3,800, softmax and order 1,400.  A step of 32
// sequences (S = 256): 48 us to 24.6.
#include "k_addr_warp.cuh"
#include "tc_common.cuh"

namespace sdm {

cudaError_t addr_p_maps(CUtensorMap (&maps)[2], const AddrArgs& a);      // k_addr_mma.cu

// Descending sort of 64 keys held two per lane (element lane in a, lane + 32 in b).
__device__ __forceinline__ void sort64_desc(uint32_t& a, uint32_t& b, int lane) {
#pragma unroll
    for (int size = 2; size <= 64; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride == 32) {
                const uint32_t hi = max(a, b), lo = min(a, b);
                a = hi; b = lo;
            } else {
                const uint32_t pa = __shfl_xor_sync(0xffffffffu, a, stride);
                const uint32_t pb = __shfl_xor_sync(0xffffffffu, b, stride);
                const bool lower = (lane & stride) == 0;
                const bool da = (lane & size) == 0, db = ((lane + 32) & size) == 0;
                a = (lower == da) ? max(a, pa) : min(a, pa);
                b = (lower == db) ? max(b, pb) : min(b, pb);
            }
        }
    }
}

// A score as the selection takes it: -0 counts as 0, a NaN (of a row of P that holds one) as -inf.
__device__ __forceinline__ float as_score(float f) { return fmaxf(f, -INFINITY) + 0.f; }

// Top L of n scores in shared memory by (score desc, index asc), sorted; short lists end in
// (-inf, INT_MAX).  cand: 64 keys of the warp's shared memory.
template <int L>
__device__ __forceinline__ void select_warp(const float* sc, int n, float* lv, int* li, unsigned long long* cand, int lane) {
    uint32_t t1 = 0u, t2 = 0u;
    for (int j0 = 0; j0 < n; j0 += 256) {                  // (eight loads in flight)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = j0 + 32 * i + lane;
            const uint32_t key = j < n ? f2key(sc[j]) : 0u;
            t2 = max(t2, min(t1, key));
            t1 = max(t1, key);
        }
    }
    sort64_desc(t1, t2, lane);
    const uint32_t ta = __shfl_sync(0xffffffffu, t1, (L - 1) & 31), tb = __shfl_sync(0xffffffffu, t2, (L - 1) & 31);
    const uint32_t theta = L - 1 < 32 ? ta : tb;
    int m = 0;
    for (int j0 = 0; j0 < n; j0 += 256) {
        uint32_t key[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = j0 + 32 * i + lane;
            key[i] = j < n ? f2key(sc[j]) : 0u;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = j0 + 32 * i + lane;
            const bool keep = j < n && key[i] >= theta;
            const unsigned mask = __ballot_sync(0xffffffffu, keep);
            const int at = m + __popc(mask & ((1u << lane) - 1u));
            if (keep && at < 64) cand[at] = static_cast<unsigned long long>(key[i]) << 32 | static_cast<uint32_t>(~j);
            m += __popc(mask);
        }
    }
    __syncwarp();
    auto put = [&](int p, unsigned long long e) {
        lv[p] = key2f(static_cast<uint32_t>(e >> 32));
        li[p] = static_cast<int>(~static_cast<uint32_t>(e));
    };
    if (m <= 64) {
        const unsigned long long e0 = lane < m ? cand[lane] : 0ull, e1 = lane + 32 < m ? cand[lane + 32] : 0ull;
        int r0 = 0, r1 = 0;
#pragma unroll 8
        for (int f = 0; f < m; ++f) {
            const unsigned long long o = cand[f];
            r0 += o > e0;
            r1 += o > e1;
        }
        if (lane < m && r0 < L) put(r0, e0);
        if (lane + 32 < m && r1 < L) put(r1, e1);
        for (int p = m + lane; p < L; p += 32) { lv[p] = -INFINITY; li[p] = INT_MAX; }
    } else {
        unsigned long long last = ~0ull;
        for (int r = 0; r < L; ++r) {
            unsigned long long best = 0ull;
            for (int j = lane; j < n; j += 32) {
                const unsigned long long e = static_cast<unsigned long long>(f2key(sc[j])) << 32 | static_cast<uint32_t>(~j);
                if (e < last && e > best) best = e;
            }
            const uint32_t hi = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(best >> 32));
            const uint32_t lo = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(best >> 32) == hi ? static_cast<uint32_t>(best) : 0u);
            last = static_cast<unsigned long long>(hi) << 32 | lo;
            if (lane == 0) put(r, last);
        }
    }
}

// Steps 2 and 3 for the CTA's tokens u0 .. u0 + nt - 1: scores in sc (token t's at t * pitch, half 1 at S).
// cand: 64 keys per warp; lv, li: [nt][2][L]; fin: [2][nt][3][64] words.  All warps of the block.
template <class D, int L>
__device__ __forceinline__ void finish_tokens(const AddrArgs& a, int z, int64_t u0, int nt, const float* sc, int pitch, const float* xnorm, float pnorm,
                                              unsigned long long* cand, float* lv, int* li, float* fin,
                                              unsigned (*wstat)[STAT_COUNT]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int S = a.S, side = z / a.H, h = z % a.H, k = a.kk[side];
    for (int e = warp; e < 2 * nt; e += W)
        select_warp<L>(sc + (e >> 1) * pitch + (e & 1) * S, S, lv + e * L, li + e * L, cand + warp * 64, lane);
    __syncthreads();
    if (warp >= nt) return;
    const int t = warp;
    const int64_t u = u0 + t, b = u / a.T, bht = (b * a.H + h) * a.T + (u - b * a.T);
    TokenCtx c;
    c.err = a.err;
    c.stat = wstat[t];
    c.count_band = true;
    c.P = a.P[side];
    c.X = a.X[side];
    c.xoff = bht * a.dk;
    c.prow0 = static_cast<int64_t>(h) * 2 * S;
    c.dk = a.dk;
    c.S = S;
    // 2 x the fp32 score error bound, rounded up
    const float e2 = c.P != nullptr ? __fmul_ru(__fmul_ru(__fmul_ru(2.f * a.cbound, pnorm), xnorm[t]), 1.f + 0x1p-12f) : 0.f;
    float* const fv = fin + t * 3 * 64;
    int* const fi = reinterpret_cast<int*>(fin + nt * 3 * 64) + t * 3 * 64;
    for (int p = lane; p < 3 * 64; p += 32) { fv[p] = 0.f; fi[p] = 0; }
    if (lane < STAT_COUNT) wstat[t][lane] = 0u;
    __syncwarp();
    auto load = [&](int hf, float& v0, int& i0, float& v1, int& i1) {
        const float* const v = lv + (t * 2 + hf) * L;
        const int* const i = li + (t * 2 + hf) * L;
        v0 = lane < L ? v[lane] : -INFINITY;           i0 = lane < L ? i[lane] : INT_MAX;
        v1 = lane + 32 < L ? v[lane + 32] : -INFINITY; i1 = lane + 32 < L ? i[lane + 32] : INT_MAX;
    };
    finalize_warp<D, L, FIN_FULL>(c, k, e2, a.idx[side] + bht * k, a.w[side] + bht * k, fv, fi, fv + 64, fi + 64, fv + 128,
                                  fi + 128, lane, load);
    __syncwarp();
    if (lane > 0 && lane < STAT_COUNT && wstat[t][lane] != 0u) stat_add(a.err, lane, wstat[t][lane]);
}

// ||x|| of the CTA's tokens, a warp per token from warp `first` on.
template <class D, class Off>
__device__ __forceinline__ void token_norms(const void* X, int dk, int nt, int first, float* xnorm, Off xoff) {
    const int lane = threadIdx.x & 31, t = (threadIdx.x >> 5) - first;
    if (t < 0 || t >= nt) return;
    float ss = 0.f;
    for (int d = lane; d < dk; d += 32) {
        const float xv = load_elem<D>(X, xoff(t) + d);
        ss = fmaf(xv, xv, ss);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    if (lane == 0) xnorm[t] = sqrtf(ss);
}

// (a row with a NaN is never selected: no part of the bound)
__device__ __forceinline__ void norm_max_to(float& mx, float ss) {
    mx = fmaxf(mx, sqrtf(ss) * (1.f + 0x1p-12f));            // (1 + 2^-12) covers the roundings of the norm
}

constexpr int AS_ROW = 144;                  // bytes between staged rows: 128 and 16 against bank conflicts
constexpr int AS_STAGE = 32 * AS_ROW;        // a warp's stage

// Shared memory of k_addr_small: x [TG][dk] (fp32), scores [TG][2S], then per warp two stages, which the
// candidates, lists and staging of the later steps take over.
__host__ __device__ constexpr int as_warps(int tg) { return tg == 1 ? 16 : 8; }
__host__ __device__ inline size_t as_smem(int tg, int S, int dk) {
    return (static_cast<size_t>(tg) * ((dk + 3) / 4 * 4) + static_cast<size_t>(tg) * 2 * S) * 4 + 16 +
           static_cast<size_t>(as_warps(tg)) * 2 * AS_STAGE;
}

template <class D, int L, int TG>
__global__ void __launch_bounds__(as_warps(TG) * 32, TG == 1 ? 1 : 2) k_addr_small(const AddrArgs a, int vec) {
    constexpr int W = as_warps(TG), E = D::E;
    extern __shared__ __align__(16) float smS[];
    __shared__ int norm_max;
    __shared__ float xnorm[TG];
    __shared__ unsigned wstat[TG][STAT_COUNT];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int S = a.S, z = blockIdx.y, side = z / a.H, h = z % a.H;
    const void* const P = a.P[side];
    const void* const X = a.X[side];
    const int dkp = P == nullptr ? 0 : (a.dk + 3) / 4 * 4;
    float* const xs = smS;                                                  // [TG][dkp]
    float* const sc = xs + TG * dkp;                                        // [TG][2S]
    unsigned char* const stage = reinterpret_cast<unsigned char*>(smS) + ((TG * dkp + TG * 2 * S) * 4 + 15) / 16 * 16;
    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    const int64_t u0 = static_cast<int64_t>(blockIdx.x) * TG;
    const int nt = static_cast<int>(BT - u0 < TG ? BT - u0 : TG);           // tokens of this CTA
    auto xoff_of = [&](int t) {
        const int64_t u = u0 + t, b = u / a.T;
        return ((b * a.H + h) * a.T + (u - b * a.T)) * a.dk;
    };
    if (tid == 0) norm_max = 0;
    if (P == nullptr) {
        for (int t = 0; t < nt; ++t) {
            const int64_t x0 = xoff_of(t);
            for (int j = tid; j < 2 * S; j += W * 32) sc[t * 2 * S + j] = as_score(load_elem<D>(X, x0 + j));
        }
    } else {
#pragma unroll
        for (int t = 0; t < TG; ++t) {
            const int64_t x0 = t < nt ? xoff_of(t) : 0;
            for (int d = tid; d < dkp; d += W * 32) xs[t * dkp + d] = t < nt && d < a.dk ? load_elem<D>(X, x0 + d) : 0.f;
        }
        __syncthreads();
        token_norms<D>(X, a.dk, nt, W - TG, xnorm, xoff_of);
        unsigned char* const mine = stage + warp * 2 * AS_STAGE;
        const uint32_t mine32 = static_cast<uint32_t>(__cvta_generic_to_shared(mine));
        const int rowbytes = a.dk * D::BYTES, npc = (rowbytes + 127) / 128;      // 128-byte pieces of a row
        const char* const Pz = static_cast<const char*>(P) + static_cast<int64_t>(h) * 2 * S * rowbytes;
        const int ngr = (2 * S + 31) / 32;                                       // groups of 32 rows
        const int total = ((ngr - warp + W - 1) / W) * npc;                      // this warp's stages (<= 0: none)
        auto issue = [&](int it) {
            if (it < total) {
                const int gi = it / npc, pc = it - gi * npc;
                const int r0 = (warp + gi * W) * 32;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int row = (lane >> 3) + 4 * i, at = pc * 128 + (lane & 7) * 16;
                    const bool in = r0 + row < 2 * S && at < rowbytes;
                    const char* src = Pz + (in ? static_cast<int64_t>(r0 + row) * rowbytes + at : 0);
                    const uint32_t off = (it & 1) * AS_STAGE + row * AS_ROW + (lane & 7) * 16;
                    if (vec) {
                        cp_async16z(mine32 + off, src, in ? 16 : 0);
                    } else {
                        float f[E];
#pragma unroll
                        for (int e = 0; e < E; ++e) f[e] = in ? load_elem<D>(src, e) : 0.f;
                        *reinterpret_cast<uint4*>(mine + off) = pack16<D>(f);      // (exact: storage values)
                    }
                }
            }
            cp_async_commit();
        };
        float acc[TG], ss = 0.f, mx = 0.f;
#pragma unroll
        for (int t = 0; t < TG; ++t) acc[t] = 0.f;
        issue(0);
        for (int it = 0; it < total; ++it) {
            issue(it + 1);
            cp_async_wait<1>();
            __syncwarp();
            const int gi = it / npc, pc = it - gi * npc;
            const unsigned char* const row = mine + (it & 1) * AS_STAGE + lane * AS_ROW;
            const int nq = min(8, (rowbytes - pc * 128) / 16);
            const float* const xq = xs + pc * (128 / D::BYTES);
#pragma unroll 2
            for (int q = 0; q < nq; ++q) {
                float f[E];
                unpack16<D>(*reinterpret_cast<const uint4*>(row + q * 16), f);
#pragma unroll
                for (int e4 = 0; e4 < E; e4 += 4) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) ss = fmaf(f[e4 + e], f[e4 + e], ss);
#pragma unroll
                    for (int t = 0; t < TG; ++t) {               // ascending d, one rounding per step
                        const float4 x4 = *reinterpret_cast<const float4*>(xq + t * dkp + q * E + e4);
                        acc[t] = fmaf(x4.x, f[e4], acc[t]);
                        acc[t] = fmaf(x4.y, f[e4 + 1], acc[t]);
                        acc[t] = fmaf(x4.z, f[e4 + 2], acc[t]);
                        acc[t] = fmaf(x4.w, f[e4 + 3], acc[t]);
                    }
                }
            }
            if (pc == npc - 1) {
                const int r = (warp + gi * W) * 32 + lane;
                norm_max_to(mx, ss);
                ss = 0.f;
#pragma unroll
                for (int t = 0; t < TG; ++t) {
                    if (r < 2 * S) sc[t * 2 * S + r] = as_score(acc[t]);
                    acc[t] = 0.f;
                }
            }
            __syncwarp();
        }
        cp_async_wait<0>();
        const int top = __reduce_max_sync(0xffffffffu, __float_as_int(mx));
        if (lane == 0) atomicMax(&norm_max, top);
    }
    __syncthreads();
    unsigned long long* const cand = reinterpret_cast<unsigned long long*>(stage);
    float* const lv = reinterpret_cast<float*>(cand + W * 64);
    finish_tokens<D, L>(a, z, u0, nt, sc, 2 * S, xnorm, __int_as_float(norm_max), cand, lv, reinterpret_cast<int*>(lv + TG * 2 * L),
                        lv + TG * 4 * L, wstat);
}

// ------------------------------------------------------------------------------------------
// bf16 shapes of the tensor-core score kernel
// ------------------------------------------------------------------------------------------
constexpr int AT_WARPS = 16;
constexpr int AT_TOK = 8;                    // tokens of a CTA at most
constexpr int AT_RING = 4;
constexpr int AT_UNIT = 256 * 128;           // 256 rows x 64 values

// Shared memory of k_addr_small_tc: x tile, ring of P units (which the later steps take over), scores with an
// odd pitch, barriers.
__host__ __device__ inline size_t at_smem(int atoms, int tg, int S) {
    return 1024 + static_cast<size_t>(atoms) * 128 * 128 + AT_RING * AT_UNIT + (static_cast<size_t>(tg) * (2 * S + 1) * 4 + 15) / 16 * 16 + 128;
}

template <int L>
__global__ void __launch_bounds__(AT_WARPS * 32, 1)
k_addr_small_tc(const __grid_constant__ CUtensorMap tp_q, const __grid_constant__ CUtensorMap tp_k, const AddrArgs a, int tg, int cl) {
    using namespace tc;
    extern __shared__ unsigned char sm_raw[];
    __shared__ int norm_max;
    __shared__ float xnorm[AT_TOK];
    __shared__ unsigned wstat[AT_TOK][STAT_COUNT];
    const uint32_t raw = smem_u32(sm_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* const sm = sm_raw + (base - raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int S = a.S, z = blockIdx.y, side = z / a.H, h = z % a.H, atoms = a.dk / 64;
    const uint32_t sA = base, sB = base + atoms * 128 * 128;
    const int pitch = 2 * S + 1;
    float* const sc = reinterpret_cast<float*>(sm + (sB - base) + AT_RING * AT_UNIT);           // [tg][pitch]
    const uint32_t bars = sB + AT_RING * AT_UNIT + (tg * pitch * 4 + 15) / 16 * 16;
    const uint32_t bar_full = bars, bar_empty = bars + 8 * AT_RING, bar_done = bars + 16 * AT_RING;
    uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(sm + (bar_done + 16 - base));
    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    const int rank = static_cast<int>(blockIdx.x) % cl;       // in the cluster: blocks rank, rank + cl, ... of P
    const int64_t u0 = static_cast<int64_t>(blockIdx.x) / cl * tg;
    const int nt = static_cast<int>(BT - u0 < tg ? BT - u0 : tg);
    const CUtensorMap* const tp = side ? &tp_k : &tp_q;
    const int pb = min(256, 2 * S), bph = (S + 255) / 256, nblk = (2 * bph - rank + cl - 1) / cl, nunit = nblk * atoms;

    uint32_t nload = 0;
    auto load_unit = [&]() {                                  // (thread 0) unit = block x 64 values of d_k
        const uint32_t s = nload % AT_RING, round = nload / AT_RING;
        if (round > 0 && !mbar_wait(bar_empty + 8 * s, (round - 1) & 1u)) return false;
        const int i = nload / atoms, at = nload - i * atoms, blk = rank + i * cl, hf = blk / bph;
        mbar_expect_tx(bar_full + 8 * s, pb * 128);
        tma_load_3d(sB + s * AT_UNIT, tp, at * 64, hf * S + (blk - hf * bph) * 256, h, bar_full + 8 * s);
        ++nload;
        return true;
    };
    if (tid == 0) {
        norm_max = 0;
        for (int i = 0; i < AT_RING; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 1 + 8); }
        mbar_init(bar_done, 1);
        mbar_init(bar_done + 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        for (int i = 0; i < AT_RING && i < nunit; ++i) load_unit();
    }
    __syncwarp();
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    // x rows of token t at tile rows t, 32 + t, 64 + t, 96 + t (the other rows hold whatever was there: a row's
    // scores depend on that row alone)
    auto xoff_of = [&](int t) {
        const int64_t u = u0 + t, b = u / a.T;
        return ((b * a.H + h) * a.T + (u - b * a.T)) * a.dk;
    };
    if (warp >= 8) {
        const int e = tid - 256;                              // at most 8 tokens x 16 pieces
        if (e < nt * (a.dk / 8)) {
            const int t = e / (a.dk / 8), q = e - t * (a.dk / 8);
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(static_cast<const char*>(a.X[side]) + xoff_of(t) * 2) + q);
#pragma unroll
            for (int r = 0; r < 4; ++r)                       // 128-byte swizzle: 16-byte piece ^ (row mod 8)
                *reinterpret_cast<uint4*>(sm + (q >> 3) * 128 * 128 + (32 * r + t) * 128 + (((q & 7) ^ (t & 7)) << 4)) = v;
        }
        token_norms<BF16>(a.X[side], a.dk, nt, 8, xnorm, xoff_of);
    }
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");      // every CTA of the cluster runs
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    auto leader = [](uint32_t at) {                           // address of the same word in the cluster's first CTA
        uint32_t r;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;\n" : "=r"(r) : "r"(at));
        return r;
    };

    uint32_t nmma = 0;
    auto run_block = [&](int blk) {                           // (thread 0) block's scores into TMEM columns 256 (blk mod 2)
        const int hb = (rank + blk * cl) % bph, npad = (S + 15) & ~15;
        const uint32_t idesc = mma_idesc(min(256, npad - hb * 256)), acc = tmem + (blk & 1) * 256;
        for (int at = 0; at < atoms; ++at) {
            const uint32_t s = nmma % AT_RING;
            if (!mbar_wait(bar_full + 8 * s, (nmma / AT_RING) & 1u)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma_bf16(acc, sw128_desc(sA + at * 128 * 128 + ks * 32), sw128_desc(sB + s * AT_UNIT + ks * 32), idesc,
                         at + ks > 0 ? 1u : 0u);
            mma_commit(bar_empty + 8 * s);
            ++nmma;
        }
        mma_commit(bar_done + 8 * (blk & 1));
        return true;
    };
    bool ok = true;
    float mx = 0.f;
    if (tid == 0) ok = run_block(0);
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");
    for (int blk = 0; blk < nblk; ++blk) {
        if (tid == 0 && ok && blk + 1 < nblk) ok = run_block(blk + 1);
        if (warp >= 8) {                                      // row norms: a thread per row, ascending d
            const int r = tid - 256;
            float ss = 0.f;
            for (int at = 0; at < atoms && ok; ++at) {
                const uint32_t un = blk * atoms + at, s = un % AT_RING;
                ok = mbar_wait(bar_full + 8 * s, (un / AT_RING) & 1u);
                ok = __all_sync(0xffffffffu, ok);
                if (ok && r < pb) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        float f[8];
                        unpack16<BF16>(*reinterpret_cast<const uint4*>(sm + (sB - base) + s * AT_UNIT + r * 128 + ((q ^ (r & 7)) << 4)), f);
#pragma unroll
                        for (int e = 0; e < 8; ++e) ss = fmaf(f[e], f[e], ss);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_empty + 8 * s);
            }
            if (r < pb) norm_max_to(mx, ss);
        } else {
            if (ok) ok = mbar_wait(bar_done + 8 * (blk & 1), (blk >> 1) & 1u);
            ok = __all_sync(0xffffffffu, ok);
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            // warps 0-3 and 4-7: lane quadrant warp mod 4, 32 of the block's columns each
            const int gb = rank + blk * cl, hf = gb / bph, hb = gb - hf * bph, nb = min(256, S - hb * 256);
            const int c0 = ((warp & 3) * 2 + (warp >> 2)) * 32;
            if (ok && c0 < nb) {
                float v[32];
                tmem_ld32(tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + (blk & 1) * 256 + c0, v);
                const uint32_t dst = leader(smem_u32(sc)) + static_cast<uint32_t>(lane * pitch + hf * S + hb * 256 + c0) * 4;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (lane < nt && c0 + j < nb)
                        asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(dst + 4 * j), "f"(as_score(v[j])) : "memory");
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        }
        // the units of block blk are free once the norms and the MMAs have read them
        if (tid == 0)
            for (int i = 0; i < atoms && ok && nload < static_cast<uint32_t>(nunit); ++i) ok = load_unit();
        ok = __syncthreads_and(ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    }
    if (!ok && tid == 0) {                                    // own copies in flight, again with a limit
        for (uint32_t un = nload > AT_RING ? nload - AT_RING : 0; un < nload; ++un)
            mbar_wait(bar_full + 8 * (un % AT_RING), (un / AT_RING) & 1u);
        flag_error(a.err, ERR_TIMEOUT);
    }
    if (warp >= 8) {
        const int top = __reduce_max_sync(0xffffffffu, __float_as_int(mx));
        if (lane == 0)
            asm volatile("red.relaxed.cluster.shared::cluster.max.s32 [%0], %1;\n" ::"r"(leader(smem_u32(&norm_max))), "r"(top) : "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");      // scores and norms are the first CTA's now
    asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");
    if (warp == AT_WARPS - 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512) : "memory");
    if (!ok || rank != 0) return;
    unsigned long long* const cand = reinterpret_cast<unsigned long long*>(sm + (sB - base));
    float* const lv = reinterpret_cast<float*>(cand + AT_WARPS * 64);
    finish_tokens<BF16, L>(a, z, u0, nt, sc, pitch, xnorm, __int_as_float(norm_max), cand, lv, reinterpret_cast<int*>(lv + AT_TOK * 2 * L),
                           lv + AT_TOK * 4 * L, wstat);
}

// Tokens per CTA: few enough that the grid fits the chip once, at most `most`, which share the reads of P.
static int small_group(int H, int64_t BT, int most, int cl = 1) {
    int tg = 1;
    while (tg < most && 2 * H * ((BT + tg - 1) / tg) * cl > PLAN_SMS) ++tg;
    return tg;
}
// Tensor-core kernel: clusters of four or two CTAs share the blocks of P while they fit the chip at once
// (one sequence of 16 heads, S = 512: the scores took 15,400 cycles of 33,000 on one CTA).
static void small_tc_shape(int H, int64_t BT, int S, int& tg, int& cl) {
    for (cl = S > 256 ? 4 : 2; cl > 1; cl /= 2) {
        tg = small_group(H, BT, AT_TOK, cl);
        if (2 * H * ((BT + tg - 1) / tg) * cl <= PLAN_SMS) return;
    }
    tg = small_group(H, BT, AT_TOK);
}

// Token-sides up to which one launch is the faster way: the passes for large problems need fewer instructions per
// token, this kernel no lists in memory and no further launches.  The kernels' times, theirs / these, us:
//   tensor cores: 32 token-sides (16 heads, S = 512, k = 32) 45 / 15; 1024 (S = 256) 48 / 25; 2048 (S = 256) 49 / 40 and
//     59 / 41, (S = 64, k = 8) 24 / 26 with three launches more; 4096 (S = 256) 59 / 69;
//   FFMA, k > 16: 512 (S = 256, f32) 112 / 20; 8192 (S = 256, d_k = 32 bf16) 191 / 87; 16384 (S = 256, f32) 446 / 323, where
//     S = 512 stays even (65536: 1940 / 1846);
//     k <= 16: 2048 (S = 128, f32) 80 / 29; 12432 (S = 128) 98 / 109; 16384 (S = 64) 70 / 123.
bool addr_small(int dtype, int direct, bool mma, int B, int H, int T, int dk, int S, int kmax) {
    const int64_t items = 2 * static_cast<int64_t>(H) * B * T;
    if (kmax > 32 || S > 1024 || 2 * H > 65535 || (!direct && dk * (dtype == 0 ? 4 : 2) % 16 != 0)) return false;
    return items <= (mma ? 2048 : kmax > 16 ? 8192 : 4096);
}

size_t addr_small_left(const AddrPlan& plan, int B, int H, int T, int dk, int S) {
    const int64_t BT = static_cast<int64_t>(B) * T;
    int tg, cl;
    small_tc_shape(H, BT, S, tg, cl);
    if (plan.mma) return 228 * 1024 - 2048 - at_smem(dk / 64, tg, S);
    tg = small_group(H, BT, 2) == 1 ? 1 : 4;
    return 228 * 1024 - (tg == 1 ? 1 : 2) * (as_smem(tg, S, dk) + 2048);
}

template <class D, int L, int TG>
static cudaError_t launch_small_t(const AddrArgs& a, cudaStream_t stream) {
    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    const size_t smem = as_smem(TG, a.S, a.P[0] != nullptr ? a.dk : 0);
    cudaError_t e = cudaFuncSetAttribute(k_addr_small<D, L, TG>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_ALLOWED);
    if (e != cudaSuccess) return e;
    const int vec = ((reinterpret_cast<uintptr_t>(a.P[0]) | reinterpret_cast<uintptr_t>(a.P[1])) & 15) == 0;
    const dim3 grid(static_cast<unsigned>((BT + TG - 1) / TG), 2 * a.H);
    k_addr_small<D, L, TG><<<grid, as_warps(TG) * 32, smem, stream>>>(a, vec);
    return cudaGetLastError();
}

template <class D, int L>
static cudaError_t launch_small_l(const AddrArgs& a, cudaStream_t stream) {
    return small_group(a.H, static_cast<int64_t>(a.B) * a.T, 2) == 1 ? launch_small_t<D, L, 1>(a, stream)
                                                                     : launch_small_t<D, L, 4>(a, stream);
}

template <int L>
static cudaError_t launch_small_tc(const AddrArgs& a, cudaStream_t stream) {
    CUtensorMap maps[2];
    if (((reinterpret_cast<uintptr_t>(a.X[0]) | reinterpret_cast<uintptr_t>(a.X[1])) & 15) != 0) return cudaErrorInvalidValue;
    cudaError_t e = addr_p_maps(maps, a);
    if (e != cudaSuccess) return e;
    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    int tg, cl;
    small_tc_shape(a.H, BT, a.S, tg, cl);
    const size_t smem = at_smem(a.dk / 64, tg, a.S);
    e = cudaFuncSetAttribute(k_addr_small_tc<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_ALLOWED);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>((BT + tg - 1) / tg * cl), 2 * a.H);
    cfg.blockDim = dim3(AT_WARPS * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = static_cast<unsigned>(cl);
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_addr_small_tc<L>, maps[0], maps[1], a, tg, cl);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_address_small(int dtype, const AddrPlan& plan, const AddrArgs& a, cudaStream_t stream) {
    if (plan.mma) return plan.L == 12 ? launch_small_tc<12>(a, stream) : plan.L == 20 ? launch_small_tc<20>(a, stream)
                                                                                       : launch_small_tc<36>(a, stream);
    switch (plan.L) {
        case 12: return dtype == 0 ? launch_small_l<F32, 12>(a, stream) : launch_small_l<BF16, 12>(a, stream);
        case 20: return dtype == 0 ? launch_small_l<F32, 20>(a, stream) : launch_small_l<BF16, 20>(a, stream);
        case 36: return dtype == 0 ? launch_small_l<F32, 36>(a, stream) : launch_small_l<BF16, 36>(a, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sdm
