// Dense contractions around the SDM path on the 5th-generation tensor cores (bf16 operands,
// fp32 accumulation in TMEM):
//
//   k_gates_tc    the gate projections of every token (Sec. 3.1, after Eq. sdm-write):
//                   [s_a | s_b] = x [W_a; W_b]^T,  x: [B*T, d_model],  N = 2H columns,
//                 with the gate nonlinearities as the epilogue:
//                   alpha = exp(-A softplus(s_a + b_dt)),  beta = sigmoid(s_b).
//   k_head_mix    the head-mixing projection o = z W_o^T ("Norm, Gating, and Head Mixing"),
//                 z: [B*T, H*d_v] (the token-major output of sdm_norm_gate), W_o: [d_model, H*d_v].
//
// Both are one kernel shape: a CTA owns 128 rows (TMEM lanes) x BN columns; TMA streams
// K-blocks of 64 bf16 (one 128-byte swizzle atom) of both operands through an S-stage ring of
// shared memory; one thread issues the loads and the tcgen05.mma (M = 128, N = BN, K = 16 per
// instruction) and releases a stage with tcgen05.commit once the MMAs that read it are done;
// after the last K-block the four warps read their 32 lanes of the accumulator with tcgen05.ld
// and run the epilogue.  Every wait is bounded; a wait that runs out sets the timeout bit of the
// status word and the CTA skips its epilogue.
#include "sdm_internal.h"
#include "tc_common.cuh"

#include <cuda.h>

#include <atomic>

namespace sdm {

namespace {

using namespace tc;

constexpr int GM_THREADS = 128;      // = rows per CTA = TMEM lanes
constexpr int GM_BK = 64;            // K per stage: one 128-byte swizzle atom of bf16

__host__ __device__ constexpr uint32_t gm_stage_bytes(int bn) { return (128u + static_cast<uint32_t>(bn)) * 128u; }
__host__ __device__ constexpr uint32_t gm_smem_bytes(int bn, int stages) {
    return 1024u + gm_stage_bytes(bn) * stages + 256u;      // alignment slack, ring, barriers
}

// 2-D bf16 tensor map of a row-major [rows, cols] matrix, box {64 columns, box_rows rows},
// 128-byte swizzle (the K-major operand layout of the MMA descriptors).
bool gm_map(CUtensorMap* m, const void* base, int64_t rows, int64_t cols, int box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encode();
    if (!enc) return false;
    cuuint64_t dim[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    cuuint64_t str[1] = {static_cast<cuuint64_t>(cols) * 2};
    cuuint32_t box[2] = {GM_BK, static_cast<cuuint32_t>(box_rows)};
    cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dim, str, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The pipelined main loop, run by thread 0: K-blocks of both operands into the ring, four
// MMAs per K-block into the accumulator at `tmem`, then a commit to `done`.  B comes from one
// map (rows n0 .. n0 + BN) or, with tb2, from two maps of BN / 2 rows each (stacked).
template <int BN, int S>
__device__ bool gm_mainloop(const CUtensorMap* ta, const CUtensorMap* tb, const CUtensorMap* tb2, int m0, int n0,
                            int nkb, uint32_t ring, uint32_t bars, uint32_t tmem) {
    const uint32_t full = bars, empty = bars + 8 * S, done = bars + 16 * S;
    const uint32_t stage = gm_stage_bytes(BN);
    const uint32_t idesc = mma_idesc(BN);
    auto load = [&](int kb, int s) {
        const uint32_t a = ring + s * stage, b = a + 128 * 128;
        mbar_expect_tx(full + 8 * s, stage);
        tma_load_2d(a, ta, kb * GM_BK, m0, full + 8 * s);
        if (tb2 == nullptr) {
            tma_load_2d(b, tb, kb * GM_BK, n0, full + 8 * s);
        } else {
            tma_load_2d(b, tb, kb * GM_BK, 0, full + 8 * s);
            tma_load_2d(b + (BN / 2) * 128, tb2, kb * GM_BK, 0, full + 8 * s);
        }
    };
    bool ok = true;
    const int pre = nkb < S ? nkb : S;
    for (int kb = 0; kb < pre; ++kb) load(kb, kb);
    for (int kb = 0; kb < nkb; ++kb) {
        const int s = kb % S;
        const uint32_t ph = static_cast<uint32_t>(kb / S) & 1u;
        if (!mbar_wait(full + 8 * s, ph)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t a = ring + s * stage, b = a + 128 * 128;
#pragma unroll
        for (int kk = 0; kk < GM_BK / 16; ++kk)
            mma_bf16(tmem, sw128_desc(a + kk * 32), sw128_desc(b + kk * 32), idesc, (kb | kk) != 0 ? 1u : 0u);
        mma_commit(empty + 8 * s);             // arrives once these MMAs have read the stage
        if (kb + S < nkb) {
            if (!mbar_wait(empty + 8 * s, ph)) { ok = false; break; }
            load(kb + S, s);
        }
    }
    mma_commit(done);                          // every MMA issued above has completed
    return ok;
}

// Shared set-up of both kernels: ring aligned to 1024 bytes, barriers, TMEM allocation.
struct GmCta {
    uint32_t ring, bars, tmem;
};

template <int BN, int S>
__device__ GmCta gm_setup(unsigned char* sm_raw) {
    const uint32_t raw = smem_u32(sm_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    const uint32_t bars = ring + gm_stage_bytes(BN) * S;       // full[S], empty[S], done, TMEM address
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm_raw + (bars - raw) + 16 * S + 8);
    const int tid = threadIdx.x;
    if (tid < 32) {
        constexpr uint32_t cols = BN < 32 ? 32 : BN;
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(bars + 8 * s, 1);
            mbar_init(bars + 8 * S + 8 * s, 1);
        }
        mbar_init(bars + 16 * S, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    return GmCta{ring, bars, *tmem_slot};
}

template <int BN>
__device__ void gm_teardown(uint32_t tmem) {
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    constexpr uint32_t cols = BN < 32 ? 32 : BN;
    if (threadIdx.x < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(cols) : "memory");
}

// Main loop, then every thread waits for the accumulator (bounded).
template <int BN, int S>
__device__ bool gm_run(const GmCta& c, const CUtensorMap* ta, const CUtensorMap* tb, const CUtensorMap* tb2, int m0,
                       int n0, int nkb) {
    bool ok = true;
    if (threadIdx.x == 0) ok = gm_mainloop<BN, S>(ta, tb, tb2, m0, n0, nkb, c.ring, c.bars, c.tmem);
    ok = __syncthreads_and(ok);
    if (!ok && threadIdx.x == 0) {              // let the copies in flight land before the CTA ends
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) __nanosleep(1000);
    }
    if (ok) ok = mbar_wait(c.bars + 16 * S, 0);
    ok = __syncthreads_and(ok);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    return ok;
}

// ------------------------------------------------------------------------------------------
// Gates: BN = 2H columns (32 or 64), rows = tokens.
// ------------------------------------------------------------------------------------------
constexpr int GATE_STAGES = 4;

template <int BN>
__global__ void __launch_bounds__(GM_THREADS) k_gates_tc(const __grid_constant__ CUtensorMap tx,
                                                         const __grid_constant__ CUtensorMap twa,
                                                         const __grid_constant__ CUtensorMap twb,
                                                         const float* __restrict__ b_dt, const float* __restrict__ A,
                                                         __nv_bfloat16* __restrict__ alpha, __nv_bfloat16* __restrict__ beta,
                                                         int64_t tokens, int T, int d, int* err) {
    constexpr int H = BN / 2;
    extern __shared__ unsigned char sm_raw[];
    const GmCta c = gm_setup<BN, GATE_STAGES>(sm_raw);
    const int m0 = blockIdx.x * 128;
    const int nkb = (d + GM_BK - 1) / GM_BK;
    const bool ok = gm_run<BN, GATE_STAGES>(c, &tx, &twa, &twb, m0, 0, nkb);
    const int warp = threadIdx.x >> 5;
    const int64_t u = m0 + threadIdx.x;                   // this thread's token row
    if (ok) {
        const uint32_t trow = c.tmem + (static_cast<uint32_t>(warp * 32) << 16);
#pragma unroll
        for (int cb = 0; cb < BN / 32; ++cb) {
            float v[32];
            tmem_ld32(trow + cb * 32, v);                  // warp-collective
            if (u < tokens) {
                const int64_t b = u / T, t = u - b * T;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int j = cb * 32 + i;
                    if (j < H) {
                        const float za = v[i] + __ldg(b_dt + j);
                        const float sp = za > 20.f ? za : log1pf(expf(za));     // softplus
                        alpha[(b * H + j) * T + t] = __float2bfloat16_rn(expf(-__ldg(A + j) * sp));
                    } else {
                        beta[(b * H + (j - H)) * T + t] = __float2bfloat16_rn(1.f / (1.f + expf(-v[i])));
                    }
                }
            }
        }
    } else if (threadIdx.x == 0) {
        flag_error(err, ERR_TIMEOUT);
    }
    gm_teardown<BN>(c.tmem);
}

// ------------------------------------------------------------------------------------------
// Head mix: BN = 256 output columns per CTA, out row-major [M, N] bf16.
// ------------------------------------------------------------------------------------------
constexpr int MIX_BN = 256;
constexpr int MIX_STAGES = 4;

__global__ void __launch_bounds__(GM_THREADS, 1) k_head_mix(const __grid_constant__ CUtensorMap tz,
                                                            const __grid_constant__ CUtensorMap tw,
                                                            __nv_bfloat16* __restrict__ out, int64_t M, int N, int K,
                                                            int* err) {
    extern __shared__ unsigned char sm_raw[];
    const GmCta c = gm_setup<MIX_BN, MIX_STAGES>(sm_raw);
    const int ntn = (N + MIX_BN - 1) / MIX_BN;
    const int m0 = static_cast<int>(blockIdx.x / ntn) * 128, n0 = static_cast<int>(blockIdx.x % ntn) * MIX_BN;
    const bool ok = gm_run<MIX_BN, MIX_STAGES>(c, &tz, &tw, nullptr, m0, n0, (K + GM_BK - 1) / GM_BK);
    const int warp = threadIdx.x >> 5;
    const int64_t r = m0 + threadIdx.x;
    if (ok) {
        const uint32_t trow = c.tmem + (static_cast<uint32_t>(warp * 32) << 16);
#pragma unroll 1
        for (int cb = 0; cb < MIX_BN / 32; ++cb) {
            float v[32];
            tmem_ld32(trow + cb * 32, v);                  // warp-collective
            const int n = n0 + cb * 32;
            if (r < M && n < N) {                          // N % 32 == 0: whole 32-column blocks
                uint4* dst = reinterpret_cast<uint4*>(out + r * N + n);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        __nv_bfloat162 p = __floats2bfloat162_rn(v[q * 8 + 2 * e], v[q * 8 + 2 * e + 1]);
                        w[e] = *reinterpret_cast<uint32_t*>(&p);
                    }
                    dst[q] = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
        }
    } else if (threadIdx.x == 0) {
        flag_error(err, ERR_TIMEOUT);
    }
    gm_teardown<MIX_BN>(c.tmem);
}

// ------------------------------------------------------------------------------------------
// Head mix on large outputs: a persistent pair of CTAs (a cluster of two on one TPC) per 256 x 256 tile.
//
// Why pairs: a 128 x 256 tile of one CTA reads (128 + 256) x 128 bytes of operands per 64 of K, 96
// bytes per clock of its tensor pipe, more than an SM gets from L2 (that kernel stays near half
// of the tensor peak whatever its pipeline).  With cta_group::2 each CTA stages its own 128 rows of z and
// half of W_o's 256 rows, 64 bytes per clock, and the pair's MMA (M = 256, N = 256) reads both halves.
// Roles: warp 0 loads (both CTAs), warp 1 issues the MMAs (the leader's only), warps 2-5 are the
// epilogue.  The accumulator is double-buffered in TMEM (2 x 256 columns), so a tile's epilogue runs
// under the next tile's main loop.  Barriers: full[s] in the leader counts the bytes of both CTAs'
// loads; empty[s] and acc_full[b] are committed by the MMA to both CTAs; acc_empty[b] in the
// leader collects the eight epilogue warps.  Every wait is bounded; a role that times out leaves its
// loop, sets the timeout bit, and the CTAs still meet at the end to free TMEM.
//
// Bound by the tensor pipe: 32,768 x 2048 x 2048 take 154 us (1.79 PFLOP/s, 0.91 of the measured peak);
// the one-CTA kernel 293 us.
// ------------------------------------------------------------------------------------------
constexpr int PR_THREADS = 192;
constexpr int PR_STAGES = 6;
constexpr uint32_t PR_STAGE_BYTES = 2u * 128u * 128u;     // z rows, W_o rows of one CTA
constexpr uint32_t PR_SMEM = 1024u + PR_STAGES * PR_STAGE_BYTES + 256u;

__device__ __forceinline__ uint32_t pr_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t pr_in_leader(uint32_t addr) {      // the same shared address in CTA 0
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(0));
    return r;
}
__device__ __forceinline__ void pr_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void pr_load(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t leader_bar) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
                 ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(leader_bar) : "memory");
}
__device__ __forceinline__ void pr_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                 ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void pr_commit(uint32_t bar) {              // arrives at `bar` in both CTAs
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n"
                 ::"r"(bar), "h"(static_cast<unsigned short>(3)) : "memory");
}
__device__ __forceinline__ void pr_arrive_leader(uint32_t leader_bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(leader_bar) : "memory");
}
// Instruction descriptor, kind::f16: bf16 A and B (K-major), fp32 D, M = 256 (both CTAs), N = 256.
__device__ __forceinline__ uint32_t pr_idesc() {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(256 >> 3) << 17) | (static_cast<uint32_t>(256 >> 4) << 24);
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PR_THREADS, 1)
k_head_mix_pair(const __grid_constant__ CUtensorMap tz, const __grid_constant__ CUtensorMap tw,
                __nv_bfloat16* __restrict__ out, int64_t M, int N, int K, int tiles, int* err) {
    extern __shared__ unsigned char sm_raw[];
    const uint32_t raw = smem_u32(sm_raw);
    const uint32_t ring = (raw + 1023u) & ~1023u;
    const uint32_t bars = ring + PR_STAGES * PR_STAGE_BYTES;
    const uint32_t full = bars, empty = bars + 8 * PR_STAGES, acc_full = bars + 16 * PR_STAGES, acc_empty = acc_full + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm_raw + (acc_empty + 16 - raw));
    const uint32_t rank = pr_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < PR_STAGES; ++i) {
            mbar_init(full + 8 * i, 1);
            mbar_init(empty + 8 * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(acc_full + 8 * i, 1);
            mbar_init(acc_empty + 8 * i, 8);
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    pr_cluster_sync();                                     // both CTAs' barriers are set up
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    const int ntn = (N + 255) / 256, nkb = (K + GM_BK - 1) / GM_BK;
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    bool ok = true;
    if (warp == 0 && lane == 0) {
        // ---- loads: this CTA's 128 rows of z and 128 rows of W_o
        uint32_t kc = 0;                                    // K-blocks so far
        for (int tile = pair; tile < tiles && ok; tile += pairs) {
            const int m0 = (tile / ntn) * 256 + static_cast<int>(rank) * 128, n0 = (tile % ntn) * 256 + static_cast<int>(rank) * 128;
            for (int kb = 0; kb < nkb; ++kb, ++kc) {
                const uint32_t s = kc % PR_STAGES, round = kc / PR_STAGES;
                if (round > 0 && !mbar_wait(empty + 8 * s, (round - 1) & 1u)) { ok = false; break; }
                if (rank == 0) mbar_expect_tx(full + 8 * s, 2 * PR_STAGE_BYTES);
                const uint32_t dst = ring + s * PR_STAGE_BYTES, bar = pr_in_leader(full + 8 * s);
                pr_load(dst, &tz, kb * GM_BK, m0, bar);
                pr_load(dst + 128 * 128, &tw, kb * GM_BK, n0, bar);
            }
        }
        // the last use of every stage: the peer's commits have arrived here before the CTA may end
        const uint32_t used = kc < PR_STAGES ? kc : PR_STAGES;
        for (uint32_t i = 0; i < used && ok; ++i) {
            const uint32_t last = kc - 1 - i;
            ok = mbar_wait(empty + 8 * (last % PR_STAGES), (last / PR_STAGES) & 1u);
        }
        if (!ok) {                                          // let the copies in flight land before the CTA ends
            const long long t0 = clock64();
            while (clock64() - t0 < 2000000) __nanosleep(1000);
        }
    } else if (warp == 1 && lane == 0 && rank == 0) {
        // ---- MMAs of the pair
        uint32_t kc = 0, it = 0;
        for (int tile = pair; tile < tiles && ok; tile += pairs, ++it) {
            const uint32_t buf = it & 1u, use = it >> 1;
            if (use > 0 && !mbar_wait(acc_empty + 8 * buf, (use - 1) & 1u)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            for (int kb = 0; kb < nkb; ++kb, ++kc) {
                const uint32_t s = kc % PR_STAGES;
                if (!mbar_wait(full + 8 * s, (kc / PR_STAGES) & 1u)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint32_t a = ring + s * PR_STAGE_BYTES, b = a + 128 * 128;
#pragma unroll
                for (int kk = 0; kk < GM_BK / 16; ++kk)
                    pr_mma(tmem + buf * 256, sw128_desc(a + kk * 32), sw128_desc(b + kk * 32), pr_idesc(), (kb | kk) != 0 ? 1u : 0u);
                pr_commit(empty + 8 * s);                   // both CTAs' stages are free once these are done
            }
            if (ok) pr_commit(acc_full + 8 * buf);
        }
    } else if (warp >= 2) {
        // ---- epilogue: TMEM lanes 32 (warp % 4) .. + 31 are this warp's rows
        const uint32_t quarter = static_cast<uint32_t>(warp & 3);
        uint32_t it = 0;
        for (int tile = pair; tile < tiles; tile += pairs, ++it) {
            const uint32_t buf = it & 1u, use = it >> 1;
            if (!__all_sync(0xffffffffu, mbar_wait(acc_full + 8 * buf, use & 1u))) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const int64_t r = static_cast<int64_t>(tile / ntn) * 256 + rank * 128 + quarter * 32 + lane;
            const int n0 = (tile % ntn) * 256;
            const uint32_t trow = tmem + buf * 256 + ((quarter * 32u) << 16);
#pragma unroll 1
            for (int cb = 0; cb < 8; ++cb) {
                float v[32];
                tmem_ld32(trow + cb * 32, v);               // warp-collective
                const int n = n0 + cb * 32;
                if (r < M && n < N) {                       // N % 32 == 0: whole 32-column blocks
                    uint4* dst = reinterpret_cast<uint4*>(out + r * N + n);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            __nv_bfloat162 p = __floats2bfloat162_rn(v[q * 8 + 2 * e], v[q * 8 + 2 * e + 1]);
                            w[e] = *reinterpret_cast<uint32_t*>(&p);
                        }
                        dst[q] = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) pr_arrive_leader(pr_in_leader(acc_empty + 8 * buf));
        }
    }
    if (!ok && lane == 0) flag_error(err, ERR_TIMEOUT);
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    pr_cluster_sync();                                      // no barrier of this CTA is in use any more
    if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512) : "memory");
}

}  // namespace

bool gates_tc_supported(int dtype, int H, int d) {
    return dtype == 1 && (H == 16 || H == 32) && d % 8 == 0 && d > 0;
}

cudaError_t launch_gates_tc(const void* x, const void* W_a, const void* W_b, const float* b_dt, const float* A,
                            void* alpha, void* beta, int B, int T, int H, int d, int* err, cudaStream_t stream) {
    const int64_t tokens = static_cast<int64_t>(B) * T;
    CUtensorMap maps[3];
    if (!gm_map(&maps[0], x, tokens, d, 128) || !gm_map(&maps[1], W_a, H, d, H) || !gm_map(&maps[2], W_b, H, d, H))
        return cudaErrorInvalidValue;
    const unsigned grid = static_cast<unsigned>((tokens + 127) / 128);
    auto* al = static_cast<__nv_bfloat16*>(alpha);
    auto* be = static_cast<__nv_bfloat16*>(beta);
    cudaError_t e;
    if (H == 16) {
        const size_t smem = gm_smem_bytes(32, GATE_STAGES);
        e = cudaFuncSetAttribute(k_gates_tc<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        k_gates_tc<32><<<grid, GM_THREADS, smem, stream>>>(maps[0], maps[1], maps[2], b_dt, A, al, be, tokens, T, d, err);
    } else {
        const size_t smem = gm_smem_bytes(64, GATE_STAGES);
        e = cudaFuncSetAttribute(k_gates_tc<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        k_gates_tc<64><<<grid, GM_THREADS, smem, stream>>>(maps[0], maps[1], maps[2], b_dt, A, al, be, tokens, T, d, err);
    }
    return cudaGetLastError();
}

// CTA pairs of k_head_mix_pair resident at once, per device (asked once).
static cudaError_t pair_clusters(int* out) {
    static std::atomic<int> known[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int n = dev >= 0 && dev < 64 ? known[dev].load(std::memory_order_relaxed) : 0;
    if (n == 0) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(2);
        cfg.blockDim = dim3(PR_THREADS);
        cfg.dynamicSmemBytes = PR_SMEM;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&n, k_head_mix_pair, &cfg);
        if (e != cudaSuccess) return e;
        if (n < 1) return cudaErrorInvalidConfiguration;
        if (dev >= 0 && dev < 64) known[dev].store(n, std::memory_order_relaxed);
    }
    *out = n;
    return cudaSuccess;
}

// Pairs of CTAs with 256 x 256 tiles once there is a tile for every pair of SMs (154 against 293 us for
// 1024 tiles); below that the one-CTA kernel's 128 x 256 tiles keep more SMs busy.
cudaError_t launch_head_mix(const void* z, const void* W_o, void* out, int64_t M, int N, int K, int* err,
                            cudaStream_t stream) {
    CUtensorMap maps[2];
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t pair_tiles = ((M + 255) / 256) * ((N + 255) / 256);
    if (pair_tiles >= sms / 2 && pair_tiles < (static_cast<int64_t>(1) << 31)) {
        if (!gm_map(&maps[0], z, M, K, 128) || !gm_map(&maps[1], W_o, N, K, 128)) return cudaErrorInvalidValue;
        e = cudaFuncSetAttribute(k_head_mix_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(PR_SMEM));
        if (e != cudaSuccess) return e;
        int clusters = 0;                        // pairs the device holds at once (a tail of late pairs would double the time)
        e = pair_clusters(&clusters);
        if (e != cudaSuccess) return e;
        const unsigned grid = 2u * static_cast<unsigned>(pair_tiles < clusters ? pair_tiles : clusters);
        k_head_mix_pair<<<grid, PR_THREADS, PR_SMEM, stream>>>(maps[0], maps[1], static_cast<__nv_bfloat16*>(out), M, N, K,
                                                             static_cast<int>(pair_tiles), err);
        return cudaGetLastError();
    }
    if (!gm_map(&maps[0], z, M, K, 128) || !gm_map(&maps[1], W_o, N, K, MIX_BN)) return cudaErrorInvalidValue;
    const int64_t tiles = ((M + 127) / 128) * ((N + MIX_BN - 1) / MIX_BN);
    const size_t smem = gm_smem_bytes(MIX_BN, MIX_STAGES);
    e = cudaFuncSetAttribute(k_head_mix, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    k_head_mix<<<static_cast<unsigned>(tiles), GM_THREADS, smem, stream>>>(maps[0], maps[1],
                                                                           static_cast<__nv_bfloat16*>(out), M, N, K, err);
    return cudaGetLastError();
}

}  // namespace sdm
