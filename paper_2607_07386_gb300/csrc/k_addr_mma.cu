// K-ADDR scores on the 5th-generation tensor cores (bf16 storage, PROJECTED addressing).
//
// The half-scores s = P x (Sec. 3.1 item 1) of 128 tokens x one half (S columns, in chunks of at
// most 512) form a dense [128 x d_k] x [d_k x S] contraction: TMA stages the x tile and units
// of 256 rows x 64 values of P in shared memory (128-byte swizzle, K-major, two units in flight), one
// thread issues tcgen05.mma (M = 128, N <= 256 per instruction, K = 16 per step, bf16 inputs, fp32
// accumulation in TMEM), and each of the 128 threads then owns one token's TMEM row.
//
// Per-token top-L selection of the half (L = k + 4; the finalize kernels certify it), all
// branch-free so a warp's 32 tokens run in lockstep; the passes over TMEM are loops over
// 32-column blocks (compact code: the kernel is instruction-fetch bound when unrolled):
//   1. the largest score of each of 64 or 128 column classes, held as truncated bf16 pairs;
//   2. theta, a lower bound on the L-th largest score: the smaller of the L/2-th largest class maxima
//      among the even and the odd columns (a pruned merge-exchange network on the pairs), so
//      that >= L distinct columns are >= it;
//   3. survivors (score >= theta), about 1.3 L of them, compacted into a per-thread shared-memory
//      buffer: every column is stored, a survivor advances the store position;
//   4. survivors sorted by 32-bit keys, the score with its low bits replaced by the buffer slot;
//      scores and columns of the first L are then read back by slot, neighbours whose keys
//      differed by less than that in the wrong order are exchanged, and the list goes to the
//      workspace.  A tie of keys at the cut after L is decided by an exact sort.
// More survivors than the buffer holds: the tile repeats with a lower bound on the L-th largest of
// those it kept as threshold; after three rounds (heavy ties) an exact insertion scan decides.
// With several chunks (S > 512) pass 1 runs over all of them and pass 3 again, the accumulators
// formed anew (the tensor cores are idle otherwise); one list per half comes out for any S.
//
// Bound by the instructions of a warp's chain (about 7,000 per token): TMEM holds one 128 x 512 tile per SM,
// so its columns are given back before the sort and a second CTA on the SM scores its tile
// meanwhile (at 97 KB of shared memory each, which leaves room for the M0 copy beside them).
// 524,288 tokens x 2 sides, S = 512, d_k = 128, L = 36: 1.30 ms (1.65 ms beside the M0 copy); 2.17
// (2.85) ms with the two largest scores of 32 classes, a sort of (score, column) pairs and one CTA per SM.
// A cycle count per tile: operands and MMA 5,500, maxima 4,000, threshold 1,700, compaction 7,500 (28
// per column with predicated stores, 14,300), then without TMEM sort 5,000, look-up 1,200, stores 3,000.
#include "sdm_internal.h"
#include "tc_common.cuh"

#include <cuda.h>

namespace sdm {

namespace {

using namespace tc;

constexpr int MM_THREADS = 128;      // = tokens per CTA = TMEM lanes
constexpr int MM_NB = 256;           // columns per MMA instruction and per staged block of P
constexpr int MM_UNIT = MM_NB * 128; // bytes of a staged unit: a block's 64 values of d_k
constexpr int MM_SLOT = MM_THREADS * 8;        // bytes of a survivor slot of all threads: (score, column) pairs

// Survivor slots per thread, packed registers of class maxima (two classes each).  With random
// scores the survivors of L = 12, 20, 36, 68 are 16 +- 3, 27 +- 4, 46 +- 5, 96 +- 8 of 512.
__host__ __device__ constexpr int mm_buf(int L) { return L <= 12 ? 40 : L <= 20 ? 56 : L <= 36 ? 72 : 121; }
__host__ __device__ constexpr int mm_pairs(int L) { return L <= 20 ? 32 : 64; }
__host__ __device__ constexpr int mm_slot_bits(int L) { return mm_buf(L) <= 64 ? 6 : 7; }
// Five more slots than survivors: the store position is held at slot BUF + 1, which marks an
// overflow, after every four columns.
__host__ __device__ constexpr uint32_t mm_buf_bytes(int L) { return static_cast<uint32_t>(mm_buf(L) + 5) * MM_SLOT; }

__device__ __forceinline__ void exchange(float& a, float& b) {           // a >= b afterwards
    const float hi = fmaxf(a, b), lo = fminf(a, b);
    a = hi;
    b = lo;
}
__device__ __forceinline__ void exchange(__nv_bfloat162& a, __nv_bfloat162& b) {
    const __nv_bfloat162 hi = __hmax2(a, b), lo = __hmin2(a, b);
    a = hi;
    b = lo;
}
// Merge-exchange sort (Batcher; Knuth vol. 3, Algorithm 5.2.2 M) of N values, descending; the
// compiler drops the exchanges that no used output needs.
template <int N, int P, int K, class T>
__device__ __forceinline__ void merge_exchange_step(T (&v)[N]) {
#pragma unroll
    for (int j = K % P; j + K < N; j += 2 * K) {
#pragma unroll
        for (int i = 0; i < K; ++i) {
            if (i + j + K < N && (i + j) / (2 * P) == (i + j + K) / (2 * P)) exchange(v[i + j], v[i + j + K]);
        }
    }
    if constexpr (K > 1) merge_exchange_step<N, P, K / 2>(v);
}
template <int N, int P = 1, class T>
__device__ __forceinline__ void sort_desc(T (&v)[N]) {
    merge_exchange_step<N, P, P>(v);
    if constexpr (2 * P < N) sort_desc<N, 2 * P>(v);
}

// Puts (v, col) at `ptr` (a shared address) and advances past it when v >= theta (a NaN on either
// side does not); a column that does not is overwritten by the next one.  No predicate, so that the
// compares of neighbouring columns overlap: 28 cycles per column with predicated stores.
__device__ __forceinline__ void put(uint32_t ptr, uint32_t v, int col) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};\n" ::"r"(ptr), "r"(v), "r"(col));
}

// The 32-column blocks of a token's row at `trow`, each handed to f(r, cb) with the next one's load in
// flight (columns past np come as `pad`).
template <class F>
__device__ __forceinline__ void tmem_blocks(uint32_t trow, int np, uint32_t pad, F&& f) {
    const int nb = (np + 31) >> 5;
    uint32_t r[2][32];
    tmem_ld32_issue(trow, r[0]);
#pragma unroll 1
    for (int cb = 0; cb < nb; cb += 2) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (cb + q < nb) {                                    // (warp-uniform)
                tmem_wait(r[q]);
                if (cb + q + 1 < nb) tmem_ld32_issue(trow + (cb + q + 1) * 32, r[q ^ 1]);
                if ((cb + q) * 32 + 32 > np) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) r[q][j] = (cb + q) * 32 + j < np ? r[q][j] : pad;
                }
                f(r[q], cb + q, q);
            }
        }
    }
}

}  // namespace

struct MmaLaunch {
    int B, H, T, dk, S;
    int bt, bb, ntt;            // token box: bt tokens x bb sequences (bt * bb <= 128); t-tiles
    int pb;                     // P box height (rows), <= 256 and <= 2S
    int atoms;                  // ceil(dk / 64)
    float* part_v;
    int* part_i;
    int* err;
    float* raw;                 // test hook: the raw fp32 scores [2H][B*T][2S] instead of the lists
    int tiles;                  // token tiles (blockIdx.x beyond them: the preparation blocks)
    const void* P[2];           // as in AddrArgs, for the row norms
    float* pnorm;
    int* queue;
};

// What the finalize passes need besides the lists, from blocks of their own in the same launch: the
// largest row norm of a head's P (rounded up, for the score error bound) and empty queues.  As a
// kernel before the scores it cost a one-token step 10 of its 65 us, and it held the SMs at the moment the M0
// copy's CTAs were placed, which then piled up on a few of them.
__device__ __forceinline__ void prepare_finalize(const MmaLaunch& a) {
    __shared__ int s_max;
    const int z = blockIdx.z, tid = threadIdx.x;
    if (blockIdx.y == 1) {
        if (z == 0 && tid < 2 && a.queue != nullptr) a.queue[tid] = 0;
        return;
    }
    if (a.pnorm == nullptr) return;
    if (tid == 0) s_max = 0;
    __syncthreads();
    const uint4* P = static_cast<const uint4*>(a.P[z / a.H]) + static_cast<int64_t>(z % a.H) * 2 * a.S * (a.dk / 8);
    float mx = 0.f;
    for (int r = tid; r < 2 * a.S; r += MM_THREADS) {
        float ss = 0.f;
        for (int q0 = 0; q0 < a.dk / 8; q0 += 8) {               // d_k is 64 or 128
            uint4 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = __ldg(P + static_cast<int64_t>(r) * (a.dk / 8) + q0 + q);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float f[8];
                unpack16<BF16>(v[q], f);
#pragma unroll
                for (int e = 0; e < 8; ++e) ss = fmaf(f[e], f[e], ss);
            }
        }
        mx = fmaxf(mx, sqrtf(ss) * (1.f + 0x1p-12f));            // (a row with a NaN is never selected: no part of the bound)
    }
    atomicMax(&s_max, __float_as_int(mx));                        // non-negative floats order as integers
    __syncthreads();
    if (tid == 0) a.pnorm[z] = __int_as_float(s_max);
}

// COLS: TMEM columns (fp32 accumulators) = maximum chunk width.  ALIAS: one chunk; the survivor
// buffer takes the place of the operands once the MMAs have read them.
template <int COLS, int L, bool ALIAS>
__global__ void __launch_bounds__(MM_THREADS, ALIAS && L <= 36 ? 2 : 1)
k_addr_mma(const __grid_constant__ CUtensorMap tx_q, const __grid_constant__ CUtensorMap tx_k,
           const __grid_constant__ CUtensorMap tp_q, const __grid_constant__ CUtensorMap tp_k, const MmaLaunch a) {
    constexpr int BUF = mm_buf(L), NQ = mm_pairs(L);
    if (static_cast<int>(blockIdx.x) >= a.tiles) {
        prepare_finalize(a);
        return;
    }
    extern __shared__ unsigned char sm_raw[];
    // 1024-byte aligned operand region (the 128-byte swizzle repeats every 8 rows = 1024 B)
    const uint32_t raw = smem_u32(sm_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* sm = sm_raw + (base - raw);
    const uint32_t sA = base;                                    // x: [atoms][128 rows][128 B]
    const uint32_t sB = sA + a.atoms * 128 * 128;                 // P: two units of [256 rows][128 B]
    const uint32_t sBuf = ALIAS ? sA : sB + 2 * MM_UNIT;          // survivors: [BUF + 5][128](score, column)
    const uint32_t end = ALIAS ? max(sB + 2 * MM_UNIT, sBuf + mm_buf_bytes(L)) : sBuf + mm_buf_bytes(L);
    const uint32_t bar_x = end, bar_full = end + 8, bar_empty = end + 24, bar_done = end + 40;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + (end - base) + 48);

    const int tid = threadIdx.x, warp = tid >> 5;
    const int side = blockIdx.z / a.H, h = blockIdx.z % a.H;
    const int hf = blockIdx.y;
    const int nchunk = ALIAS ? 1 : (a.S + COLS - 1) / COLS;
    const int ti = blockIdx.x % a.ntt, bi = blockIdx.x / a.ntt;
    const int t0 = ti * a.bt, b0 = bi * a.bb;
    const CUtensorMap* tx = side ? &tx_k : &tx_q;
    const CUtensorMap* tp = side ? &tp_k : &tp_q;

    // ---- thread 0 stages units of P (a block of columns x 64 values of d_k, in the order the MMAs
    // take them) and issues the MMAs; nload, nmma: units so far
    uint32_t nload = 0, nmma = 0;
    auto chunk_cols = [&](int ch) { return min(a.S - ch * COLS, COLS); };
    auto chunk_units = [&](int ch) { return (chunk_cols(ch) + MM_NB - 1) / MM_NB * a.atoms; };
    auto load_unit = [&](int ch, int unit) {
        const uint32_t s = nload & 1u;
        const int blk = unit / a.atoms, at = unit - blk * a.atoms;
        if (nload >= 2 && !mbar_wait(bar_empty + 8 * s, ((nload >> 1) - 1) & 1u)) return false;
        mbar_expect_tx(bar_full + 8 * s, a.pb * 128);
        tma_load_3d(sB + s * MM_UNIT, tp, at * 64, hf * a.S + ch * COLS + blk * MM_NB, h, bar_full + 8 * s);
        ++nload;
        return true;
    };
    auto run_chunk = [&](int ch, int loaded, uint32_t acc) {       // `loaded` units are on their way already
        const int npad = (chunk_cols(ch) + 15) & ~15, nu = chunk_units(ch);
        bool ok = true;
        for (int unit = loaded; unit < min(nu, 2) && ok; ++unit) ok = load_unit(ch, unit);
        for (int unit = 0; unit < nu && ok; ++unit) {
            const uint32_t s = nmma & 1u;
            const int blk = unit / a.atoms, at = unit - blk * a.atoms;
            ok = mbar_wait(bar_full + 8 * s, (nmma >> 1) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t idesc = mma_idesc(min(MM_NB, npad - blk * MM_NB));
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma_bf16(acc + blk * MM_NB, sw128_desc(sA + at * 128 * 128 + ks * 32), sw128_desc(sB + s * MM_UNIT + ks * 32),
                         idesc, at + ks > 0 ? 1u : 0u);
            mma_commit(bar_empty + 8 * s);
            ++nmma;
            if (unit + 2 < nu) ok = load_unit(ch, unit + 2);
        }
        mma_commit(bar_done);
        return ok;
    };

    bool ok = true;
    int pre = 0;
    if (tid == 0) {
        mbar_init(bar_x, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 1); }
        mbar_init(bar_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        // x tile: rows = (b0 .. b0+bb-1) x (t0 .. t0+bt-1) of head h, and the first blocks of P, under the
        // wait for TMEM columns
        mbar_expect_tx(bar_x, a.atoms * a.bt * a.bb * 128);
        for (int at = 0; at < a.atoms; ++at) tma_load_4d(sA + at * 128 * 128, tx, at * 64, t0, h, b0, bar_x);
        for (; pre < min(2, chunk_units(0)); ++pre) load_unit(0, pre);
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    // chunk ch's scores in TMEM (block-uniform; false after a wait that ran out)
    int held = -1;
    uint32_t ndone = 0;
    auto need = [&](int ch) {
        if (!ok || ch == held) return ok;
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();                                          // the chunk before has been read
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (tid == 0) {
            if (held < 0) ok = mbar_wait(bar_x, 0);
            if (ok) ok = run_chunk(ch, held < 0 ? pre : 0, tmem);
            if (!ok) {                                            // own copies in flight, again with a limit
                if (held < 0) mbar_wait(bar_x, 0);
                for (uint32_t u = nload > 2 ? nload - 2 : 0; u < nload; ++u) mbar_wait(bar_full + 8 * (u & 1u), (u >> 1) & 1u);
            }
        }
        ok = __syncthreads_and(ok);
        if (ok) ok = mbar_wait(bar_done, ndone & 1u);
        ok = __syncthreads_and(ok);
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        ++ndone;
        held = ch;
        return ok;
    };
    bool freed = false;
    auto free_tmem = [&]() {                                      // (after a block barrier)
        if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(COLS) : "memory");
        freed = true;
    };

    const int64_t BT = static_cast<int64_t>(a.B) * a.T;
    const int b = b0 + tid / a.bt, t = t0 + tid % a.bt;
    const bool mine = b < a.B && t < a.T;
    const uint32_t trow = tmem + (static_cast<uint32_t>(warp * 32) << 16);

    if (a.raw != nullptr) {
        // test hook: the accumulators themselves, one token row per thread, no selection
        float* dst = a.raw + (static_cast<int64_t>(blockIdx.z) * BT + static_cast<int64_t>(b) * a.T + t) * (2 * a.S) + hf * a.S;
        for (int ch = 0; ch < nchunk && need(ch); ++ch) {
            const int np = chunk_cols(ch);
#pragma unroll 1
            for (int cb = 0; cb * 32 < np; ++cb) {
                float v[32];
                tmem_ld32(trow + cb * 32, v);                        // warp-collective: every lane loads
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (mine && cb * 32 + j < np) dst[ch * COLS + cb * 32 + j] = v[j];
            }
        }
        if (!ok && tid == 0) flag_error(a.err, ERR_TIMEOUT);
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
        free_tmem();
        return;
    }

    // Rows past the batch (a tile of fewer than 128 tokens) hold zeros or stale operands: they
    // select nothing, and a warp of them skips the passes (warp-uniform, so the warp-collective
    // TMEM loads stay whole).  Left in, S equal scores a row ran every retry and the insertion
    // scan: 0.29 ms for one token of 16 heads.
    const bool work = __any_sync(0xffffffffu, mine);

    // 1-2. class maxima, truncated to bf16 (pairs of neighbouring columns), then the threshold
    float theta = __int_as_float(0x7fffffff);                     // NaN: selects nothing
    {
        __nv_bfloat162 m[NQ];
        const uint32_t ninf = 0xff80ff80u;
#pragma unroll
        for (int i = 0; i < NQ; ++i) m[i] = *reinterpret_cast<const __nv_bfloat162*>(&ninf);
        for (int ch = 0; ch < nchunk && need(ch); ++ch) {
            const int np = chunk_cols(ch);
            if (!work) continue;
            // blocks 2 i and 2 i + 1 fill the registers of 64 classes; with 128 classes, odd i the others
            int half = 0;
            tmem_blocks(trow, np, 0xff800000u, [&](uint32_t (&r)[32], int, int q) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const uint32_t w = __byte_perm(r[2 * j], r[2 * j + 1], 0x7632);
                    const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162*>(&w);
                    if constexpr (NQ == 32) {
                        m[q * 16 + j] = __hmax2(m[q * 16 + j], x);
                    } else {
                        if (half) m[32 + q * 16 + j] = __hmax2(m[32 + q * 16 + j], x);
                        else m[q * 16 + j] = __hmax2(m[q * 16 + j], x);
                    }
                }
                if (q == 1) half ^= 1;
            });
        }
        if (work && mine && ok) {
            sort_desc<NQ>(m);                                     // even and odd columns side by side
            const float th = fminf(__low2float(m[L / 2 - 1]), __high2float(m[L / 2 - 1]));
            // truncation raised a negative bound by less than 2^-7 of it
            theta = a.S < L ? -INFINITY : th > 0.f ? th : fmaf(th, 1.f + 0x1p-7f, -0x1p-126f);
        }
    }

    // 3-4. compaction of survivors, then the sort; on overflow the tile repeats with a lower bound on
    // the L-th largest survivor kept so far (still one on the L-th largest score)
    const uint32_t my_buf = sBuf + tid * 8, last = my_buf + (BUF + 1) * MM_SLOT;
    const float* buf_v = reinterpret_cast<const float*>(sm + (sBuf - base)) + 2 * tid;    // [slot * 256]
    const int* buf_i = reinterpret_cast<const int*>(sm + (sBuf - base) + 4) + 2 * tid;
    constexpr uint32_t SLOT_MASK = (1u << mm_slot_bits(L)) - 1u;
    float key[BUF];
    int cnt = 0;
    bool exact = false;
    for (int round = 0; round < 3; ++round) {
        uint32_t ptr = my_buf;
        const int first = held < 0 ? 0 : held;
        for (int i = 0; i < nchunk; ++i) {
            const int ch = first + i < nchunk ? first + i : first + i - nchunk;
            if (!need(ch)) break;
            const int np = chunk_cols(ch);
            if (!work) continue;
            tmem_blocks(trow, np, 0x7fffffffu, [&](uint32_t (&r)[32], int cb, int) {
                const int col = ch * COLS + cb * 32;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    put(ptr, r[j], col + j);
                    uint32_t over;                                 // all ones when the score reaches theta
                    asm("set.ge.u32.f32 %0, %1, %2;" : "=r"(over) : "f"(__uint_as_float(r[j])), "f"(theta));
                    ptr -= over * MM_SLOT;
                    if (j % 4 == 3) ptr = min(ptr, last);
                }
            });
        }
        const bool overflow = ptr == last;
        cnt = overflow ? BUF : static_cast<int>((ptr - my_buf) / MM_SLOT);
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        const bool again = __syncthreads_or(overflow);
        if (!again) free_tmem();                                  // the next tile's CTA may score now
        if (work) {
#pragma unroll
            for (int i = 0; i < BUF; ++i) {
                const float v = fminf(fmaxf(i < cnt ? buf_v[i * 256] : -INFINITY, -3.4028234e38f), 3.4028234e38f);
                key[i] = __uint_as_float((__float_as_uint(v) & ~SLOT_MASK) | i);
            }
            sort_desc<BUF>(key);
        }
        if (!again) break;
        if ((tid & 31) == 0 && work) stat_add(a.err, STAT_SELECT_RETRY);
        if (overflow) {
            const uint32_t kb = __float_as_uint(key[L - 1]);
            theta = __uint_as_float(kb >> 31 ? kb | SLOT_MASK : kb & ~SLOT_MASK);
            if (round == 2) exact = true;
        }
    }
    float outv[L];
    int outi[L];
    if (work) {
        // keys that tie across the cut (their scores differ by less than the slot bits): exact order
        // of this thread's survivors by selection in its buffer column (rare)
        const bool tie = cnt > L && ((__float_as_uint(key[L - 1]) ^ __float_as_uint(key[L])) & ~SLOT_MASK) == 0u && !exact;
        if (__any_sync(0xffffffffu, tie)) {
            if (tie) {
                float* bv = const_cast<float*>(buf_v);
                int* bx = const_cast<int*>(buf_i);
                for (int r = 0; r < L; ++r) {
                    int best = r;
                    float bvv = bv[r * 256];
                    for (int p = r + 1; p < cnt; ++p) {
                        const float x = bv[p * 256];
                        if (x > bvv) { bvv = x; best = p; }
                    }
                    const float ov = bv[r * 256];
                    const int oi = bx[r * 256], ob = bx[best * 256];
                    bv[r * 256] = bvv; bx[r * 256] = ob;
                    bv[best * 256] = ov; bx[best * 256] = oi;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < L; ++i) {
            const int slot = tie ? i : static_cast<int>(__float_as_uint(key[i]) & SLOT_MASK);
            outv[i] = i < cnt ? buf_v[slot * 256] : -INFINITY;
            outi[i] = i < cnt ? buf_i[slot * 256] : 0x7fffffff;
        }
        // neighbours closer than the slot bits may stand in the wrong order
        while (true) {
            bool wrong = false;
#pragma unroll
            for (int i = 0; i + 1 < L; ++i) wrong |= outv[i] < outv[i + 1];
            if (!__any_sync(0xffffffffu, wrong)) break;
#pragma unroll
            for (int par = 0; par < 2; ++par)
#pragma unroll
                for (int i = par; i + 1 < L; i += 2) {
                    const bool sw = outv[i] < outv[i + 1];
                    const float x = outv[i];
                    const int ix = outi[i];
                    outv[i] = sw ? outv[i + 1] : x; outi[i] = sw ? outi[i + 1] : ix;
                    outv[i + 1] = sw ? x : outv[i + 1]; outi[i + 1] = sw ? ix : outi[i + 1];
                }
        }
    }
    if (__syncthreads_or(exact)) {
        // heavy ties: exact top-L by insertion over the half (rare, slow).  Every lane of a working
        // warp runs the TMEM loads (they are warp-collective); only flagged lanes insert.
        float lv[L];
        int li[L];
        for (int i = 0; i < L; ++i) { lv[i] = -INFINITY; li[i] = 0x7fffffff; }
        for (int ch = 0; ch < nchunk && need(ch); ++ch) {
            for (int col = 0; col < chunk_cols(ch) && work; ++col) {
                uint32_t xb;
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n" : "=r"(xb) : "r"(trow + col));
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                const float x = __uint_as_float(xb);
                if (exact && x > lv[L - 1]) {
                    int p = L - 1;
                    while (p > 0 && x > lv[p - 1]) { lv[p] = lv[p - 1]; li[p] = li[p - 1]; --p; }
                    lv[p] = x; li[p] = ch * COLS + col;
                }
            }
        }
        if (exact) {
            for (int i = 0; i < L; ++i) { outv[i] = lv[i]; outi[i] = li[i]; }
        }
    }
    if (ok && mine) {   // the token's L entries are contiguous (L % 4 == 0): 16-byte stores
        const int64_t u = static_cast<int64_t>(b) * a.T + t;
        const int64_t lbase = ((static_cast<int64_t>(blockIdx.z) * 2 + hf) * BT + u) * L;
        float4* pv = reinterpret_cast<float4*>(a.part_v + lbase);
        int4* pi = reinterpret_cast<int4*>(a.part_i + lbase);
#pragma unroll
        for (int i = 0; i < L; i += 4) {
            pv[i / 4] = make_float4(outv[i], outv[i + 1], outv[i + 2], outv[i + 3]);
            pi[i / 4] = make_int4(outi[i], outi[i + 1], outi[i + 2], outi[i + 3]);
        }
    }
    if (!ok && tid == 0) flag_error(a.err, ERR_TIMEOUT);
    if (!freed) {                                                 // (block-uniform)
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
        free_tmem();
    }
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
namespace {

// P of one side: dims {dk, 2S, H}; box {64, min(256, 2S), 1}
CUresult encode_p(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap* map, const void* P, int dk, int S, int H) {
    cuuint64_t dim[3] = {static_cast<cuuint64_t>(dk), static_cast<cuuint64_t>(2 * S), static_cast<cuuint64_t>(H)};
    cuuint64_t str[2] = {static_cast<cuuint64_t>(dk) * 2, static_cast<cuuint64_t>(dk) * 2 * 2 * S};
    cuuint32_t box[3] = {64, static_cast<cuuint32_t>(2 * S < MM_NB ? 2 * S : MM_NB), 1};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(P), dim, str, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

}  // namespace

cudaError_t addr_p_maps(CUtensorMap (&maps)[2], const AddrArgs& a) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tc::tensor_map_encode();
    if (!enc) return cudaErrorNotSupported;
    for (int s = 0; s < 2; ++s)
        if (encode_p(enc, &maps[s], a.P[s], a.dk, a.S, a.H) != CUDA_SUCCESS) return cudaErrorInvalidValue;
    return cudaSuccess;
}

bool mma_path_supported(int dtype, int direct, int dk, int S, int kmax) {
    return dtype == 1 && !direct && (dk == 64 || dk == 128) && kmax <= 64 && S >= 16;
}

namespace {

size_t mma_smem(int atoms, int L, bool alias) {
    const size_t ops = static_cast<size_t>(atoms) * 128 * 128 + 2 * MM_UNIT, buf = mm_buf_bytes(L);
    return 1024 + (alias ? (ops > buf ? ops : buf) : ops + buf) + 64;
}

template <int COLS, int L, bool ALIAS>
cudaError_t launch_mma(const MmaLaunch& a, const CUtensorMap (&maps)[4], cudaStream_t stream) {
    const size_t smem = mma_smem(a.atoms, L, ALIAS);
    cudaError_t e = cudaFuncSetAttribute(k_addr_mma<COLS, L, ALIAS>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_ALLOWED);
    // the whole carveout, so that what these CTAs leave of it is there for the M0 copy beside them
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_addr_mma<COLS, L, ALIAS>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    k_addr_mma<COLS, L, ALIAS><<<dim3(static_cast<unsigned>(a.tiles) + 1, 2, 2 * a.H), MM_THREADS, smem, stream>>>(maps[0], maps[1], maps[2], maps[3], a);
    return cudaGetLastError();
}

// 256 TMEM columns hold a whole half up to S = 256 (two tiles at once on an SM), 512 above; halves
// of more than 512 columns go through in chunks.
template <int L>
cudaError_t launch_mma_cols(const MmaLaunch& a, const CUtensorMap (&maps)[4], cudaStream_t stream) {
    if (a.S <= 256) return launch_mma<256, L, true>(a, maps, stream);
    if (a.S <= 512) return launch_mma<512, L, true>(a, maps, stream);
    return launch_mma<512, L, false>(a, maps, stream);
}

}  // namespace

size_t addr_smem_left(const AddrPlan& plan, int dk, int S) {
    if (!plan.mma) return 0;
    const size_t sm = 228 * 1024, cta = mma_smem((dk + 63) / 64, plan.L, S <= 512) + 1024 + 64;    // with the system's and static
    return sm - (sm / cta < 2 ? sm / cta : 2) * cta;
}

cudaError_t launch_address_mma(const AddrPlan& plan, const AddrArgs& aa, cudaStream_t stream) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tc::tensor_map_encode();
    if (!enc) return cudaErrorNotSupported;
    MmaLaunch a{};
    a.B = aa.B; a.H = aa.H; a.T = aa.T; a.dk = aa.dk; a.S = aa.S;
    a.bt = 1;
    while (a.bt * 2 <= aa.T && a.bt < 128) a.bt *= 2;     // largest power of two <= min(T, 128)
    a.bb = 128 / a.bt;
    if (a.bb > aa.B) a.bb = aa.B;                          // boxes never exceed the tensor
    a.ntt = (aa.T + a.bt - 1) / a.bt;
    const int nbt = (aa.B + a.bb - 1) / a.bb;
    a.pb = 2 * aa.S < MM_NB ? 2 * aa.S : MM_NB;
    a.atoms = (aa.dk + 63) / 64;
    a.part_v = aa.part_v;
    a.part_i = aa.part_i;
    a.err = aa.err;
    a.raw = aa.raw;

    CUtensorMap maps[4];
    for (int s = 0; s < 2; ++s) {
        // x: dims {dk, T, H, B}; box {64, bt, 1, bb}
        cuuint64_t gdim[4] = {static_cast<cuuint64_t>(aa.dk), static_cast<cuuint64_t>(aa.T), static_cast<cuuint64_t>(aa.H),
                              static_cast<cuuint64_t>(aa.B)};
        cuuint64_t gstr[3] = {static_cast<cuuint64_t>(aa.dk) * 2, static_cast<cuuint64_t>(aa.dk) * 2 * aa.T,
                              static_cast<cuuint64_t>(aa.dk) * 2 * aa.T * aa.H};
        cuuint32_t box[4] = {64, static_cast<cuuint32_t>(a.bt), 1, static_cast<cuuint32_t>(a.bb)};
        cuuint32_t es[4] = {1, 1, 1, 1};
        CUresult r = enc(&maps[s], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(aa.X[s]), gdim, gstr, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
        r = encode_p(enc, &maps[2 + s], aa.P[s], aa.dk, aa.S, aa.H);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    a.tiles = a.ntt * nbt;
    a.P[0] = aa.P[0];
    a.P[1] = aa.P[1];
    a.pnorm = aa.pnorm;
    a.queue = aa.queue;
    switch (plan.L) {
        case 12: return launch_mma_cols<12>(a, maps, stream);
        case 20: return launch_mma_cols<20>(a, maps, stream);
        case 36: return launch_mma_cols<36>(a, maps, stream);
        case 68: return launch_mma_cols<68>(a, maps, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sdm
