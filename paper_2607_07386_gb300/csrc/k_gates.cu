// The steps on either side of the SDM path in a layer (Sec. 3.1):
//
//   k_gates      per-head gates of every token from the layer input x_t (after Eq. sdm-write):
//                  alpha_t = exp(-A softplus(W_a x_t + b_dt)),  beta_t = sigmoid(W_b x_t)
//                One warp per token: lanes split x_t into 16-byte vectors, every lane
//                accumulates all 2H dot products against W_a and W_b (staged in shared memory
//                when they fit), warp reductions finish them, and lane j writes gate j.  x is
//                read once: 2H * d FMAs per token, B*T*d*elem bytes of HBM.
//   k_norm_gate  z = g (.) RMSNorm(y) per head ("Norm, Gating, and Head Mixing"), with the
//                RMSNorm scale gamma: z = g * gamma * y / sqrt(mean(y^2) + eps).  z is written
//                token-major [B, T, H, d_v], the layout in which the head-mixing projection W_o
//                is one plain GEMM.  HBM-bound: y and g read once, z written once.
#include "sdm_internal.h"

namespace sdm {

constexpr int GT_THREADS = 256;        // k_norm_gate
constexpr int GG_THREADS = 512;        // k_gates: 16 warps share one copy of W_a, W_b per SM
constexpr size_t GT_SMEM_MAX = 200 * 1024;

template <class D> __device__ __forceinline__ void store_elem(void* base, int64_t i, float v);
template <> __device__ __forceinline__ void store_elem<F32>(void* base, int64_t i, float v) {
    reinterpret_cast<float*>(base)[i] = v;
}
template <> __device__ __forceinline__ void store_elem<BF16>(void* base, int64_t i, float v) {
    reinterpret_cast<__nv_bfloat16*>(base)[i] = __float2bfloat16_rn(v);
}

// NH >= 2H accumulators per lane.
template <class D, int NH>
__global__ void __launch_bounds__(GG_THREADS) k_gates(const void* __restrict__ x, const void* __restrict__ W_a,
                                                      const void* __restrict__ W_b, const float* __restrict__ b_dt,
                                                      const float* __restrict__ A, void* __restrict__ alpha,
                                                      void* __restrict__ beta, int64_t tokens, int T, int H, int d,
                                                      int use_smem) {
    extern __shared__ __align__(16) unsigned char smG[];
    const int nq = d * D::BYTES / 16;                       // 16-byte vectors per row
    const int rows = 2 * H;
    const uint4* Wg_a = static_cast<const uint4*>(W_a);
    const uint4* Wg_b = static_cast<const uint4*>(W_b);
    uint4* Ws = reinterpret_cast<uint4*>(smG);              // [2H][nq]: W_a rows, then W_b rows
    if (use_smem) {
        for (int i = threadIdx.x; i < rows * nq; i += GG_THREADS) {
            const int r = i / nq, q = i - r * nq;
            Ws[i] = r < H ? __ldg(Wg_a + static_cast<int64_t>(r) * nq + q) : __ldg(Wg_b + static_cast<int64_t>(r - H) * nq + q);
        }
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int64_t wstride = static_cast<int64_t>(gridDim.x) * (GG_THREADS / 32);
    for (int64_t u = static_cast<int64_t>(blockIdx.x) * (GG_THREADS / 32) + (threadIdx.x >> 5); u < tokens; u += wstride) {
        const uint4* xr = static_cast<const uint4*>(x) + u * nq;
        float acc[NH];
#pragma unroll
        for (int r = 0; r < NH; ++r) acc[r] = 0.f;
        for (int q = lane; q < nq; q += 32) {
            float fx[D::E];
            unpack16<D>(__ldg(xr + q), fx);
#pragma unroll
            for (int r = 0; r < NH; ++r) {
                if (r < rows) {
                    const uint4 wv = use_smem ? Ws[r * nq + q]
                                              : (r < H ? __ldg(Wg_a + static_cast<int64_t>(r) * nq + q)
                                                       : __ldg(Wg_b + static_cast<int64_t>(r - H) * nq + q));
                    float fw[D::E];
                    unpack16<D>(wv, fw);
#pragma unroll
                    for (int e = 0; e < D::E; ++e) acc[r] = fmaf(fw[e], fx[e], acc[r]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < NH; ++r) {
            if (r < rows) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off);
            }
        }
        const int64_t b = u / T, t = u - b * T;
        for (int j = lane; j < rows; j += 32) {
            float z = 0.f;
#pragma unroll
            for (int r = 0; r < NH; ++r) z = (r == j) ? acc[r] : z;
            if (j < H) {
                const float za = z + __ldg(b_dt + j);
                const float sp = za > 20.f ? za : log1pf(expf(za));     // softplus
                store_elem<D>(alpha, (b * H + j) * T + t, expf(-__ldg(A + j) * sp));
            } else {
                store_elem<D>(beta, (b * H + (j - H)) * T + t, 1.f / (1.f + expf(-z)));
            }
        }
    }
}

// Division of row numbers below 2^31 by a fixed divisor: (n + mulhi(n, m)) >> s.
struct RowDiv {
    uint32_t m, s;
};
static RowDiv row_div(uint32_t d) {
    uint32_t s = 0;
    while (s < 31 && (1u << s) < d) ++s;
    return RowDiv{static_cast<uint32_t>((((1ull << s) - d) << 32) / d + 1), s};
}

// CPL: 16-byte vectors per lane.  A row is spread over LPR neighbouring lanes (a power of two at
// least its vectors, at most 32), so a warp covers 32 / LPR rows at once and every thread keeps NG_ROWS of
// them, y and g, in flight.  Bound by HBM: 64 us for 524,288 rows of 128 bf16 (6.3 TB/s); 107 us with
// 8-byte vectors, one row in flight per warp and two 64-bit divisions per row.
template <class D, int CPL>
__global__ void __launch_bounds__(GT_THREADS) k_norm_gate(const uint4* __restrict__ y, const uint4* __restrict__ g,
                                                          const float* __restrict__ gamma, float eps, uint4* __restrict__ z,
                                                          int64_t rows, int H, int T, int dv, int lpr_log2, RowDiv by_t,
                                                          RowDiv by_h) {
    constexpr int E = D::E;
    constexpr int NG_ROWS = CPL == 1 ? 4 : 2;
    const int lpr = 1 << lpr_log2, l = threadIdx.x & (lpr - 1);
    const int nv = dv / E;                                  // vectors per row
    const int pass = GT_THREADS >> lpr_log2;                // rows a CTA loads at once
    const int64_t u0 = static_cast<int64_t>(blockIdx.x) * pass * NG_ROWS + (threadIdx.x >> lpr_log2);
    float gm[CPL][E];
#pragma unroll
    for (int c = 0; c < CPL; ++c)
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int v = l + c * lpr;
            gm[c][e] = v < nv ? __ldg(gamma + v * E + e) : 0.f;
        }
    uint4 yr[NG_ROWS][CPL], gr[NG_ROWS][CPL];
#pragma unroll
    for (int q = 0; q < NG_ROWS; ++q) {
        const int64_t u = u0 + q * pass, at = u * nv + l;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const bool in = u < rows && l + c * lpr < nv;
            yr[q][c] = in ? __ldcs(y + at + c * lpr) : make_uint4(0u, 0u, 0u, 0u);
            gr[q][c] = in ? __ldcs(g + at + c * lpr) : make_uint4(0u, 0u, 0u, 0u);
        }
    }
#pragma unroll
    for (int q = 0; q < NG_ROWS; ++q) {
        const int64_t u = u0 + q * pass;
        float ss = 0.f;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            float f[E];
            unpack16<D>(yr[q][c], f);
#pragma unroll
            for (int e = 0; e < E; ++e) ss = fmaf(f[e], f[e], ss);
        }
        for (int off = lpr >> 1; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
        const float inv = 1.f / sqrtf(ss / static_cast<float>(dv) + eps);
        // row u = (b * H + h) * T + t  ->  z row (b * T + t) * H + h
        int64_t bh, b;
        if (rows < (1ll << 31)) {
            const uint32_t n = static_cast<uint32_t>(u);
            const uint32_t q1 = (n + __umulhi(n, by_t.m)) >> by_t.s;
            bh = q1;
            b = (q1 + __umulhi(q1, by_h.m)) >> by_h.s;
        } else {
            bh = u / T;
            b = bh / H;
        }
        uint4* zr = z + ((b * T + (u - bh * T)) * H + (bh - b * H)) * nv + l;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            if (u < rows && l + c * lpr < nv) {
                float f[E], w[E], o[E];
                unpack16<D>(yr[q][c], f);
                unpack16<D>(gr[q][c], w);
#pragma unroll
                for (int e = 0; e < E; ++e) o[e] = w[e] * gm[c][e] * (f[e] * inv);
                zr[c * lpr] = pack16<D>(o);
            }
        }
    }
}

namespace {
unsigned persistent_grid(int64_t warps_wanted, int threads = GT_THREADS) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t grid = (warps_wanted + threads / 32 - 1) / (threads / 32);
    const int64_t cap = static_cast<int64_t>(sms > 0 ? sms : 1) * (2048 / threads);   // a full SM of threads
    return static_cast<unsigned>(grid < 1 ? 1 : (grid < cap ? grid : cap));
}

template <class D, int NH>
cudaError_t gates_nh(const void* x, const void* W_a, const void* W_b, const float* b_dt, const float* A, void* alpha,
                     void* beta, int B, int T, int H, int d, cudaStream_t s) {
    const size_t wbytes = static_cast<size_t>(2) * H * d * D::BYTES;
    const int use_smem = wbytes <= GT_SMEM_MAX;
    const size_t smem = use_smem ? wbytes : 0;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_gates<D, NH>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_ALLOWED);
        if (e != cudaSuccess) return e;
    }
    const int64_t tokens = static_cast<int64_t>(B) * T;
    k_gates<D, NH><<<persistent_grid(tokens, GG_THREADS), GG_THREADS, smem, s>>>(x, W_a, W_b, b_dt, A, alpha, beta, tokens, T, H, d,
                                                                    use_smem);
    return cudaGetLastError();
}

template <class D>
cudaError_t gates_dtype(const void* x, const void* W_a, const void* W_b, const float* b_dt, const float* A, void* alpha,
                        void* beta, int B, int T, int H, int d, cudaStream_t s) {
    const int rows = 2 * H;
    if (rows <= 2) return gates_nh<D, 2>(x, W_a, W_b, b_dt, A, alpha, beta, B, T, H, d, s);
    if (rows <= 8) return gates_nh<D, 8>(x, W_a, W_b, b_dt, A, alpha, beta, B, T, H, d, s);
    if (rows <= 16) return gates_nh<D, 16>(x, W_a, W_b, b_dt, A, alpha, beta, B, T, H, d, s);
    if (rows <= 32) return gates_nh<D, 32>(x, W_a, W_b, b_dt, A, alpha, beta, B, T, H, d, s);
    return gates_nh<D, 64>(x, W_a, W_b, b_dt, A, alpha, beta, B, T, H, d, s);
}

template <class D, int CPL>
cudaError_t norm_gate_cpl(const void* y, const void* g, const float* gamma, float eps, void* z, int B, int H, int T, int dv,
                          int lpr_log2, cudaStream_t s) {
    const int64_t rows = static_cast<int64_t>(B) * H * T;
    const int64_t per_cta = (GT_THREADS >> lpr_log2) * (CPL == 1 ? 4 : 2);
    const int64_t ctas = (rows + per_cta - 1) / per_cta;
    if (ctas > INT32_MAX) return cudaErrorInvalidConfiguration;
    k_norm_gate<D, CPL><<<static_cast<unsigned>(ctas), GT_THREADS, 0, s>>>(
        static_cast<const uint4*>(y), static_cast<const uint4*>(g), gamma, eps, static_cast<uint4*>(z), rows, H, T, dv,
        lpr_log2, row_div(static_cast<uint32_t>(T)), row_div(static_cast<uint32_t>(H)));
    return cudaGetLastError();
}

template <class D>
cudaError_t norm_gate_dtype(const void* y, const void* g, const float* gamma, float eps, void* z, int B, int H, int T,
                            int dv, cudaStream_t s) {
    const int nv = dv / D::E;                                            // vectors per row, 1 .. 64
    int lg = 0;
    while (lg < 5 && (1 << lg) < nv) ++lg;
    return nv <= 32 ? norm_gate_cpl<D, 1>(y, g, gamma, eps, z, B, H, T, dv, lg, s)
                    : norm_gate_cpl<D, 2>(y, g, gamma, eps, z, B, H, T, dv, lg, s);
}
}  // namespace

cudaError_t launch_gates(int dtype, const void* x, const void* W_a, const void* W_b, const float* b_dt, const float* A,
                         void* alpha, void* beta, int B, int T, int H, int d, cudaStream_t stream) {
    return dtype == 0 ? gates_dtype<F32>(x, W_a, W_b, b_dt, A, alpha, beta, B, T, H, d, stream)
                      : gates_dtype<BF16>(x, W_a, W_b, b_dt, A, alpha, beta, B, T, H, d, stream);
}

cudaError_t launch_norm_gate(int dtype, const void* y, const void* g, const float* gamma, float eps, void* z, int B, int H,
                             int T, int dv, cudaStream_t stream) {
    return dtype == 0 ? norm_gate_dtype<F32>(y, g, gamma, eps, z, B, H, T, dv, stream)
                      : norm_gate_dtype<BF16>(y, g, gamma, eps, z, B, H, T, dv, stream);
}

}  // namespace sdm
