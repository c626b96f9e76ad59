// Device helpers shared by the fp32 CUDA-core chunk kernels.
#pragma once
#include "sla_internal.h"

#include <math.h>

namespace sla {
namespace detail {

constexpr int CMAX = 64;       // largest chunk
constexpr int VS = 16;         // state columns owned by one CTA of the scan kernels
constexpr unsigned FULL = 0xffffffffu;

template <typename T> __device__ __forceinline__ float ldf(const T *p, size_t i);
template <> __device__ __forceinline__ float ldf<float>(const float *p, size_t i) { return p[i]; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16 *p, size_t i) {
    return __bfloat162float(p[i]);
}
template <typename T> __device__ __forceinline__ void stf(T *p, size_t i, float v);
template <> __device__ __forceinline__ void stf<float>(float *p, size_t i, float v) { p[i] = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16 *p, size_t i, float v) {
    p[i] = __float2bfloat16_rn(v);
}

__device__ __forceinline__ size_t tok_row(const Dims &d, int b, int t, int h) {
    return ((size_t)b * d.T + t) * d.H + h;
}
// chunk-local cumulative log-decay of token row `row`, key dimension dd
__device__ __forceinline__ float bcum_at(const Dims &d, const float *bcum, size_t row, int dd) {
    return d.variant == SLA_GLA ? bcum[row * d.dk + dd] : bcum[row];
}
__device__ __forceinline__ size_t state_off(const Dims &d, int bh, int n, int slots) {
    return ((size_t)bh * slots + n) * d.dk * d.dv;
}

// ------------------------------------------------------------------------------------------
// Shared-memory tile product used by the per-tile kernels.  256 threads: ty = warp (0..7),
// tx = lane.  Thread (ty,tx) owns rows ty+8r (r<8) and columns tx+32cb (cb<NB) of a 64 x N tile:
//   acc[r][cb] += sum_k A[(ty+8r)*sa_i + k*sa_k] * Bm[k*sb_k + (tx+32cb)*sb_j]
// A reads are warp-wide broadcasts; Bm reads are conflict-free when the stride that multiplies
// the lane index is odd (all tiles are stored with an odd leading dimension).
// Four k-steps are unrolled so that their shared-memory reads overlap (rolled, each step waited out its own read latency), and
// the column blocks past a 64-wide tile are left out instead of multiplied by zero.
template <int NB, int NE>
__device__ __forceinline__ void tile_gemm_blocks(float (&acc)[8][NB], const float *A, int sa_i, int sa_k, const float *Bm, int sb_k, int sb_j, int K,
                                                 int N, int ty, int tx) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        float a[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) a[r] = A[(ty + 8 * r) * sa_i + k * sa_k];
#pragma unroll
        for (int cb = 0; cb < NE; ++cb) {
            int j = tx + 32 * cb;
            float bv = (j < N) ? Bm[k * sb_k + j * sb_j] : 0.f;
#pragma unroll
            for (int r = 0; r < 8; ++r) acc[r][cb] = fmaf(a[r], bv, acc[r][cb]);
        }
    }
}
template <int NB>
__device__ __forceinline__ void tile_gemm(float (&acc)[8][NB], const float *A, int sa_i, int sa_k,
                                          const float *Bm, int sb_k, int sb_j, int K, int N, int ty,
                                          int tx) {
    if (NB > 2 && N <= 64) tile_gemm_blocks<NB, (NB > 2 ? 2 : NB)>(acc, A, sa_i, sa_k, Bm, sb_k, sb_j, K, N, ty, tx);
    else tile_gemm_blocks<NB, NB>(acc, A, sa_i, sa_k, Bm, sb_k, sb_j, K, N, ty, tx);
}

template <int NB> __device__ __forceinline__ void zero_acc(float (&acc)[8][NB]) {
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int cb = 0; cb < NB; ++cb) acc[r][cb] = 0.f;
}

// four consecutive elements of a row (head widths are multiples of 16, tensors 16-byte aligned)
__device__ __forceinline__ float4 ldf4(const float *p, size_t i) { return *reinterpret_cast<const float4 *>(p + i); }
__device__ __forceinline__ float4 ldf4(const __nv_bfloat16 *p, size_t i) {
    const uint2 u = *reinterpret_cast<const uint2 *>(p + i);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 bcum_at4(const Dims &d, const float *bcum, size_t row, int dd) {
    if (d.variant == SLA_GLA) return ldf4(bcum, row * d.dk + dd);
    const float v = bcum[row];
    return make_float4(v, v, v, v);
}
__device__ __forceinline__ void put4(float *dst, float4 v) { dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w; }

// Fill shared memory from global memory: for every index of 0 .. total-1 store(idx, load(idx)), the loads of U indices of
// a thread in flight together; an index stands for four elements of a row.  (A plain loop over single elements keeps one read
// in flight, as the compiler does not move a global read above a shared-memory write: a tile of 16 elements a thread then
// cost 16 memory latencies.)
template <int U = 4, class Load, class Store>
__device__ __forceinline__ void fill(int total, Load load, Store store) {
    using V = decltype(load(0));
    for (int base = threadIdx.x; base < total; base += U * blockDim.x) {
        V v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * blockDim.x;
            if (idx < total) v[u] = load(idx);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * blockDim.x;
            if (idx < total) store(idx, v[u]);
        }
    }
}
// rows 0 .. rows-1 of a tile into shared memory (leading dimension ld), row i from src + row(i); rows from cn on are zero
template <typename T, class Row>
__device__ __forceinline__ void fill_rows(float *dst, int ld, const T *src, int rows, int cn, int width, Row row) {
    const int w4 = width >> 2;
    fill(rows * w4,
         [&](int idx) { const int i = idx / w4; return i < cn ? ldf4(src, row(i) + 4 * (idx - i * w4)) : make_float4(0.f, 0.f, 0.f, 0.f); },
         [&](int idx, float4 v) { const int i = idx / w4; put4(dst + i * ld + 4 * (idx - i * w4), v); });
}

// Load the decayed, gated operands of one chunk into shared memory (rows >= cn zero-filled).
//   Qs[i][dd] = scale*Gq_i*q*exp(b)   Ks[i][dd] = gk_i*k*exp(-b)   (gk_i = Gk_i, or 1 for GDN)
template <typename TIO>
__device__ __forceinline__ void load_qk_hat(const Dims &d, const TIO *q, const TIO *k,
                                            const float *Gq, const float *Gk, const float *bcum, int b,
                                            int h, int t0, int cn, float *Qs, float *Ks, int ld) {
    struct In { float4 q, k, b; float gq, gk; };
    const int w4 = d.dk >> 2;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    fill<2>(CMAX * w4,
        [&](int idx) {
            const int i = idx / w4, dd = 4 * (idx - i * w4);
            In x{zero, zero, zero, 0.f, 0.f};
            if (i < cn) {
                const size_t row = tok_row(d, b, t0 + i, h);
                x.b = bcum_at4(d, bcum, row, dd);
                x.gk = d.variant == SLA_GDN ? 1.f : Gk[row];
                x.gq = Gq[row];
                x.q = ldf4(q, row * d.dk + dd);
                x.k = ldf4(k, row * d.dk + dd);
            }
            return x;
        },
        [&](int idx, const In &x) {
            const int i = idx / w4, o = i * ld + 4 * (idx - i * w4);
            const float gq = d.scale * x.gq;
            put4(Qs + o, i < cn ? make_float4(gq * x.q.x * expf(x.b.x), gq * x.q.y * expf(x.b.y), gq * x.q.z * expf(x.b.z), gq * x.q.w * expf(x.b.w)) : zero);
            put4(Ks + o, i < cn ? make_float4(x.gk * x.k.x * expf(-x.b.x), x.gk * x.k.y * expf(-x.b.y), x.gk * x.k.z * expf(-x.b.z), x.gk * x.k.w * expf(-x.b.w)) : zero);
        });
}


template <typename F> inline bool set_smem(F *fn, size_t bytes) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

}  // namespace detail
}  // namespace sla
