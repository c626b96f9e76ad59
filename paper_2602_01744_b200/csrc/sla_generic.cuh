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

// ------------------------------------------------------------------------------------------
// The same products from 4 x 4 register tiles and 16-byte shared-memory reads, for the Softmax-RetNet / -GLA kernels: 8 reads for 64
// multiply-adds where tile_gemm issues 40, whole 16-byte pieces into shared memory and out to global memory.  Both are bound by
// the shared-memory pipe (a 16-byte read takes it four cycles: 4,100 for a 64 x 64 x 64 product, 5,100 for tile_gemm).  2 x 1000 tokens x 4 heads of
// 64: k_grads_lin 63 -> 41 us, k_output 18 -> 16.  256 threads: thread (tr, tc)
// owns rows tr + 16 a and columns 64 blk + 4 tc + b (a, b < 4) of a 64 x N tile, acc[a][4 blk + b].  Operands are stored with
// leading dimensions pad4(width): 16-byte rows, and eight neighbouring rows start in different groups of four banks.
__host__ __device__ constexpr int pad4(int width) { return width + 4; }
struct Tile {
    int tr, tc;
    __device__ __forceinline__ explicit Tile(int tid = threadIdx.x) {
        const int w = tid >> 5, lane = tid & 31;
        tr = (lane >> 2) + 8 * (w & 1);
        tc = (lane & 3) + 4 * (w >> 1);
    }
    __device__ __forceinline__ int row(int a) const { return tr + 16 * a; }
    __device__ __forceinline__ int col(int blk) const { return 64 * blk + 4 * tc; }
};
// acc += A[i][k] B: A has its rows along k.  BT: B[k][j], else B[j][k].  K a multiple of four (rows past the last token are zero).
// Only the row groups a = A0 .. A1 - 1 (rows 16 A0 .. 16 A1 - 1) where A is triangular, see mm_lower, mm_upper.
template <int NB, bool BT, int A0 = 0, int A1 = 4>
__device__ __forceinline__ void mm(float (&acc)[4][4 * NB], const Tile &t, const float *A, int lda, const float *B, int ldb, int K, int N) {
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float4 a[4];
#pragma unroll
        for (int x = A0; x < A1; ++x) a[x] = *reinterpret_cast<const float4 *>(A + t.row(x) * lda + k);
#pragma unroll
        for (int blk = 0; blk < NB; ++blk) {
            if (t.col(blk) >= N) continue;
            float4 b[4];
#pragma unroll
            for (int y = 0; y < 4; ++y)
                b[y] = *reinterpret_cast<const float4 *>(BT ? B + (k + y) * ldb + t.col(blk) : B + (t.col(blk) + y) * ldb + k);
#pragma unroll
            for (int x = A0; x < A1; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    float &c = acc[x][4 * blk + y];
                    if (BT) {
                        const float *b0 = reinterpret_cast<const float *>(&b[0]), *b1 = reinterpret_cast<const float *>(&b[1]),
                                    *b2 = reinterpret_cast<const float *>(&b[2]), *b3 = reinterpret_cast<const float *>(&b[3]);
                        c = fmaf(a[x].x, b0[y], c); c = fmaf(a[x].y, b1[y], c); c = fmaf(a[x].z, b2[y], c); c = fmaf(a[x].w, b3[y], c);
                    } else {
                        c = fmaf(a[x].x, b[y].x, c); c = fmaf(a[x].y, b[y].y, c); c = fmaf(a[x].z, b[y].z, c); c = fmaf(a[x].w, b[y].w, c);
                    }
                }
        }
    }
}
// acc += A B with A lower (upper) triangular [64][64], K of its columns and of B's rows: the 16 x 16 blocks of zeros are left out.
template <int S = 0>
__device__ __forceinline__ void mm_lower(float (&acc)[4][4], const Tile &t, const float *A, int lda, const float *B, int ldb, int K, int N) {
    if (K <= 16 * S) return;
    mm<1, true, S, 4>(acc, t, A + 16 * S, lda, B + 16 * S * ldb, ldb, min(K - 16 * S, 16), N);
    if constexpr (S < 3) mm_lower<S + 1>(acc, t, A, lda, B, ldb, K, N);
}
template <int S = 0>
__device__ __forceinline__ void mm_upper(float (&acc)[4][4], const Tile &t, const float *A, int lda, const float *B, int ldb, int K, int N) {
    if (K <= 16 * S) return;
    mm<1, true, 0, S + 1>(acc, t, A + 16 * S, lda, B + 16 * S * ldb, ldb, min(K - 16 * S, 16), N);
    if constexpr (S < 3) mm_upper<S + 1>(acc, t, A, lda, B, ldb, K, N);
}
// acc = tril(X Y^T), 64 x 64: a warp's 16 columns meet the row groups from its own on
__device__ __forceinline__ void mm_tril(float (&acc)[4][4], const Tile &t, const float *X, int ldx, const float *Y, int ldy, int K) {
    switch (t.tc >> 2) {
        case 0: mm<1, false, 0>(acc, t, X, ldx, Y, ldy, K, CMAX); break;
        case 1: mm<1, false, 1>(acc, t, X, ldx, Y, ldy, K, CMAX); break;
        case 2: mm<1, false, 2>(acc, t, X, ldx, Y, ldy, K, CMAX); break;
        default: mm<1, false, 3>(acc, t, X, ldx, Y, ldy, K, CMAX);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (t.col(0) + c > t.row(a)) acc[a][c] = 0.f;
}
// acc += X^T Y over the tokens: X[k][i], Y[k][j]; thread (tr, tc) owns rows 4 tr + a instead.
template <int NB>
__device__ __forceinline__ void mm_outer(float (&acc)[4][4 * NB], const Tile &t, const float *X, int ldx, const float *Y, int ldy, int K, int M, int N) {
    if (4 * t.tr >= M) return;
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float4 x4 = *reinterpret_cast<const float4 *>(X + k * ldx + 4 * t.tr);
        const float x[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
        for (int blk = 0; blk < NB; ++blk) {
            if (t.col(blk) >= N) continue;
            const float4 y4 = *reinterpret_cast<const float4 *>(Y + k * ldy + t.col(blk));
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                acc[a][4 * blk] = fmaf(x[a], y4.x, acc[a][4 * blk]);         acc[a][4 * blk + 1] = fmaf(x[a], y4.y, acc[a][4 * blk + 1]);
                acc[a][4 * blk + 2] = fmaf(x[a], y4.z, acc[a][4 * blk + 2]); acc[a][4 * blk + 3] = fmaf(x[a], y4.w, acc[a][4 * blk + 3]);
            }
        }
    }
}
template <int NC> __device__ __forceinline__ void zero_acc(float (&acc)[4][NC]) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[a][c] = 0.f;
}
// four neighbouring results of a tile in the I/O dtype
__device__ __forceinline__ void stf4(float *p, size_t i, float4 v) { *reinterpret_cast<float4 *>(p + i) = v; }
__device__ __forceinline__ void stf4(__nv_bfloat16 *p, size_t i, float4 v) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2 *>(p + i) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
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

// The same for tiles with 16-byte rows (ld a multiple of four), without waiting: fp32 rows travel by asynchronous copies, so that the
// tiles a kernel starts from are all on their way together; copies_wait() (and a barrier) before they are read.  bf16 rows are widened on
// the way and take fill_rows.  (A training step of 2 x 1000 tokens x 4 heads of 64, every tile waited for by itself: 93 us, 88 so.)
__device__ __forceinline__ void copy_rows(float *dst, int ld, const float *src, int rows, int cn, int width, size_t row0, size_t stride) {
    const int w4 = width >> 2;
    for (int idx = threadIdx.x; idx < rows * w4; idx += blockDim.x) {
        const int i = idx / w4, c = 4 * (idx - i * w4);
        float *d = dst + i * ld + c;
        if (i < cn)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(d)), "l"(src + row0 + i * stride + c) : "memory");
        else
            *reinterpret_cast<float4 *>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
__device__ __forceinline__ void copy_rows(float *dst, int ld, const __nv_bfloat16 *src, int rows, int cn, int width, size_t row0, size_t stride) {
    fill_rows(dst, ld, src, rows, cn, width, [&](int i) { return row0 + i * stride; });
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Load the decayed, gated operands of one chunk into shared memory (rows >= cn zero-filled).
//   Qs[i][dd] = scale*Gq_i*q*exp(b)   Ks[i][dd] = gk_i*k*exp(-b)   (gk_i = Gk_i, or 1 for GDN)
// U: reads in flight together (see fill)
template <int U = 2, typename TIO>
__device__ __forceinline__ void load_qk_hat(const Dims &d, const TIO *q, const TIO *k,
                                            const float *Gq, const float *Gk, const float *bcum, int b,
                                            int h, int t0, int cn, float *Qs, float *Ks, int ld) {
    struct In { float4 q, k, b; float gq, gk; };
    const int w4 = d.dk >> 2;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    fill<U>(CMAX * w4,
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
