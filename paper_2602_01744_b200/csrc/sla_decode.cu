// Recurrent decode (Eq. 5-6 with the instantiations of Eq. 10-16 at single tokens) as a streaming kernel.
//
// A decode step moves the whole fp32 state once in and once out and does two FLOP per byte: it is HBM-bound, so the
// kernel is built like a copy.  One work item is CW columns of the [d_k x d_v] state of one (sequence, head) (columns of a
// state do not meet in a step, with or without the delta rule).  Persistent CTAs walk their items with a ring of three
// shared-memory stages and three roles.  One token a call: CW = 64, two CTAs per SM, whose loads and stores cover one
// another's barriers and whose smaller items fill the last wave (64 streams of 16 heads 25.5 -> 24.6 us, one stream 5.1 -> 4.4).
// Several tokens a call: CW = 128, one CTA per SM, two operand warps - then preparing the operands, which does not shrink
// with the slice, sets the pace (16 streams x 8 tokens of the delta rule: 22.6 us; 30.7 with one operand warp, 34.8 in slices
// of 64).  Both add up the rows of a state in the
// same order - even and odd rows of a warp apart, then the warps - so that n tokens in one call give the bits of n calls.
//   TMA lane          tile loads up to three items ahead of the arithmetic; the updated state leaves through a TMA
//                     store from the same stage, and the stage takes the next load as soon as the store has read it
//   operand warps     per token: the H gate logits -> head-softmax gates (Eq. 4), decay factors exp(g), and the
//                     operand vectors scale*Gq*q, Gk*k (or k), v (or Gk*v) as fp32 in a ring of blocks, a step ahead
//                     each; the raw operands arrive by asynchronous 4-byte copies requested three or four tokens ahead
//   arithmetic warps  the state in registers (warp w owns row pairs w, w+NW, ..; a lane four columns of one row
//                     of the pair, or of both): decay, the delta
//                     rule's k S (GDN), the rank-1 write, the read-out o = q S
// so loads, arithmetic and stores of neighbouring items overlap all the time.
// n_tok consecutive tokens of a sequence are applied while its state sits in registers (multi-token decode).
#include "sla_gla_tc.cuh"

namespace sla {
namespace {

using namespace ptx;

namespace dc {
constexpr int STAGES = 3;                // states in flight per CTA
constexpr int NW = 8;                    // arithmetic warps
constexpr int NCONS = NW * 32;
constexpr int W_TMA = NW, W_OPS = NW + 1;
constexpr int DMAX = 128;
// operand block (floats): q'[128] k'[128] a[128] beta, u[CW] last
constexpr int OP_Q = 0, OP_K = DMAX, OP_A = 2 * DMAX, OP_BETA = 3 * DMAX, OP_U = 3 * DMAX + 4;
// raw operand block (byte offsets): q, k (I/O dtype, up to 512 B each), log-decay vector (GLA), the two logit rows, beta and the
// scalar log-decay (RETNET, GDN), and last the item's columns of v
constexpr uint32_t RAW_Q = 0, RAW_K = 512, RAW_G = 1024, RAW_LQ = 1536, RAW_LK = 1664, RAW_BETA = 1792, RAW_V = 1808;
template <int CW> struct Lay {
    static constexpr int RP = DMAX / CW;                     // state rows a warp takes at a time
    static constexpr int RPT = DMAX / (RP * NW);             // ... and how many times
    static constexpr int LPR = 32 / RP;                      // lanes per row
    static constexpr uint32_t TILE = DMAX * CW * 4;          // 64 or 32 KiB
    // operand warps: warp x takes the steps n with n % NOPS == x, cooked NOPS steps ahead into one of NOPS + 1 blocks; raw
    // operands are requested AHEAD of the warp's own steps before they are cooked
    static constexpr int NOPS = CW == DMAX ? 2 : 1, AHEAD = CW == DMAX ? 2 : 3, RAWBLOCKS = AHEAD + 1, OPBLOCKS = NOPS + 1;
    static constexpr int NTHREADS = NCONS + 32 + 32 * NOPS;
    static constexpr int OP_FLOATS = OP_U + CW;
    static constexpr uint32_t RAW_BYTES = RAW_V + CW * 4;
    static constexpr uint32_t OFF_OP = STAGES * TILE;                        // [OPBLOCKS] operand blocks
    static constexpr uint32_t OFF_RAW = OFF_OP + OPBLOCKS * OP_FLOATS * 4;   // [NOPS][RAWBLOCKS] raw operand blocks
    static constexpr uint32_t OFF_RED = OFF_RAW + NOPS * RAWBLOCKS * RAW_BYTES;     // [2][NW][LPR] float4 partial sums
    static constexpr uint32_t OFF_BAR = OFF_RED + 2 * NW * LPR * 16;         // STAGES "full" + STAGES "ready to store" barriers
    static constexpr uint32_t SMEM = OFF_BAR + 2 * STAGES * 8 + 16 + 128;    // + abort flag, + slack to align the base to 128 B
    static constexpr int CTAS = DMAX / CW;                   // per SM
    static_assert(CTAS * (SMEM + 1024) <= 233472, "shared memory budget");
};
}  // namespace dc

// four consecutive outputs (16-byte aligned position)
template <typename T> __device__ __forceinline__ void st_io4(T *p, size_t i, float4 v);
template <> __device__ __forceinline__ void st_io4<float>(float *p, size_t i, float4 v) {
    *reinterpret_cast<float4 *>(p + i) = v;
}
template <> __device__ __forceinline__ void st_io4<__nv_bfloat16>(__nv_bfloat16 *p, size_t i, float4 v) {
    *reinterpret_cast<uint2 *>(p + i) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
}

// (states move by 2-D tiled TMA: coordinates are column, row of the [Bdec*H*d_k, d_v] view)
struct DecParams {
    const void *q, *k, *v;
    const float *log_decay, *beta, *lq, *lk;
    void *o;
    int *status;
    int variant, H, dk, dv, n_tok;
    int n_items, nsl;                           // Bdec * H * nsl items, nsl = slices of dc::CW columns per state
    float scale;
};

// ---- raw per-token operands: asynchronous 4-byte copies global -> shared by the operand warp, several tokens ahead ----
__device__ __forceinline__ void cp_async4(void *dst_smem, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
template <typename TIO> __device__ __forceinline__ float io_at(const uint8_t *blk, int i) {
    if (sizeof(TIO) == 4) return reinterpret_cast<const float *>(blk)[i];
    return __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(blk)[i]);
}
// The operand warp's copies of the operands of token row `tok` = b*n_tok + t, head h into raw block `blk` (bytes in the
// I/O dtype for q, k, v; fp32 for decay, beta, logits); of v the columns from c0 on.
template <typename TIO, int CW>
__device__ __forceinline__ void issue_raw(const DecParams &p, uint8_t *blk, size_t tok, int h, int c0, int lane) {
    const size_t th = tok * p.H + h;
    const int nq = p.dk * (int)sizeof(TIO) / 4, nv = min(CW, p.dv - c0) * (int)sizeof(TIO) / 4;     // 4-byte words of a q / k row, of v
    for (int i = lane; i < nq; i += 32) {
        cp_async4(blk + dc::RAW_Q + 4 * i, (const uint8_t *)p.q + (th * p.dk) * sizeof(TIO) + 4 * i);
        cp_async4(blk + dc::RAW_K + 4 * i, (const uint8_t *)p.k + (th * p.dk) * sizeof(TIO) + 4 * i);
    }
    for (int i = lane; i < nv; i += 32)
        cp_async4(blk + dc::RAW_V + 4 * i, (const uint8_t *)p.v + (th * p.dv + c0) * sizeof(TIO) + 4 * i);
    if (p.variant == SLA_GLA)
        for (int i = lane; i < p.dk; i += 32) cp_async4(blk + dc::RAW_G + 4 * i, p.log_decay + th * p.dk + i);
    if (lane < p.H) {
        cp_async4(blk + dc::RAW_LQ + 4 * lane, p.lq + tok * p.H + lane);
        cp_async4(blk + dc::RAW_LK + 4 * lane, p.lk + tok * p.H + lane);
    }
    if (lane == 0) {
        if (p.variant == SLA_GDN) {
            cp_async4(blk + dc::RAW_BETA, p.beta + th);
            cp_async4(blk + dc::RAW_BETA + 4, p.log_decay + th);
        } else if (p.variant == SLA_RETNET) {
            cp_async4(blk + dc::RAW_BETA + 4, p.log_decay + h);
        }
    }
}
// Gates (Eq. 4) and the operand vectors the arithmetic warps use, from raw block `raw` into operand block `op`.
template <typename TIO, int CW>
__device__ __forceinline__ void cook_ops(const DecParams &p, const uint8_t *raw, float *op, int h, int c0, int lane) {
    const float *rf = reinterpret_cast<const float *>(raw);
    const float xq = lane < p.H ? rf[dc::RAW_LQ / 4 + lane] : -INFINITY, xk = lane < p.H ? rf[dc::RAW_LK / 4 + lane] : -INFINITY;
    float mq = xq, mk = xk;
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) {
        mq = fmaxf(mq, __shfl_xor_sync(0xffffffffu, mq, o2));
        mk = fmaxf(mk, __shfl_xor_sync(0xffffffffu, mk, o2));
    }
    const float eq = expf(xq - mq), ek = expf(xk - mk);          // exp(-inf) = 0 on the padding lanes
    float sq = eq, sk = ek;
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) {
        sq += __shfl_xor_sync(0xffffffffu, sq, o2);
        sk += __shfl_xor_sync(0xffffffffu, sk, o2);
    }
    const float Gq = __shfl_sync(0xffffffffu, eq, h) / sq, Gk = __shfl_sync(0xffffffffu, ek, h) / sk;
    const bool gdn = p.variant == SLA_GDN;
    const float fq = p.scale * Gq, fk = gdn ? 1.f : Gk, fv = gdn ? Gk : 1.f;
    const float a_scalar = p.variant == SLA_GLA ? 0.f : expf(rf[dc::RAW_BETA / 4 + 1]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int i = lane + 32 * e;
        // (all entries are written: the arithmetic warps read rows and columns past d_k, d_v as zeros)
        const bool rk = i < p.dk;
        op[dc::OP_Q + i] = rk ? fq * io_at<TIO>(raw + dc::RAW_Q, i) : 0.f;
        op[dc::OP_K + i] = rk ? fk * io_at<TIO>(raw + dc::RAW_K, i) : 0.f;
        op[dc::OP_A + i] = rk ? (p.variant == SLA_GLA ? expf(rf[dc::RAW_G / 4 + i]) : a_scalar) : 0.f;
        if (e < CW / 32) op[dc::OP_U + i] = c0 + i < p.dv ? fv * io_at<TIO>(raw + dc::RAW_V, i) : 0.f;
    }
    if (lane == 0) op[dc::OP_BETA] = gdn ? rf[dc::RAW_BETA / 4] : 0.f;
}

template <typename TIO, int CW>
__global__ void __launch_bounds__(dc::Lay<CW>::NTHREADS, dc::Lay<CW>::CTAS)
k_decode_stream(const __grid_constant__ CUtensorMap tm_s, DecParams p) {
    using namespace dc;
    using L = Lay<CW>;
    constexpr int RPT = L::RPT, RP = L::RP, LPR = L::LPR;
    constexpr uint32_t TILE_BYTES = L::TILE, OFF_OP = L::OFF_OP, OFF_RAW = L::OFF_RAW, OFF_RED = L::OFF_RED, OFF_BAR = L::OFF_BAR,
                       RAW_BYTES = L::RAW_BYTES;
    constexpr int OP_FLOATS = L::OP_FLOATS, NOPS = L::NOPS, AHEAD = L::AHEAD, RAWBLOCKS = L::RAWBLOCKS, OPBLOCKS = L::OPBLOCKS;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 127u) & ~127u;
    uint8_t *sm = smem_raw + (base - raw);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    float *ops = reinterpret_cast<float *>(sm + OFF_OP);
    float4 *red = reinterpret_cast<float4 *>(sm + OFF_RED);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + OFF_BAR + 2 * STAGES * 8);
    auto bar = [&](int i) { return base + OFF_BAR + 8u * i; };       // FULL[s] = s, READY[s] = STAGES + s
    const int cw = min(CW, p.dv);               // columns of a tile in shared memory (past d_v: zeros, dropped by the store)
    const uint32_t tile_bytes = (uint32_t)p.dk * cw * 4;

    // this CTA's items (bh * nsl + slice): blockIdx.x, + gridDim.x, ...
    const int first = blockIdx.x, stride = gridDim.x;
    const int nj = first < p.n_items ? (p.n_items - first + stride - 1) / stride : 0;
    const int nsteps = nj * p.n_tok;            // steps (item j, token t) in processing order: n = j * n_tok + t

    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(bar(i), 1);
            mbar_init(bar(STAGES + i), NCONS);
        }
        fence_mbar_init();
        tma_prefetch_desc(&tm_s);
    }
    __syncthreads();

    if (w == W_TMA) {
        // ---------------- TMA lane: state loads ahead of the arithmetic, stores behind it ----------------
        if (lane == 0) {
            bool failed = false;
            auto issue_load = [&](int j) {          // state of item j -> stage j % STAGES
                const int s = j % STAGES, item = first + j * stride;
                mbar_expect_tx(bar(s), tile_bytes);
                tma_load_2d(base + s * TILE_BYTES, &tm_s, (item % p.nsl) * CW, (item / p.nsl) * p.dk, bar(s));
            };
            for (int j = 0; j < STAGES && j < nj; ++j) issue_load(j);
            for (int j = 0; j < nj; ++j) {
                const int s = j % STAGES, item = first + j * stride;
                if (!mbar_wait_bounded(bar(STAGES + s), (uint32_t)(j / STAGES) & 1, abort_flag)) { failed = true; *abort_flag = 1; break; }
                tma_store_2d(&tm_s, base + s * TILE_BYTES, (item % p.nsl) * CW, (item / p.nsl) * p.dk);     // the updated state goes back
                bulk_commit();
                if (j + STAGES < nj) {              // once the store has read the stage, the stage takes the next load
                    bulk_wait_read0();
                    issue_load(j + STAGES);
                }
            }
            bulk_wait0();
            if (failed) {   // give loads that are still in flight time to land before shared memory goes away
                atomicOr(p.status, STATUS_TIMEOUT);
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
            }
        }
        return;
    }
    if (w >= W_OPS) {
        // ---------------- operand warps ----------------
        // Warp x walks its steps n = x, x + NOPS, ..  It meets the arithmetic warps at the start of step n (on a barrier of its
        // own); they have then finished step n - 1, the last to read the block of step n + NOPS, which may be cooked now.
        // These warps set the pace of a call with many tokens: what an item fixes is worked out once per item.
        const int ow = w - W_OPS;
        uint8_t *rawb = sm + OFF_RAW + (uint32_t)(ow * RAWBLOCKS) * RAW_BYTES;
        struct Where { size_t tok; int h, c0; };
        struct Pos { int j, t, raw; Where w; };      // item, token and raw block of a step
        auto locate = [&](Pos &q) {
            const int item = first + q.j * stride, bh = item / p.nsl, b = bh / p.H;
            q.w = Where{(size_t)b * p.n_tok, bh - b * p.H, (item - bh * p.nsl) * CW};
        };
        auto advance = [&](Pos &q) {                 // to this warp's next step
            if (++q.raw == RAWBLOCKS) q.raw = 0;
            q.t += NOPS;
            if (q.t < p.n_tok) return;
            while (q.t >= p.n_tok) { q.t -= p.n_tok; ++q.j; }
            if (q.j < nj) locate(q);
        };
        Pos rq{0, ow - NOPS, RAWBLOCKS - 1, {}}, ck;  // the next step to request, to cook
        if (nj > 0) locate(rq);
        advance(rq);
        ck = rq;
        auto request = [&]() {                       // always commits a group, empty past the last step
            if (rq.j < nj) {
                issue_raw<TIO, CW>(p, rawb + (uint32_t)rq.raw * RAW_BYTES, rq.w.tok + rq.t, rq.w.h, rq.w.c0, lane);
                advance(rq);
            }
            cp_async_commit();
        };
        auto cook = [&](int m) {                     // step m: its raw operands have landed but for the AHEAD - 1 later requests
            cp_async_wait<AHEAD - 1>();
            __syncwarp();
            cook_ops<TIO, CW>(p, rawb + (uint32_t)ck.raw * RAW_BYTES, ops + (m % OPBLOCKS) * OP_FLOATS, ck.w.h, ck.w.c0, lane);
            advance(ck);
        };
        for (int m = 0; m < AHEAD; ++m) request();
        if (ow < nsteps) cook(ow);
        for (int n = ow; n < nsteps; n += NOPS) {
            named_bar_sync(1 + 2 * ow, NCONS + 32);  // step n starts
            request();                               // (its raw block was cooked from before this barrier)
            if (n + NOPS < nsteps) cook(n + NOPS);
        }
        cp_async_wait<0>();
        return;
    }

    // ---------------- arithmetic warps ----------------
    bool failed = false;
    const bool gdn = p.variant == SLA_GDN;
    const int hl = lane / LPR, cl = lane % LPR;     // row of the group, column quad
    const bool in_tile = 4 * cl < cw;
    const int ld4 = cw >> 2;                        // float4s per tile row
    constexpr int NS = 2 / RP;                      // rows of a pair this lane holds: sums of its even and odd rows apart
    auto row = [&](int i) { return 2 * (w + NW * (i / NS)) + (RP == 2 ? hl : i % NS); };
    auto fold = [&](float4 (&vs)[NS]) {             // the two rows of a pair: in one lane, or in lanes l and l + 16
        float4 v = vs[0];
        if (RP == 1) {
            const float4 y = vs[NS - 1];
            v.x += y.x; v.y += y.y; v.z += y.z; v.w += y.w;
            return v;
        }
        v.x += __shfl_xor_sync(0xffffffffu, v.x, 16); v.y += __shfl_xor_sync(0xffffffffu, v.y, 16);
        v.z += __shfl_xor_sync(0xffffffffu, v.z, 16); v.w += __shfl_xor_sync(0xffffffffu, v.w, 16);
        return v;
    };
    int n = 0;
    for (int j = 0; j < nj; ++j) {
        const int item = first + j * stride, bh = item / p.nsl, c0 = (item % p.nsl) * CW, b = bh / p.H, h = bh % p.H, s = j % STAGES;
        float4 *tile = reinterpret_cast<float4 *>(sm + s * TILE_BYTES);
        if (!failed && !mbar_wait_bounded(bar(s), (uint32_t)(j / STAGES) & 1, abort_flag)) { failed = true; *abort_flag = 1; }
        float4 S[RPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = row(i);
            S[i] = (r < p.dk && in_tile) ? tile[r * ld4 + cl] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int t = 0; t < p.n_tok; ++t, ++n) {
            named_bar_sync(1 + 2 * (n % NOPS), NCONS + 32);   // the operand block of this step is complete
            const float *op = ops + (n % OPBLOCKS) * OP_FLOATS;
            float4 u = *reinterpret_cast<const float4 *>(op + OP_U + 4 * cl);
            float kr[RPT];
#pragma unroll
            for (int i = 0; i < RPT; ++i) {         // Sbar = diag(a) S
                const int r = row(i);
                const float a = op[OP_A + r];
                kr[i] = op[OP_K + r];
                S[i].x *= a; S[i].y *= a; S[i].z *= a; S[i].w *= a;
            }
            if (gdn) {                              // u = beta (Gk v - k Sbar)
                float4 part[NS] = {};
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    float4 &q = part[i % NS];
                    q.x = fmaf(kr[i], S[i].x, q.x); q.y = fmaf(kr[i], S[i].y, q.y);
                    q.z = fmaf(kr[i], S[i].z, q.z); q.w = fmaf(kr[i], S[i].w, q.w);
                }
                const float4 sum = fold(part);
                if (hl == 0) red[w * LPR + cl] = sum;
                named_bar_sync(2, NCONS);
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int ww = 0; ww < NW; ++ww) {
                    const float4 x = red[ww * LPR + cl];
                    acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
                }
                const float beta = op[OP_BETA];
                u.x = beta * (u.x - acc.x); u.y = beta * (u.y - acc.y); u.z = beta * (u.z - acc.z); u.w = beta * (u.w - acc.w);
            }
            float4 part[NS] = {};
#pragma unroll
            for (int i = 0; i < RPT; ++i) {         // write: S = Sbar + k^T u ; read: o = q S
                const int r = row(i);
                const float qr = op[OP_Q + r];
                S[i].x = fmaf(kr[i], u.x, S[i].x); S[i].y = fmaf(kr[i], u.y, S[i].y);
                S[i].z = fmaf(kr[i], u.z, S[i].z); S[i].w = fmaf(kr[i], u.w, S[i].w);
                float4 &y = part[i % NS];
                y.x = fmaf(qr, S[i].x, y.x); y.y = fmaf(qr, S[i].y, y.y);
                y.z = fmaf(qr, S[i].z, y.z); y.w = fmaf(qr, S[i].w, y.w);
            }
            const float4 sum = fold(part);
            if (hl == 0) red[(NW + w) * LPR + cl] = sum;
            if (t == p.n_tok - 1) {                 // after the last token the state goes back: registers -> stage
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int r = row(i);
                    if (r < p.dk && in_tile) tile[r * ld4 + cl] = S[i];
                }
                fence_proxy_async();
                mbar_arrive(bar(STAGES + s));       // (the TMA lane stores it and reloads the stage)
            }
            named_bar_sync(2, NCONS);
            if (w == 0 && hl == 0 && c0 + 4 * cl < p.dv) {
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int ww = 0; ww < NW; ++ww) {
                    const float4 x = red[(NW + ww) * LPR + cl];
                    acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
                }
                st_io4((TIO *)p.o, (((size_t)b * p.n_tok + t) * p.H + h) * p.dv + c0 + 4 * cl, acc);
            }
        }
    }
}

bool make_state_map(CUtensorMap *m, float *state, long rows, int dv, int dk, int cw) {
    tc::EncodeFn fn = tc::encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)dv, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)dv * 4};
    cuuint32_t box[2] = {(cuuint32_t)(dv < cw ? dv : cw), (cuuint32_t)dk};
    cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, state, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int decode_sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 148;
    }
    return n;
}

}  // namespace

template <typename TIO, int CW>
static bool decode_configure_one() {
    return cudaFuncSetAttribute(k_decode_stream<TIO, CW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dc::Lay<CW>::SMEM) == cudaSuccess;
}
int decode_configure() {
    if (!tc::encode_fn()) return -1;
    return decode_configure_one<float, 64>() && decode_configure_one<float, 128>() && decode_configure_one<__nv_bfloat16, 64>() &&
                   decode_configure_one<__nv_bfloat16, 128>() ? 0 : -1;
}

template <int CW>
static int decode_launch(const Dims &d, const DecArgs &a, int *status, cudaStream_t st) {
    CUtensorMap ms;
    if (!make_state_map(&ms, a.state, (long)a.Bdec * d.H * d.dk, d.dv, d.dk, CW)) return -1;
    const int nsl = (d.dv + CW - 1) / CW;                // (Bdec H d_k fits an int, and nsl < d_k)
    DecParams p{a.q, a.k, a.v, a.log_decay, a.beta, a.lq, a.lk, a.o, status, d.variant, d.H, d.dk, d.dv, a.n_tok,
                a.Bdec * d.H * nsl, nsl, d.scale};
    const long want = (long)dc::Lay<CW>::CTAS * decode_sm_count();     // persistent CTAs
    const unsigned grid = (unsigned)(p.n_items < want ? p.n_items : want);
    if (d.io_bf16)
        k_decode_stream<__nv_bfloat16, CW><<<grid, dc::Lay<CW>::NTHREADS, dc::Lay<CW>::SMEM, st>>>(ms, p);
    else
        k_decode_stream<float, CW><<<grid, dc::Lay<CW>::NTHREADS, dc::Lay<CW>::SMEM, st>>>(ms, p);
    return 0;
}

int decode_step(const Dims &d, const DecArgs &a, int *status, cudaStream_t st, Tracer &tr) {
    if ((a.n_tok == 1 ? decode_launch<64>(d, a, status, st) : decode_launch<128>(d, a, status, st)) < 0) return -1;
    tr.mark("decode");
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace sla
