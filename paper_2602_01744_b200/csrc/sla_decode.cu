// Recurrent decode (Eq. 5-6 with the instantiations of Eq. 10-16 at single tokens) as a streaming kernel.
//
// A decode step moves the whole fp32 state once in and once out and does two FLOP per byte: it is HBM-bound, so the
// kernel is built like a copy.  One work item is CW columns of the [d_k x d_v] state of one (sequence, head) (columns of a
// state do not meet in a step, with or without the delta rule).  Persistent CTAs walk their items with a ring of three
// shared-memory stages and three roles:
//   TMA lane          tile loads up to three items ahead of the arithmetic; the updated state leaves through a TMA
//                     store from the same stage, and the stage takes the next load as soon as the store has read it
//   operand warps     per token: the H gate logits -> head-softmax gates (Eq. 4), decay factors exp(g), and the
//                     operand vectors scale*Gq*q, Gk*k (or k), v (or Gk*v) as fp32 in a ring of blocks, several steps ahead
//   arithmetic warps  the state in registers: decay, the delta rule's k S (GDN), the rank-1 write, the read-out o = q S
// so loads, arithmetic and stores of neighbouring items overlap all the time.
// n_tok consecutive tokens of a sequence are applied while its state sits in registers (multi-token decode).
//
// An arithmetic warp owns CW / 8 columns and all rows of them, so that a token's sums over the rows stay inside the warp
// (three shuffle steps) and the warps meet nobody but the operand ring: the delta rule's chain from token to token has no
// block-wide barrier.  A lane holds 16 rows (lane group x: x, x + 8, x + 16 ..) of CW / 32 columns, as pairs of rows in packed
// fp32 registers (two multiply-adds an instruction).  With the rows spread over the warps, three block barriers and two trips
// through shared memory a token set the pace.  Device time of a call, before and now, 16 heads of 128, states in turn (256 MiB and more), delta rule:
// 16 streams x 8 tokens 23.8 -> 17.4 us, 64 x 8 69.8 -> 47.1, 64 x 4 41.6 -> 30.9, one stream x 8 12.2 -> 8.7; one token: 1 stream 4.5 -> 3.9, 16 streams
// 10.4 -> 9.3, 64 streams 23.6 -> 23.4.  Softmax-GLA, one token: 4.4 -> 3.7, 10.1 -> 8.7, 64 streams 23.3 -> 23.6 (HBM: 5.7 TB/s; 20.1 -> 14.9
// where the 64 MiB of states stay in L2).
// A single token takes slices of 64 columns and two CTAs per SM, whose loads and stores cover one another's barriers and whose
// smaller items fill the last wave; several tokens take 128 columns, because preparing the operands does not shrink with the slice.
// Both add up the rows of a state in the same order, so that n tokens in one call give the bits of n calls.
#include "sla_gla_tc.cuh"

namespace sla {
namespace {

using namespace ptx;

namespace dc {
constexpr int STAGES = 3;                // states in flight per CTA
constexpr int NW = 8;                    // arithmetic warps
constexpr int W_TMA = NW, W_OPS = NW + 1;
constexpr int DMAX = 128;
constexpr int PANEL = 32;                // columns of a 128-byte-swizzled line of a tile
// operand block (floats): q' k' a, each [128] in lane order (op_pos), then (a, beta) as scalars, u[CW] last
constexpr int OP_VEC = 4 * 36, OP_Q = 0, OP_K = OP_VEC, OP_A = 2 * OP_VEC, OP_SC = 3 * OP_VEC, OP_U = OP_SC + 4;
// Element r of an operand vector: the 16 rows x + 8 i of lane group x stand in four runs of four, the runs of the eight groups
// side by side, so that a lane reads four rows at a time and a warp's read is one run of 128 bytes; 36: the operand warps'
// writes (four neighbouring rows a lane) then fall into different banks.
__device__ __forceinline__ constexpr int op_pos(int r) { return (r >> 5) * 36 + (r & 7) * 4 + ((r >> 3) & 3); }
template <int CW> struct Lay {
    static constexpr int NC = CW / 32;                       // columns a lane
    static constexpr uint32_t TILE = DMAX * CW * 4;          // 64 or 32 KiB
    // operand warps: warp x takes the steps n with n % NOPS == x.  (Two of them beside the narrow slices leave 80 registers a thread, which
    // spill: one token for 64 streams 23.4 us with one, 25.5 with two.)
    static constexpr int NOPS = CW == DMAX ? 3 : 1, BLOCKS = CW == DMAX ? 6 : 4;
    static constexpr int NTHREADS = 32 * (NW + 1 + NOPS);
    static constexpr int OP_FLOATS = OP_U + CW;
    static constexpr uint32_t OFF_OP = STAGES * TILE;                        // [BLOCKS] operand blocks
    static constexpr uint32_t OFF_BAR = OFF_OP + BLOCKS * OP_FLOATS * 4;
    static constexpr int B_FULL = 0, B_READY = STAGES, B_OPFULL = 2 * STAGES, B_OPFREE = B_OPFULL + BLOCKS, NBAR = B_OPFREE + BLOCKS;
    static constexpr uint32_t SMEM = OFF_BAR + NBAR * 8 + 16 + 1024;         // + abort flag, + slack to align the base to 1 KiB
    static constexpr int CTAS = DMAX / CW;                   // per SM
    static_assert(OP_FLOATS % 4 == 0 && OFF_BAR % 8 == 0, "alignment");
    static_assert(CTAS * (SMEM + 1024) <= 233472, "shared memory budget");
};
}  // namespace dc

// States move by tiled TMA in lines of 32 columns, 128-byte swizzled in shared memory.  d_v a multiple of 32: one 3-D copy an item,
// dims (32 columns, lines of a row, rows of the [Bdec*H*d_k, d_v] view), so that a row's lines are fetched together; otherwise one
// 2-D copy per panel of 32 columns, because a line across the end of a row would be stored into the next one.  (Panels for every
// width fetch a row in pieces of 128 bytes: one token for 64 streams 24.9 us instead of 23.4.)
struct DecParams {
    const void *q, *k, *v;
    const float *log_decay, *beta, *lq, *lk;
    void *o;
    int *status;
    int H, dk, dv, n_tok;
    int n_items, nsl;                           // Bdec * H * nsl items, nsl = slices of CW columns per state
    float scale;
};

// ---- packed fp32: two values of neighbouring rows in one 64-bit register ----
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 up2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// ---- operands of one step as a lane of an operand warp fetches them: elements 4 lane .. 4 lane + 3 of the vectors ----
template <typename TIO> struct Quad;
template <> struct Quad<float> {
    float4 v;
    __device__ __forceinline__ void load(const void *p, size_t i, bool ok) {
        v = ok ? __ldg(reinterpret_cast<const float4 *>((const float *)p + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ float4 get() const { return v; }
};
template <> struct Quad<__nv_bfloat16> {
    uint2 v;
    __device__ __forceinline__ void load(const void *p, size_t i, bool ok) {
        v = ok ? __ldg(reinterpret_cast<const uint2 *>((const __nv_bfloat16 *)p + i)) : make_uint2(0u, 0u);
    }
    __device__ __forceinline__ float4 get() const {
        const float2 a = unpack_bf16(v.x), b = unpack_bf16(v.y);
        return make_float4(a.x, a.y, b.x, b.y);
    }
};
template <typename TIO> struct RawOps {
    Quad<TIO> q, k, v;
    float4 g;                                   // log-decay vector (GLA)
    float xq, xk, gs, beta;                     // logits of head `lane`, scalar log-decay (RetNet, GDN), beta (GDN)
};
// step's token row `tok` = b*n_tok + t, head h; of v the columns from c0 on
template <typename TIO, int CW, int VAR>
__device__ __forceinline__ void fetch_ops(const DecParams &p, RawOps<TIO> &r, size_t tok, int h, int c0, int lane) {
    const size_t th = tok * p.H + h;
    const int e = 4 * lane;
    r.q.load(p.q, th * p.dk + e, e < p.dk);
    r.k.load(p.k, th * p.dk + e, e < p.dk);
    r.v.load(p.v, th * p.dv + c0 + e, e < CW && c0 + e < p.dv);
    if (VAR == SLA_GLA) r.g = e < p.dk ? __ldg(reinterpret_cast<const float4 *>(p.log_decay + th * p.dk + e)) : make_float4(0.f, 0.f, 0.f, 0.f);
    else r.gs = __ldg(p.log_decay + (VAR == SLA_GDN ? th : (size_t)h));
    if (VAR == SLA_GDN) r.beta = __ldg(p.beta + th);
    r.xq = lane < p.H ? __ldg(p.lq + tok * p.H + lane) : -INFINITY;
    r.xk = lane < p.H ? __ldg(p.lk + tok * p.H + lane) : -INFINITY;
}
// Gates (Eq. 4) and the operand vectors the arithmetic warps use, into operand block `op`.
template <typename TIO, int CW, int VAR>
__device__ __forceinline__ void cook_ops(const DecParams &p, const RawOps<TIO> &r, float *op, int h, int lane) {
    float mq = r.xq, mk = r.xk;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mq = fmaxf(mq, __shfl_xor_sync(0xffffffffu, mq, o));
        mk = fmaxf(mk, __shfl_xor_sync(0xffffffffu, mk, o));
    }
    const float eq = expf(r.xq - mq), ek = expf(r.xk - mk);      // exp(-inf) = 0 on the padding lanes
    float sq = eq, sk = ek;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sq += __shfl_xor_sync(0xffffffffu, sq, o);
        sk += __shfl_xor_sync(0xffffffffu, sk, o);
    }
    const float Gq = __shfl_sync(0xffffffffu, eq, h) / sq, Gk = __shfl_sync(0xffffffffu, ek, h) / sk;
    const float fq = p.scale * Gq, fk = VAR == SLA_GDN ? 1.f : Gk, fv = VAR == SLA_GDN ? Gk : 1.f;
    // (all entries are written: the arithmetic warps take rows past d_k as zeros)
    const float4 q = r.q.get(), k = r.k.get(), v = r.v.get();
    const bool rk = 4 * lane < p.dk;
    const int o = dc::op_pos(4 * lane);          // rows 4 lane + e: four groups' runs, 4 floats apart
    const float qv[4] = {q.x, q.y, q.z, q.w}, kv[4] = {k.x, k.y, k.z, k.w}, gv[4] = {r.g.x, r.g.y, r.g.z, r.g.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        op[dc::OP_Q + o + 4 * e] = rk ? fq * qv[e] : 0.f;
        op[dc::OP_K + o + 4 * e] = rk ? fk * kv[e] : 0.f;
        if (VAR == SLA_GLA) op[dc::OP_A + o + 4 * e] = rk ? expf(gv[e]) : 0.f;
    }
    if (4 * lane < CW) *reinterpret_cast<float4 *>(op + dc::OP_U + 4 * lane) = make_float4(fv * v.x, fv * v.y, fv * v.z, fv * v.w);
    if (VAR != SLA_GLA && lane == 0) *reinterpret_cast<float2 *>(op + dc::OP_SC) = make_float2(expf(r.gs), VAR == SLA_GDN ? r.beta : 0.f);
}

template <typename TIO, int CW, int VAR>
__global__ void __launch_bounds__(dc::Lay<CW>::NTHREADS, dc::Lay<CW>::CTAS)
k_decode_stream(const __grid_constant__ CUtensorMap tm_s, const __grid_constant__ DecParams p) {
    using namespace dc;
    using L = Lay<CW>;
    constexpr int NC = L::NC, NOPS = L::NOPS, BLOCKS = L::BLOCKS, OP_FLOATS = L::OP_FLOATS;
    constexpr uint32_t TILE_BYTES = L::TILE;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    float *ops = reinterpret_cast<float *>(sm + L::OFF_OP);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + L::OFF_BAR + L::NBAR * 8);
    auto bar = [&](int i) { return base + L::OFF_BAR + 8u * i; };
    const bool rows_whole = p.dv % PANEL == 0;
    const uint32_t panel_bytes = (uint32_t)p.dk * PANEL * 4;     // (columns past d_v: zeros, dropped by the store)

    // this CTA's items (bh * nsl + slice): blockIdx.x, + gridDim.x, ...
    const int first = blockIdx.x, stride = gridDim.x;
    const int nj = first < p.n_items ? (p.n_items - first + stride - 1) / stride : 0;
    const int nsteps = nj * p.n_tok;            // steps (item j, token t) in processing order: n = j * n_tok + t

    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < L::NBAR; ++i)
            mbar_init(bar(i), ((i >= L::B_READY && i < L::B_OPFULL) || i >= L::B_OPFREE) ? NW : 1);
        fence_mbar_init();
        tma_prefetch_desc(&tm_s);
    }
    __syncthreads();
    bool failed = false;
    auto wait = [&](int i, uint32_t parity) {
        if (!failed && !mbar_wait_bounded(bar(i), parity, abort_flag)) { failed = true; *abort_flag = 1; }
    };

    if (w == W_TMA) {
        // ---------------- TMA lane: state loads ahead of the arithmetic, stores behind it ----------------
        if (lane == 0) {
            auto panels = [&](int c0) { return (min(CW, p.dv - c0) + PANEL - 1) / PANEL; };
            auto issue_load = [&](int j) {          // state of item j -> stage j % STAGES
                const int s = j % STAGES, item = first + j * stride, c0 = (item % p.nsl) * CW, r0 = (item / p.nsl) * p.dk;
                const int np = rows_whole ? CW / PANEL : panels(c0);
                const uint32_t dst = base + s * TILE_BYTES, full = bar(L::B_FULL + s);
                mbar_expect_tx(full, np * panel_bytes);
                if (rows_whole) tma_load_3d(dst, &tm_s, 0, c0 / PANEL, r0, full);
                else for (int x = 0; x < np; ++x) tma_load_2d(dst + x * panel_bytes, &tm_s, c0 + x * PANEL, r0, full);
            };
            auto issue_store = [&](int j) {         // the updated state goes back
                const int item = first + j * stride, c0 = (item % p.nsl) * CW, r0 = (item / p.nsl) * p.dk;
                const uint32_t src = base + (j % STAGES) * TILE_BYTES;
                if (rows_whole) tma_store_3d(&tm_s, src, 0, c0 / PANEL, r0);
                else for (int x = 0; x < panels(c0); ++x) tma_store_2d(&tm_s, src + x * panel_bytes, c0 + x * PANEL, r0);
                bulk_commit();
            };
            for (int j = 0; j < STAGES && j < nj; ++j) issue_load(j);
            for (int j = 0; j < nj; ++j) {
                wait(L::B_READY + j % STAGES, (uint32_t)(j / STAGES) & 1);
                if (failed) break;
                issue_store(j);
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
        // Warp x walks its steps n = x, x + NOPS, ..: the next one's operands are requested before the present one's are
        // cooked into block n % BLOCKS, as soon as the arithmetic warps are done with what was there.
        struct Pos { int j, t, h, c0; size_t tok; };
        auto locate = [&](Pos &q) {
            const int item = first + q.j * stride, bh = item / p.nsl, b = bh / p.H;
            q.tok = (size_t)b * p.n_tok;
            q.h = bh - b * p.H;
            q.c0 = (item - bh * p.nsl) * CW;
        };
        auto settle = [&](Pos &q) {                  // q.t counts on past the item: into the item it belongs to
            if (q.t < p.n_tok) return;
            do { q.t -= p.n_tok; ++q.j; } while (q.t >= p.n_tok);
            if (q.j < nj) locate(q);
        };
        Pos at{0, w - W_OPS, 0, 0, 0};
        RawOps<TIO> cur, nxt;
        if (nj > 0) locate(at);
        settle(at);
        if (at.j < nj) fetch_ops<TIO, CW, VAR>(p, nxt, at.tok + at.t, at.h, at.c0, lane);
        for (int n = w - W_OPS; n < nsteps; n += NOPS) {
            cur = nxt;
            const int h = at.h, blk = n % BLOCKS;
            at.t += NOPS;
            settle(at);
            if (at.j < nj) fetch_ops<TIO, CW, VAR>(p, nxt, at.tok + at.t, at.h, at.c0, lane);
            if (n >= BLOCKS) wait(L::B_OPFREE + blk, (uint32_t)(n / BLOCKS - 1) & 1);
            cook_ops<TIO, CW, VAR>(p, cur, ops + blk * OP_FLOATS, h, lane);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(L::B_OPFULL + blk));
        }
        return;
    }

    // ---------------- arithmetic warps ----------------
    const int cl = lane & 3, g = lane >> 2;          // this lane: rows g + 8 i of ..
    const int col0 = w * (CW / 8) + cl * NC;         // .. its columns of the slice
    // In shared memory a 16-byte piece of a line stands at its position XOR (line % 8).  Lines of a row side by side: the rows that
    // lanes read in one cycle (two neighbouring ones of 4 lines, four of 2) then lie in different banks.
    constexpr int LR = CW / PANEL;                   // lines of a row
    const int line0 = rows_whole ? g * LR + col0 / PANEL : g;
    const uint32_t row8 = 8 * 128 * (rows_whole ? LR : 1);       // bytes from row r to row r + 8
    const uint32_t tile_off = (rows_whole ? 0 : (col0 / PANEL) * panel_bytes) + line0 * 128 + ((((col0 % PANEL) >> 2) ^ (line0 & 7)) << 4) + (col0 & 3) * 4;
    const int npair = p.dk >> 4;                     // row pairs (g + 16 m, g + 16 m + 8) that exist
    auto rows_sum = [&](uint64_t v) {                // over the lanes' sums of their even and odd rows, then the lane groups
        const float2 f = up2(v);
        float s = f.x + f.y;
#pragma unroll
        for (int o = 16; o >= 4; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };
    int n = 0;
    for (int j = 0; j < nj; ++j) {
        const int item = first + j * stride, bh = item / p.nsl, c0 = (item % p.nsl) * CW, b = bh / p.H, h = bh % p.H, s = j % STAGES;
        uint8_t *tile = sm + s * TILE_BYTES + tile_off;
        const bool active = c0 + w * (CW / 8) < p.dv;    // (d_v is a multiple of 16: a warp's columns exist or not, together)
        wait(L::B_FULL + s, (uint32_t)(j / STAGES) & 1);
        uint64_t S[8][NC];                           // [row pair][column]
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            float lo[NC] = {}, hi[NC] = {};
            if (active && m < npair) {
                if (NC == 4) {
                    const float4 a = *reinterpret_cast<const float4 *>(tile + 2 * m * row8), c = *reinterpret_cast<const float4 *>(tile + (2 * m + 1) * row8);
                    lo[0] = a.x; lo[1] = a.y; lo[NC - 2] = a.z; lo[NC - 1] = a.w;
                    hi[0] = c.x; hi[1] = c.y; hi[NC - 2] = c.z; hi[NC - 1] = c.w;
                } else {
                    const float2 a = *reinterpret_cast<const float2 *>(tile + 2 * m * row8), c = *reinterpret_cast<const float2 *>(tile + (2 * m + 1) * row8);
                    lo[0] = a.x; lo[1] = a.y;
                    hi[0] = c.x; hi[1] = c.y;
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) S[m][c] = pk2(lo[c], hi[c]);
        }
        size_t orow = ((size_t)b * p.n_tok * p.H + h) * p.dv + c0 + w * (CW / 8);
        for (int t = 0; t < p.n_tok; ++t, ++n, orow += (size_t)p.H * p.dv) {
            const int blk = n % BLOCKS;
            wait(L::B_OPFULL + blk, (uint32_t)(n / BLOCKS) & 1);
            const float *op = ops + blk * OP_FLOATS;
            const float *vec = op + 4 * g;           // run m of this lane's rows: + 36 m
            auto pairs = [&](int off, int m2, uint64_t (&x)[2]) {
                const ulonglong2 y = *reinterpret_cast<const ulonglong2 *>(vec + off + 36 * m2);
                x[0] = y.x; x[1] = y.y;
            };
            float u[NC];
            if (NC == 4) {
                const float4 x = *reinterpret_cast<const float4 *>(op + OP_U + col0);
                u[0] = x.x; u[1] = x.y; u[NC - 2] = x.z; u[NC - 1] = x.w;
            } else {
                const float2 x = *reinterpret_cast<const float2 *>(op + OP_U + col0);
                u[0] = x.x; u[1] = x.y;
            }
            uint64_t kr[8], a1 = 0;
            const float2 sc = VAR == SLA_GLA ? make_float2(0.f, 0.f) : *reinterpret_cast<const float2 *>(op + OP_SC);
            if (VAR != SLA_GLA) a1 = pk2(sc.x, sc.x);
            uint64_t part[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) part[c] = 0;
#pragma unroll
            for (int m2 = 0; m2 < 4; ++m2) {        // Sbar = diag(a) S;  k Sbar for the delta rule
                uint64_t k2[2], a2[2] = {a1, a1};
                pairs(OP_K, m2, k2);
                if (VAR == SLA_GLA) pairs(OP_A, m2, a2);
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    kr[2 * m2 + x] = k2[x];
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        S[2 * m2 + x][c] = mul2(a2[x], S[2 * m2 + x][c]);
                        if (VAR == SLA_GDN) part[c] = fma2(k2[x], S[2 * m2 + x][c], part[c]);
                    }
                }
            }
            if (VAR == SLA_GDN) {                   // u = beta (Gk v - k Sbar)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    u[c] = sc.y * (u[c] - rows_sum(part[c]));
                    part[c] = 0;
                }
            }
            uint64_t u2[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) u2[c] = pk2(u[c], u[c]);
#pragma unroll
            for (int m2 = 0; m2 < 4; ++m2) {        // write: S = Sbar + k^T u ; read: o = q S
                uint64_t q2[2];
                pairs(OP_Q, m2, q2);
#pragma unroll
                for (int x = 0; x < 2; ++x)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        S[2 * m2 + x][c] = fma2(kr[2 * m2 + x], u2[c], S[2 * m2 + x][c]);
                        part[c] = fma2(q2[x], S[2 * m2 + x][c], part[c]);
                    }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(L::B_OPFREE + blk));
            if (t == p.n_tok - 1) {                 // after the last token the state goes back: registers -> stage
                if (active)
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        if (m >= npair) break;
                        float2 f[NC];
#pragma unroll
                        for (int c = 0; c < NC; ++c) f[c] = up2(S[m][c]);
                        if (NC == 4) {
                            *reinterpret_cast<float4 *>(tile + 2 * m * row8) = make_float4(f[0].x, f[1].x, f[NC - 2].x, f[NC - 1].x);
                            *reinterpret_cast<float4 *>(tile + (2 * m + 1) * row8) = make_float4(f[0].y, f[1].y, f[NC - 2].y, f[NC - 1].y);
                        } else {
                            *reinterpret_cast<float2 *>(tile + 2 * m * row8) = make_float2(f[0].x, f[1].x);
                            *reinterpret_cast<float2 *>(tile + (2 * m + 1) * row8) = make_float2(f[0].y, f[1].y);
                        }
                    }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(L::B_READY + s));       // (the TMA lane stores it and reloads the stage)
            }
            // o: each step of the sum over the lane groups also halves the columns a lane is in charge of, down to one
            float y[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float2 f = up2(part[c]);
                y[c] = f.x + f.y;
            }
            int oc = 0, nc = NC;                    // first of the columns left, their number
#pragma unroll
            for (int o = 16; o >= 4; o >>= 1) {
                if (nc > 1) {
                    nc >>= 1;
                    const bool up = lane & o;
#pragma unroll
                    for (int c = 0; c < NC / 2; ++c) {
                        if (c >= nc) break;
                        const float keep = up ? y[c + nc] : y[c], send = up ? y[c] : y[c + nc];
                        y[c] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                    oc += up ? nc : 0;
                } else {
                    y[0] += __shfl_xor_sync(0xffffffffu, y[0], o);
                }
            }
            constexpr int REST = NC == 4 ? 4 : 12;  // lanes that differ in these bits hold the same column
            if (active && (lane & REST) == 0) {
                TIO *dst = (TIO *)p.o + orow + cl * NC + oc;
                if (sizeof(TIO) == 4) *reinterpret_cast<float *>(dst) = y[0];
                else *reinterpret_cast<__nv_bfloat16 *>(dst) = __float2bfloat16_rn(y[0]);
            }
        }
    }
}

bool make_state_map(CUtensorMap *m, float *state, long rows, int dv, int dk, int cw) {
    tc::EncodeFn fn = tc::encode_fn();
    if (!fn) return false;
    const bool rows_whole = dv % dc::PANEL == 0;
    const cuuint64_t dims3[3] = {dc::PANEL, (cuuint64_t)(dv / dc::PANEL), (cuuint64_t)rows}, strides3[2] = {dc::PANEL * 4, (cuuint64_t)dv * 4};
    const cuuint32_t box3[3] = {dc::PANEL, (cuuint32_t)(cw / dc::PANEL), (cuuint32_t)dk};
    const cuuint64_t dims2[2] = {(cuuint64_t)dv, (cuuint64_t)rows}, strides2[1] = {(cuuint64_t)dv * 4};
    const cuuint32_t box2[2] = {dc::PANEL, (cuuint32_t)dk}, estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, rows_whole ? 3 : 2, state, rows_whole ? dims3 : dims2, rows_whole ? strides3 : strides2,
              rows_whole ? box3 : box2, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
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

// f(kernel) for the I/O type, slice width and variant at hand
template <int CW, class F>
bool with_kernel(bool bf16, int variant, F f) {
    if (variant == SLA_GDN) return bf16 ? f(k_decode_stream<__nv_bfloat16, CW, SLA_GDN>) : f(k_decode_stream<float, CW, SLA_GDN>);
    if (variant == SLA_GLA) return bf16 ? f(k_decode_stream<__nv_bfloat16, CW, SLA_GLA>) : f(k_decode_stream<float, CW, SLA_GLA>);
    return bf16 ? f(k_decode_stream<__nv_bfloat16, CW, SLA_RETNET>) : f(k_decode_stream<float, CW, SLA_RETNET>);
}
template <int CW>
bool decode_configure_one(bool bf16, int variant) {
    return with_kernel<CW>(bf16, variant, [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dc::Lay<CW>::SMEM) == cudaSuccess;
    });
}

}  // namespace

int decode_configure(int variant, bool bf16) {
    return tc::encode_fn() && decode_configure_one<64>(bf16, variant) && decode_configure_one<128>(bf16, variant) ? 0 : -1;
}

template <int CW>
static int decode_launch(const Dims &d, const DecArgs &a, int *status, cudaStream_t st) {
    CUtensorMap ms;
    if (!make_state_map(&ms, a.state, (long)a.Bdec * d.H * d.dk, d.dv, d.dk, CW)) return -1;
    const int nsl = (d.dv + CW - 1) / CW;                // (Bdec H d_k fits an int, and nsl < d_k)
    DecParams p{a.q, a.k, a.v, a.log_decay, a.beta, a.lq, a.lk, a.o, status, d.H, d.dk, d.dv, a.n_tok, a.Bdec * d.H * nsl, nsl, d.scale};
    const long want = (long)dc::Lay<CW>::CTAS * decode_sm_count();     // persistent CTAs
    const unsigned grid = (unsigned)(p.n_items < want ? p.n_items : want);
    with_kernel<CW>(d.io_bf16, d.variant, [&](auto kernel) {
        kernel<<<grid, dc::Lay<CW>::NTHREADS, dc::Lay<CW>::SMEM, st>>>(ms, p);
        return true;
    });
    return 0;
}

// One token, or states of one narrow slice: 64 columns an item.  Several tokens of wider states: 128 (in slices of 64 the operands of
// a token are prepared twice).
int decode_step(const Dims &d, const DecArgs &a, int *status, cudaStream_t st, Tracer &tr) {
    if ((a.n_tok == 1 || d.dv <= 64 ? decode_launch<64>(d, a, status, st) : decode_launch<128>(d, a, status, st)) < 0) return -1;
    tr.mark("decode");
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace sla
