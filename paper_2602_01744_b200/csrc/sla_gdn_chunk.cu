// Softmax-GatedDeltaNet on the 5th-generation tensor cores, chunk-parallel form (bf16 I/O, d_k and d_v 128 or 64, chunk 64).
//
// The delta rule's chunk recurrence carries only a d_k x d_v state; everything else a chunk needs depends on its own
// tokens.  The one-CTA-per-sequence kernels (sla_gdn_tc.cu, sla_gdn_tc_bwd.cu) put all of it on the serial chain; here
// it runs in parallel over the chunks and only two products a chunk stay serial:
//
//   prep_worker   every chunk: A = tril(Qg K^T), the triangular inverse, We, T2 (below), the per-token factors
//   scan_item     chunks in order, one CTA per (sequence, head, 64 value columns), state in fp32 registers:
//                   Ue = T2 V - We S            S' = e^{b_last} (S + K^T Ue)           o = fq (q S) + A Ue
//   bscan_item    chunks in reverse, same split, state gradient in fp32 registers (dZ = e^{b_last} dS'):
//                   dUe = A^T dO + K dZ         dS = dZ + Qg^T dO - We^T dUe
//   bgrad_chunks  every chunk: all input gradients from S, Ue, dUe, dZ
//
// Notation, token i of a chunk: b_i cumulative log-decay, Gam = e^b, fq = scale Gq Gam, Qg = fq q, L = strict_tril(beta_i
// e^{b_i - b_j} (k_i . k_j)), T = (I + L)^{-1}.  Eq. 14-15 in WY form give U = T(beta Gk V - beta Gam K S); with
// Ue_j = e^{-b_j} U_j (a row scaling, no loss of relative precision) all decays inside the chunk fold into
//   Te = diag(e^{-b}) T      T2 = Te diag(beta Gk)      We = Te diag(beta Gam) K
// and the forward's operands enter the tensor core as they stand in memory: no tile is rescaled, which leaves the two
// serial products a chunk (We S and K^T Ue), one 64x64 and one 128x64 accumulator read between them.
// Range: e^b is kept as 2^k e^b, with 2^-k the power of two nearest to half a chunk's whole decay, and S, dS as 2^-k S, 2^k dS: the
// formulas keep their form, every factor is exact (the bits are those of k = 0), and a state goes from one chunk's scale to the next one's
// inside its decay.  At the decay limit the factors that bf16 operands carry (e^b in A and dUe, e^-b in T2 and Ue) then span e^-38 .. e^38.
// With k = 0 A and dUe carried e^-76 = 1e-33: for dO of 1e-6, the size a mean-reduced loss leaves, their products were bf16 subnormals and dv
// was off by 1.5 % (26 % at 1e-9; one-CTA kernels 1.0 and 3.5 %; 0.3 % now at every scale).
// Gradients (chain rule, X = dUe):  dR = Te^T X (T's unit diagonal in fp32, only the part below it as bf16),  dA = tril(dO Ue^T),  P = strict_tril(dR Ue^T),  M = -beta Gam P,
//   aq = dO S^T + dA K               dq = fq aq               dv = beta Gk dR
//   kd = Ue dZ^T + dA^T Qg + M^T K   Y = dR S^T + P K         dk = kd - beta Gam Y
//   dbeta = Gk (dR.v) - Gam (k.Y)    db = Qg.aq - k.kd - beta Gam (k.Y)  (+ <dS', S'> on the last row)
//   dlog_decay = suffix sum of db;   Gq dGq = Qg.aq,  Gk dGk = beta Gk (dR.v)
// T's diagonal is one, but e^{-b} is not a bf16 number: with the whole of Te as the operand dR's dominant term was rounded once more than
// in the one-CTA kernels, which hold T itself (dv 4.00e-3 against 3.60e-3 on feature-map keys, and 3.41e-3 with the diagonal in fp32,
// which costs the training step 1 %: 4 x 4096 x 16 heads 512 -> 517 us).
// Qg.aq and k.kd cancel in the suffix sum, so both sides take the same rounded Qg and the same rounded dA.
#include "sla_gla_tc.cuh"
#include "sla_gdn_route.h"

#include <algorithm>
#include <cooperative_groups.h>

namespace sla {
namespace {

using namespace ptx;
using namespace tc;

// Per-chunk record in the workspace (byte offsets).  Training keeps what the backward pass reads; inference only what the
// scan reads.  T2 is dead once the scan has read it and shares its place with dUe.  We, A, scalars and T2 are contiguous.
struct Rec {
    uint32_t bytes, s, u, te, w, a, sc, t2, du, dz;
};
constexpr uint32_t SC_BYTES = 2048;                  // [6][64] floats, at float 384 (2^k e^{b_last}, 2^-k), at float 388 the 16 partial sums of <dS', S'>
enum Sc { SC_FQ = 0, SC_BG, SC_FV, SC_GAM, SC_GK, SC_IG, SC_NARR };
constexpr uint32_t SC_END = SC_NARR * C, SC_DOT = SC_END + 4, SC_LOAD = SC_DOT * 4;
static_assert(SC_LOAD % 16 == 0 && (SC_DOT + 16) * 4 <= SC_BYTES, "scalars of a record");
constexpr uint32_t PREP_BYTES = TILE_BF16 + HALF_BF16 + SC_BYTES + HALF_BF16;                        // We | A | scalars | T2
constexpr Rec REC_INFER = {PREP_BYTES, 0, 0, 0, 0, TILE_BF16, TILE_BF16 + HALF_BF16, TILE_BF16 + HALF_BF16 + SC_BYTES, 0, 0};
constexpr uint32_t R_U = STATE_BF16, R_TE = R_U + TILE_BF16, R_W = R_TE + HALF_BF16, R_A = R_W + TILE_BF16, R_SC = R_A + HALF_BF16,
                   R_DU = R_SC + SC_BYTES, R_DZ = R_DU + TILE_BF16, R_BYTES = R_DZ + STATE_BF16;
constexpr Rec REC_TRAIN = {R_BYTES, 0, R_U, R_TE, R_W, R_A, R_SC, R_DU, R_DU, R_DZ};

struct ChunkParams {
    const float *lq, *lk, *g, *beta;    // logits, log-decay, beta
    const float *h0, *dht;
    float *ht, *dh0;
    float *dg, *dbeta, *pq, *pk;
    uint8_t *rec;
    Rec L;
    int *status;
    int T, H, NT, n_rows;               // n_rows: batch rows (a packed batch: n_seq sequences instead)
    int slots;                          // (chunks + 1) summed over the (sequence, head) pairs
    float scale;
    int save, write_o;
    const SeqInfo *seqs;                // packed variable-length batch: per-sequence table and tensor maps, else nullptr
    int n_seq;
    const CUtensorMap *vmaps;
    int dk, dv;
};

// One (sequence, head): where its tokens, records and tensor maps are.
struct SeqHead {
    int b, h, T, NT;
    int slot;                           // first record
    size_t tok, sbh;                    // first token, index into the state tensors
    const CUtensorMap *vm;              // its own tensor maps (packed batch; batch coordinate 0), else nullptr
};
__device__ __forceinline__ SeqHead seq_head(const ChunkParams &p, int s, int h) {
    SeqHead q{s, h, p.T, p.NT, (s * p.H + h) * (p.NT + 1), (size_t)s * p.T, (size_t)s * p.H + h, nullptr};
    if (p.seqs) {
        const SeqInfo si = p.seqs[s];
        q.b = 0; q.T = si.T; q.NT = si.NT;
        q.tok = (size_t)si.t0;
        q.slot = si.slot0 * p.H + h * (si.NT + 1);
        q.sbh = (size_t)si.id * p.H + h;
        q.vm = p.vmaps + (size_t)s * Varlen::MAPS_PER_SEQ;
    }
    return q;
}
// The (sequence, head) that record slot `slot` belongs to (the table's slot0 ascend).
__device__ __forceinline__ SeqHead slot_owner(const ChunkParams &p, int slot) {
    if (!p.seqs) {
        const uint32_t bh = (uint32_t)slot / (uint32_t)(p.NT + 1), b = bh / (uint32_t)p.H;
        return seq_head(p, (int)b, (int)(bh - b * (uint32_t)p.H));
    }
    int lo = 0, hi = p.n_seq - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.seqs[mid].slot0 * p.H <= slot) lo = mid; else hi = mid - 1;
    }
    const SeqInfo si = p.seqs[lo];
    return seq_head(p, lo, (slot - si.slot0 * p.H) / (si.NT + 1));
}
// The first chunk among record slots slot, slot + step, ... (the slot after a sequence's last chunk holds only the final
// state); its owner in s.  p.slots if there is none.
__device__ __forceinline__ int next_chunk(const ChunkParams &p, int slot, int step, SeqHead &s) {
    for (; slot < p.slots; slot += step) {
        s = slot_owner(p, slot);
        if (slot - s.slot < s.NT) break;
    }
    return min(slot, p.slots);
}

// K extent of 128 (8 steps of 16) or 64 (4), unrolled: a rolled loop costs the issuing lane about 130 cycles a step
template <class F>
__device__ __forceinline__ void ksteps(bool wide, F step) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) step(kk);
    if (wide) {
#pragma unroll
        for (int kk = 4; kk < 8; ++kk) step(kk);
    }
}
// loads still in flight when a wait gave up get time to land before shared memory is used for other things
__device__ __forceinline__ void let_copies_land() {
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
}

// ------------------------------------------------------------------------------------------------
// every chunk: A, T and its scaled forms, We, per-token factors.  Three workers of four warps per CTA, each with its own
// shared memory, tensor-memory columns and named barrier: a chunk is a chain of small dependent steps (gates, products,
// triangular inverse, product), and three chains side by side fill one another's gaps.
namespace pr {
constexpr int LDL = 68;                                 // row stride (floats) of the fp32 64x64 work arrays
constexpr uint32_t MAT = 64 * LDL * 4;                  // 17 KiB
constexpr uint32_t OFF_Q = 0;                           // q tile -> fp32 T
constexpr uint32_t OFF_K = OFF_Q + MAT;
constexpr uint32_t OFF_L = OFF_K + TILE_BF16;           // fp32 L -> Te below its diagonal | T2 (bf16)
constexpr uint32_t OFF_A = OFF_L + MAT;                 // bf16 A; afterwards A and TW hold We staged for the store
constexpr uint32_t OFF_TW = OFF_A + HALF_BF16;          // bf16 -Te diag(beta Gam)
constexpr uint32_t OFF_X = OFF_TW + HALF_BF16;          // [4 warps][32][8] block-product scratch
constexpr uint32_t OFF_SC = OFF_X + 4 * 32 * 8 * 4;     // b, e^-b, scale Gq (then fq), beta Gam, beta Gk, Gk, beta, log-decay: 8 x 64 floats
constexpr uint32_t WORKER = (OFF_SC + 8 * C * 4 + 1023) & ~1023u;
constexpr int NWORK = 3, NTH = 128;
enum Bar { FULL = 0, M1, M2, NBAR };
static_assert(MAT % 1024 == 0, "tile alignment");
}  // namespace pr

// wid: this worker's number in the CTA; bars: its NBAR barriers (initialised, one arrival each)
__device__ __forceinline__ void prep_worker(const CUtensorMap &gm_q, const CUtensorMap &gm_k, const ChunkParams &p, uint8_t *sm, uint32_t base,
                                            uint32_t bars, uint32_t tmem, int wid, int tid, volatile int *abort_flag, bool &failed) {
    using namespace pr;
    const int warp = tid >> 5, lane = tid & 31;
    const uint32_t bFULL = bars + 8 * FULL, bM1 = bars + 8 * M1, bM2 = bars + 8 * M2;
    float *sc = reinterpret_cast<float *>(sm + OFF_SC);
    float *s_b = sc, *s_ig = sc + C, *s_fq = sc + 2 * C, *s_bg = sc + 3 * C, *s_fv = sc + 4 * C, *s_gk = sc + 5 * C, *s_beta = sc + 6 * C,
          *s_g = sc + 7 * C;
    float *Ls = reinterpret_cast<float *>(sm + OFF_L), *Ts = reinterpret_cast<float *>(sm + OFF_Q);
    auto wait = [&](uint32_t bar, uint32_t par) {
        if (!failed && !mbar_wait_bounded(bar, par, abort_flag)) { failed = true; *abort_flag = 1; }
    };
    auto sync = [&] { named_bar_sync(2 + wid, NTH); };
    const bool leader = warp == 0 && elect_lane();      // issues this worker's copies and products
    uint32_t par = 0;
    const int step = (int)gridDim.x * NWORK;
    SeqHead s, sn;
    int slot = next_chunk(p, (int)blockIdx.x * NWORK + wid, step, s), slot_n;
    auto load = [&](const SeqHead &o, int n) {              // q, k of a chunk (by the leader)
        mbar_expect_tx(bFULL, 2 * TILE_BF16);
        tma_load_5d(base + OFF_K, o.vm ? o.vm + 1 : &gm_k, 0, n * C, 0, o.h, o.b, bFULL);
        tma_load_5d(base + OFF_Q, o.vm ? o.vm : &gm_q, 0, n * C, 0, o.h, o.b, bFULL);
    };
    GateAhead gates;                                        // of the chunk to come, one token's logits spread over its lanes
    float xv = 0.f;                                         // its log-decay (threads 0..63) or beta of token tid % 64
    auto fetch_gates = [&](const SeqHead &o, int n) {
        const int t = tid & (C - 1), cn = min(C, o.T - n * C);
        const size_t t0 = o.tok + (size_t)n * C;
        gates.fetch((tid < C ? p.lq : p.lk) + t0 * p.H, p.H, cn, t);
        xv = t < cn ? (tid < C ? p.g : p.beta)[(t0 + t) * p.H + o.h] : 0.f;
    };
    if (slot < p.slots) {
        if (leader) load(s, slot - s.slot);
        fetch_gates(s, slot - s.slot);
    }
    for (; slot < p.slots; slot = slot_n, s = sn) {
        const int n = slot - s.slot;
        {
            const int t = tid & (C - 1), cn = min(C, s.T - n * C);
            gates.finish((tid < C ? p.lq : p.lk) + (s.tok + (size_t)n * C) * p.H, p.H, cn, s.h, tid < C ? p.scale : 1.f, tid < C ? s_fq : s_gk, t);
            (tid < C ? s_g : s_beta)[t] = xv;
        }
        // The next chunk's logits, log-decay and beta into registers, its tiles into L2 (their copies start when this chunk's last product
        // has read k).  Logits requested where they are used cost 4,600 of a chunk's 15,000 cycles: with the tiles' early request 3 x 2500
        // tokens x 16 heads forward 109 -> 100 us, 4 x 4096 x 16 forward and backward 517 -> 506.
        slot_n = next_chunk(p, slot + step, step, sn);
        if (slot_n < p.slots) {
            const int nn = slot_n - sn.slot;
            if (leader) {
                tma_prefetch_l2_5d(sn.vm ? sn.vm + 1 : &gm_k, 0, nn * C, 0, sn.h, sn.b);
                tma_prefetch_l2_5d(sn.vm ? sn.vm : &gm_q, 0, nn * C, 0, sn.h, sn.b);
            }
            fetch_gates(sn, nn);
        }
        sync();
        if (warp == 0) {
            constexpr uint32_t ID = idesc_bf16(64, 64, 0, 0);
            const uint64_t kQ = desc_kmajor(base + OFF_Q), kK = desc_kmajor(base + OFF_K);
            wait(bFULL, par);
            tc_fence_after();
            if (leader) {
                if (!failed) ksteps(p.dk > 64, [&](int kk) {
                    const uint64_t st = kstep_kmajor(kk, HALF_BF16);
                    tc_mma_bf16(tmem, kK + st, kK + st, ID, kk > 0);                // K K^T
                    tc_mma_bf16(tmem + 64, kQ + st, kK + st, ID, kk > 0);           // q K^T
                });
                tc_commit(bM1);
            }
        } else if (warp == 1) {      // inclusive scan of the 64 log-decays: lane l owns tokens 2l, 2l+1
            const float g0 = s_g[2 * lane], g1 = s_g[2 * lane + 1];
            float incl = g0 + g1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            s_b[2 * lane] = incl - g1;
            s_b[2 * lane + 1] = incl;
        }
        sync();
        if (tid >= C) {
            const int t = tid - C;
            const float b = s_b[t], beta = s_beta[t];
            const int k = min(max(__float2int_rn(s_b[C - 1] * (-0.5f * LOG2E)), -60), 60);
            const float up = __int_as_float((127 + k) << 23), down = __int_as_float((127 - k) << 23);          // 2^k, 2^-k
            const float gam = __expf(b) * up, fq = s_fq[t] * gam, bg = beta * gam, fv = beta * s_gk[t], ig = __expf(-b) * down;
            s_ig[t] = ig;
            s_fq[t] = fq;
            s_bg[t] = bg;
            s_fv[t] = fv;
            float *out = reinterpret_cast<float *>(p.rec + (size_t)slot * p.L.bytes + p.L.sc);
            out[SC_FQ * C + t] = fq;
            out[SC_BG * C + t] = bg;
            out[SC_FV * C + t] = fv;
            out[SC_GAM * C + t] = gam;
            out[SC_GK * C + t] = s_gk[t];
            out[SC_IG * C + t] = ig;
            if (t == C - 1) {
                *reinterpret_cast<float2 *>(out + SC_END) = make_float2(gam, down);
                if (b < -SLA_MAX_CHUNK_DECAY) atomicOr(p.status, STATUS_RANGE);
            }
        }
        if (leader) bulk_wait_read0();                      // the previous chunk's We, Te, T2 have left the buffers of A, TW and L
        sync();
        wait(bM1, par);
        tc_fence_after();
        const uint32_t tw = tmem + ((uint32_t)(32 * warp) << 16);
        const int r = 16 * warp + (lane >> 2), c0 = 2 * (lane & 3);
        {
            float v[32];
            tmem_ld_frag8(tw, v);                           // K K^T -> L
            tmem_wait_ld();
            const float f0 = s_bg[r], f1 = s_bg[r + 8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int j = 8 * i + c0;
                if (i < 2 * warp + 2) {                     // (blocks above the diagonal are never read)
                    const float2 g = *reinterpret_cast<const float2 *>(s_ig + j);
                    *reinterpret_cast<float2 *>(Ls + r * LDL + j) =
                        make_float2(j < r ? f0 * g.x * v[4 * i] : 0.f, j + 1 < r ? f0 * g.y * v[4 * i + 1] : 0.f);
                    *reinterpret_cast<float2 *>(Ls + (r + 8) * LDL + j) =
                        make_float2(j < r + 8 ? f1 * g.x * v[4 * i + 2] : 0.f, j + 1 < r + 8 ? f1 * g.y * v[4 * i + 3] : 0.f);
                }
            }
            tmem_ld_frag8(tw + 64, v);                      // q K^T -> A
            tmem_wait_ld();
            const float q0 = s_fq[r], q1 = s_fq[r + 8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int j = 8 * i + c0;
                const uint32_t off = frag_off(warp, lane, 0, i);
                *reinterpret_cast<uint32_t *>(sm + OFF_A + off) = pack_bf16(j <= r ? q0 * v[4 * i] : 0.f, j + 1 <= r ? q0 * v[4 * i + 1] : 0.f);
                *reinterpret_cast<uint32_t *>(sm + OFF_A + off + 1024) =
                    pack_bf16(j <= r + 8 ? q1 * v[4 * i + 2] : 0.f, j + 1 <= r + 8 ? q1 * v[4 * i + 3] : 0.f);
            }
        }
        fence_proxy_async();
        tc_fence_before();
        sync();
        uint8_t *rec = p.rec + (size_t)slot * p.L.bytes;
        if (leader) {
            bulk_store(rec + p.L.a, base + OFF_A, HALF_BF16);
            bulk_commit();
        }
        if (tid < C) {        // diagonal 16x16 blocks: column c of (I + L_bb)^{-1} by forward substitution
            const int bb = tid >> 4, c = tid & 15;
            const float *Lb = Ls + (16 * bb) * LDL + 16 * bb;
            float x[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                float acc = i == c ? 1.f : 0.f;
#pragma unroll
                for (int j = 0; j < i; ++j) acc = fmaf(-Lb[i * LDL + j], x[j], acc);
                x[i] = acc;
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) Ts[(16 * bb + i) * LDL + 16 * bb + c] = x[i];
        }
        sync();
        // Off-diagonal blocks by doubling, [[T1, 0], [T21, T2]] with T21 = -T2 (L21 T1): first inside the two 32x32 diagonal
        // blocks, then the 32x32 block between them, on the warp-level tf32 MMA (T is rounded to bf16 afterwards).  A column
        // of T21 needs only that column of T1, so a warp takes eight columns through both products without a barrier:
        // 2 + 2 and 4 + 4 dependent steps.
        {
            const int g = lane >> 2, t = lane & 3;
            float *Xw = reinterpret_cast<float *>(sm + OFF_X) + warp * 32 * 8;
            auto mac = [&](float (&x)[4], const float *M, const float *N, int ldn) {      // x += M[16 x 8] N[8 x 8]
                const uint32_t fa[4] = {to_tf32(M[g * LDL + t]), to_tf32(M[(g + 8) * LDL + t]), to_tf32(M[g * LDL + t + 4]), to_tf32(M[(g + 8) * LDL + t + 4])};
                const uint32_t fb[2] = {to_tf32(N[t * ldn + g]), to_tf32(N[(t + 4) * ldn + g])};
                mma_tf32_16x8x8(x, fa, fb);
            };
            auto put = [&](float *D, int ldd, const float (&x)[4], float sign) {
                *reinterpret_cast<float2 *>(D + g * ldd + 2 * t) = make_float2(sign * x[0], sign * x[1]);
                *reinterpret_cast<float2 *>(D + (g + 8) * ldd + 2 * t) = make_float2(sign * x[2], sign * x[3]);
            };
            {
                const int o = 32 * (warp >> 1), col = o + 8 * (warp & 1);
                float x[4] = {0.f, 0.f, 0.f, 0.f}, y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) mac(x, Ls + (o + 16) * LDL + o + 8 * ks, Ts + (o + 8 * ks) * LDL + col, LDL);
                put(Xw, 8, x, 1.f);
                __syncwarp();
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) mac(y, Ts + (o + 16) * LDL + o + 16 + 8 * ks, Xw + 8 * ks * 8, 8);
                put(Ts + (o + 16) * LDL + col, LDL, y, -1.f);
            }
            sync();
            {
                const int col = 8 * warp;
                float x[2][4] = {}, y[2][4] = {};
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    if (ks < 2 && col >= 16) continue;      // (T1 has no entries above its diagonal blocks)
                    mac(x[0], Ls + 32 * LDL + 8 * ks, Ts + 8 * ks * LDL + col, LDL);
                    mac(x[1], Ls + 48 * LDL + 8 * ks, Ts + 8 * ks * LDL + col, LDL);
                }
                put(Xw, 8, x[0], 1.f);
                put(Xw + 16 * 8, 8, x[1], 1.f);
                __syncwarp();
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    if (ks < 2) mac(y[0], Ts + 32 * LDL + 32 + 8 * ks, Xw + 8 * ks * 8, 8);
                    mac(y[1], Ts + 48 * LDL + 32 + 8 * ks, Xw + 8 * ks * 8, 8);
                }
                put(Ts + 32 * LDL + col, LDL, y[0], -1.f);
                put(Ts + 48 * LDL + col, LDL, y[1], -1.f);
            }
        }
        sync();
        {   // Te without its diagonal, T2 over L; -Te diag(beta Gam): thread = (row i, every other 16-byte chunk)
            const int i = tid >> 1;
            const float gi = s_ig[i];
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                const int ch = 2 * cc + (tid & 1), j0 = 8 * ch;
                uint4 e, t2, tn;
                uint32_t *ew = reinterpret_cast<uint32_t *>(&e), *t2w = reinterpret_cast<uint32_t *>(&t2), *tnw = reinterpret_cast<uint32_t *>(&tn);
                const bool have = (j0 >> 4) <= (i >> 4);     // (blocks above the diagonal were never written)
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int j = j0 + 4 * x;
                    float4 a = have ? *reinterpret_cast<const float4 *>(Ts + i * LDL + j) : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 fv = *reinterpret_cast<const float4 *>(s_fv + j), bg = *reinterpret_cast<const float4 *>(s_bg + j);
                    a.x *= gi; a.y *= gi; a.z *= gi; a.w *= gi;
                    ew[2 * x] = pack_bf16(a.x, a.y);
                    ew[2 * x + 1] = pack_bf16(a.z, a.w);
                    t2w[2 * x] = pack_bf16(a.x * fv.x, a.y * fv.y);
                    t2w[2 * x + 1] = pack_bf16(a.z * fv.z, a.w * fv.w);
                    tnw[2 * x] = pack_bf16(-a.x * bg.x, -a.y * bg.y);
                    tnw[2 * x + 1] = pack_bf16(-a.z * bg.z, -a.w * bg.w);
                }
                *reinterpret_cast<uint4 *>(sm + OFF_L + swz(i, ch)) = e;
                *reinterpret_cast<uint4 *>(sm + OFF_L + HALF_BF16 + swz(i, ch)) = t2;
                *reinterpret_cast<uint4 *>(sm + OFF_TW + swz(i, ch)) = tn;
            }
            if ((tid & 1) == ((i >> 3) & 1)) *reinterpret_cast<__nv_bfloat16 *>(sm + OFF_L + swz(i, i >> 3) + 2 * (i & 7)) = __float2bfloat16_rn(0.f);
        }
        fence_proxy_async();
        tc_fence_before();
        if (leader) bulk_wait_read0();                      // A has left: We goes there
        sync();
        if (warp == 0) {
            constexpr uint32_t ID = idesc_bf16(64, 128, 0, 1);
            const uint64_t kT = desc_kmajor(base + OFF_TW), mK = desc_mnmajor(base + OFF_K, HALF_BF16);
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem, kT + kstep_kmajor(kk, 0), mK + kstep_mnmajor(kk), ID, kk > 0);   // -We
                tc_commit(bM2);
            }
        }
        wait(bM2, par);
        tc_fence_after();
        // k has been read for the last time and T before the last barrier: the next chunk's tiles land while We leaves.  (Requested at the
        // top of the next chunk, behind the stores of We out of q's place, they cost 6,000 of a chunk's 15,700 cycles.)
        if (leader && slot_n < p.slots) load(sn, slot_n - sn.slot);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            float v[32];
            tmem_ld_frag8(tw + 64 * hf, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t off = frag_off(warp, lane, 64 * hf, i);
                *reinterpret_cast<uint32_t *>(sm + OFF_A + off) = pack_bf16(v[4 * i], v[4 * i + 1]);
                *reinterpret_cast<uint32_t *>(sm + OFF_A + off + 1024) = pack_bf16(v[4 * i + 2], v[4 * i + 3]);
            }
        }
        fence_proxy_async();
        tc_fence_before();
        sync();
        tc_fence_after();
        if (leader) {
            bulk_store(rec + p.L.w, base + OFF_A, TILE_BF16);
            bulk_store(rec + p.L.t2, base + OFF_L + HALF_BF16, HALF_BF16);
            if (p.save) bulk_store(rec + p.L.te, base + OFF_L, HALF_BF16);
            bulk_commit();
        }
        par ^= 1;
    }
    if (leader) {
        bulk_wait0();
        if (failed) let_copies_land();
    }
}

// ------------------------------------------------------------------------------------------------
// What the two scans share: 8 compute warps (state slice [128][64] in fp32 registers: warp w owns rows 32 (w % 4) + lane,
// columns 32 (w / 4) .. + 31), a warp each for MMA issue, loads and stores, four helper warps; every operand has two
// buffers.  A buffer is loaded again as soon as its own last reader is done, not when the chunk is: that keeps close to two
// chunks of time between the request for a tile and its use.  The issuing warps walk their loops converged: with a
// single lane in a branch of its own the issue of the 28 MMAs set the pace (2.0 us a chunk against 1.5).
namespace scn {
constexpr int NTHREADS = NCOMPUTE + 32 + 32 + 128 + 32; // warps 0..7 compute, 8 MMA issue, 9 loads, 10..13 helpers, 14 stores
constexpr uint32_t SLICE = STATE_HALF;                  // bf16 [128][64] state slice
// pairs: one barrier per buffer
enum Bar { F0 = 0, F1 = 2, F2 = 4, F3 = 6, E0 = 8, E1 = 10, E2 = 12, E3 = 14, UREADY = 16, HELP = 18, SAVED = 20, SREADY = 22, C1, C2, FINAL, DRAIN,
           NBAR };
constexpr uint32_t TM_ACC = 0, TM_D = 64, TM_O = 128 /* [2][q S | A Ue] */;
}  // namespace scn

// this thread's 32 state columns -> bf16 into a [128][64] swizzled slice
__device__ __forceinline__ void store_slice(uint8_t *dst, int row, int ch, const float (&v)[32]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint4 w;
        w.x = pack_bf16(v[8 * c + 0], v[8 * c + 1]);
        w.y = pack_bf16(v[8 * c + 2], v[8 * c + 3]);
        w.z = pack_bf16(v[8 * c + 4], v[8 * c + 5]);
        w.w = pack_bf16(v[8 * c + 6], v[8 * c + 7]);
        *reinterpret_cast<uint4 *>(dst + swz(row, 4 * ch + c)) = w;
    }
}
__device__ __forceinline__ void frag16_to_tile(uint8_t *dst, int quarter, int lane, int col0, const float (&v)[16]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t off = frag_off(quarter, lane, col0, i);
        *reinterpret_cast<uint32_t *>(dst + off) = pack_bf16(v[4 * i], v[4 * i + 1]);
        *reinterpret_cast<uint32_t *>(dst + off + 1024) = pack_bf16(v[4 * i + 2], v[4 * i + 3]);
    }
}

// Barriers for one (sequence, head, slice): they start from phase 0 for every item a CTA takes.
__device__ __forceinline__ void scan_barriers(uint32_t bars, bool first) {
    using namespace scn;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 0; i < NBAR; ++i) {
            const bool compute = i == SREADY || i == UREADY || i == UREADY + 1 || i == FINAL;
            if (!first) mbar_inval(bars + 8 * i);
            mbar_init(bars + 8 * i, compute ? NCOMPUTE / 32 : (i == HELP || i == HELP + 1) ? 4 : 1);
        }
        fence_mbar_init();
    }
    __syncthreads();
}

namespace fs {
constexpr uint32_t B_W = 0, B_K = B_W + 2 * TILE_BF16, B_Q = B_K + 2 * TILE_BF16, B_T2 = B_Q + 2 * TILE_BF16, B_V = B_T2 + 2 * HALF_BF16,
                   B_A = B_V + 2 * HALF_BF16;           // [2] each: 144 KiB
constexpr uint32_t OFF_S = B_A + 2 * HALF_BF16;         // [2] state slice
constexpr uint32_t OFF_U = OFF_S + 2 * scn::SLICE;      // [2] Ue
constexpr uint32_t OFF_O = OFF_U + 2 * HALF_BF16;       // [2] o staged for the store
constexpr uint32_t BYTES = OFF_O + 2 * HALF_BF16;
// F0/E0: T2, V full / read; F1/E1: We; F2/E2: q; F3/E3: K, A (E3: o complete, too)
}  // namespace fs

__device__ __forceinline__ void scan_item(int item, const CUtensorMap &gm_q, const CUtensorMap &gm_k, const CUtensorMap &gm_v, const CUtensorMap &gm_o,
                                          const ChunkParams &p, uint8_t *sm, uint32_t base, uint32_t bars, bool first, uint32_t tmem,
                                          volatile int *abort_flag, bool &failed) {
    using namespace scn;
    using namespace fs;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nsl = p.dv / 64, sl = item % nsl, bh = item / nsl;     // (slices of a head side by side: they share tiles in L2)
    const SeqHead s = seq_head(p, bh / p.H, bh % p.H);
    const int NT = s.NT;
    const CUtensorMap &tm_q = s.vm ? s.vm[0] : gm_q, &tm_k = s.vm ? s.vm[1] : gm_k, &tm_v = s.vm ? s.vm[2] : gm_v, &tm_o = s.vm ? s.vm[3] : gm_o;
    uint8_t *rec0 = p.rec + (size_t)s.slot * p.L.bytes;
    auto bar = [&](int i) { return bars + 8u * i; };
    auto wait = [&](int i, uint32_t parity) {
        if (!failed && !mbar_wait_bounded(bar(i), parity, abort_flag)) { failed = true; *abort_flag = 1; }
    };
    scan_barriers(bars, first);
    auto scalars = [&](int n) { return reinterpret_cast<const float *>(rec0 + (size_t)n * p.L.bytes + p.L.sc); };
    auto end_of = [&](int n) { return *reinterpret_cast<const float2 *>(scalars(n) + SC_END); };

    if (warp == 8) {
        // ---------------- MMA issue ----------------
        const bool leader = elect_lane();
        constexpr uint32_t ID_KM = idesc_bf16(64, 64, 0, 1), ID_S = idesc_bf16(128, 64, 1, 1);
        const bool wide = p.dk > 64;
        auto t2v = [&](int n) {                    // acc = T2 V
            const int x = n & 1;
            const uint64_t a = desc_kmajor(base + B_T2 + x * HALF_BF16), b = desc_mnmajor(base + B_V + x * HALF_BF16, HALF_BF16);
            wait(F0 + x, (n >> 1) & 1);
            if (failed) return;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_ACC, a + kstep_kmajor(kk, 0), b + kstep_mnmajor(kk), ID_KM, kk > 0);
                tc_commit(bar(E0 + x));
            }
        };
        t2v(0);
        for (int n = 0; n < NT && !failed; ++n) {
            const int x = n & 1;
            const uint32_t ph = (n >> 1) & 1, acc_o = tmem + TM_O + 128 * x;
            const uint64_t mS = desc_mnmajor(base + OFF_S + x * SLICE, HALF_BF16), mU = desc_mnmajor(base + OFF_U + x * HALF_BF16, HALF_BF16),
                           kW = desc_kmajor(base + B_W + x * TILE_BF16), kQ = desc_kmajor(base + B_Q + x * TILE_BF16),
                           mK = desc_mnmajor(base + B_K + x * TILE_BF16, HALF_BF16), kA = desc_kmajor(base + B_A + x * HALF_BF16);
            // (the operands' waits come before the state's, while this warp has nothing else to do)
            wait(F1 + x, ph);
            wait(F2 + x, ph);
            wait(F3 + x, ph);
            if (n >= 2) wait(HELP + x, ((n - 2) >> 1) & 1);                   // o of chunk n-2 has been read out
            wait(SREADY, n & 1);
            if (failed) break;
            tc_fence_after();
            if (leader) {
                ksteps(wide, [&](int kk) {             // Ue = T2 V - We S
                    tc_mma_bf16(tmem + TM_ACC, kW + kstep_kmajor(kk, HALF_BF16), mS + kstep_mnmajor(kk), ID_KM, 1);
                });
                tc_commit(bar(C1));
                tc_commit(bar(E1 + x));                // (same event on a per-buffer barrier for the loads)
                ksteps(wide, [&](int kk) {             // q S
                    tc_mma_bf16(acc_o, kQ + kstep_kmajor(kk, HALF_BF16), mS + kstep_mnmajor(kk), ID_KM, kk > 0);
                });
                tc_commit(bar(E2 + x));
            }
            wait(UREADY + x, ph);
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_D, mK + kstep_mnmajor(kk), mU + kstep_mnmajor(kk), ID_S, kk > 0);    // K^T Ue
                tc_commit(bar(C2));
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(acc_o + 64, kA + kstep_kmajor(kk, 0), mU + kstep_mnmajor(kk), ID_KM, kk > 0);  // A Ue
                tc_commit(bar(E3 + x));
            }
            if (n + 1 < NT) t2v(n + 1);
        }
        if (leader) tc_commit(bar(DRAIN));
        mbar_wait_bounded(bar(DRAIN), 0, nullptr, 20000000ull);
    } else if (warp == 9) {
        // ---------------- loads ----------------
        const bool leader = elect_lane();
        auto load_t = [&](int n) {
            if (n >= NT || !leader) return;
            const int x = n & 1;
            const uint8_t *rec = rec0 + (size_t)n * p.L.bytes;
            mbar_expect_tx(bar(F0 + x), 2 * HALF_BF16);
            bulk_load(base + B_T2 + x * HALF_BF16, rec + p.L.t2, HALF_BF16, bar(F0 + x));
            tma_load_5d(base + B_V + x * HALF_BF16, &tm_v, 0, n * C, sl, s.h, s.b, bar(F0 + x));
        };
        auto load_w = [&](int n) {
            if (n >= NT || !leader) return;
            mbar_expect_tx(bar(F1 + (n & 1)), TILE_BF16);
            bulk_load(base + B_W + (n & 1) * TILE_BF16, rec0 + (size_t)n * p.L.bytes + p.L.w, TILE_BF16, bar(F1 + (n & 1)));
        };
        auto load_q = [&](int n) {
            if (n >= NT || !leader) return;
            mbar_expect_tx(bar(F2 + (n & 1)), TILE_BF16);
            tma_load_5d(base + B_Q + (n & 1) * TILE_BF16, &tm_q, 0, n * C, 0, s.h, s.b, bar(F2 + (n & 1)));
        };
        auto load_k = [&](int n) {
            if (n >= NT || !leader) return;
            const int x = n & 1;
            mbar_expect_tx(bar(F3 + x), TILE_BF16 + HALF_BF16);
            tma_load_5d(base + B_K + x * TILE_BF16, &tm_k, 0, n * C, 0, s.h, s.b, bar(F3 + x));
            bulk_load(base + B_A + x * HALF_BF16, rec0 + (size_t)n * p.L.bytes + p.L.a, HALF_BF16, bar(F3 + x));
        };
        auto prefetch = [&](int n) {               // (one slice of the head asks for the tiles both read)
            if (n >= NT || !leader) return;
            if (sl == 0) {
                bulk_prefetch_l2(rec0 + (size_t)n * p.L.bytes + p.L.w, PREP_BYTES);
                tma_prefetch_l2_5d(&tm_k, 0, n * C, 0, s.h, s.b);
                tma_prefetch_l2_5d(&tm_q, 0, n * C, 0, s.h, s.b);
            }
            tma_prefetch_l2_5d(&tm_v, 0, n * C, sl, s.h, s.b);
        };
        for (int n = 0; n < 2; ++n) {
            load_t(n);
            load_w(n);
            load_q(n);
            load_k(n);
        }
        prefetch(2);
        prefetch(3);
        wait(E0, 0);
        if (!failed) load_t(2);
        for (int n = 0; n < NT && !failed; ++n) {
            const int x = n & 1;
            const uint32_t ph = (n >> 1) & 1;
            prefetch(n + 4);
            wait(E1 + x, ph);
            if (failed) break;
            load_w(n + 2);
            wait(E2 + x, ph);
            if (failed) break;
            load_q(n + 2);
            wait(E3 + x, ph);
            if (failed) break;
            load_k(n + 2);
            if (n + 1 < NT) wait(E0 + (x ^ 1), ((n + 1) >> 1) & 1);
            if (failed) break;
            load_t(n + 3);
        }
        if (failed) let_copies_land();
    } else if (warp == 14) {
        // ---------------- stores: Ue and S of the chunk (training), o ----------------
        const bool leader = elect_lane();
        for (int n = 0; n < NT && !failed; ++n) {
            const int x = n & 1;
            const uint32_t ph = (n >> 1) & 1;
            if (p.save) {
                wait(UREADY + x, ph);                  // Ue of chunk n (and long before it S_n) stand in shared memory
                if (failed) break;
                if (leader) {
                    uint8_t *rec = rec0 + (size_t)n * p.L.bytes;
                    bulk_store(rec + p.L.s + sl * SLICE, base + OFF_S + x * SLICE, SLICE);
                    bulk_store(rec + p.L.u + sl * HALF_BF16, base + OFF_U + x * HALF_BF16, HALF_BF16);
                    bulk_commit();
                }
            }
            wait(HELP + x, ph);                        // o staged
            if (failed) break;
            if (leader) {
                if (p.write_o) tma_store_5d(&tm_o, base + OFF_O + x * HALF_BF16, 0, n * C, sl, s.h, s.b);
                bulk_commit();
                bulk_wait_read1();
                mbar_arrive(bar(SAVED + x));           // chunk n's Ue and S and chunk n-1's o have left their buffers
            }
        }
        if (p.save) {
            wait(FINAL, 0);
            if (!failed && leader) {
                bulk_store(rec0 + (size_t)NT * p.L.bytes + p.L.s + sl * SLICE, base + OFF_S + (NT & 1) * SLICE, SLICE);
                bulk_commit();
            }
        }
        if (leader) bulk_wait0();
    } else if (warp >= 10) {
        // ---------------- o = fq (q S) + A Ue ----------------
        const int qr = warp & 3, r = 16 * qr + (lane >> 2);
        float f0 = scalars(0)[SC_FQ * C + r], f1 = scalars(0)[SC_FQ * C + r + 8];
        for (int n = 0; n < NT; ++n) {
            const int x = n & 1;
            const float *nx = scalars(n + 1 < NT ? n + 1 : n) + SC_FQ * C;        // (a chunk ahead of their use)
            const float g0 = nx[r], g1 = nx[r + 8];
            wait(E3 + x, (n >> 1) & 1);
            if (n >= 2) wait(SAVED + (x ^ 1), ((n - 1) >> 1) & 1);                // o of chunk n-2 has left the staging buffer
            if (failed) break;
            tc_fence_after();
            float v[32], w[32];
            const uint32_t ta = tmem + ((uint32_t)(32 * qr) << 16) + TM_O + 128 * x;
            tmem_ld_frag8(ta, v);
            tmem_ld_frag8(ta + 64, w);
            tmem_wait_ld();
            uint8_t *dst = sm + OFF_O + x * HALF_BF16;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t off = frag_off(qr, lane, 0, i);
                *reinterpret_cast<uint32_t *>(dst + off) = pack_bf16(fmaf(f0, v[4 * i], w[4 * i]), fmaf(f0, v[4 * i + 1], w[4 * i + 1]));
                *reinterpret_cast<uint32_t *>(dst + off + 1024) =
                    pack_bf16(fmaf(f1, v[4 * i + 2], w[4 * i + 2]), fmaf(f1, v[4 * i + 3], w[4 * i + 3]));
            }
            fence_proxy_async();
            tc_fence_before();
            warp_arrive(bar(HELP + x), lane);
            f0 = g0;
            f1 = g1;
        }
    } else {
        // ---------------- compute warps: Ue, and the state in registers ----------------
        const int qr = warp & 3, ch = warp >> 2, row = 32 * qr + lane;
        const uint32_t tq = tmem + ((uint32_t)(32 * qr) << 16);
        float S[32];
        float2 e = end_of(0);
        {
            const float *src = state_row(p.h0, s.sbh, row, sl, p.dk, p.dv);
            load_state32(src ? src + 32 * ch : nullptr, S);
#pragma unroll
            for (int j = 0; j < 32; ++j) S[j] *= e.y;
        }
        store_slice(sm + OFF_S, row, ch, S);
        fence_proxy_async();
        warp_arrive(bar(SREADY), lane);
        for (int n = 0; n < NT; ++n) {
            const int x = n & 1;
            const float2 en = end_of(n + 1 < NT ? n + 1 : n);
            wait(C1, n & 1);
            tc_fence_after();
            {
                float v[16];
                tmem_ld_frag4(tq + TM_ACC + 32 * ch, v);
                tmem_wait_ld();
                frag16_to_tile(sm + OFF_U + x * HALF_BF16, qr, lane, 32 * ch, v);
            }
            fence_proxy_async();
            tc_fence_before();
            warp_arrive(bar(UREADY + x), lane);
            wait(C2, n & 1);
            tc_fence_after();
            {
                float v[32];
                tmem_ld32(tq + TM_D + 32 * ch, v);
                tmem_wait_ld();
                const float dec = n + 1 < NT ? e.x * en.y : e.x;     // (the final state leaves unscaled)
#pragma unroll
                for (int j = 0; j < 32; ++j) S[j] = dec * (S[j] + v[j]);
            }
            if (p.save && n >= 1) wait(SAVED + (x ^ 1), ((n - 1) >> 1) & 1);         // S_{n-1} and Ue of chunk n-1 have left their buffers
            store_slice(sm + OFF_S + (x ^ 1) * SLICE, row, ch, S);
            fence_proxy_async();
            tc_fence_before();
            if (n + 1 < NT) warp_arrive(bar(SREADY), lane);
            e = en;
        }
        warp_arrive(bar(FINAL), lane);
        if (float *dst = state_row(p.ht, s.sbh, row, sl, p.dk, p.dv)) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) *reinterpret_cast<float4 *>(dst + 32 * ch + j) = make_float4(S[j], S[j + 1], S[j + 2], S[j + 3]);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// reverse scan: dUe and dZ of every chunk
namespace bs {
constexpr uint32_t B_K = 0, B_Q = B_K + 2 * TILE_BF16, B_W = B_Q + 2 * TILE_BF16, B_S = B_W + 2 * TILE_BF16, B_A = B_S + 2 * scn::SLICE,
                   B_DO = B_A + 2 * HALF_BF16;          // [2] each: 160 KiB
constexpr uint32_t OFF_Z = B_DO + 2 * HALF_BF16;        // [2] dZ slice
constexpr uint32_t OFF_U = OFF_Z + 2 * scn::SLICE;      // [2] dUe
constexpr uint32_t BYTES = OFF_U + 2 * HALF_BF16;
// F0/E0: A, K full / read; F1/E1: dO, q; F2/E2: We; F3: S_{n+1} (read by the time dUe stands)
}  // namespace bs

__device__ __forceinline__ void bscan_item(int item, const CUtensorMap &gm_q, const CUtensorMap &gm_k, const CUtensorMap &gm_do, const ChunkParams &p,
                                           uint8_t *sm, uint32_t base, uint32_t bars, bool first, uint32_t tmem, volatile int *abort_flag,
                                           bool &failed) {
    using namespace scn;
    using namespace bs;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nsl = p.dv / 64, sl = item % nsl, bh = item / nsl;
    const SeqHead s = seq_head(p, bh / p.H, bh % p.H);
    const int NT = s.NT;
    const CUtensorMap &tm_q = s.vm ? s.vm[0] : gm_q, &tm_k = s.vm ? s.vm[1] : gm_k, &tm_do = s.vm ? s.vm[7] : gm_do;
    uint8_t *rec0 = p.rec + (size_t)s.slot * p.L.bytes;
    auto bar = [&](int i) { return bars + 8u * i; };
    auto wait = [&](int i, uint32_t parity) {
        if (!failed && !mbar_wait_bounded(bar(i), parity, abort_flag)) { failed = true; *abort_flag = 1; }
    };
    scan_barriers(bars, first);
    // chunks are visited in the order n = NT-1 ... 0; x = NT-1-n is the visit number that drives buffers and parities
    auto scalars = [&](int x) { return reinterpret_cast<const float *>(rec0 + (size_t)(NT - 1 - x) * p.L.bytes + p.L.sc); };
    auto end_of = [&](int x) { return *reinterpret_cast<const float2 *>(scalars(x) + SC_END); };

    if (warp == 8) {
        // ---------------- MMA issue ----------------
        const bool leader = elect_lane();
        constexpr uint32_t ID_MM = idesc_bf16(64, 64, 1, 1), ID_KM = idesc_bf16(64, 64, 0, 1), ID_S = idesc_bf16(128, 64, 1, 1);
        const bool wide = p.dk > 64;
        auto atdo = [&](int x) {                   // acc = A^T dO
            const int y = x & 1;
            const uint64_t a = desc_mnmajor(base + B_A + y * HALF_BF16, HALF_BF16), b = desc_mnmajor(base + B_DO + y * HALF_BF16, HALF_BF16);
            wait(F0 + y, (x >> 1) & 1);
            wait(F1 + y, (x >> 1) & 1);
            if (failed) return;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_ACC, a + kstep_mnmajor(kk), b + kstep_mnmajor(kk), ID_MM, kk > 0);
            }
        };
        atdo(0);
        for (int x = 0; x < NT && !failed; ++x) {
            const int y = x & 1;
            const uint32_t ph = (x >> 1) & 1;
            const uint64_t mZ = desc_mnmajor(base + OFF_Z + y * SLICE, HALF_BF16), mU = desc_mnmajor(base + OFF_U + y * HALF_BF16, HALF_BF16),
                           kK = desc_kmajor(base + B_K + y * TILE_BF16), mQ = desc_mnmajor(base + B_Q + y * TILE_BF16, HALF_BF16),
                           mDO = desc_mnmajor(base + B_DO + y * HALF_BF16, HALF_BF16), mW = desc_mnmajor(base + B_W + y * TILE_BF16, HALF_BF16);
            wait(F2 + y, ph);
            wait(SREADY, x & 1);
            if (failed) break;
            tc_fence_after();
            if (leader) {
                ksteps(wide, [&](int kk) {             // dUe = A^T dO + K dZ
                    tc_mma_bf16(tmem + TM_ACC, kK + kstep_kmajor(kk, HALF_BF16), mZ + kstep_mnmajor(kk), ID_KM, 1);
                });
                tc_commit(bar(C1));
                tc_commit(bar(E0 + y));                // (same event on a per-buffer barrier for the loads)
            }
            wait(HELP + y, ph);                        // Qg stands in place of q
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_D, mQ + kstep_mnmajor(kk), mDO + kstep_mnmajor(kk), ID_S, kk > 0);   // Qg^T dO
                tc_commit(bar(E1 + y));
            }
            wait(UREADY + y, ph);
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_D, mW + kstep_mnmajor(kk), mU + kstep_mnmajor(kk), ID_S, 1);         // - We^T dUe
                tc_commit(bar(C2));
                tc_commit(bar(E2 + y));
            }
            if (x + 1 < NT) atdo(x + 1);
        }
        if (leader) tc_commit(bar(DRAIN));
        mbar_wait_bounded(bar(DRAIN), 0, nullptr, 20000000ull);
    } else if (warp == 9) {
        // ---------------- loads ----------------
        const bool leader = elect_lane();
        auto load_ak = [&](int x) {
            if (x >= NT || !leader) return;
            const int y = x & 1, n = NT - 1 - x;
            mbar_expect_tx(bar(F0 + y), HALF_BF16 + TILE_BF16);
            bulk_load(base + B_A + y * HALF_BF16, rec0 + (size_t)n * p.L.bytes + p.L.a, HALF_BF16, bar(F0 + y));
            tma_load_5d(base + B_K + y * TILE_BF16, &tm_k, 0, n * C, 0, s.h, s.b, bar(F0 + y));
        };
        auto load_dq = [&](int x) {
            if (x >= NT || !leader) return;
            const int y = x & 1, n = NT - 1 - x;
            mbar_expect_tx(bar(F1 + y), HALF_BF16 + TILE_BF16);
            tma_load_5d(base + B_DO + y * HALF_BF16, &tm_do, 0, n * C, sl, s.h, s.b, bar(F1 + y));
            tma_load_5d(base + B_Q + y * TILE_BF16, &tm_q, 0, n * C, 0, s.h, s.b, bar(F1 + y));
        };
        auto load_w = [&](int x) {
            if (x >= NT || !leader) return;
            mbar_expect_tx(bar(F2 + (x & 1)), TILE_BF16);
            bulk_load(base + B_W + (x & 1) * TILE_BF16, rec0 + (size_t)(NT - 1 - x) * p.L.bytes + p.L.w, TILE_BF16, bar(F2 + (x & 1)));
        };
        auto load_s = [&](int x) {
            if (x >= NT || !leader) return;
            mbar_expect_tx(bar(F3 + (x & 1)), SLICE);
            bulk_load(base + B_S + (x & 1) * SLICE, rec0 + (size_t)(NT - x) * p.L.bytes + p.L.s + sl * SLICE, SLICE, bar(F3 + (x & 1)));   // S_{n+1}
        };
        auto prefetch = [&](int x) {
            if (x >= NT || !leader) return;
            const int n = NT - 1 - x;
            const uint8_t *rec = rec0 + (size_t)n * p.L.bytes;
            if (sl == 0) {
                tma_prefetch_l2_5d(&tm_k, 0, n * C, 0, s.h, s.b);
                tma_prefetch_l2_5d(&tm_q, 0, n * C, 0, s.h, s.b);
                bulk_prefetch_l2(rec + p.L.w, TILE_BF16 + HALF_BF16 + SC_LOAD);
            }
            tma_prefetch_l2_5d(&tm_do, 0, n * C, sl, s.h, s.b);
            bulk_prefetch_l2(rec + p.L.bytes + p.L.s + sl * SLICE, SLICE);
        };
        for (int x = 0; x < 2; ++x) {
            load_ak(x);
            load_dq(x);
            load_w(x);
            load_s(x);
        }
        prefetch(2);
        prefetch(3);
        for (int x = 0; x < NT && !failed; ++x) {
            const int y = x & 1;
            const uint32_t ph = (x >> 1) & 1;
            prefetch(x + 4);
            wait(E0 + y, ph);
            if (failed) break;
            load_ak(x + 2);
            wait(E1 + y, ph);
            if (failed) break;
            load_dq(x + 2);
            wait(UREADY + y, ph);
            if (failed) break;
            load_s(x + 2);
            wait(E2 + y, ph);
            if (failed) break;
            load_w(x + 2);
        }
        if (failed) let_copies_land();
    } else if (warp == 14) {
        // ---------------- stores ----------------
        const bool leader = elect_lane();
        for (int x = 0; x < NT && !failed; ++x) {
            const int y = x & 1;
            wait(UREADY + y, (x >> 1) & 1);            // dUe (and long before it dZ) stand in shared memory
            if (failed) break;
            if (leader) {
                uint8_t *rec = rec0 + (size_t)(NT - 1 - x) * p.L.bytes;
                bulk_store(rec + p.L.dz + sl * SLICE, base + OFF_Z + y * SLICE, SLICE);
                bulk_store(rec + p.L.du + sl * HALF_BF16, base + OFF_U + y * HALF_BF16, HALF_BF16);
                bulk_commit();
                bulk_wait_read0();
                mbar_arrive(bar(SAVED + y));
            }
        }
        if (leader) bulk_wait0();
    } else if (warp >= 10) {
        // ---------------- Qg = fq q, in place ----------------
        const int t = tid - (NCOMPUTE + 64), r = t >> 1;
        float f = scalars(0)[SC_FQ * C + r];
        for (int x = 0; x < NT; ++x) {
            const float fn = scalars(x + 1 < NT ? x + 1 : x)[SC_FQ * C + r];
            wait(F1 + (x & 1), (x >> 1) & 1);
            if (failed) break;
            uint8_t *tile = sm + B_Q + (x & 1) * TILE_BF16;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                uint4 *w4 = reinterpret_cast<uint4 *>(tile + (c >> 2) * HALF_BF16 + swz(r, 2 * (c & 3) + (t & 1)));
                uint4 v = *w4;
                uint32_t *w = reinterpret_cast<uint32_t *>(&v);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 y = unpack_bf16(w[e]);
                    w[e] = pack_bf16(f * y.x, f * y.y);
                }
                *w4 = v;
            }
            fence_proxy_async();
            warp_arrive(bar(HELP + (x & 1)), lane);
            f = fn;
        }
    } else {
        // ---------------- compute warps: the state gradient in registers, dUe ----------------
        const int qr = warp & 3, ch = warp >> 2, row = 32 * qr + lane;
        const uint32_t tq = tmem + ((uint32_t)(32 * qr) << 16);
        float S[32];                                   // dS of the state after the current chunk
        {
            const float *src = state_row(p.dht, s.sbh, row, sl, p.dk, p.dv);
            load_state32(src ? src + 32 * ch : nullptr, S);
        }
        float2 e = end_of(0);
        float d = 1.f;                                 // 2^-k of the chunk visited before (the gradient of the final state comes unscaled)
        for (int x = 0; x < NT; ++x) {
            const int y = x & 1;
            const uint32_t ph = (x >> 1) & 1;
            if (x >= 2) wait(SAVED + y, ((x - 2) >> 1) & 1);            // dZ and dUe of visit x-2 have left their buffers
            float part = 0.f;
            {   // dZ = e^{b_last} dS' as an operand; <dS', S'> beside the first product
                float z[32];
                const float dec = e.x * d;             // (here and not where e is read: the read is under way until now)
#pragma unroll
                for (int j = 0; j < 32; ++j) z[j] = dec * S[j];
                store_slice(sm + OFF_Z + y * SLICE, row, ch, z);
                fence_proxy_async();
                tc_fence_before();
                warp_arrive(bar(SREADY), lane);
                wait(F3 + y, ph);
                const uint8_t *img = sm + B_S + y * SLICE;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint4 a = *reinterpret_cast<const uint4 *>(img + swz(row, 4 * ch + c));
                    const uint32_t *aw = reinterpret_cast<const uint32_t *>(&a);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 w = unpack_bf16(aw[q]);
                        part = fmaf(S[8 * c + 2 * q], w.x, part);
                        part = fmaf(S[8 * c + 2 * q + 1], w.y, part);
                    }
                }
#pragma unroll
                for (int j = 0; j < 32; ++j) S[j] = z[j];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            if (lane == 0) const_cast<float *>(scalars(x))[SC_DOT + 8 * sl + warp] = part;
            d = e.y;
            e = end_of(x + 1 < NT ? x + 1 : x);
            wait(C1, x & 1);
            tc_fence_after();
            {
                float v[16];
                tmem_ld_frag4(tq + TM_ACC + 32 * ch, v);
                tmem_wait_ld();
                frag16_to_tile(sm + OFF_U + y * HALF_BF16, qr, lane, 32 * ch, v);
            }
            fence_proxy_async();
            tc_fence_before();
            warp_arrive(bar(UREADY + y), lane);
            wait(C2, x & 1);
            tc_fence_after();
            {
                float v[32];
                tmem_ld32(tq + TM_D + 32 * ch, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) S[j] += v[j];
            }
        }
        if (float *dst = state_row(p.dh0, s.sbh, row, sl, p.dk, p.dv)) {
#pragma unroll
            for (int j = 0; j < 32; j += 4)
                *reinterpret_cast<float4 *>(dst + 32 * ch + j) = make_float4(d * S[j], d * S[j + 1], d * S[j + 2], d * S[j + 3]);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// every chunk: the input gradients.  Warps 0..7 compute, 8 MMA issue, 9 copies; a chunk's tiles are reloaded for the
// CTA's next chunk as soon as their last reader is done.
namespace bg {
constexpr uint32_t OFF_Q = 0;                           // q -> Qg -> dq staged
constexpr uint32_t OFF_K = OFF_Q + TILE_BF16;           // k -> dk staged
constexpr uint32_t OFF_V = OFF_K + TILE_BF16;           // v -> dv staged
constexpr uint32_t OFF_DO = OFF_V + TILE_BF16;
constexpr uint32_t OFF_S = OFF_DO + TILE_BF16;
constexpr uint32_t OFF_DZ = OFF_S + STATE_BF16;
constexpr uint32_t OFF_U = OFF_DZ + STATE_BF16;
constexpr uint32_t OFF_X = OFF_U + TILE_BF16;           // dUe
constexpr uint32_t OFF_TE = OFF_X + TILE_BF16;
constexpr uint32_t OFF_DR = OFF_TE + HALF_BF16;         // bf16 dR
constexpr uint32_t OFF_DA = OFF_DR + TILE_BF16;         // bf16 dA
constexpr uint32_t OFF_P = OFF_DA + HALF_BF16;          // bf16 P
constexpr uint32_t OFF_M = OFF_P + HALF_BF16;           // bf16 -beta Gam P
constexpr uint32_t OFF_SC = OFF_M + HALF_BF16;          // [2] scalars of the chunk
constexpr uint32_t OFF_PART = OFF_SC + 2 * SC_BYTES;    // [2][4][2][64]: dR.v, Qg.aq, k.kd, k.Y per column half
constexpr uint32_t BYTES = OFF_PART + 2 * 4 * 2 * C * 4;
enum Bar { FA = 0, FV, FQ, FK, C1, C1B, C2, C3, E1R, E2R, DQS, DKS, TFREE, DRAIN, NBAR };
constexpr uint32_t TM_R = 0 /* dR, then Y */, TM_A = 128 /* dA, then P */, TM_Q = 192, TM_K = 320;
}  // namespace bg

__device__ __forceinline__ void bgrad_chunks(const CUtensorMap &gm_q, const CUtensorMap &gm_k, const CUtensorMap &gm_v, const CUtensorMap &gm_do,
                                             const CUtensorMap &gm_dq, const CUtensorMap &gm_dk, const CUtensorMap &gm_dv, const ChunkParams &p,
                                             uint8_t *sm, uint32_t base, uint32_t bars, uint32_t tmem, volatile int *abort_flag, bool &failed) {
    using namespace bg;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto bar = [&](int i) { return bars + 8u * i; };
    auto wait = [&](int i, uint32_t parity) {
        if (!failed && !mbar_wait_bounded(bar(i), parity, abort_flag)) { failed = true; *abort_flag = 1; }
    };
    const int nh = p.dv / 64, step = (int)gridDim.x;
    const bool wide = nh > 1;

    if (warp == 8) {
        // ---------------- MMA issue ----------------
        const bool leader = elect_lane();
        const uint32_t nbits = (uint32_t)(p.dv >> 3) << 17;       // N = d_v in the instruction descriptor
        constexpr uint32_t NMASK = ~(0x3Fu << 17);
        const uint32_t ID_DR = (idesc_bf16(64, 128, 1, 1) & NMASK) | nbits;
        constexpr uint32_t ID_64 = idesc_bf16(64, 64, 0, 0), ID_KK = idesc_bf16(64, 128, 0, 0), ID_KM = idesc_bf16(64, 128, 0, 1),
                           ID_MM = idesc_bf16(64, 128, 1, 1);
        const uint64_t mTE = desc_mnmajor(base + OFF_TE, HALF_BF16), mX = desc_mnmajor(base + OFF_X, HALF_BF16),
                       kDO = desc_kmajor(base + OFF_DO), kU = desc_kmajor(base + OFF_U), kS = desc_kmajor(base + OFF_S),
                       kDZ = desc_kmajor(base + OFF_DZ), kDR = desc_kmajor(base + OFF_DR), kDA = desc_kmajor(base + OFF_DA),
                       mDA = desc_mnmajor(base + OFF_DA, HALF_BF16), kP = desc_kmajor(base + OFF_P), mM = desc_mnmajor(base + OFF_M, HALF_BF16),
                       mK = desc_mnmajor(base + OFF_K, HALF_BF16), mQ = desc_mnmajor(base + OFF_Q, HALF_BF16);
        SeqHead s;
        int it = 0;
        for (int slot = next_chunk(p, blockIdx.x, step, s); slot < p.slots && !failed; slot = next_chunk(p, slot + step, step, s), ++it) {
            const uint32_t par = it & 1;
            wait(FA, par);
            if (it > 0) wait(TFREE, par ^ 1);                     // the accumulators of the previous chunk have been read
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_R, mTE + kstep_mnmajor(kk), mX + kstep_mnmajor(kk), ID_DR, kk > 0);   // dR = Te^T X, but for the diagonal
                ksteps(wide, [&](int kk) {                        // dA = dO Ue^T
                    tc_mma_bf16(tmem + TM_A, kDO + kstep_kmajor(kk, HALF_BF16), kU + kstep_kmajor(kk, HALF_BF16), ID_64, kk > 0);
                });
                tc_commit(bar(C1));
                ksteps(wide, [&](int kk) {                        // aq = dO S^T
                    tc_mma_bf16(tmem + TM_Q, kDO + kstep_kmajor(kk, HALF_BF16), kS + kstep_kmajor(kk, STATE_HALF), ID_KK, kk > 0);
                });
                ksteps(wide, [&](int kk) {                        // kd = Ue dZ^T
                    tc_mma_bf16(tmem + TM_K, kU + kstep_kmajor(kk, HALF_BF16), kDZ + kstep_kmajor(kk, STATE_HALF), ID_KK, kk > 0);
                });
                tc_commit(bar(C1B));
            }
            wait(FK, par);
            wait(E1R, par);                                       // dR, dA, Qg in place
            if (failed) break;
            tc_fence_after();
            if (leader) {
                ksteps(wide, [&](int kk) {                        // P = dR Ue^T
                    tc_mma_bf16(tmem + TM_A, kDR + kstep_kmajor(kk, HALF_BF16), kU + kstep_kmajor(kk, HALF_BF16), ID_64, kk > 0);
                });
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_Q, kDA + kstep_kmajor(kk, 0), mK + kstep_mnmajor(kk), ID_KM, 1);      // aq += dA K
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_K, mDA + kstep_mnmajor(kk), mQ + kstep_mnmajor(kk), ID_MM, 1);        // kd += dA^T Qg
                ksteps(wide, [&](int kk) {                        // Y = dR S^T
                    tc_mma_bf16(tmem + TM_R, kDR + kstep_kmajor(kk, HALF_BF16), kS + kstep_kmajor(kk, STATE_HALF), ID_KK, kk > 0);
                });
                tc_commit(bar(C2));
            }
            wait(E2R, par);
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_R, kP + kstep_kmajor(kk, 0), mK + kstep_mnmajor(kk), ID_KM, 1);       // Y += P K
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) tc_mma_bf16(tmem + TM_K, mM + kstep_mnmajor(kk), mK + kstep_mnmajor(kk), ID_MM, 1);         // kd += M^T K
                tc_commit(bar(C3));
            }
        }
        if (leader) tc_commit(bar(DRAIN));
        mbar_wait_bounded(bar(DRAIN), 0, nullptr, 20000000ull);
    } else if (warp == 9) {
        // ---------------- loads and stores ----------------
        const bool leader = elect_lane();
        auto mp = [&](const SeqHead &s, int i, const CUtensorMap *g) { return s.vm ? s.vm + i : g; };
        auto load_a1 = [&](const SeqHead &s, int slot) {           // what the first products read
            if (!leader) return;
            const int n = slot - s.slot;
            const uint8_t *rec = p.rec + (size_t)slot * p.L.bytes;
            mbar_expect_tx(bar(FA), HALF_BF16 + TILE_BF16 + nh * (HALF_BF16 + HALF_BF16 + STATE_HALF + STATE_HALF));
            bulk_load(base + OFF_TE, rec + p.L.te, HALF_BF16, bar(FA));
            tma_load_5d(base + OFF_DO, mp(s, 3, &gm_do), 0, n * C, 0, s.h, s.b, bar(FA));
            bulk_load(base + OFF_DZ, rec + p.L.dz, nh * STATE_HALF, bar(FA));
        };
        auto load_x = [&](int slot) {                              // (X: the compute warps read it, too)
            if (leader) bulk_load(base + OFF_X, p.rec + (size_t)slot * p.L.bytes + p.L.du, nh * HALF_BF16, bar(FA));
        };
        auto load_a2 = [&](int slot) {                             // ... and what the later ones read as well
            if (!leader) return;
            const uint8_t *rec = p.rec + (size_t)slot * p.L.bytes;
            bulk_load(base + OFF_U, rec + p.L.u, nh * HALF_BF16, bar(FA));
            bulk_load(base + OFF_S, rec + p.L.s, nh * STATE_HALF, bar(FA));
        };
        auto load_v = [&](const SeqHead &s, int slot, int it) {
            if (!leader) return;
            mbar_expect_tx(bar(FV), TILE_BF16 + SC_BYTES);
            bulk_load(base + OFF_SC + (it & 1) * SC_BYTES, p.rec + (size_t)slot * p.L.bytes + p.L.sc, SC_BYTES, bar(FV));
            tma_load_5d(base + OFF_V, mp(s, 2, &gm_v), 0, (slot - s.slot) * C, 0, s.h, s.b, bar(FV));
        };
        auto load_q = [&](const SeqHead &s, int slot) {
            if (!leader) return;
            mbar_expect_tx(bar(FQ), TILE_BF16);
            tma_load_5d(base + OFF_Q, mp(s, 0, &gm_q), 0, (slot - s.slot) * C, 0, s.h, s.b, bar(FQ));
        };
        auto load_k = [&](const SeqHead &s, int slot) {
            if (!leader) return;
            mbar_expect_tx(bar(FK), TILE_BF16);
            tma_load_5d(base + OFF_K, mp(s, 1, &gm_k), 0, (slot - s.slot) * C, 0, s.h, s.b, bar(FK));
        };
        auto store = [&](const CUtensorMap *map, uint32_t off, const SeqHead &s, int n) {
            if (!leader) return;
            tma_store_5d(map, base + off, 0, n * C, 0, s.h, s.b);
            bulk_commit();
        };
        SeqHead s, sn;
        int slot = next_chunk(p, blockIdx.x, step, s);
        if (slot < p.slots) {
            load_a1(s, slot);
            load_x(slot);
            load_a2(slot);
            load_v(s, slot, 0);
            load_k(s, slot);
            load_q(s, slot);
        }
        for (int it = 0; slot < p.slots && !failed; ++it) {
            const uint32_t par = it & 1;
            const int n = slot - s.slot;
            const int sl2 = next_chunk(p, slot + step, step, sn);
            const bool more = sl2 < p.slots;
            if (more && leader) {   // q, k, v and the second group of the next chunk load late: have them in L2 by then
                const int n2 = sl2 - sn.slot;
                const uint8_t *rec = p.rec + (size_t)sl2 * p.L.bytes;
                bulk_prefetch_l2(rec + p.L.s, nh * STATE_HALF);
                bulk_prefetch_l2(rec + p.L.u, nh * HALF_BF16);
                bulk_prefetch_l2(rec + p.L.du, nh * HALF_BF16);
                tma_prefetch_l2_5d(mp(sn, 2, &gm_v), 0, n2 * C, 0, sn.h, sn.b);
                tma_prefetch_l2_5d(mp(sn, 0, &gm_q), 0, n2 * C, 0, sn.h, sn.b);
                tma_prefetch_l2_5d(mp(sn, 1, &gm_k), 0, n2 * C, 0, sn.h, sn.b);
            }
            wait(C1B, par);
            if (failed) break;
            if (more) load_a1(sn, sl2);
            wait(E1R, par);                        // dv staged over v
            if (failed) break;
            store(mp(s, 6, &gm_dv), OFF_V, s, n);
            if (more) load_x(sl2);
            wait(C2, par);
            if (failed) break;
            if (more) load_a2(sl2);
            if (leader) bulk_wait_read0();
            if (more) load_v(sn, sl2, it + 1);
            wait(DQS, par);                        // dq staged over q
            if (failed) break;
            store(mp(s, 4, &gm_dq), OFF_Q, s, n);
            if (leader) bulk_wait_read0();
            if (more) load_q(sn, sl2);
            wait(DKS, par);                        // dk staged over k
            if (failed) break;
            store(mp(s, 5, &gm_dk), OFF_K, s, n);
            if (leader) bulk_wait_read0();
            if (more) load_k(sn, sl2);
            slot = sl2;
            s = sn;
        }
        if (leader) bulk_wait0();
        if (failed) let_copies_land();
    } else if (warp < 8) {
        // ---------------- compute warps ----------------
        const int qr = warp & 3, ch = warp >> 2, r = 16 * qr + (lane >> 2);
        const uint32_t tq = tmem + ((uint32_t)(32 * qr) << 16);
        // this thread's words of a tile: rows r, r + 8 of its eight column blocks
        auto read_tile = [&](uint32_t tile, uint32_t (&w)[16]) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t off = tile + frag_off(qr, lane, 64 * ch, i);
                w[2 * i] = *reinterpret_cast<const uint32_t *>(sm + off);
                w[2 * i + 1] = *reinterpret_cast<const uint32_t *>(sm + off + 1024);
            }
        };
        // row sums of (fragment * tile) over this warp's 64 columns; lanes of a quad share a row
        auto quad_store = [&](float a0, float a1, float *dst) {
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                a0 += __shfl_xor_sync(0xffffffffu, a0, o);
                a1 += __shfl_xor_sync(0xffffffffu, a1, o);
            }
            if ((lane & 3) == 0) { dst[ch * C + r] = a0; dst[ch * C + r + 8] = a1; }
        };
        SeqHead s;
        int it = 0;
        for (int slot = next_chunk(p, blockIdx.x, step, s); slot < p.slots; slot = next_chunk(p, slot + step, step, s), ++it) {
            const uint32_t par = it & 1;
            const float *sc = reinterpret_cast<const float *>(sm + OFF_SC + par * SC_BYTES);
            float *part = reinterpret_cast<float *>(sm + OFF_PART) + par * 8 * C;
            // ---- Qg; dR, dv; dA ----
            wait(FV, par);
            const float fq0 = sc[SC_FQ * C + r], fq1 = sc[SC_FQ * C + r + 8], bg0 = sc[SC_BG * C + r], bg1 = sc[SC_BG * C + r + 8];
            wait(FQ, par);
            uint32_t tw[16];                           // (read whole, then written: no read is moved above a write of these tiles)
            read_tile(OFF_Q, tw);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t off = frag_off(qr, lane, 64 * ch, i);
                const float2 y0 = unpack_bf16(tw[2 * i]), y1 = unpack_bf16(tw[2 * i + 1]);
                *reinterpret_cast<uint32_t *>(sm + OFF_Q + off) = pack_bf16(fq0 * y0.x, fq0 * y0.y);
                *reinterpret_cast<uint32_t *>(sm + OFF_Q + off + 1024) = pack_bf16(fq1 * y1.x, fq1 * y1.y);
            }
            read_tile(OFF_V, tw);
            uint32_t xw[16];                           // X: T's unit diagonal is added to dR here, in fp32
            wait(FA, par);
            if (ch < nh) read_tile(OFF_X, xw);
            wait(C1, par);
            tc_fence_after();
            {
                float a0 = 0.f, a1 = 0.f;
                if (ch < nh) {
                    const float fv0 = sc[SC_FV * C + r], fv1 = sc[SC_FV * C + r + 8], ig0 = sc[SC_IG * C + r], ig1 = sc[SC_IG * C + r + 8];
                    float v[32];
                    tmem_ld_frag8(tq + TM_R + 64 * ch, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t off = frag_off(qr, lane, 64 * ch, i);
                        uint32_t *x0 = reinterpret_cast<uint32_t *>(sm + OFF_V + off), *x1 = reinterpret_cast<uint32_t *>(sm + OFF_V + off + 1024);
                        const float2 y0 = unpack_bf16(tw[2 * i]), y1 = unpack_bf16(tw[2 * i + 1]), x2 = unpack_bf16(xw[2 * i]), x3 = unpack_bf16(xw[2 * i + 1]);
                        v[4 * i] = fmaf(ig0, x2.x, v[4 * i]);         v[4 * i + 1] = fmaf(ig0, x2.y, v[4 * i + 1]);
                        v[4 * i + 2] = fmaf(ig1, x3.x, v[4 * i + 2]); v[4 * i + 3] = fmaf(ig1, x3.y, v[4 * i + 3]);
                        a0 = fmaf(v[4 * i], y0.x, a0);     a0 = fmaf(v[4 * i + 1], y0.y, a0);
                        a1 = fmaf(v[4 * i + 2], y1.x, a1); a1 = fmaf(v[4 * i + 3], y1.y, a1);
                        *reinterpret_cast<uint32_t *>(sm + OFF_DR + off) = pack_bf16(v[4 * i], v[4 * i + 1]);
                        *reinterpret_cast<uint32_t *>(sm + OFF_DR + off + 1024) = pack_bf16(v[4 * i + 2], v[4 * i + 3]);
                        *x0 = pack_bf16(fv0 * v[4 * i], fv0 * v[4 * i + 1]);
                        *x1 = pack_bf16(fv1 * v[4 * i + 2], fv1 * v[4 * i + 3]);
                    }
                }
                quad_store(a0, a1, part);
                float w[16];
                tmem_ld_frag4(tq + TM_A + 32 * ch, w);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int j = 32 * ch + 8 * i + 2 * (lane & 3);
                    const uint32_t off = frag_off(qr, lane, 32 * ch, i);
                    *reinterpret_cast<uint32_t *>(sm + OFF_DA + off) = pack_bf16(j <= r ? w[4 * i] : 0.f, j + 1 <= r ? w[4 * i + 1] : 0.f);
                    *reinterpret_cast<uint32_t *>(sm + OFF_DA + off + 1024) =
                        pack_bf16(j <= r + 8 ? w[4 * i + 2] : 0.f, j + 1 <= r + 8 ? w[4 * i + 3] : 0.f);
                }
            }
            fence_proxy_async();
            tc_fence_before();
            warp_arrive(bar(E1R), lane);
            // ---- P and M; dq ----
            wait(C2, par);
            tc_fence_after();
            {
                float w[16];
                tmem_ld_frag4(tq + TM_A + 32 * ch, w);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int j = 32 * ch + 8 * i + 2 * (lane & 3);
                    const uint32_t off = frag_off(qr, lane, 32 * ch, i);
                    const float x00 = j < r ? w[4 * i] : 0.f, x01 = j + 1 < r ? w[4 * i + 1] : 0.f,
                                x10 = j < r + 8 ? w[4 * i + 2] : 0.f, x11 = j + 1 < r + 8 ? w[4 * i + 3] : 0.f;
                    *reinterpret_cast<uint32_t *>(sm + OFF_P + off) = pack_bf16(x00, x01);
                    *reinterpret_cast<uint32_t *>(sm + OFF_P + off + 1024) = pack_bf16(x10, x11);
                    *reinterpret_cast<uint32_t *>(sm + OFF_M + off) = pack_bf16(-bg0 * x00, -bg0 * x01);
                    *reinterpret_cast<uint32_t *>(sm + OFF_M + off + 1024) = pack_bf16(-bg1 * x10, -bg1 * x11);
                }
                fence_proxy_async();
                tc_fence_before();
                warp_arrive(bar(E2R), lane);
                float v[32], a0 = 0.f, a1 = 0.f;
                tmem_ld_frag8(tq + TM_Q + 64 * ch, v);
                read_tile(OFF_Q, tw);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t off = frag_off(qr, lane, 64 * ch, i);
                    uint32_t *x0 = reinterpret_cast<uint32_t *>(sm + OFF_Q + off), *x1 = reinterpret_cast<uint32_t *>(sm + OFF_Q + off + 1024);
                    const float2 y0 = unpack_bf16(tw[2 * i]), y1 = unpack_bf16(tw[2 * i + 1]);
                    a0 = fmaf(v[4 * i], y0.x, a0);     a0 = fmaf(v[4 * i + 1], y0.y, a0);
                    a1 = fmaf(v[4 * i + 2], y1.x, a1); a1 = fmaf(v[4 * i + 3], y1.y, a1);
                    *x0 = pack_bf16(fq0 * v[4 * i], fq0 * v[4 * i + 1]);
                    *x1 = pack_bf16(fq1 * v[4 * i + 2], fq1 * v[4 * i + 3]);
                }
                quad_store(a0, a1, part + 2 * C);
            }
            fence_proxy_async();
            warp_arrive(bar(DQS), lane);
            // ---- dk ----
            wait(FK, par);
            wait(C3, par);
            tc_fence_after();
            {
                float v[32], y[32], a0 = 0.f, a1 = 0.f, e0 = 0.f, e1 = 0.f;
                tmem_ld_frag8(tq + TM_K + 64 * ch, v);
                tmem_ld_frag8(tq + TM_R + 64 * ch, y);
                read_tile(OFF_K, tw);
                tmem_wait_ld();
                tc_fence_before();
                warp_arrive(bar(TFREE), lane);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t off = frag_off(qr, lane, 64 * ch, i);
                    uint32_t *x0 = reinterpret_cast<uint32_t *>(sm + OFF_K + off), *x1 = reinterpret_cast<uint32_t *>(sm + OFF_K + off + 1024);
                    const float2 k0 = unpack_bf16(tw[2 * i]), k1 = unpack_bf16(tw[2 * i + 1]);
                    a0 = fmaf(v[4 * i], k0.x, a0);     a0 = fmaf(v[4 * i + 1], k0.y, a0);
                    a1 = fmaf(v[4 * i + 2], k1.x, a1); a1 = fmaf(v[4 * i + 3], k1.y, a1);
                    e0 = fmaf(y[4 * i], k0.x, e0);     e0 = fmaf(y[4 * i + 1], k0.y, e0);
                    e1 = fmaf(y[4 * i + 2], k1.x, e1); e1 = fmaf(y[4 * i + 3], k1.y, e1);
                    *x0 = pack_bf16(fmaf(-bg0, y[4 * i], v[4 * i]), fmaf(-bg0, y[4 * i + 1], v[4 * i + 1]));
                    *x1 = pack_bf16(fmaf(-bg1, y[4 * i + 2], v[4 * i + 2]), fmaf(-bg1, y[4 * i + 3], v[4 * i + 3]));
                }
                quad_store(a0, a1, part + 4 * C);
                quad_store(e0, e1, part + 6 * C);
            }
            fence_proxy_async();
            warp_arrive(bar(DKS), lane);
            named_bar_sync(1, NCOMPUTE);               // the partial row sums are complete
            if (warp == 0) {      // per-token scalars; lane l owns tokens 2l, 2l+1
                float db[2], dbt[2], pqv[2], pkv[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i = 2 * lane + e;
                    const float pv = part[i] + part[C + i], qd = part[2 * C + i] + part[3 * C + i], kd = part[4 * C + i] + part[5 * C + i],
                                ky = part[6 * C + i] + part[7 * C + i];
                    db[e] = qd - kd - sc[SC_BG * C + i] * ky;
                    dbt[e] = sc[SC_GK * C + i] * pv - sc[SC_GAM * C + i] * ky;
                    pqv[e] = qd;
                    pkv[e] = sc[SC_FV * C + i] * pv;
                }
                float dot = lane < 8 * nh ? sc[SC_DOT + lane] : 0.f;
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                dot = __shfl_sync(0xffffffffu, dot, 0);
                if (lane == 31) db[1] += dot;                             // <dS', S'> enters at the last token
                float suf = db[0] + db[1];                                // inclusive suffix sum over the lanes
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float t = __shfl_down_sync(0xffffffffu, suf, o);
                    if (lane + o < 32) suf += t;
                }
                const int n = slot - s.slot, cn = min(C, s.T - n * C);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i = 2 * lane + e;
                    if (i < cn) {
                        const size_t o = (s.tok + (size_t)n * C + i) * p.H + s.h;
                        p.dg[o] = e ? suf - db[0] : suf;
                        p.dbeta[o] = dbt[e];
                        p.pq[o] = pqv[e];
                        p.pk[o] = pkv[e];
                    }
                }
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------
// The two launches.  Each is one cooperative kernel, one CTA per SM, in two phases with a grid-wide barrier between them:
// what one phase leaves in the records the other CTAs read.
namespace kn {
constexpr uint32_t cmax(uint32_t a, uint32_t b) { return a > b ? a : b; }
constexpr uint32_t FWD_DATA = cmax(pr::NWORK * pr::WORKER, fs::BYTES), BWD_DATA = cmax(bs::BYTES, bg::BYTES);
// behind the data: the scan's barriers, the other phase's barriers, the TMEM base address, the abort flag
constexpr uint32_t TAIL_B0 = 0, TAIL_B1 = 32 * 8, TAIL_TM = TAIL_B1 + 16 * 8, TAIL = TAIL_TM + 16;
constexpr uint32_t FWD_SMEM = FWD_DATA + TAIL + 1024, BWD_SMEM = BWD_DATA + TAIL + 1024;
static_assert(FWD_SMEM <= 232448 && BWD_SMEM <= 232448, "shared memory budget");
static_assert(scn::NBAR <= 32 && pr::NWORK * pr::NBAR <= 16 && bg::NBAR <= 16, "barrier slots");
}  // namespace kn

// Records written through both proxies (bulk stores, plain stores) and read by other CTAs' bulk loads.
__device__ __forceinline__ void grid_handover() {
    fence_proxy_async_all();
    cooperative_groups::this_grid().sync();
    fence_proxy_async_all();
}

__global__ void __launch_bounds__(scn::NTHREADS, 1)
k_gdn_chunk_fwd(const __grid_constant__ CUtensorMap gm_q, const __grid_constant__ CUtensorMap gm_k, const __grid_constant__ CUtensorMap gm_v,
                const __grid_constant__ CUtensorMap gm_o, const __grid_constant__ ChunkParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    const int tid = threadIdx.x, warp = tid >> 5;
    constexpr uint32_t TAIL = kn::FWD_DATA;
    const uint32_t bars0 = base + TAIL + kn::TAIL_B0, bars1 = base + TAIL + kn::TAIL_B1;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + TAIL + kn::TAIL_TM + 8);
    bool failed = false;
    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < pr::NWORK * pr::NBAR; ++i) mbar_init(bars1 + 8 * i, 1);
        fence_mbar_init();
    }
    if (warp == 8) tmem_alloc(base + TAIL + kn::TAIL_TM, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(sm + TAIL + kn::TAIL_TM);
    if (warp < 4 * pr::NWORK) {
        const int wid = warp >> 2;
        prep_worker(gm_q, gm_k, p, sm + wid * pr::WORKER, base + wid * pr::WORKER, bars1 + 8 * pr::NBAR * wid, tmem + 128 * wid, wid, tid & 127,
                    abort_flag, failed);
    }
    tc_fence_before();
    grid_handover();
    tc_fence_after();
    const int items = (p.seqs ? p.n_seq : p.n_rows) * p.H * (p.dv / 64);
    for (int item = blockIdx.x; item < items; item += gridDim.x)
        scan_item(item, gm_q, gm_k, gm_v, gm_o, p, sm, base, bars0, item == (int)blockIdx.x, tmem, abort_flag, failed);
    if (failed) atomicOr(p.status, STATUS_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

__global__ void __launch_bounds__(scn::NTHREADS, 1)
k_gdn_chunk_bwd(const __grid_constant__ CUtensorMap gm_q, const __grid_constant__ CUtensorMap gm_k, const __grid_constant__ CUtensorMap gm_v,
                const __grid_constant__ CUtensorMap gm_do, const __grid_constant__ CUtensorMap gm_dq, const __grid_constant__ CUtensorMap gm_dk,
                const __grid_constant__ CUtensorMap gm_dv, const __grid_constant__ CUtensorMap gm_doh, const __grid_constant__ ChunkParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    const int tid = threadIdx.x, warp = tid >> 5;
    constexpr uint32_t TAIL = kn::BWD_DATA;
    const uint32_t bars0 = base + TAIL + kn::TAIL_B0, bars1 = base + TAIL + kn::TAIL_B1;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + TAIL + kn::TAIL_TM + 8);
    bool failed = false;
    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < bg::NBAR; ++i) mbar_init(bars1 + 8 * i, (i >= bg::E1R && i <= bg::TFREE) ? NCOMPUTE / 32 : 1);
        fence_mbar_init();
    }
    if (warp == 8) tmem_alloc(base + TAIL + kn::TAIL_TM, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(sm + TAIL + kn::TAIL_TM);
    const int items = (p.seqs ? p.n_seq : p.n_rows) * p.H * (p.dv / 64);
    for (int item = blockIdx.x; item < items; item += gridDim.x)
        bscan_item(item, gm_q, gm_k, gm_doh, p, sm, base, bars0, item == (int)blockIdx.x, tmem, abort_flag, failed);
    tc_fence_before();
    grid_handover();
    tc_fence_after();
    bgrad_chunks(gm_q, gm_k, gm_v, gm_do, gm_dq, gm_dk, gm_dv, p, sm, base, bars1, tmem, abort_flag, failed);
    if (failed) atomicOr(p.status, STATUS_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 8) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// Tensor map over a bf16 [B,T,H,d] tensor that moves 64 tokens x 64 features (one half of make_tile_map's tile).
// Coordinates: (0, token, half, head, batch).
bool make_half_map(CUtensorMap *m, const void *ptr, int B, int T, int H, int d) {
    EncodeFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[5] = {64, (cuuint64_t)T, (cuuint64_t)(d / 64), (cuuint64_t)H, (cuuint64_t)B};
    cuuint64_t strides[4] = {(cuuint64_t)H * d * 2, 128, (cuuint64_t)d * 2, (cuuint64_t)T * H * d * 2};
    cuuint32_t box[5] = {64, (cuuint32_t)C, 1, 1, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// record slots (one per chunk plus one per sequence) over all (sequence, head) pairs
// (a record is at least 34 KiB, so their number fits an int long before their size fits the device)
long chunk_slots(const Dims &d, const Varlen *vl) {
    return (vl && vl->n_seq) ? vl->slots * d.H : (long)d.B * d.H * (d.NT + 1);
}

// The maps of one kernel: per-sequence device arrays for a packed batch (region r), else the kernel parameters alone.
struct MapSpec { const void *ptr; int width; bool half; };
template <int N>
bool chunk_maps(const Dims &d, Varlen *vl, int r, const MapSpec (&spec)[N], CUtensorMap (&maps)[N], const CUtensorMap **dev, cudaStream_t st) {
    auto one = [&](CUtensorMap *m, const MapSpec &e, size_t tok, int B, int T) {
        const void *ptr = (const __nv_bfloat16 *)e.ptr + tok * d.H * e.width;
        return e.half ? make_half_map(m, ptr, B, T, d.H, e.width) : make_tile_map(m, ptr, B, T, d.H, e.width);
    };
    for (int i = 0; i < N; ++i)
        if (!one(&maps[i], spec[i], 0, d.B, d.T)) return false;
    *dev = nullptr;
    if (!vl) return true;
    const void *key[N + 1];
    for (int i = 0; i < N; ++i) key[i] = spec[i].ptr;
    static const char kind = 0;
    key[N] = &kind;                                     // (other kernels keep other maps of the same tensors in this region)
    *dev = varlen_maps(*vl, r, key, N + 1, st, [&](const SeqInfo &si, CUtensorMap *m) {
        for (int i = 0; i < N; ++i)
            if (!one(m + i, spec[i], (size_t)si.t0, 1, si.T)) return false;
        return true;
    });
    return *dev != nullptr;
}

}  // namespace

static gdn::Load chunk_load(const Dims &d, const Varlen *vl) {
    if (vl && vl->n_seq) return {vl->seqs[0].NT, (vl->slots - vl->n_seq) * d.H, (long)vl->n_seq * d.H, d.coop_sms, d.dv > 64};      // (kept longest first)
    return {d.NT, (long)d.B * d.H * d.NT, (long)d.B * d.H, d.coop_sms, d.dv > 64};
}
bool gdn_chunk_selected(const Dims &d, const Varlen *vl) { return gdn::chunk_parallel_step(chunk_load(d, vl)); }
bool gdn_chunk_forward_selected(const Dims &d, const Varlen *vl) { return gdn::chunk_parallel_forward(chunk_load(d, vl)); }

int gdn_chunk_sms() {
    int dev = 0, sms = 0, coop = 0, fwd = 0, bwd = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fwd, k_gdn_chunk_fwd, scn::NTHREADS, kn::FWD_SMEM) == cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bwd, k_gdn_chunk_bwd, scn::NTHREADS, kn::BWD_SMEM) == cudaSuccess)
        return coop && fwd > 0 && bwd > 0 ? sms : 0;
    cudaGetLastError();
    return 0;
}

// One of the two kernels on a cooperative grid of at most one CTA per SM
static int launch_cooperative(const void *kernel, long grid, void **args, uint32_t smem, cudaStream_t st) {
    const cudaError_t e = cudaLaunchCooperativeKernel(kernel, dim3((unsigned)grid), dim3(scn::NTHREADS), args, smem, st);
    if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported) return e == cudaSuccess ? 0 : -1;
    cudaGetLastError();
    return gdn::REFUSED;
}

int gdn_chunk_configure() {
    constexpr cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return cudaFuncSetAttribute(k_gdn_chunk_fwd, A, (int)kn::FWD_SMEM) == cudaSuccess &&
                   cudaFuncSetAttribute(k_gdn_chunk_bwd, A, (int)kn::BWD_SMEM) == cudaSuccess ? 0 : -1;
}

size_t gdn_chunk_forward_workspace_bytes(const Dims &d, const Varlen *vl) { return (size_t)chunk_slots(d, vl) * REC_INFER.bytes; }
size_t gdn_chunk_record_bytes(const Dims &d, const Varlen *vl) { return (size_t)chunk_slots(d, vl) * REC_TRAIN.bytes; }

static ChunkParams chunk_params(const Dims &d, const FwdArgs &a, uint8_t *rec, bool save, int *status) {
    const Varlen *vl = (a.vl && a.vl->n_seq) ? a.vl : nullptr;
    ChunkParams p{};
    p.lq = a.lq; p.lk = a.lk; p.g = a.log_decay; p.beta = a.beta; p.h0 = a.h0; p.ht = a.ht;
    p.rec = rec;
    p.L = save ? REC_TRAIN : REC_INFER;
    p.status = status;
    p.T = d.T; p.H = d.H; p.NT = d.NT; p.n_rows = d.B;
    p.slots = (int)chunk_slots(d, vl);
    p.scale = d.scale;
    p.save = save;
    p.write_o = a.o != nullptr;
    p.seqs = vl ? vl->d_seqs : nullptr;
    p.n_seq = vl ? vl->n_seq : 0;
    p.dk = d.dk; p.dv = d.dv;
    return p;
}

// a.o == nullptr: the records only (the backward's own recomputation), in region 1 of a packed batch's maps
int gdn_chunk_forward(const Dims &d, const FwdArgs &a, uint8_t *rec, bool save, int *status, cudaStream_t st, Tracer &tr) {
    Varlen *vl = (a.vl && a.vl->n_seq) ? a.vl : nullptr;
    ChunkParams p = chunk_params(d, a, rec, save, status);
    const MapSpec spec[4] = {{a.q, d.dk, false}, {a.k, d.dk, false}, {a.v, d.dv, true}, {a.o ? a.o : a.v, d.dv, true}};
    CUtensorMap m[4];
    if (!chunk_maps(d, vl, a.o ? 0 : 1, spec, m, &p.vmaps, st)) return -1;
    const long items = (long)(vl ? vl->n_seq : d.B) * d.H * (d.dv / 64);
    const long grid = std::min<long>(d.coop_sms, std::max<long>((p.slots + pr::NWORK - 1) / pr::NWORK, items));
    void *args[] = {&m[0], &m[1], &m[2], &m[3], &p};
    if (const int e = launch_cooperative((const void *)k_gdn_chunk_fwd, grid, args, kn::FWD_SMEM, st)) return e;
    tr.mark(a.o ? "gdn_chunk_fwd" : "gdn_chunk_records");
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int gdn_chunk_backward(const Dims &d, const BwdArgs &a, bool have_records, int *status, cudaStream_t st, Tracer &tr) {
    Varlen *vl = (a.vl && a.vl->n_seq) ? a.vl : nullptr;
    const size_t bth = (size_t)d.B * d.T * d.H;
    uint8_t *rec = reinterpret_cast<uint8_t *>(a.ws);
    FwdArgs f{a.q, a.k, a.v, a.log_decay, a.beta, a.lq, a.lk, a.h0, nullptr, nullptr, a.ws, a.status, vl};
    int n = 0;
    if (!have_records) {
        n = gdn_chunk_forward(d, f, rec, true, status, st, tr);
        if (n < 0) return n;
    }
    ChunkParams p = chunk_params(d, f, rec, true, status);
    p.dht = a.dht; p.dh0 = a.dh0;
    p.dg = a.dlog_decay; p.dbeta = a.dbeta;
    p.pq = reinterpret_cast<float *>(rec + gdn_chunk_record_bytes(d, vl));
    p.pk = p.pq + ((bth + 63) & ~(size_t)63);
    const MapSpec spec[8] = {{a.q, d.dk, false}, {a.k, d.dk, false}, {a.v, d.dv, false}, {a.dO, d.dv, false},
                             {a.dq, d.dk, false}, {a.dk, d.dk, false}, {a.dv, d.dv, false}, {a.dO, d.dv, true}};
    CUtensorMap m[8];
    if (!chunk_maps(d, vl, 2, spec, m, &p.vmaps, st)) return -1;
    const long items = (long)(vl ? vl->n_seq : d.B) * d.H * (d.dv / 64);
    const long grid = std::min<long>(d.coop_sms, std::max<long>(p.slots, items));
    void *args[] = {&m[0], &m[1], &m[2], &m[3], &m[4], &m[5], &m[6], &m[7], &p};
    if (const int e = launch_cooperative((const void *)k_gdn_chunk_bwd, grid, args, kn::BWD_SMEM, st)) return e;
    tr.mark("gdn_chunk_bwd");
    if (gate_bwd_prod(a.lq, a.lk, p.pq, p.pk, a.dlq, a.dlk, (long)d.B * d.T, d.H, st) < 0) return -1;
    tr.mark("gate_bwd");
    return cudaGetLastError() == cudaSuccess ? n + 2 : -1;
}

}  // namespace sla
