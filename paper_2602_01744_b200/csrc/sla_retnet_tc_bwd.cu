// Softmax-RetNet gradient sweep on the 5th-generation tensor cores (bf16 I/O, d_k and d_v 128 - or 64: two heads side by side, or one with zero padding
// supplied by the tensor maps -, chunk 64).  The formulas are Softmax-GLA's (sla_gla_tc_bwd.cu: one CTA per sequence, chunks in
// reverse, dS in TMEM),
//     qh_i = f_i q_i, f_i = scale*Gq_i e^{b_i}        kh_j = c_j k_j, c_j = Gk_j e^{-b_j}        dZ = e^{b_last} dS_{n+1}
//     A = tril(qh kh^T)   dA = tril(dO V^T)   dqh = dA kh + dO S_n^T   dkh = dA^T qh + V dZ^T   dV = A^T dO + kh dZ   dS_n = dZ + qh^T dO
//     dq = f dqh          dk = c dkh          Gq dGq = sum_d qh dqh     Gk dGk = sum_d kh dkh
// but with a constant decay per head (Eq. 10) b_i is a number a token: the factors f, c come ready from the gate warps, the
// prologue only scales rows, the read-out needs two numbers a token instead of a tile of factors, and there is no log-decay to
// read and none whose gradient has to be summed up.  What that leaves of shared memory (68 KiB) holds the four input tiles of
// TWO chunks, so that a chunk's tiles are requested a whole chunk before their use, and the prologue of the next chunk runs
// while the tensor core works on this one's products: A and dA of the next chunk start the moment their columns are free.
// 8 x 4096 tokens x 16 heads: 366 us on Softmax-GLA's kernel, 262 here (2 320 bytes a token and head with the state image: 4.6 TB/s);
// bound by the chain of a chunk's phases in the eight compute warps, about 4 us a chunk.
#include "sla_gla_tc.cuh"

namespace sla {
namespace {

using namespace ptx;
using namespace tc;

constexpr uint32_t T_Q = 0, T_K = TILE_BF16, T_V = 2 * TILE_BF16, T_DO = 3 * TILE_BF16;
constexpr uint32_t STAGE = 4 * TILE_BF16;               // [2]: q -> qh -> dq staged, k -> kh -> dk staged, v, dO
constexpr uint32_t OFF_S = 2 * STAGE;                   // bf16 S_n image
constexpr uint32_t OFF_DZ = OFF_S + STATE_BF16;         // bf16 dZ operand
constexpr uint32_t OFF_A = OFF_DZ + STATE_BF16;         // masked A, [64 rows][128 B]
constexpr uint32_t OFF_DA = OFF_A + HALF_BF16;          // masked dA; afterwards A|dA hold the dv tile staged for the store
constexpr uint32_t OFF_GATE = OFF_DA + HALF_BF16;       // [4][heads][2][64]: f, c of four chunks
constexpr uint32_t OFF_RED = OFF_GATE + 4 * 2 * 2 * C * 4;  // [2][2 column halves][64] gate partial sums
constexpr uint32_t OFF_BAR = OFF_RED + 2 * 2 * C * 4;
constexpr uint32_t OFF_TMEM = OFF_BAR + 32 * 8;         // TMEM base address, then the abort flag
constexpr uint32_t SMEM_BYTES = OFF_TMEM + 16 + 1024;
constexpr uint32_t TMEM_COLS = 512;
constexpr int NTHREADS = NCOMPUTE + 32 + NGATE + 32;    // warps 0..7 compute, 8 MMA issue, 9..12 gates, 13 TMA
enum Bar { FULL_QK = 0 /*[2]*/, FULL_VO = 2 /*[2]*/, FULL_S = 4, OPR, GREADY = 6 /*[4]*/, GFREE = 10 /*[4]*/, ZREADY = 14, AREADY, OUT1, OUT2,
           DVREAD, DVFREE, BAR_A, BAR_M1, BAR_M2, ALLREAD, SFREE, DRAIN, NBAR };
static_assert(SMEM_BYTES <= 232448, "shared memory budget");
static_assert(NBAR <= 32, "barrier slots");

// PAIR: two 64-wide heads a CTA, as in k_gla_bwd_tc.
template <bool PAIR>
__global__ void __launch_bounds__(NTHREADS, 1)
k_retnet_bwd_tc(const __grid_constant__ CUtensorMap gm_q, const __grid_constant__ CUtensorMap gm_k, const __grid_constant__ CUtensorMap gm_v,
                const __grid_constant__ CUtensorMap gm_do, const __grid_constant__ CUtensorMap gm_dq, const __grid_constant__ CUtensorMap gm_dk,
                const __grid_constant__ CUtensorMap gm_dv, BwdParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int HPC = PAIR ? 2 : 1;                       // heads per CTA
    constexpr uint32_t COL_DS = 0, COL_A = 128, COL_DA = PAIR ? 256 : 192, COL_DV = 128 /* once A and dA are read */, COL_DQ = PAIR ? 384 : 256,
                       COL_DK = PAIR ? 256 /* once dA is read */ : 384;
    const int hg = p.H / HPC, h = blockIdx.x % hg;          // h: head, or pair of heads, as the tensor maps count them
    int b = blockIdx.x / hg;
    const int bh = b * p.H + h * HPC;
    size_t tokb = (size_t)b * p.T, slot = (size_t)bh * (p.NT + 1);
    size_t sbh = (size_t)bh, hbh = sbh;                     // (sequence, head) index into dht, into dh0
    int img_n0 = 0;
    const CUtensorMap *vm = nullptr;
    if (p.seqs) {                                           // packed batch: see k_gla_fwd_tc
        const SeqInfo si = p.seqs[b];
        vm = p.vmaps + (size_t)b * Varlen::MAPS_PER_SEQ;
        p.T = si.T; p.NT = si.NT;
        tokb = (size_t)si.t0;
        slot = (size_t)si.slot0 * p.H + (size_t)h * HPC * (si.img_NT + 1);
        img_n0 = si.img_n0;
        hbh = (size_t)max(si.dh0_id, 0) * p.H + h * HPC;
        if (si.dh0_id < 0) p.dh0 = nullptr;
        if (si.ht_id < 0) p.dht = p.edge;
        sbh = (size_t)(si.ht_id < 0 ? si.id : si.ht_id) * p.H + h * HPC;        // (the table is ordered longest first, the state tensors as the caller gave them)
        b = 0;
    }
    const CUtensorMap &tm_q = vm ? vm[0] : gm_q, &tm_k = vm ? vm[1] : gm_k, &tm_v = vm ? vm[2] : gm_v, &tm_do = vm ? vm[3] : gm_do,
                      &tm_dq = vm ? vm[5] : gm_dq, &tm_dk = vm ? vm[6] : gm_dk, &tm_dv = vm ? vm[7] : gm_dv;
    auto bar = [&](int i) { return base + OFF_BAR + 8u * i; };
    float *gate_s = reinterpret_cast<float *>(sm + OFF_GATE);
    float *red = reinterpret_cast<float *>(sm + OFF_RED);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + OFF_TMEM + 8);
    bool failed = false;
    auto wait = [&](int i, uint32_t parity) {
        if (!failed && !mbar_wait_bounded(bar(i), parity, abort_flag)) { failed = true; *abort_flag = 1; }
    };
    auto wait_relaxed = [&](int i, uint32_t parity) {
        if (!failed && !mbar_wait_bounded<128>(bar(i), parity, abort_flag)) { failed = true; *abort_flag = 1; }
    };

    if (tid == 0) {
        *abort_flag = 0;
        for (int i = 0; i < NBAR; ++i) {
            const bool warps = i == OPR || (i >= GFREE && i <= DVREAD);            // one arrival per compute warp
            mbar_init(bar(i), warps ? NCOMPUTE / 32 : (i >= GREADY && i < GFREE) ? NGATE / 32 : 1);
        }
        fence_mbar_init();
        tma_prefetch_desc(&tm_q);
        tma_prefetch_desc(&tm_k);
        tma_prefetch_desc(&tm_v);
        tma_prefetch_desc(&tm_do);
        tma_prefetch_desc(&tm_dq);
        tma_prefetch_desc(&tm_dk);
        tma_prefetch_desc(&tm_dv);
        for (int x = 0; x < HPC; ++x) check_scalar_range(p.log_gamma[HPC * h + x], p.T, p.status);
    }
    if (warp == 0) tmem_alloc(base + OFF_TMEM, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(sm + OFF_TMEM);
    const uint8_t *img0 = p.simg + slot * STATE_BF16 + (size_t)img_n0 * (PAIR ? PAIR_STATE : STATE_BF16);
    const int NT = p.NT;
    // chunks are visited in the order n = NT-1 ... 0; k = NT-1-n is the visit number that drives every buffer and parity

    if (warp == 8) {
        // ---------------- MMA issue (the warp walks the loop together, one lane issues) ----------------
        const bool leader = elect_lane();
        // (the whole warp gives up together: it votes)
        auto wait = [&](int i, uint32_t parity) {
            if (!failed && !__all_sync(0xffffffffu, mbar_wait_bounded(bar(i), parity, abort_flag))) { failed = true; *abort_flag = 1; }
        };
        constexpr uint32_t ID_A = idesc_bf16(64, 64, 0, 0);
        constexpr uint32_t ID_KK = idesc_bf16(64, 128, 0, 0), ID_KM = idesc_bf16(64, 128, 0, 1),
                           ID_MM = idesc_bf16(64, 128, 1, 1), ID_S = idesc_bf16(128, 128, 1, 1);
        constexpr uint32_t ID_KM64 = idesc_bf16(64, 64, 0, 1), ID_MM64 = idesc_bf16(64, 64, 1, 1);
        const uint64_t kS = desc_kmajor(base + OFF_S), kDZ = desc_kmajor(base + OFF_DZ),
                       mDZ = desc_mnmajor(base + OFF_DZ, STATE_HALF), mA = desc_mnmajor(base + OFF_A, HALF_BF16),
                       kDA = desc_kmajor(base + OFF_DA), mDA = desc_mnmajor(base + OFF_DA, HALF_BF16);
        for (int k = 0; k < NT; ++k) {
            const uint32_t par = k & 1, ph = (k >> 1) & 1, st = base + (k & 1) * STAGE;
            const uint64_t kQ = desc_kmajor(st + T_Q), kK = desc_kmajor(st + T_K), kV = desc_kmajor(st + T_V), kDO = desc_kmajor(st + T_DO),
                           mQ = desc_mnmajor(st + T_Q, HALF_BF16), mK = desc_mnmajor(st + T_K, HALF_BF16),
                           mDO = desc_mnmajor(st + T_DO, HALF_BF16);
            wait(FULL_VO + (k & 1), ph);
            wait(OPR, par);                            // qh, kh (a chunk ahead of their use, but for the first)
            if (k > 0) wait(DVREAD, (k - 1) & 1);      // dV of the previous chunk, in the columns of A and dA, has been read out
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {       // A = qh kh^T,  dA = dO V^T
                    const uint32_t hc = PAIR ? 64 * (kk >> 2) : 0, acc = PAIR ? (kk & 3) > 0 : kk > 0;      // (a pair: head kk / 4)
                    tc_mma_bf16(tmem + COL_A + hc, kQ + kstep_kmajor(kk, HALF_BF16), kK + kstep_kmajor(kk, HALF_BF16), ID_A, acc);
                    tc_mma_bf16(tmem + COL_DA + hc, kDO + kstep_kmajor(kk, HALF_BF16), kV + kstep_kmajor(kk, HALF_BF16), ID_A, acc);
                }
                tc_commit(bar(BAR_A));
            }
            wait(FULL_S, par);
            if (k > 0) wait(OUT1, (k - 1) & 1);        // dqh, dkh of the previous chunk have been read out (before its dV)
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {       // dqh = dO S_n^T ...
                    if (PAIR)
                        tc_mma_bf16(tmem + COL_DQ + 64 * (kk >> 2), kDO + kstep_kmajor(kk, HALF_BF16),
                                    desc_kmajor(base + OFF_S + pair_block(kk >> 2)) + kstep_kmajor(kk & 3, 0), ID_A, (kk & 3) > 0);
                    else
                        tc_mma_bf16(tmem + COL_DQ, kDO + kstep_kmajor(kk, HALF_BF16), kS + kstep_kmajor(kk, STATE_HALF), ID_KK, kk > 0);
                }
                tc_commit(bar(SFREE));                 // (for the TMA lane: the next image may land)
            }
            wait(ZREADY, par);                         // dZ: fp32 in TMEM, bf16 in shared memory
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {       // two independent accumulation chains, interleaved
                    if (!PAIR) tc_mma_bf16(tmem + COL_DK, kV + kstep_kmajor(kk, HALF_BF16), kDZ + kstep_kmajor(kk, STATE_HALF), ID_KK, kk > 0);   // dkh = V dZ^T ...
                    if (kk < 4) tc_mma_bf16(tmem + COL_DS, mQ + kstep_mnmajor(kk), mDO + kstep_mnmajor(kk), ID_S, 1);                // dS_n = dZ + qh^T dO
                }
            }
            wait(AREADY, par);                         // masked A, dA in shared memory
            if (failed) break;
            tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {       // dV = kh dZ ... (A and dA have been read; before M1, after which dk goes over kh)
                    if (PAIR) {                        // (head kk / 4; and dkh = V dZ^T)
                        const uint32_t dz = base + OFF_DZ + pair_block(kk >> 2);
                        tc_mma_bf16(tmem + COL_DV + 64 * (kk >> 2), kK + kstep_kmajor(kk, HALF_BF16), desc_mnmajor(dz, STATE_HALF) + kstep_mnmajor(kk & 3), ID_KM64, (kk & 3) > 0);
                        tc_mma_bf16(tmem + COL_DK + 64 * (kk >> 2), kV + kstep_kmajor(kk, HALF_BF16), desc_kmajor(dz) + kstep_kmajor(kk & 3, 0), ID_A, (kk & 3) > 0);
                    } else {
                        tc_mma_bf16(tmem + COL_DV, kK + kstep_kmajor(kk, HALF_BF16), mDZ + kstep_mnmajor(kk), ID_KM, kk > 0);
                    }
                }
                // ... + dA kh  and  ... + dA^T qh, interleaved; a pair: head x's tile and its half of kh, qh
                auto head = [&](int x, uint32_t sDA, int kk) {
                    tc_mma_bf16(tmem + COL_DQ + 64 * x, desc_kmajor(sDA) + kstep_kmajor(kk, 0), desc_mnmajor(st + T_K + x * HALF_BF16, HALF_BF16) + kstep_mnmajor(kk), ID_KM64, 1);
                    tc_mma_bf16(tmem + COL_DK + 64 * x, desc_mnmajor(sDA, HALF_BF16) + kstep_mnmajor(kk), desc_mnmajor(st + T_Q + x * HALF_BF16, HALF_BF16) + kstep_mnmajor(kk), ID_MM64, 1);
                };
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    if (PAIR) {
                        head(0, base + OFF_DA, kk);
                        head(1, base + OFF_S + PAIR_FREE1, kk);
                    } else {
                        tc_mma_bf16(tmem + COL_DQ, kDA + kstep_kmajor(kk, 0), mK + kstep_mnmajor(kk), ID_KM, 1);
                        tc_mma_bf16(tmem + COL_DK, mDA + kstep_mnmajor(kk), mQ + kstep_mnmajor(kk), ID_MM, 1);
                    }
                }
                tc_commit(bar(BAR_M1));
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {       // ... + A^T dO
                    if (PAIR) {
                        tc_mma_bf16(tmem + COL_DV, mA + kstep_mnmajor(kk), mDO + kstep_mnmajor(kk), ID_MM64, 1);
                        tc_mma_bf16(tmem + COL_DV + 64, desc_mnmajor(base + OFF_S + PAIR_FREE0, HALF_BF16) + kstep_mnmajor(kk),
                                    desc_mnmajor(st + T_DO + HALF_BF16, HALF_BF16) + kstep_mnmajor(kk), ID_MM64, 1);
                    } else {
                        tc_mma_bf16(tmem + COL_DV, mA + kstep_mnmajor(kk), mDO + kstep_mnmajor(kk), ID_MM, 1);
                    }
                }
                tc_commit(bar(BAR_M2));
                tc_commit(bar(ALLREAD));               // (same event, for the TMA lane)
            }
        }
        if (leader) tc_commit(bar(DRAIN));
        mbar_wait_bounded(bar(DRAIN), 0, nullptr, 20000000ull);
    } else if (warp == 13) {
        // ---------------- TMA (one lane) ----------------
        if (lane == 0) {
            auto load_tiles = [&](int k) {
                const int n = NT - 1 - k;
                const uint32_t dst = base + (k & 1) * STAGE, qk = bar(FULL_QK + (k & 1)), vo = bar(FULL_VO + (k & 1));
                mbar_expect_tx(qk, 2 * TILE_BF16);
                tma_load_5d(dst + T_Q, &tm_q, 0, n * C, 0, h, b, qk);
                tma_load_5d(dst + T_K, &tm_k, 0, n * C, 0, h, b, qk);
                mbar_expect_tx(vo, 2 * TILE_BF16);
                tma_load_5d(dst + T_V, &tm_v, 0, n * C, 0, h, b, vo);
                tma_load_5d(dst + T_DO, &tm_do, 0, n * C, 0, h, b, vo);
            };
            constexpr uint32_t IMAGE = PAIR ? PAIR_STATE : STATE_BF16;
            auto load_s = [&](int n) {
                mbar_expect_tx(bar(FULL_S), IMAGE);
                if (PAIR) {
                    bulk_load(base + OFF_S + pair_block(0), img0 + (size_t)n * IMAGE, STATE_BLOCK, bar(FULL_S));
                    bulk_load(base + OFF_S + pair_block(1), img0 + (size_t)n * IMAGE + STATE_BLOCK, STATE_BLOCK, bar(FULL_S));
                } else {
                    bulk_load(base + OFF_S, img0 + (size_t)n * IMAGE, IMAGE, bar(FULL_S));
                }
            };
            load_tiles(0);
            load_s(NT - 1);
            if (NT > 1) load_tiles(1);
            for (int k = 0; k < NT && !failed; ++k) {
                const int n = NT - 1 - k;
                const uint32_t par = k & 1, st = base + (k & 1) * STAGE;
                if (n > 1) {      // the tiles of the chunk after next load when this one's buffers fall free: have them in L2 by then
                    tma_prefetch_l2_5d(&tm_q, 0, (n - 2) * C, 0, h, b);
                    tma_prefetch_l2_5d(&tm_k, 0, (n - 2) * C, 0, h, b);
                    tma_prefetch_l2_5d(&tm_v, 0, (n - 2) * C, 0, h, b);
                    tma_prefetch_l2_5d(&tm_do, 0, (n - 2) * C, 0, h, b);
                    bulk_prefetch_l2(img0 + (size_t)(n - 2) * IMAGE, IMAGE);
                }
                if (n > 0) {
                    wait(SFREE, par);                  // S_n has been read
                    if (failed) break;
                    load_s(n - 1);
                }
                wait(OUT1, par);                       // dq, dk staged over qh, kh
                if (failed) break;
                tma_store_5d(&tm_dq, st + T_Q, 0, n * C, 0, h, b);
                tma_store_5d(&tm_dk, st + T_K, 0, n * C, 0, h, b);
                bulk_commit();
                wait(ALLREAD, par);                    // every product of the chunk is done with v, dO, too
                if (failed) break;
                bulk_wait_read0();
                if (k + 2 < NT) load_tiles(k + 2);
                wait(OUT2, par);                       // dv staged
                if (failed) break;
                tma_store_5d(&tm_dv, base + OFF_A, 0, n * C, 0, h, b);
                bulk_commit();
                bulk_wait_read0();
                mbar_arrive(bar(DVFREE));
            }
            bulk_wait0();
            if (failed) {   // give loads that are still in flight time to land before shared memory goes away
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
            }
        }
    } else if (warp >= 9) {
        // ---------------- gates with the tokens' decay, up to four chunks ahead ----------------
        const int g = tid - (NCOMPUTE + 32), t = g & (C - 1);
        const float *l = g < C ? p.lq : p.lk;
        const float mult = g < C ? p.scale : 1.f, sign = g < C ? LOG2E : -LOG2E;
        const DecayFactor f{mult, sign * p.log_gamma[HPC * h]}, f2{mult, PAIR ? sign * p.log_gamma[2 * h + 1] : 0.f};
        for (int k = 0; k < NT; ++k) {
            const int n = NT - 1 - k;
            if (k >= 4) wait_relaxed(GFREE + (k & 3), ((k >> 2) - 1) & 1);
            if (failed) break;
            const int cn = min(C, p.T - n * C);
            float *dst = gate_s + (k & 3) * HPC * 2 * C + (g < C ? 0 : C);
            chunk_gate_by<64, HPC>(l + (tokb + (size_t)n * C) * p.H, p.H, cn, HPC * h, f, dst, t, f2, dst + 2 * C);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(GREADY + (k & 3)));
        }
    } else {
        // ---------------- compute warps ----------------
        const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
        const int wh = warp >> 2;                       // column half, of the state and of the gradient tiles
        const int row = 32 * (warp & 3) + lane;         // state row of this thread (its TMEM lane)
        const int qr = warp & 3, tr = 16 * qr + (lane >> 2);       // gradient tiles: tokens tr, tr + 8
        const bool holds = !PAIR || pair_diagonal(warp & 3, wh);   // (a pair's threads off the diagonal blocks have no state)
        const float lg = LOG2E * p.log_gamma[HPC * h + (PAIR ? row >> 6 : 0)];
        auto prologue = [&](int k) {
            wait(GREADY + (k & 3), (k >> 2) & 1);
            wait(FULL_QK + (k & 1), (k >> 1) & 1);
            uint8_t *qk = sm + (k & 1) * STAGE;
            const float *g = gate_s + (k & 3) * HPC * 2 * C;
            scale_rows(qk + T_Q, g, tid, PAIR ? 2 * C : 0);
            scale_rows(qk + T_K, g + C, tid, PAIR ? 2 * C : 0);
            fence_proxy_async();
            warp_arrive(bar(OPR), lane);
        };
        {   // dS_NT = dht (or zero) into TMEM
            const float *src = PAIR ? pair_state_row(p.dht, sbh, row, wh) : state_row(p.dht, sbh, row, wh, p.dk, p.dv);
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                float v[32];
                load_state32(src ? src + 32 * part : nullptr, v);
                tmem_st32(tmem + lane_base + COL_DS + 64 * wh + 32 * part, v);
            }
            tmem_wait_st();
        }
        prologue(0);
        for (int k = 0; k < NT; ++k) {
            const int n = NT - 1 - k, t0 = n * C, cn = min(C, p.T - t0);
            const uint32_t par = k & 1;
            uint8_t *qk = sm + (k & 1) * STAGE;
            const float *gate = gate_s + ((k & 3) * HPC + (PAIR ? wh : 0)) * 2 * C;       // (of the head whose columns this warp reads out)

            // ---- dZ = e^{b_last} dS_{n+1}: fp32 back into TMEM (dS_n accumulates on it), bf16 operand copy (every product of the
            // previous chunk is complete, see BAR_M2 below) ----
            if (holds) {
                const float e = ex2f(lg * (float)cn);
                float v0[32], v1[32];
                const uint32_t ta = tmem + lane_base + COL_DS + 64 * wh;
                tmem_ld32(ta, v0);
                tmem_ld32(ta + 32, v1);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) { v0[j] *= e; v1[j] *= e; }
                tmem_st32(ta, v0);
                tmem_st32(ta + 32, v1);
                uint8_t *img = sm + OFF_DZ + wh * STATE_HALF;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    *reinterpret_cast<uint4 *>(img + swz(row, c)) =
                        make_uint4(pack_bf16(v0[8 * c], v0[8 * c + 1]), pack_bf16(v0[8 * c + 2], v0[8 * c + 3]),
                                   pack_bf16(v0[8 * c + 4], v0[8 * c + 5]), pack_bf16(v0[8 * c + 6], v0[8 * c + 7]));
                    *reinterpret_cast<uint4 *>(img + swz(row, 4 + c)) =
                        make_uint4(pack_bf16(v1[8 * c], v1[8 * c + 1]), pack_bf16(v1[8 * c + 2], v1[8 * c + 3]),
                                   pack_bf16(v1[8 * c + 4], v1[8 * c + 5]), pack_bf16(v1[8 * c + 6], v1[8 * c + 7]));
                }
                tmem_wait_st();
            }
            fence_proxy_async();
            tc_fence_before();
            warp_arrive(bar(ZREADY), lane);

            // ---- A, dA: TMEM -> causal mask -> bf16 -> shared memory ----
            wait(BAR_A, par);
            tc_fence_after();
            {
#pragma unroll
                for (int x = 0; x < HPC; ++x) {
                    uint8_t *dst = sm + (x == 0 ? (wh ? OFF_DA : OFF_A) : OFF_S + (wh ? PAIR_FREE1 : PAIR_FREE0));
                    float v[32];
                    tmem_ld_frag8(tmem + lane_base + (wh ? COL_DA : COL_A) + 64 * x, v);
                    tmem_wait_ld();
                    if (x == 0 && k > 0) wait(DVFREE, (k - 1) & 1);   // the staged dv of the previous chunk has left A|dA
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int j = 8 * i + 2 * (lane & 3);
                        const uint32_t off = frag_off(qr, lane, 0, i);
                        *reinterpret_cast<uint32_t *>(dst + off) = pack_bf16(j <= tr ? v[4 * i] : 0.f, j + 1 <= tr ? v[4 * i + 1] : 0.f);
                        *reinterpret_cast<uint32_t *>(dst + off + 1024) = pack_bf16(j <= tr + 8 ? v[4 * i + 2] : 0.f, j + 1 <= tr + 8 ? v[4 * i + 3] : 0.f);
                    }
                }
            }
            fence_proxy_async();
            tc_fence_before();
            warp_arrive(bar(AREADY), lane);

            // ---- qh, kh of the next chunk, while the tensor core works on the products with the masked tiles ----
            if (k + 1 < NT) prologue(k + 1);

            // ---- dqh, dkh: tokens tr, tr + 8, pairs of features of column half wh ----
            wait(BAR_M1, par);
            tc_fence_after();
            {
                const float f0 = gate[tr], f1 = gate[tr + 8], c0 = gate[C + tr], c1 = gate[C + tr + 8];
                float sq0 = 0.f, sq1 = 0.f, sk0 = 0.f, sk1 = 0.f;
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {       // 32 features at a time; every read of a batch is in flight before its first write
                    float dqh[16], dkh[16];
                    uint32_t qw[8], kw[8];
                    tmem_ld_frag4(tmem + lane_base + COL_DQ + 64 * wh + 32 * hf, dqh);
                    tmem_ld_frag4(tmem + lane_base + COL_DK + 64 * wh + 32 * hf, dkh);
#pragma unroll
                    for (int y = 0; y < 8; ++y) {      // feature block y / 2, token tr + 8 (y % 2)
                        const uint32_t off = frag_off(qr, lane, 64 * wh + 32 * hf, y >> 1) + 1024 * (y & 1);
                        qw[y] = *reinterpret_cast<const uint32_t *>(qk + T_Q + off);
                        kw[y] = *reinterpret_cast<const uint32_t *>(qk + T_K + off);
                    }
                    tmem_wait_ld();
#pragma unroll
                    for (int y = 0; y < 8; ++y) {
                        const uint32_t off = frag_off(qr, lane, 64 * wh + 32 * hf, y >> 1) + 1024 * (y & 1);
                        const float2 qv = unpack_bf16(qw[y]), kv = unpack_bf16(kw[y]);
                        const float a0 = dqh[2 * y], a1 = dqh[2 * y + 1], e0 = dkh[2 * y], e1 = dkh[2 * y + 1];
                        const float f = (y & 1) ? f1 : f0, c = (y & 1) ? c1 : c0;
                        float &sq = (y & 1) ? sq1 : sq0, &sk = (y & 1) ? sk1 : sk0;
                        sq = fmaf(qv.x, a0, fmaf(qv.y, a1, sq));
                        sk = fmaf(kv.x, e0, fmaf(kv.y, e1, sk));
                        *reinterpret_cast<uint32_t *>(qk + T_Q + off) = pack_bf16(f * a0, f * a1);      // dq (over qh, for the store)
                        *reinterpret_cast<uint32_t *>(qk + T_K + off) = pack_bf16(c * e0, c * e1);      // dk
                    }
                }
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {      // a token's features: four lanes, two column halves
                    sq0 += __shfl_xor_sync(0xffffffffu, sq0, o); sq1 += __shfl_xor_sync(0xffffffffu, sq1, o);
                    sk0 += __shfl_xor_sync(0xffffffffu, sk0, o); sk1 += __shfl_xor_sync(0xffffffffu, sk1, o);
                }
                if ((lane & 3) == 0) {
                    red[wh * C + tr] = sq0;
                    red[wh * C + tr + 8] = sq1;
                    red[(2 + wh) * C + tr] = sk0;
                    red[(2 + wh) * C + tr + 8] = sk1;
                }
            }
            fence_proxy_async();
            tc_fence_before();
            warp_arrive(bar(OUT1), lane);
            if (lane == 0) mbar_arrive(bar(GFREE + (k & 3)));

            // ---- dV -> dv tile; gate products ----
            wait(BAR_M2, par);
            tc_fence_after();
            {
                float v[32];
                tmem_ld_frag8(tmem + lane_base + COL_DV + 64 * wh, v);
                tmem_wait_ld();
                tc_fence_before();
                warp_arrive(bar(DVREAD), lane);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t off = frag_off(qr, lane, 64 * wh, i);
                    *reinterpret_cast<uint32_t *>(sm + OFF_A + off) = pack_bf16(v[4 * i], v[4 * i + 1]);
                    *reinterpret_cast<uint32_t *>(sm + OFF_A + off + 1024) = pack_bf16(v[4 * i + 2], v[4 * i + 3]);
                }
            }
            fence_proxy_async();
            warp_arrive(bar(OUT2), lane);
            named_bar_sync(1, NCOMPUTE);                // red is complete
            if (PAIR && tid < 2 * C) {        // Gq*dGq and Gk*dGk of token tid % 64: a head's sums are one column half's
                const int x = tid / C, i = tid % C;
                if (i < cn) {
                    p.pq[(tokb + t0 + i) * p.H + 2 * h + x] = red[x * C + i];
                    p.pk[(tokb + t0 + i) * p.H + 2 * h + x] = red[(2 + x) * C + i];
                }
            }
            if (!PAIR && tid < cn) {          // ... of token tid: sum over the two column halves
                p.pq[(tokb + t0 + tid) * p.H + h] = red[tid] + red[C + tid];
                p.pk[(tokb + t0 + tid) * p.H + h] = red[2 * C + tid] + red[3 * C + tid];
            }
        }

        if (p.dh0) {   // dS_0, fp32 (the last chunk's MMAs were waited for above)
            float *dst = PAIR ? pair_state_row(p.dh0, hbh, row, wh) : state_row(p.dh0, hbh, row, wh, p.dk, p.dv);
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                float v[32];
                tmem_ld32(tmem + lane_base + COL_DS + 64 * wh + 32 * part, v);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    if (dst) *reinterpret_cast<float4 *>(dst + 32 * part + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            }
        }
    }
    if (failed) atomicOr(p.status, STATUS_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

}  // namespace

namespace tc {

int retnet_tc_bwd_configure() {
    constexpr cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return cudaFuncSetAttribute(k_retnet_bwd_tc<false>, A, (int)SMEM_BYTES) == cudaSuccess &&
                   cudaFuncSetAttribute(k_retnet_bwd_tc<true>, A, (int)SMEM_BYTES) == cudaSuccess ? 0 : -1;
}

void retnet_tc_bwd_launch(const CUtensorMap (&m)[7], const BwdParams &p, bool pair, int ctas, cudaStream_t st) {
    (pair ? k_retnet_bwd_tc<true> : k_retnet_bwd_tc<false>)<<<ctas, NTHREADS, SMEM_BYTES, st>>>(m[0], m[1], m[2], m[3], m[4], m[5], m[6], p);
}

}  // namespace tc
}  // namespace sla
