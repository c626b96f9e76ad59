// Chunkwise Softmax-Linear-Attention on CUDA cores, fp32 arithmetic, for every variant and
// both I/O dtypes.  This is the precision path (fp32 I/O needs more than bf16 tensor-core
// operands give) and the path for shapes the tensor-core kernels do not cover.
//
// Per (batch, head) sequence and chunk of C tokens (local index i), with
//   b_i   inclusive cumulative log-decay inside the chunk (per key dimension for GLA),
//   qh_i = scale*Gq_i*q_i*exp(b_i),   kh_j = Gk_j*k_j*exp(-b_j)   (GDN: kh_j = k_j*exp(-b_j)),
//   S     state at the chunk start,
// the chunk computes  A = tril(qh kh^T),  O = A V + qh S,  S' = diag(exp(b_last)) S + kbar^T V
// with kbar_j = kh_j*exp(b_last)  (GDN: V is replaced by U = U0 - W S from the WY solve).
// All of these are exact re-associations of the recurrence (Eq. 5-6, 10-16).
#include "sla_generic.cuh"

namespace sla {
namespace {

using namespace detail;

// ------------------------------------------------------------------------------------------
// a1 + a2 in one launch (the two do not meet; a launch costs more than either).  Blocks 0 .. gate_blocks-1: head-softmax gates, HP
// lanes per token (HP = power of two >= H), max and sum by shuffles, the two gates side by side.  The others: chunk-local
// inclusive cumulative log-decay of one chunk of one (batch, head) sequence (Softmax-GLA, a lane four key dimensions) or of eight
// (a warp each, by shuffles).  A chunk whose cumulative log-decay is beyond the range of the e^{b}, e^{-b} factors raises STATUS_RANGE.
template <int HP>
__global__ void __launch_bounds__(256)
k_gates_decay(Dims d, const float *__restrict__ lq, const float *__restrict__ lk, float *__restrict__ Gq, float *__restrict__ Gk,
              const float *__restrict__ log_decay, float *__restrict__ bcum, int gate_blocks, int *status) {
    if ((int)blockIdx.x < gate_blocks) {
        const long n_tok = (long)d.B * d.T, gt = (long)blockIdx.x * 256 + threadIdx.x, tok = gt / HP;
        const int h = (int)(gt % HP);
        const bool valid = tok < n_tok && h < d.H;
        const float x0 = valid ? lq[tok * d.H + h] : -INFINITY, x1 = valid ? lk[tok * d.H + h] : -INFINITY;
        float m0 = x0, m1 = x1;
#pragma unroll
        for (int o = HP / 2; o > 0; o >>= 1) {
            m0 = fmaxf(m0, __shfl_xor_sync(FULL, m0, o));
            m1 = fmaxf(m1, __shfl_xor_sync(FULL, m1, o));
        }
        const float e0 = valid ? expf(x0 - m0) : 0.f, e1 = valid ? expf(x1 - m1) : 0.f;
        float s0 = e0, s1 = e1;
#pragma unroll
        for (int o = HP / 2; o > 0; o >>= 1) {
            s0 += __shfl_xor_sync(FULL, s0, o);
            s1 += __shfl_xor_sync(FULL, s1, o);
        }
        if (valid) {
            Gq[tok * d.H + h] = e0 / s0;
            Gk[tok * d.H + h] = e1 / s1;
        }
        return;
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, blk = (int)blockIdx.x - gate_blocks;
    const long chunks = (long)d.B * d.H * d.NT;
    const long c = d.variant == SLA_GLA ? blk : 8L * blk + w;
    if (c >= chunks) return;
    const int n = (int)(c % d.NT), bh = (int)(c / d.NT), b = bh / d.H, h = bh % d.H, t0 = n * d.C, cn = min(d.C, d.T - t0);
    if (d.variant == SLA_GLA) {             // warp w the tokens 8w .. 8w+7 of all key dimensions, two levels
        __shared__ float4 tot[8][32];
        const bool live = 4 * lane < d.dk;
        float4 g[8], run = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            g[i] = live && 8 * w + i < cn ? ldf4(log_decay, tok_row(d, b, t0 + 8 * w + i, h) * d.dk + 4 * lane) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 8; ++i) { run.x += g[i].x; run.y += g[i].y; run.z += g[i].z; run.w += g[i].w; }
        tot[w][lane] = run;
        __syncthreads();
        run = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int x = 0; x < w; ++x) { const float4 a = tot[x][lane]; run.x += a.x; run.y += a.y; run.z += a.z; run.w += a.w; }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            run.x += g[i].x; run.y += g[i].y; run.z += g[i].z; run.w += g[i].w;
            if (live && 8 * w + i < cn) stf4(bcum, tok_row(d, b, t0 + 8 * w + i, h) * d.dk + 4 * lane, run);
        }
        if (w == 7 && live && fminf(fminf(run.x, run.y), fminf(run.z, run.w)) < -SLA_MAX_CHUNK_DECAY) atomicOr(status, STATUS_RANGE);
        return;
    }
    auto at = [&](int i) { return i >= cn ? 0.f : d.variant == SLA_RETNET ? log_decay[h] : log_decay[tok_row(d, b, t0 + i, h)]; };
    const float g0 = at(2 * lane), g1 = at(2 * lane + 1);      // lane l owns tokens 2l, 2l + 1
    float incl = g0 + g1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
    }
    const float before = __shfl_up_sync(FULL, incl, 1);        // (the first of the two not as incl - g1, which keeps only what g1 leaves of it)
    if (2 * lane < cn) bcum[tok_row(d, b, t0 + 2 * lane, h)] = lane ? before + g0 : g0;
    if (2 * lane + 1 < cn) bcum[tok_row(d, b, t0 + 2 * lane + 1, h)] = incl;
    if (lane == 31 && incl < -SLA_MAX_CHUNK_DECAY) atomicOr(status, STATUS_RANGE);
}

// gate backward: dl_h = G_h (dG_h - sum_h' G_h' dG_h')
template <int HP>
__global__ void k_gate_bwd(const float *__restrict__ Gq, const float *__restrict__ Gk,
                           const float *__restrict__ dGq, const float *__restrict__ dGk,
                           float *__restrict__ dlq, float *__restrict__ dlk, long n_tok, int H) {
    const float *G = blockIdx.y ? Gk : Gq;
    const float *dG = blockIdx.y ? dGk : dGq;
    float *dl = blockIdx.y ? dlk : dlq;
    long gt = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long tok = gt / HP;
    int h = (int)(gt % HP);
    bool valid = tok < n_tok && h < H;
    float g = valid ? G[tok * H + h] : 0.f;
    float dg = valid ? dG[tok * H + h] : 0.f;
    float s = g * dg;
#pragma unroll
    for (int o = HP / 2; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
    if (valid) dl[tok * H + h] = g * (dg - s);
}

// ------------------------------------------------------------------------------------------
// GDN WY preparation (per tile): L_ij = beta_i exp(b_i-b_j) (k_i.k_j), j<i; forward substitution
// (I+L)[W|U0] = [diag(beta exp(b)) K | diag(beta Gk) V].  One thread per right-hand-side column.
template <typename TIO>
__global__ void __launch_bounds__(256)
k_gdn_prepare(Dims d, const TIO *__restrict__ k, const TIO *__restrict__ v,
              const float *__restrict__ beta, const float *__restrict__ Gk,
              const float *__restrict__ bcum, float *__restrict__ Wout, float *__restrict__ U0out) {
    extern __shared__ float sm[];
    int n = blockIdx.x, bh = blockIdx.y, b = bh / d.H, h = bh % d.H;
    int t0 = n * d.C, cn = min(d.C, d.T - t0);
    int ldk = d.dk + 1, ldl = CMAX + 1, ldx = d.dk + d.dv;
    float *Ks = sm;                       // [CMAX][ldk]   raw keys
    float *Ls = Ks + CMAX * ldk;          // [CMAX][ldl]
    float *Xs = Ls + CMAX * ldl;          // [CMAX][ldx]
    float *bs = Xs + CMAX * ldx;          // [CMAX] cumulative log-decay
    float *bt = bs + CMAX;                // [CMAX] beta
    for (int i = threadIdx.x; i < CMAX; i += blockDim.x) {
        bool ok = i < cn;
        size_t row = ok ? tok_row(d, b, t0 + i, h) : 0;
        bs[i] = ok ? bcum[row] : 0.f;
        bt[i] = ok ? beta[row] : 0.f;
    }
    fill_rows(Ks, ldk, k, CMAX, cn, d.dk, [&](int i) { return tok_row(d, b, t0 + i, h) * d.dk; });
    __syncthreads();
    for (int idx = threadIdx.x; idx < CMAX * d.dk; idx += blockDim.x) {
        int i = idx / d.dk, dd = idx % d.dk;
        Xs[i * ldx + dd] = bt[i] * expf(bs[i]) * Ks[i * ldk + dd];
    }
    const int v4 = d.dv >> 2;
    struct In { float4 v; float g; };
    fill(CMAX * v4,
        [&](int idx) {
            const int i = idx / v4;
            In x{make_float4(0.f, 0.f, 0.f, 0.f), 0.f};
            if (i < cn) {
                const size_t row = tok_row(d, b, t0 + i, h);
                x.v = ldf4(v, row * d.dv + 4 * (idx - i * v4));
                x.g = Gk[row];
            }
            return x;
        },
        [&](int idx, const In &x) {
            const int i = idx / v4;
            const float f = bt[i] * x.g;
            put4(Xs + i * ldx + d.dk + 4 * (idx - i * v4), make_float4(f * x.v.x, f * x.v.y, f * x.v.z, f * x.v.w));
        });
    for (int idx = threadIdx.x; idx < CMAX * CMAX; idx += blockDim.x) {
        int i = idx % CMAX, j = idx / CMAX;
        float acc = 0.f;
        if (j < i) {
            for (int dd = 0; dd < d.dk; ++dd) acc = fmaf(Ks[i * ldk + dd], Ks[j * ldk + dd], acc);
            acc *= bt[i] * expf(bs[i] - bs[j]);
        }
        Ls[i * ldl + j] = acc;
    }
    __syncthreads();
    for (int col = threadIdx.x; col < ldx; col += blockDim.x) {
        for (int i = 1; i < cn; ++i) {
            float acc = Xs[i * ldx + col];
            for (int j = 0; j < i; ++j) acc = fmaf(-Ls[i * ldl + j], Xs[j * ldx + col], acc);
            Xs[i * ldx + col] = acc;
        }
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < cn * d.dk; idx += blockDim.x) {
        int i = idx / d.dk, dd = idx % d.dk;
        Wout[tok_row(d, b, t0 + i, h) * d.dk + dd] = Xs[i * ldx + dd];
    }
    for (int idx = threadIdx.x; idx < cn * d.dv; idx += blockDim.x) {
        int i = idx / d.dv, j = idx % d.dv;
        U0out[tok_row(d, b, t0 + i, h) * d.dv + j] = Xs[i * ldx + d.dk + j];
    }
}

// ------------------------------------------------------------------------------------------
// a4 for GDN: inter-chunk state pass, chunk after chunk.  grid (dv/VS, B*H), 256 threads on a [dk x VS] slice of S.  Stores
// the state before every chunk (slot n) and the final state (slot NT, and ht), and U = U0 - W S.
// Serial over the chunks, so what counts is the time of one: four neighbouring columns a thread (float4 reads of the
// shared operand) and the next chunk's tiles in flight in registers while this one computes (28 -> 4.4 us a chunk at d = 64).
template <typename TIO>
__global__ void __launch_bounds__(256)
k_state_scan(Dims d, const TIO *__restrict__ k, const float *__restrict__ bcum,
             const float *__restrict__ h0, float *__restrict__ states, float *__restrict__ ht,
             const float *__restrict__ Wws, const float *__restrict__ U0ws, float *__restrict__ Uws) {
    extern __shared__ float sm[];
    const int vs0 = blockIdx.x * VS, bh = blockIdx.y, b = bh / d.H, h = bh % d.H, ldk = d.dk + 1, tid = threadIdx.x;
    float *Ss = sm;                         // [dk][VS]
    float *Vs = Ss + d.dk * VS;             // [CMAX][VS]   U0, then U
    float *es = Vs + CMAX * VS;             // [CMAX]       e^{b_last - b}
    float *Ks = es + CMAX;                  // [CMAX][ldk]
    float *Ws = Ks + CMAX * ldk;            // [CMAX][ldk]
    const int i0 = tid >> 2, jq = 4 * (tid & 3), w4 = d.dk >> 2;   // this thread's token and state rows (i0, i0 + 64), its columns
    float4 S[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int dd = i0 + 64 * x;
        S[x] = (dd < d.dk && h0) ? ldf4(h0, ((size_t)bh * d.dk + dd) * d.dv + vs0 + jq) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float4 kr[8], wr[8], ur;
    float br = 0.f, bl = 0.f;
    auto fetch = [&](int n) {
        const int t0 = n * d.C, cn = min(d.C, d.T - t0);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int idx = tid + 256 * u, i = idx / w4;
            if (i >= cn) continue;
            const size_t o = tok_row(d, b, t0 + i, h) * d.dk + 4 * (idx - i * w4);
            kr[u] = ldf4(k, o);
            wr[u] = ldf4(Wws, o);
        }
        if (i0 < cn) ur = ldf4(U0ws, tok_row(d, b, t0 + i0, h) * d.dv + vs0 + jq);
        if (tid < cn) br = bcum[tok_row(d, b, t0 + tid, h)];
        bl = bcum[tok_row(d, b, t0 + cn - 1, h)];
    };
    fetch(0);
    for (int n = 0; n < d.NT; ++n) {
        const int t0 = n * d.C, cn = min(d.C, d.T - t0);
        const float dec = expf(bl);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int dd = i0 + 64 * x;
            if (dd >= d.dk) continue;
            *reinterpret_cast<float4 *>(states + state_off(d, bh, n, d.NT + 1) + (size_t)dd * d.dv + vs0 + jq) = S[x];
            *reinterpret_cast<float4 *>(Ss + dd * VS + jq) = S[x];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int idx = tid + 256 * u, i = idx / w4, o = i * ldk + 4 * (idx - i * w4);
            if (i >= cn) continue;
            put4(Ks + o, kr[u]);
            put4(Ws + o, wr[u]);
        }
        if (tid < cn) es[tid] = expf(bl - br);
        float4 acc = ur;
        __syncthreads();
        if (n + 1 < d.NT) fetch(n + 1);
        if (i0 < cn) {
#pragma unroll 4
            for (int c = 0; c < d.dk; ++c) {
                const float w = -Ws[i0 * ldk + c];
                const float4 sv = *reinterpret_cast<const float4 *>(Ss + c * VS + jq);
                acc.x = fmaf(w, sv.x, acc.x); acc.y = fmaf(w, sv.y, acc.y); acc.z = fmaf(w, sv.z, acc.z); acc.w = fmaf(w, sv.w, acc.w);
            }
            *reinterpret_cast<float4 *>(Vs + i0 * VS + jq) = acc;
            *reinterpret_cast<float4 *>(Uws + tok_row(d, b, t0 + i0, h) * d.dv + vs0 + jq) = acc;
        }
        __syncthreads();
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int dd = i0 + 64 * x;
            if (dd >= d.dk) continue;
            S[x].x *= dec; S[x].y *= dec; S[x].z *= dec; S[x].w *= dec;
#pragma unroll 4
            for (int i = 0; i < cn; ++i) {
                const float kb = Ks[i * ldk + dd] * es[i];
                const float4 u = *reinterpret_cast<const float4 *>(Vs + i * VS + jq);
                S[x].x = fmaf(kb, u.x, S[x].x); S[x].y = fmaf(kb, u.y, S[x].y); S[x].z = fmaf(kb, u.z, S[x].z); S[x].w = fmaf(kb, u.w, S[x].w);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int dd = i0 + 64 * x;
        if (dd >= d.dk) continue;
        *reinterpret_cast<float4 *>(states + state_off(d, bh, d.NT, d.NT + 1) + (size_t)dd * d.dv + vs0 + jq) = S[x];
        if (ht) *reinterpret_cast<float4 *>(ht + ((size_t)bh * d.dk + dd) * d.dv + vs0 + jq) = S[x];
    }
}

// ------------------------------------------------------------------------------------------
// a4 for RETNET / GLA, whose state transition is a diagonal: what a chunk adds to the state, and to the state gradient,
// does not depend on the state, so those products run in parallel over the chunks and only an elementwise recurrence
// is left for the walk along the sequence (k_state_fold).  One CTA per sequence walking the chunks through shared memory
// took 19 us a chunk; at 2 x 1000 x 4 heads of 64 both kernels together take 20 us where the scan took 300 (reverse: 250).
// GRAD = false: KV_n = (Gk k e^{b_last - b})^T V into state slot n + 1;  GRAD = true: qh^T dO into slot n - 1 of the state
// gradients (n = 0: into dh0 - ADD: on top of what is there - if wanted).  grid (NT, B*H, ceil(dk / 64)).
template <typename TIO, bool GRAD, bool ADD = false>
__global__ void __launch_bounds__(256)
k_chunk_outer(Dims d, const TIO *__restrict__ x, const TIO *__restrict__ y, const float *__restrict__ gate, const float *__restrict__ bcum,
              float *__restrict__ out, float *__restrict__ dh0) {
    extern __shared__ float sm[];
    const int n = blockIdx.x, bh = blockIdx.y, b = bh / d.H, h = bh % d.H, r0 = 64 * blockIdx.z, nr = min(64, d.dk - r0);
    float *dst = !GRAD ? out + state_off(d, bh, n + 1, d.NT + 1) : n > 0 ? out + state_off(d, bh, n - 1, d.NT) : dh0 ? dh0 + state_off(d, bh, 0, 1) : nullptr;
    if (!dst) return;
    const int t0 = n * d.C, cn = min(d.C, d.T - t0), ldv = pad4(d.dv);
    constexpr int ldx = pad4(64);
    float *Xs = sm;                          // [CMAX][ldx]
    float *Ys = Xs + CMAX * ldx;             // [CMAX][ldv]
    const size_t row_last = tok_row(d, b, t0 + cn - 1, h);
    copy_rows(Ys, ldv, y, cn, cn, d.dv, tok_row(d, b, t0, h) * d.dv, (size_t)d.H * d.dv);
    struct In { float4 x, b, bl; float g; };
    const int w4 = nr >> 2;
    fill<2>(cn * w4,
        [&](int idx) {
            const int i = idx / w4, c = r0 + 4 * (idx - i * w4);
            const size_t row = tok_row(d, b, t0 + i, h);
            In v;
            v.x = ldf4(x, row * d.dk + c);
            v.b = bcum_at4(d, bcum, row, c);
            v.g = GRAD ? d.scale * gate[row] : gate[row];
            v.bl = GRAD ? v.b : bcum_at4(d, bcum, row_last, c);
            return v;
        },
        [&](int idx, const In &v) {
            const int i = idx / w4;
            const float4 e = GRAD ? v.b : make_float4(v.bl.x - v.b.x, v.bl.y - v.b.y, v.bl.z - v.b.z, v.bl.w - v.b.w);
            stf4(Xs, i * ldx + 4 * (idx - i * w4), make_float4(v.g * v.x.x * expf(e.x), v.g * v.x.y * expf(e.y), v.g * v.x.z * expf(e.z), v.g * v.x.w * expf(e.w)));
        });
    copies_wait();
    __syncthreads();
    const Tile t;
    auto emit = [&](const auto &acc) {
        if (4 * t.tr >= nr) return;
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int blk = 0; blk < (int)(sizeof(acc[0]) / 16); ++blk) {
                if (t.col(blk) >= d.dv) continue;
                float *e = dst + (size_t)(r0 + 4 * t.tr + a) * d.dv + t.col(blk);
                float4 v = make_float4(acc[a][4 * blk], acc[a][4 * blk + 1], acc[a][4 * blk + 2], acc[a][4 * blk + 3]);
                if (ADD) {
                    const float4 w = *reinterpret_cast<const float4 *>(e);
                    v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
                }
                *reinterpret_cast<float4 *>(e) = v;
            }
    };
    if (d.dv <= 64) {
        float acc[4][4];
        zero_acc(acc);
        mm_outer<1>(acc, t, Xs, ldx, Ys, ldv, cn, nr, d.dv);
        emit(acc);
    } else {
        float acc[4][8];
        zero_acc(acc);
        mm_outer<2>(acc, t, Xs, ldx, Ys, ldv, cn, nr, d.dv);
        emit(acc);
    }
}

// The walk along the sequence, one thread per state element, in place over what k_chunk_outer left:
// GRAD = false: S_0 = h0, S_{n+1} = e^{b_last} S_n + KV_n (slot n: the state before chunk n; the last also to ht);
// GRAD = true, in reverse: slot NT-1 = dht, slot n-1 = e^{b_last,n} slot n + (qh^T dO)_n (n = 0: dh0, whose product lies in prod0 or,
// nullptr, comes later).  first and last may be one buffer.
template <bool GRAD>
__global__ void __launch_bounds__(256)
k_state_fold(Dims d, const float *__restrict__ bcum, const float *first, float *__restrict__ st, float *last, const float *prod0) {
    const int sz = d.dk * d.dv, e = blockIdx.x * blockDim.x + threadIdx.x, bh = blockIdx.y, b = bh / d.H, h = bh % d.H;
    if (e >= sz) return;
    const int c = e / d.dv, NT = d.NT, slots = GRAD ? NT : NT + 1;
    float *p = st + (size_t)bh * slots * sz + e;
    auto dec = [&](int n) { return bcum_at(d, bcum, tok_row(d, b, min((n + 1) * d.C, d.T) - 1, h), c); };
    float S = first ? first[(size_t)bh * sz + e] : 0.f;
    constexpr int U = 8;                     // chunks whose reads are in flight together
    for (int m0 = 0; m0 < NT; m0 += U) {
        float add[U], dc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int m = m0 + u, n = GRAD ? NT - 1 - m : m;
            add[u] = dc[u] = 0.f;
            if (m >= NT) continue;
            dc[u] = dec(n);
            add[u] = !GRAD ? p[(size_t)(n + 1) * sz] : n > 0 ? p[(size_t)(n - 1) * sz] : prod0 ? prod0[(size_t)bh * sz + e] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int m = m0 + u, n = GRAD ? NT - 1 - m : m;
            if (m >= NT) continue;
            p[(size_t)n * sz] = S;
            S = fmaf(expf(dc[u]), S, add[u]);
        }
    }
    if (!GRAD) p[(size_t)NT * sz] = S;
    if (last) last[(size_t)bh * sz + e] = S;
}

// ------------------------------------------------------------------------------------------
// a3 + a5: per tile, A = tril(qh kh^T) ; O = A V + qh S ; store in the I/O dtype (heads concatenated).
template <typename TIO>
__global__ void __launch_bounds__(256)
k_output(Dims d, const TIO *__restrict__ q, const TIO *__restrict__ k, const TIO *__restrict__ v,
         const float *__restrict__ Gq, const float *__restrict__ Gk, const float *__restrict__ bcum,
         const float *__restrict__ states, const float *__restrict__ Uws, TIO *__restrict__ o) {
    extern __shared__ float sm[];
    int n = blockIdx.x, bh = blockIdx.y, b = bh / d.H, h = bh % d.H;
    int t0 = n * d.C, cn = min(d.C, d.T - t0);
    const int ldk = pad4(d.dk), ldv = pad4(d.dv), cn4 = (cn + 3) & ~3;
    constexpr int lda = pad4(CMAX);
    float *Qs = sm;
    float *Ks = Qs + CMAX * ldk;
    float *Vs = Ks + CMAX * ldk;
    float *As = Vs + CMAX * ldv;
    float *Ss = As + CMAX * lda;             // [dk][ldv]
    const bool gdn = d.variant == SLA_GDN;
    const Tile t;

    const size_t v0 = tok_row(d, b, t0, h) * d.dv, vs = (size_t)d.H * d.dv;
    if (gdn) copy_rows(Vs, ldv, Uws, CMAX, cn, d.dv, v0, vs);
    else copy_rows(Vs, ldv, v, CMAX, cn, d.dv, v0, vs);
    copy_rows(Ss, ldv, states + state_off(d, bh, n, d.NT + 1), d.dk, d.dk, d.dv, 0, d.dv);
    load_qk_hat(d, q, k, Gq, Gk, bcum, b, h, t0, cn, Qs, Ks, ldk);
    copies_wait();
    __syncthreads();
    {
        float A[4][4];
        zero_acc(A);
        mm<1, false>(A, t, Qs, ldk, Ks, ldk, d.dk, CMAX);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = t.row(a), j = t.col(0);
            stf4(As, i * lda + j, make_float4(j <= i ? A[a][0] : 0.f, j + 1 <= i ? A[a][1] : 0.f, j + 2 <= i ? A[a][2] : 0.f, j + 3 <= i ? A[a][3] : 0.f));
        }
    }
    __syncthreads();
    auto emit = [&](const auto &acc) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = t.row(a);
            if (i >= cn) continue;
            const size_t row = tok_row(d, b, t0 + i, h) * d.dv;
#pragma unroll
            for (int blk = 0; blk < (int)(sizeof(acc[0]) / 16); ++blk)
                if (t.col(blk) < d.dv) stf4(o, row + t.col(blk), make_float4(acc[a][4 * blk], acc[a][4 * blk + 1], acc[a][4 * blk + 2], acc[a][4 * blk + 3]));
        }
    };
    if (d.dv <= 64) {
        float acc[4][4];
        zero_acc(acc);
        mm<1, true>(acc, t, As, lda, Vs, ldv, cn4, d.dv);
        mm<1, true>(acc, t, Qs, ldk, Ss, ldv, d.dk, d.dv);
        emit(acc);
    } else {
        float acc[4][8];
        zero_acc(acc);
        mm<2, true>(acc, t, As, lda, Vs, ldv, cn4, d.dv);
        mm<2, true>(acc, t, Qs, ldk, Ss, ldv, d.dk, d.dv);
        emit(acc);
    }
}

// The same for heads of at most 64 x 64, 512 threads in two groups of 256: the masked product beside qh S, then A V with the contraction
// halved; the groups' sums meet in shared memory, two row groups each.
template <typename TIO>
__global__ void __launch_bounds__(512)
k_output_narrow(Dims d, const TIO *__restrict__ q, const TIO *__restrict__ k, const TIO *__restrict__ v,
                const float *__restrict__ Gq, const float *__restrict__ Gk, const float *__restrict__ bcum,
                const float *__restrict__ states, const float *__restrict__ Uws, TIO *__restrict__ o) {
    extern __shared__ float sm[];
    const int n = blockIdx.x, bh = blockIdx.y, b = bh / d.H, h = bh % d.H;
    const int t0 = n * d.C, cn = min(d.C, d.T - t0), cn4 = (cn + 3) & ~3;
    const int ldk = pad4(d.dk), ldv = pad4(d.dv);
    constexpr int lda = pad4(CMAX);
    float *Qs = sm;
    float *Ks = Qs + CMAX * ldk;
    float *Vs = Ks + CMAX * ldk;
    float *As = Vs + CMAX * ldv;
    float *Ss = As + CMAX * lda;             // [dk][ldv]
    float *Xs = Ss + d.dk * ldv;             // [64][lda]: what a group hands the other
    const int grp = threadIdx.x >> 8;
    const Tile t(threadIdx.x & 255);

    const size_t v0 = tok_row(d, b, t0, h) * d.dv, vs = (size_t)d.H * d.dv;
    if (d.variant == SLA_GDN) copy_rows(Vs, ldv, Uws, CMAX, cn, d.dv, v0, vs);
    else copy_rows(Vs, ldv, v, CMAX, cn, d.dv, v0, vs);
    copy_rows(Ss, ldv, states + state_off(d, bh, n, d.NT + 1), d.dk, d.dk, d.dv, 0, d.dv);
    load_qk_hat(d, q, k, Gq, Gk, bcum, b, h, t0, cn, Qs, Ks, ldk);
    copies_wait();
    __syncthreads();
    float acc[4][4];
    zero_acc(acc);
    if (grp == 0) {
        float A[4][4];
        zero_acc(A);
        mm_tril(A, t, Qs, ldk, Ks, ldk, d.dk);
#pragma unroll
        for (int a = 0; a < 4; ++a) stf4(As, t.row(a) * lda + t.col(0), make_float4(A[a][0], A[a][1], A[a][2], A[a][3]));
    } else {
        mm<1, true>(acc, t, Qs, ldk, Ss, ldv, d.dk, d.dv);
    }
    __syncthreads();
    if (grp == 0) {                          // tokens 0 .. 31 of v
        mm<1, true, 0>(acc, t, As, lda, Vs, ldv, min(cn4, 16), d.dv);
        if (cn4 > 16) mm<1, true, 1>(acc, t, As + 16, lda, Vs + 16 * ldv, ldv, min(cn4 - 16, 16), d.dv);
    } else {
        if (cn4 > 32) mm<1, true, 2>(acc, t, As + 32, lda, Vs + 32 * ldv, ldv, min(cn4 - 32, 16), d.dv);
        if (cn4 > 48) mm<1, true, 3>(acc, t, As + 48, lda, Vs + 48 * ldv, ldv, cn4 - 48, d.dv);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
        if ((a >> 1) != grp) stf4(Xs, t.row(a) * lda + t.col(0), make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]));
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int i = t.row(a);
        if ((a >> 1) != grp || i >= cn || t.col(0) >= d.dv) continue;
        const float4 x = *reinterpret_cast<const float4 *>(Xs + i * lda + t.col(0));
        stf4(o, tok_row(d, b, t0 + i, h) * d.dv + t.col(0), make_float4(acc[a][0] + x.x, acc[a][1] + x.y, acc[a][2] + x.z, acc[a][3] + x.w));
    }
}

// ------------------------------------------------------------------------------------------
// backward for GDN, state-gradient pass (reverse chunk order).  grid (dv/VS, B*H), 256 threads on a [dk x VS] slice of dS.
// Stores dS entering each chunk from the right (slot n = gradient w.r.t. the state after chunk n) and
//   dU = Pq^T dO + diag(E) K dS ;  dS' = exp(b_last) dS + qh^T dO - W^T dU.
// Thread layout and reason as in k_state_scan (52 -> 11 us a chunk at d = 64).
template <typename TIO>
__global__ void __launch_bounds__(256)
k_dstate_scan(Dims d, const TIO *__restrict__ q, const TIO *__restrict__ k, const TIO *__restrict__ dO,
              const float *__restrict__ Gq, const float *__restrict__ bcum,
              const float *__restrict__ dht, float *__restrict__ dstates, float *__restrict__ dh0,
              const float *__restrict__ Wws, float *__restrict__ dUws) {
    extern __shared__ float sm[];
    const int vs0 = blockIdx.x * VS, bh = blockIdx.y, b = bh / d.H, h = bh % d.H, ldk = d.dk + 1, lda = CMAX + 1, tid = threadIdx.x;
    float *dSs = sm;                         // [dk][VS]
    float *dOs = dSs + d.dk * VS;            // [CMAX][VS]
    float *dUs = dOs + CMAX * VS;            // [CMAX][VS]
    float *Qs = dUs + CMAX * VS;             // [CMAX][ldk]  qh
    float *Ks = Qs + CMAX * ldk;             // [CMAX][ldk]  k*exp(-b)
    float *Ws = Ks + CMAX * ldk;             // [CMAX][ldk]
    float *Ps = Ws + CMAX * ldk;             // [CMAX][lda]  Pq
    const int i0 = tid >> 2, jq = 4 * (tid & 3), w4 = d.dk >> 2, ty = tid >> 5, tx = tid & 31;
    float4 dS[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int dd = i0 + 64 * x;
        dS[x] = (dd < d.dk && dht) ? ldf4(dht, ((size_t)bh * d.dk + dd) * d.dv + vs0 + jq) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    struct In { float4 q, k, w; float b, g; };
    for (int n = d.NT - 1; n >= 0; --n) {
        const int t0 = n * d.C, cn = min(d.C, d.T - t0);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int dd = i0 + 64 * x;
            if (dd >= d.dk) continue;
            *reinterpret_cast<float4 *>(dstates + state_off(d, bh, n, d.NT) + (size_t)dd * d.dv + vs0 + jq) = dS[x];
            *reinterpret_cast<float4 *>(dSs + dd * VS + jq) = dS[x];
        }
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        fill<4>(CMAX * w4,
            [&](int idx) {
                const int i = idx / w4;
                In x{zero, zero, zero, 0.f, 0.f};
                if (i < cn) {
                    const size_t row = tok_row(d, b, t0 + i, h), o = row * d.dk + 4 * (idx - i * w4);
                    x.q = ldf4(q, o);
                    x.k = ldf4(k, o);
                    x.w = ldf4(Wws, o);
                    x.b = bcum[row];
                    x.g = Gq[row];
                }
                return x;
            },
            [&](int idx, const In &x) {
                const int i = idx / w4, o = i * ldk + 4 * (idx - i * w4);
                const float g = d.scale * x.g, e = expf(x.b), m = expf(-x.b);
                put4(Qs + o, make_float4(g * x.q.x * e, g * x.q.y * e, g * x.q.z * e, g * x.q.w * e));
                put4(Ks + o, make_float4(x.k.x * m, x.k.y * m, x.k.z * m, x.k.w * m));
                put4(Ws + o, x.w);
            });
        *reinterpret_cast<float4 *>(dOs + i0 * VS + jq) = i0 < cn ? ldf4(dO, tok_row(d, b, t0 + i0, h) * d.dv + vs0 + jq) : zero;
        const float dec = expf(bcum[tok_row(d, b, t0 + cn - 1, h)]);
        __syncthreads();
        {
            float a[8][2];
            zero_acc(a);
            tile_gemm<2>(a, Qs, ldk, 1, Ks, 1, ldk, d.dk, CMAX, ty, tx);
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) {
                    const int i = ty + 8 * r, j = tx + 32 * cb;
                    Ps[i * lda + j] = (j <= i && i < cn) ? a[r][cb] : 0.f;
                }
        }
        __syncthreads();
        if (i0 < cn) {
            float4 acc = zero, acc2 = zero;
#pragma unroll 4
            for (int i2 = i0; i2 < cn; ++i2) {
                const float pv = Ps[i2 * lda + i0];
                const float4 g = *reinterpret_cast<const float4 *>(dOs + i2 * VS + jq);
                acc.x = fmaf(pv, g.x, acc.x); acc.y = fmaf(pv, g.y, acc.y); acc.z = fmaf(pv, g.z, acc.z); acc.w = fmaf(pv, g.w, acc.w);
            }
#pragma unroll 4
            for (int c = 0; c < d.dk; ++c) {
                const float kv = Ks[i0 * ldk + c];
                const float4 sv = *reinterpret_cast<const float4 *>(dSs + c * VS + jq);
                acc2.x = fmaf(kv, sv.x, acc2.x); acc2.y = fmaf(kv, sv.y, acc2.y); acc2.z = fmaf(kv, sv.z, acc2.z); acc2.w = fmaf(kv, sv.w, acc2.w);
            }
            acc.x = fmaf(dec, acc2.x, acc.x); acc.y = fmaf(dec, acc2.y, acc.y); acc.z = fmaf(dec, acc2.z, acc.z); acc.w = fmaf(dec, acc2.w, acc.w);
            *reinterpret_cast<float4 *>(dUs + i0 * VS + jq) = acc;
            *reinterpret_cast<float4 *>(dUws + tok_row(d, b, t0 + i0, h) * d.dv + vs0 + jq) = acc;
        }
        __syncthreads();
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int dd = i0 + 64 * x;
            if (dd >= d.dk) continue;
            float4 v = dS[x];
            v.x *= dec; v.y *= dec; v.z *= dec; v.w *= dec;
#pragma unroll 4
            for (int i = 0; i < cn; ++i) {
                const float qv = Qs[i * ldk + dd];
                const float4 g = *reinterpret_cast<const float4 *>(dOs + i * VS + jq);
                v.x = fmaf(qv, g.x, v.x); v.y = fmaf(qv, g.y, v.y); v.z = fmaf(qv, g.z, v.z); v.w = fmaf(qv, g.w, v.w);
            }
#pragma unroll 4
            for (int i = 0; i < cn; ++i) {
                const float wv = -Ws[i * ldk + dd];
                const float4 u = *reinterpret_cast<const float4 *>(dUs + i * VS + jq);
                v.x = fmaf(wv, u.x, v.x); v.y = fmaf(wv, u.y, v.y); v.z = fmaf(wv, u.z, v.z); v.w = fmaf(wv, u.w, v.w);
            }
            dS[x] = v;
        }
        __syncthreads();
    }
    if (dh0) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int dd = i0 + 64 * x;
            if (dd < d.dk) *reinterpret_cast<float4 *>(dh0 + ((size_t)bh * d.dk + dd) * d.dv + vs0 + jq) = dS[x];
        }
    }
}

// ------------------------------------------------------------------------------------------
// backward, per-tile gradients for RETNET / GLA.
//   dA = tril(dO V^T) ; dZ = diag(exp(b_last)) dS_next
//   dqh = dA kh + dO S^T ; dkh = dA^T qh + V dZ^T ; dV = A^T dO + kh dZ
//   db = qh*dqh - kh*dkh (+ rowsum(dS_next*S_next) on the last row) ; dlog_decay = suffix sum of db
// The three matrices dA, dA^T, A^T take turns in one buffer (heads of 128 leave room for one), kept in registers meanwhile.
// NB: 64-column blocks of the wider of the two head widths.
template <typename TIO, int NB>
__global__ void __launch_bounds__(256)
k_grads_lin(Dims d, const TIO *__restrict__ q, const TIO *__restrict__ k, const TIO *__restrict__ v,
            const TIO *__restrict__ dO, const float *__restrict__ Gq, const float *__restrict__ Gk,
            const float *__restrict__ bcum, const float *__restrict__ states,
            const float *__restrict__ dstates, TIO *__restrict__ dq, TIO *__restrict__ dk,
            TIO *__restrict__ dv, float *__restrict__ dlog_decay, float *__restrict__ dGq,
            float *__restrict__ dGk) {
    extern __shared__ float sm[];
    const int n = blockIdx.x, bh = blockIdx.y, b = bh / d.H, h = bh % d.H;
    const int t0 = n * d.C, cn = min(d.C, d.T - t0), cn4 = (cn + 3) & ~3;
    const int ldk = pad4(d.dk), ldv = pad4(d.dv);
    constexpr int lda = pad4(CMAX);
    float *Qs = sm;
    float *Ks = Qs + CMAX * ldk;
    float *Vs = Ks + CMAX * ldk;
    float *dOs = Vs + CMAX * ldv;
    float *Ms = dOs + CMAX * ldv;             // dA, then dA^T, then A^T
    float *Ss = Ms + CMAX * lda;              // [dk][ldv]: S, then dZ
    float *Rs = Ss + d.dk * ldv;              // [dk]
    float *red = Rs + d.dk;                   // [2][4][CMAX] a token's gate sums, by quarter of the columns
    const int ty = threadIdx.x >> 5, tx = threadIdx.x & 31;
    const Tile t;
    const size_t row_last = tok_row(d, b, t0 + cn - 1, h);

    const size_t v0 = tok_row(d, b, t0, h) * d.dv, vs = (size_t)d.H * d.dv;
    copy_rows(Vs, ldv, v, CMAX, cn, d.dv, v0, vs);
    copy_rows(dOs, ldv, dO, CMAX, cn, d.dv, v0, vs);
    copy_rows(Ss, ldv, states + state_off(d, bh, n, d.NT + 1), d.dk, d.dk, d.dv, 0, d.dv);
    load_qk_hat<4>(d, q, k, Gq, Gk, bcum, b, h, t0, cn, Qs, Ks, ldk);
    copies_wait();
    __syncthreads();
    float A[4][4], dA[4][4];
    zero_acc(A);
    zero_acc(dA);
    mm<1, false>(A, t, Qs, ldk, Ks, ldk, d.dk, CMAX);
    mm<1, false>(dA, t, dOs, ldv, Vs, ldv, d.dv, CMAX);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (t.col(0) + c > t.row(a)) A[a][c] = dA[a][c] = 0.f;
#pragma unroll
    for (int a = 0; a < 4; ++a) stf4(Ms, t.row(a) * lda + t.col(0), make_float4(dA[a][0], dA[a][1], dA[a][2], dA[a][3]));
    auto transposed = [&](const float (&m)[4][4]) {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) Ms[(t.col(0) + c) * lda + t.row(a)] = m[a][c];
    };
    // a token's sum over this thread's columns -> its quarter's slot (four lanes share a row)
    auto row_sum = [&](float s, int which, int i) {
        s += __shfl_xor_sync(FULL, s, 1);
        s += __shfl_xor_sync(FULL, s, 2);
        if ((tx & 3) == 0) red[(4 * which + (ty >> 1)) * CMAX + i] = s;
    };
    __syncthreads();
    float db[4][4 * NB];
    {   // dqh and the query-side outputs
        float acc[4][4 * NB];
        zero_acc(acc);
        mm<NB, true>(acc, t, Ms, lda, Ks, ldk, cn4, d.dk);
        mm<NB, false>(acc, t, dOs, ldv, Ss, ldv, d.dv, d.dk);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = t.row(a);
            const size_t row = i < cn ? tok_row(d, b, t0 + i, h) : 0;
            const float gq = i < cn ? Gq[row] : 0.f;
            float gsum = 0.f;
#pragma unroll
            for (int blk = 0; blk < NB; ++blk) {
                const int c = t.col(blk);
                float *dbv = &db[a][4 * blk], *y = &acc[a][4 * blk];
#pragma unroll
                for (int e = 0; e < 4; ++e) dbv[e] = 0.f;
                if (i >= cn || c >= d.dk) continue;
                const float4 qh = *reinterpret_cast<const float4 *>(Qs + i * ldk + c), bc = bcum_at4(d, bcum, row, c), qv = ldf4(q, row * d.dk + c);
                dbv[0] = qh.x * y[0]; dbv[1] = qh.y * y[1]; dbv[2] = qh.z * y[2]; dbv[3] = qh.w * y[3];
                const float4 g = make_float4(y[0] * expf(bc.x), y[1] * expf(bc.y), y[2] * expf(bc.z), y[3] * expf(bc.w));
                gsum = fmaf(d.scale * qv.x, g.x, fmaf(d.scale * qv.y, g.y, fmaf(d.scale * qv.z, g.z, fmaf(d.scale * qv.w, g.w, gsum))));
                const float f = d.scale * gq;
                stf4(dq, row * d.dk + c, make_float4(f * g.x, f * g.y, f * g.z, f * g.w));
            }
            row_sum(gsum, 0, i);
        }
    }
    __syncthreads();
    transposed(dA);
    {   // Ss <- dZ = diag(exp(b_last)) dS_next ; Rs <- rowsum(dS_next * S_next)
        const float *dSg = dstates + state_off(d, bh, n, d.NT);
        const float *Sn = states + state_off(d, bh, n + 1, d.NT + 1);
#pragma unroll 4
        for (int r0 = ty; r0 < d.dk; r0 += 8) {
            const float e = expf(bcum_at(d, bcum, row_last, r0));
            float part = 0.f;
            const int j = 4 * tx;
            if (j < d.dv) {
                const float4 g = ldf4(dSg, (size_t)r0 * d.dv + j), s = ldf4(Sn, (size_t)r0 * d.dv + j);
                part = fmaf(g.x, s.x, fmaf(g.y, s.y, fmaf(g.z, s.z, g.w * s.w)));
                stf4(Ss, r0 * ldv + j, make_float4(e * g.x, e * g.y, e * g.z, e * g.w));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
            if (tx == 0) Rs[r0] = part;
        }
    }
    __syncthreads();
    {   // dkh and the key-side outputs
        float acc[4][4 * NB];
        zero_acc(acc);
        mm<NB, true>(acc, t, Ms, lda, Qs, ldk, cn4, d.dk);
        mm<NB, false>(acc, t, Vs, ldv, Ss, ldv, d.dv, d.dk);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = t.row(a);
            const size_t row = i < cn ? tok_row(d, b, t0 + i, h) : 0;
            const float gk = i < cn ? Gk[row] : 0.f;
            float gsum = 0.f;
#pragma unroll
            for (int blk = 0; blk < NB; ++blk) {
                const int c = t.col(blk);
                if (i >= cn || c >= d.dk) continue;
                float *dbv = &db[a][4 * blk], *y = &acc[a][4 * blk];
                const float4 kh = *reinterpret_cast<const float4 *>(Ks + i * ldk + c), bc = bcum_at4(d, bcum, row, c), kv = ldf4(k, row * d.dk + c);
                dbv[0] -= kh.x * y[0]; dbv[1] -= kh.y * y[1]; dbv[2] -= kh.z * y[2]; dbv[3] -= kh.w * y[3];
                const float4 g = make_float4(y[0] * expf(-bc.x), y[1] * expf(-bc.y), y[2] * expf(-bc.z), y[3] * expf(-bc.w));
                gsum = fmaf(kv.x, g.x, fmaf(kv.y, g.y, fmaf(kv.z, g.z, fmaf(kv.w, g.w, gsum))));
                stf4(dk, row * d.dk + c, make_float4(gk * g.x, gk * g.y, gk * g.z, gk * g.w));
            }
            row_sum(gsum, 1, i);
        }
    }
    __syncthreads();
    transposed(A);
    if (threadIdx.x < 2 * CMAX) {     // the gates' gradients: a token's four quarters
        const int which = threadIdx.x / CMAX, i = threadIdx.x % CMAX;
        const float *r = red + 4 * which * CMAX + i;
        if (i < cn) (which ? dGk : dGq)[tok_row(d, b, t0 + i, h)] = (r[0] + r[CMAX]) + (r[2 * CMAX] + r[3 * CMAX]);
    }
    __syncthreads();
    {   // dV = A^T dO + kh dZ
        float acc[4][4 * NB];
        zero_acc(acc);
        mm<NB, true>(acc, t, Ms, lda, dOs, ldv, cn4, d.dv);
        mm<NB, true>(acc, t, Ks, ldk, Ss, ldv, d.dk, d.dv);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = t.row(a);
            if (i >= cn) continue;
            const size_t row = tok_row(d, b, t0 + i, h) * d.dv;
#pragma unroll
            for (int blk = 0; blk < NB; ++blk)
                if (t.col(blk) < d.dv) stf4(dv, row + t.col(blk), make_float4(acc[a][4 * blk], acc[a][4 * blk + 1], acc[a][4 * blk + 2], acc[a][4 * blk + 3]));
        }
    }
    if (d.variant != SLA_GLA || !dlog_decay) return;
    // db over Qs, whose last reader was the key side; warp w the suffix sums of tokens 8w .. 8w+7, the warps' totals over Vs
    float *dbs = Qs, *tot = Vs;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int blk = 0; blk < NB; ++blk)
            if (t.col(blk) < d.dk)
                stf4(dbs, t.row(a) * ldk + t.col(blk), make_float4(db[a][4 * blk], db[a][4 * blk + 1], db[a][4 * blk + 2], db[a][4 * blk + 3]));
    __syncthreads();
    const int c = 4 * tx;
    float4 x[8], run = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < d.dk) {
#pragma unroll
        for (int i = 7; i >= 0; --i) {
            x[i] = *reinterpret_cast<const float4 *>(dbs + (8 * ty + i) * ldk + c);
            run.x += x[i].x; run.y += x[i].y; run.z += x[i].z; run.w += x[i].w;
        }
        stf4(tot, ty * ldk + c, run);
    }
    __syncthreads();
    if (c >= d.dk) return;
    run = *reinterpret_cast<const float4 *>(Rs + c);
    for (int g = 7; g > ty; --g) {
        const float4 y = *reinterpret_cast<const float4 *>(tot + g * ldk + c);
        run.x += y.x; run.y += y.y; run.z += y.z; run.w += y.w;
    }
#pragma unroll
    for (int i = 7; i >= 0; --i) {
        run.x += x[i].x; run.y += x[i].y; run.z += x[i].z; run.w += x[i].w;
        if (8 * ty + i < cn) stf4(dlog_decay, tok_row(d, b, t0 + 8 * ty + i, h) * d.dk + c, run);
    }
}

// The same for heads of at most 64 x 64: everything has room at once, so 512 threads in two groups of 256 take a product of every result
// each - A beside dA; then dA kh, dA^T qh, A^T dO (triangular: their blocks of zeros are left out) beside dO S^T, V dZ^T, kh dZ -
// without a barrier in between, and finish two row groups each after one exchange.  k_grads_lin's one group runs through eight phases with
// eight warps on an SM; what bounds both is the shared-memory pipe and, with so few warps, its latency.  2 x 1000 tokens x 4 heads of 64 (128 chunks): 37 ->
// 28 us, k_output 15 -> 12.  (The blocks of zeros left out in k_output and k_grads_lin, too: 4 x 2048 tokens x 8 heads of 32 slower by 6 to 10 %, 8 x 2048 x 16
// of 64 forward 424 -> 409 us, backward 974 -> 1008.)
template <typename TIO>
__global__ void __launch_bounds__(512)
k_grads_narrow(Dims d, const TIO *__restrict__ q, const TIO *__restrict__ k, const TIO *__restrict__ v,
               const TIO *__restrict__ dO, const float *__restrict__ Gq, const float *__restrict__ Gk,
               const float *__restrict__ bcum, const float *__restrict__ states,
               const float *__restrict__ dstates, TIO *__restrict__ dq, TIO *__restrict__ dk,
               TIO *__restrict__ dv, float *__restrict__ dlog_decay, float *__restrict__ dGq,
               float *__restrict__ dGk) {
    extern __shared__ float sm[];
    const int n = blockIdx.x, bh = blockIdx.y, b = bh / d.H, h = bh % d.H;
    const int t0 = n * d.C, cn = min(d.C, d.T - t0), cn4 = (cn + 3) & ~3;
    const int ldk = pad4(d.dk), ldv = pad4(d.dv);
    constexpr int lda = pad4(CMAX);
    float *Qs = sm;
    float *Ks = Qs + CMAX * ldk;
    float *Vs = Ks + CMAX * ldk;
    float *dOs = Vs + CMAX * ldv;
    float *Ss = dOs + CMAX * ldv;             // [dk][ldv]
    float *Zs = Ss + d.dk * ldv;              // [dk][ldv]: dZ
    float *Ms = Zs + d.dk * ldv;              // [3][64][lda]: dA, dA^T, A^T; then the exchange of dqh, dkh, dV
    float *Rs = Ms + 3 * CMAX * lda;          // [dk]
    float *red = Rs + d.dk;                   // [2][4][CMAX] a token's gate sums, by quarter of the columns
    const int grp = threadIdx.x >> 8, warp = threadIdx.x >> 5, tx = threadIdx.x & 31;
    const Tile t(threadIdx.x & 255);
    const size_t row_last = tok_row(d, b, t0 + cn - 1, h);
    const bool decay_grad = d.variant == SLA_GLA && dlog_decay;

    const size_t v0 = tok_row(d, b, t0, h) * d.dv, vs = (size_t)d.H * d.dv;
    copy_rows(Vs, ldv, v, CMAX, cn, d.dv, v0, vs);
    copy_rows(dOs, ldv, dO, CMAX, cn, d.dv, v0, vs);
    copy_rows(Ss, ldv, states + state_off(d, bh, n, d.NT + 1), d.dk, d.dk, d.dv, 0, d.dv);
    load_qk_hat(d, q, k, Gq, Gk, bcum, b, h, t0, cn, Qs, Ks, ldk);
    {   // Zs <- dZ = diag(exp(b_last)) dS_next ; Rs <- rowsum(dS_next * S_next); half a warp a row
        const float *dSg = dstates + state_off(d, bh, n, d.NT);
        const float *Sn = states + state_off(d, bh, n + 1, d.NT + 1);
        const int j = 4 * (tx & 15);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int r0 = 32 * x + 2 * warp + (tx >> 4);
            float part = 0.f;
            if (r0 < d.dk && j < d.dv) {
                const float e = expf(bcum_at(d, bcum, row_last, r0));
                const float4 g = ldf4(dSg, (size_t)r0 * d.dv + j);
                if (decay_grad) {
                    const float4 y = ldf4(Sn, (size_t)r0 * d.dv + j);
                    part = fmaf(g.x, y.x, fmaf(g.y, y.y, fmaf(g.z, y.z, g.w * y.w)));
                }
                stf4(Zs, r0 * ldv + j, make_float4(e * g.x, e * g.y, e * g.z, e * g.w));
            }
            if (decay_grad) {
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
                if ((tx & 15) == 0 && r0 < d.dk) Rs[r0] = part;
            }
        }
    }
    copies_wait();
    __syncthreads();
    {
        float A[4][4];                        // A; the second group: dA
        zero_acc(A);
        if (grp == 0) mm_tril(A, t, Qs, ldk, Ks, ldk, d.dk);
        else mm_tril(A, t, dOs, ldv, Vs, ldv, d.dv);
        float *Mt = Ms + (grp == 0 ? 2 : 1) * CMAX * lda;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            if (grp) stf4(Ms, t.row(a) * lda + t.col(0), make_float4(A[a][0], A[a][1], A[a][2], A[a][3]));
#pragma unroll
            for (int c = 0; c < 4; ++c) Mt[(t.col(0) + c) * lda + t.row(a)] = A[a][c];
        }
    }
    __syncthreads();
    float acc[3][4][4];                       // this group's half of dqh, dkh, dV
#pragma unroll
    for (int x = 0; x < 3; ++x) zero_acc(acc[x]);
    if (grp == 0) {
        mm_lower(acc[0], t, Ms, lda, Ks, ldk, cn4, d.dk);
        mm_upper(acc[1], t, Ms + CMAX * lda, lda, Qs, ldk, cn4, d.dk);
        mm_upper(acc[2], t, Ms + 2 * CMAX * lda, lda, dOs, ldv, cn4, d.dv);
    } else {
        mm<1, false>(acc[0], t, dOs, ldv, Ss, ldv, d.dv, d.dk);
        mm<1, false>(acc[1], t, Vs, ldv, Zs, ldv, d.dv, d.dk);
        mm<1, true>(acc[2], t, Ks, ldk, Zs, ldv, d.dk, d.dv);
    }
    const int c = t.col(0);
    struct Raw { float4 q, k, b; float gq, gk; } in[2];      // of the two rows this thread finishes, on their way during the exchange
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int i = t.row(0) + 16 * (2 * grp + x);
        if (i < cn && c < d.dk) {
            const size_t row = tok_row(d, b, t0 + i, h);
            in[x].q = ldf4(q, row * d.dk + c);
            in[x].k = ldf4(k, row * d.dk + c);
            in[x].b = bcum_at4(d, bcum, row, c);
            in[x].gq = Gq[row];
            in[x].gk = Gk[row];
        }
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if ((a >> 1) != grp) stf4(Ms, (x * CMAX + t.row(a)) * lda + c, make_float4(acc[x][a][0], acc[x][a][1], acc[x][a][2], acc[x][a][3]));
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        const int i = t.row(0) + 16 * (2 * grp + x);
        auto sum = [&](int m) {
            const float4 y = *reinterpret_cast<const float4 *>(Ms + (m * CMAX + i) * lda + c);
            const float (&lo)[4] = acc[m][x], (&hi)[4] = acc[m][2 + x];
            return make_float4((grp ? hi[0] : lo[0]) + y.x, (grp ? hi[1] : lo[1]) + y.y, (grp ? hi[2] : lo[2]) + y.z, (grp ? hi[3] : lo[3]) + y.w);
        };
        float sq = 0.f, sk = 0.f;
        float4 db = make_float4(0.f, 0.f, 0.f, 0.f);
        const size_t row = i < cn ? tok_row(d, b, t0 + i, h) : 0;
        if (i < cn && c < d.dk) {
            const Raw &r = in[x];
            const float4 yq = sum(0), yk = sum(1);
            const float4 qh = *reinterpret_cast<const float4 *>(Qs + i * ldk + c), kh = *reinterpret_cast<const float4 *>(Ks + i * ldk + c);
            db = make_float4(qh.x * yq.x - kh.x * yk.x, qh.y * yq.y - kh.y * yk.y, qh.z * yq.z - kh.z * yk.z, qh.w * yq.w - kh.w * yk.w);
            const float4 g = make_float4(yq.x * expf(r.b.x), yq.y * expf(r.b.y), yq.z * expf(r.b.z), yq.w * expf(r.b.w));
            sq = fmaf(d.scale * r.q.x, g.x, fmaf(d.scale * r.q.y, g.y, fmaf(d.scale * r.q.z, g.z, d.scale * r.q.w * g.w)));
            const float f = d.scale * r.gq;
            stf4(dq, row * d.dk + c, make_float4(f * g.x, f * g.y, f * g.z, f * g.w));
            const float4 u = make_float4(yk.x * expf(-r.b.x), yk.y * expf(-r.b.y), yk.z * expf(-r.b.z), yk.w * expf(-r.b.w));
            sk = fmaf(r.k.x, u.x, fmaf(r.k.y, u.y, fmaf(r.k.z, u.z, r.k.w * u.w)));
            stf4(dk, row * d.dk + c, make_float4(r.gk * u.x, r.gk * u.y, r.gk * u.z, r.gk * u.w));
        }
        if (i < cn && c < d.dv) stf4(dv, row * d.dv + c, sum(2));
        if (decay_grad && c < d.dk) stf4(Qs, i * ldk + c, db);          // its own elements: nobody else reads them here
        // a token's sums over this thread's columns -> its quarter's slots (four lanes share a row)
        sq += __shfl_xor_sync(FULL, sq, 1);
        sk += __shfl_xor_sync(FULL, sk, 1);
        sq += __shfl_xor_sync(FULL, sq, 2);
        sk += __shfl_xor_sync(FULL, sk, 2);
        if ((tx & 3) == 0) {
            red[(t.tc >> 2) * CMAX + i] = sq;
            red[(4 + (t.tc >> 2)) * CMAX + i] = sk;
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 * CMAX) {     // the gates' gradients: a token's four quarters
        const int which = threadIdx.x / CMAX, i = threadIdx.x % CMAX;
        const float *r = red + 4 * which * CMAX + i;
        if (i < cn) (which ? dGk : dGq)[tok_row(d, b, t0 + i, h)] = (r[0] + r[CMAX]) + (r[2 * CMAX] + r[3 * CMAX]);
    }
    if (!decay_grad) return;
    // warp w the suffix sums of tokens 4w .. 4w+3, the warps' totals over Vs
    float *tot = Vs;
    const int e = 4 * tx;
    float4 x[4], run = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < d.dk) {
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            x[i] = *reinterpret_cast<const float4 *>(Qs + (4 * warp + i) * ldk + e);
            run.x += x[i].x; run.y += x[i].y; run.z += x[i].z; run.w += x[i].w;
        }
        stf4(tot, warp * ldk + e, run);
    }
    __syncthreads();
    if (e >= d.dk) return;
    run = *reinterpret_cast<const float4 *>(Rs + e);
    for (int g = 15; g > warp; --g) {
        const float4 y = *reinterpret_cast<const float4 *>(tot + g * ldk + e);
        run.x += y.x; run.y += y.y; run.z += y.z; run.w += y.w;
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) {
        run.x += x[i].x; run.y += x[i].y; run.z += x[i].z; run.w += x[i].w;
        if (4 * warp + i < cn) stf4(dlog_decay, tok_row(d, b, t0 + 4 * warp + i, h) * d.dk + e, run);
    }
}

// ------------------------------------------------------------------------------------------
// host side
size_t smem_prepare(const Dims &d) {
    return sizeof(float) * (CMAX * (d.dk + 1) + CMAX * (CMAX + 1) + CMAX * (d.dk + d.dv) + 2 * CMAX);
}
size_t smem_scan(const Dims &d) {
    return sizeof(float) * (2 * CMAX * (d.dk + 1) + CMAX * VS + d.dk * VS + CMAX);
}
size_t smem_outer(const Dims &d) { return sizeof(float) * CMAX * (pad4(64) + pad4(d.dv)); }
size_t smem_output(const Dims &d) {
    return sizeof(float) * (2 * CMAX * pad4(d.dk) + CMAX * pad4(d.dv) + CMAX * pad4(CMAX) + d.dk * pad4(d.dv));
}
size_t smem_output_narrow(const Dims &d) { return smem_output(d) + sizeof(float) * CMAX * pad4(CMAX); }
size_t smem_grads_narrow(const Dims &d) {
    return sizeof(float) * (2 * CMAX * pad4(d.dk) + 2 * CMAX * pad4(d.dv) + 3 * CMAX * pad4(CMAX) + 2 * d.dk * pad4(d.dv) + d.dk + 8 * CMAX);
}
// Heads of at most 64 x 64 on few chunks: no SM gets a second CTA.  Softmax-RetNet, 4 heads x 2 sequences, forward and step, us, general -> narrow:
// 128 chunks of 64 x 64 26.9 and 85.6 -> 24.9 and 75.9, 144 27.2 and 89.6 -> 25.4 and 78.0, of 32 x 32 20.2 and 63.7 -> 19.8 and 60.2; past one a SM two CTAs of
// the general kernels hide one another's phases: 152 chunks 36.4 and 117.5 -> 36.9 and 117.8 (32 x 32: 23.8 and 73.5 -> 25.3 and 78.6), 256
// 38.7 and 125.2 -> 40.0 and 126.3, 512 64.4 and 214 -> 67.6 and 222.
bool narrow(const Dims &d) {
    static const int sms = [] {
        int dev = 0, n = 0;
        return cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0 ? n : 148;
    }();
    return d.dk <= 64 && d.dv <= 64 && (long)d.NT * d.B * d.H <= sms;
}
size_t smem_dscan(const Dims &d) {
    return sizeof(float) * (3 * CMAX * (d.dk + 1) + 2 * CMAX * VS + CMAX * (CMAX + 1) + d.dk * VS);
}
size_t smem_grads_lin(const Dims &d) {
    return sizeof(float) * (2 * CMAX * pad4(d.dk) + 2 * CMAX * pad4(d.dv) + CMAX * pad4(CMAX) + d.dk * pad4(d.dv) + d.dk + 8 * CMAX);
}

template <int HP>
void launch_gates_decay(const Dims &d, const Workspace &w, const FwdArgs &a, cudaStream_t st) {
    const long chunks = (long)d.B * d.H * d.NT;
    const int gate_blocks = (int)(((long)d.B * d.T * HP + 255) / 256);
    const long decay_blocks = d.variant == SLA_GLA ? chunks : (chunks + 7) / 8;
    k_gates_decay<HP><<<(unsigned)(gate_blocks + decay_blocks), 256, 0, st>>>(d, a.lq, a.lk, a.ws + w.Gq, a.ws + w.Gk, a.log_decay, a.ws + w.bcum,
                                                                              gate_blocks, a.status);
}
template <int HP>
void launch_gate_bwd(const float *Gq, const float *Gk, const float *dGq, const float *dGk, float *dlq,
                     float *dlk, long n_tok, int H, cudaStream_t st) {
    long threads = n_tok * HP;
    dim3 grid((unsigned)((threads + 255) / 256), 2);
    k_gate_bwd<HP><<<grid, 256, 0, st>>>(Gq, Gk, dGq, dGk, dlq, dlk, n_tok, H);
}

template <typename TIO>
int forward_t(const Dims &d, const Workspace &w, const FwdArgs &a, bool write_o, cudaStream_t st, Tracer &tr) {
    float *ws = a.ws;
    float *Gq = ws + w.Gq, *Gk = ws + w.Gk, *bcum = ws + w.bcum, *states = ws + w.states;
    float *Wws = ws + w.W, *U0ws = ws + w.U0, *Uws = ws + w.U;
    int launches = 0;
    int hp = 1;
    while (hp < d.H) hp <<= 1;
    switch (hp) {
        case 1: launch_gates_decay<1>(d, w, a, st); break;
        case 2: launch_gates_decay<2>(d, w, a, st); break;
        case 4: launch_gates_decay<4>(d, w, a, st); break;
        case 8: launch_gates_decay<8>(d, w, a, st); break;
        case 16: launch_gates_decay<16>(d, w, a, st); break;
        default: launch_gates_decay<32>(d, w, a, st); break;
    }
    tr.mark("gates_decay");
    ++launches;
    const dim3 tiles(d.NT, d.B * d.H);
    const TIO *q = (const TIO *)a.q, *k = (const TIO *)a.k, *v = (const TIO *)a.v;
    if (d.variant == SLA_GDN) {
        k_gdn_prepare<TIO><<<tiles, 256, smem_prepare(d), st>>>(d, k, v, a.beta, Gk, bcum, Wws, U0ws);
        tr.mark("gdn_prepare");
        ++launches;
    }
    if (d.variant == SLA_GDN) {
        dim3 slices(d.dv / VS, d.B * d.H);
        k_state_scan<TIO><<<slices, 256, smem_scan(d), st>>>(d, k, bcum, a.h0, states, a.ht, Wws, U0ws, Uws);
        tr.mark("state_scan");
        ++launches;
    } else {
        k_chunk_outer<TIO, false><<<dim3(d.NT, d.B * d.H, (d.dk + 63) / 64), 256, smem_outer(d), st>>>(d, k, v, Gk, bcum, states, nullptr);
        tr.mark("chunk_outer");
        k_state_fold<false><<<dim3((d.dk * d.dv + 255) / 256, d.B * d.H), 256, 0, st>>>(d, bcum, a.h0, states, a.ht, nullptr);
        tr.mark("state_fold");
        launches += 2;
    }
    if (write_o) {
        if (narrow(d)) k_output_narrow<TIO><<<tiles, 512, smem_output_narrow(d), st>>>(d, q, k, v, Gq, Gk, bcum, states, Uws, (TIO *)a.o);
        else k_output<TIO><<<tiles, 256, smem_output(d), st>>>(d, q, k, v, Gq, Gk, bcum, states, Uws, (TIO *)a.o);
        tr.mark("output");
        ++launches;
    }
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

template <typename TIO>
int backward_lin_t(const Dims &d, const Workspace &w, const BwdArgs &a, cudaStream_t st, Tracer &tr) {
    float *ws = a.ws;
    float *Gq = ws + w.Gq, *Gk = ws + w.Gk, *bcum = ws + w.bcum, *states = ws + w.states;
    float *dstates = ws + w.dstates, *dGq = ws + w.dGq, *dGk = ws + w.dGk;
    int launches = 0;
    const TIO *q = (const TIO *)a.q, *k = (const TIO *)a.k, *v = (const TIO *)a.v, *dO = (const TIO *)a.dO;
    dim3 tiles(d.NT, d.B * d.H);
    // dh0 may be dht's own buffer: the first chunk's product must not go there before dht has been read
    const bool in_place = a.dh0 && a.dh0 == a.dht;
    float *prod0 = in_place ? nullptr : a.dh0;
    k_chunk_outer<TIO, true><<<dim3(d.NT, d.B * d.H, (d.dk + 63) / 64), 256, smem_outer(d), st>>>(d, q, dO, Gq, bcum, dstates, prod0);
    tr.mark("chunk_outer");
    k_state_fold<true><<<dim3((d.dk * d.dv + 255) / 256, d.B * d.H), 256, 0, st>>>(d, bcum, a.dht, dstates, a.dh0, prod0);
    tr.mark("state_fold");
    launches += 2;
    if (in_place) {
        k_chunk_outer<TIO, true, true><<<dim3(1, d.B * d.H, (d.dk + 63) / 64), 256, smem_outer(d), st>>>(d, q, dO, Gq, bcum, nullptr, a.dh0);
        tr.mark("chunk_outer");
        ++launches;
    }
    (narrow(d) ? k_grads_narrow<TIO> : d.dk <= 64 && d.dv <= 64 ? k_grads_lin<TIO, 1> : k_grads_lin<TIO, 2>)<<<tiles, narrow(d) ? 512 : 256, narrow(d) ? smem_grads_narrow(d) : smem_grads_lin(d), st>>>(
        d, q, k, v, dO, Gq, Gk, bcum, states, dstates, (TIO *)a.dq, (TIO *)a.dk, (TIO *)a.dv, a.dlog_decay, dGq, dGk);
    tr.mark("grads_lin");
    ++launches;
    return cudaGetLastError() == cudaSuccess ? launches : -1;
}

template <typename TIO> bool configure_t() {
    Dims d{};
    d.dk = d.dv = 128;
    bool ok = true;
    ok &= set_smem(k_gdn_prepare<TIO>, smem_prepare(d));
    ok &= set_smem(k_state_scan<TIO>, smem_scan(d));
    ok &= set_smem(k_output<TIO>, smem_output(d));
    ok &= set_smem(k_chunk_outer<TIO, false>, smem_outer(d)) && set_smem(k_chunk_outer<TIO, true>, smem_outer(d)) &&
          set_smem(k_chunk_outer<TIO, true, true>, smem_outer(d));
    ok &= set_smem(k_dstate_scan<TIO>, smem_dscan(d));
    ok &= set_smem(k_grads_lin<TIO, 1>, smem_grads_lin(d)) && set_smem(k_grads_lin<TIO, 2>, smem_grads_lin(d));
    d.dk = d.dv = 64;
    ok &= set_smem(k_output_narrow<TIO>, smem_output_narrow(d)) && set_smem(k_grads_narrow<TIO>, smem_grads_narrow(d));
    return ok;
}

}  // namespace

int generic_configure(bool bf16) { return (bf16 ? configure_t<__nv_bfloat16>() : configure_t<float>()) ? 0 : -1; }

int generic_forward(const Dims &d, const Workspace &w, const FwdArgs &a, bool write_o, cudaStream_t st, Tracer &tr) {
    return d.io_bf16 ? forward_t<__nv_bfloat16>(d, w, a, write_o, st, tr) : forward_t<float>(d, w, a, write_o, st, tr);
}

int generic_backward(const Dims &d, const Workspace &w, const BwdArgs &a, cudaStream_t st, Tracer &tr) {
    // recompute gates, cumulative decays and the per-chunk states (no output store)
    FwdArgs f{a.q, a.k, a.v, a.log_decay, a.beta, a.lq, a.lk, a.h0, nullptr, nullptr, a.ws, a.status};
    int n1 = generic_forward(d, w, f, false, st, tr);
    if (n1 < 0) return -1;
    int n2;
    if (d.variant == SLA_GDN) {
        float *ws = a.ws;
        dim3 slices(d.dv / VS, d.B * d.H);
        if (d.io_bf16)
            k_dstate_scan<__nv_bfloat16><<<slices, 256, smem_dscan(d), st>>>(
                d, (const __nv_bfloat16 *)a.q, (const __nv_bfloat16 *)a.k, (const __nv_bfloat16 *)a.dO, ws + w.Gq,
                ws + w.bcum, a.dht, ws + w.dstates, a.dh0, ws + w.W, ws + w.dU);
        else
            k_dstate_scan<float><<<slices, 256, smem_dscan(d), st>>>(
                d, (const float *)a.q, (const float *)a.k, (const float *)a.dO, ws + w.Gq, ws + w.bcum, a.dht,
                ws + w.dstates, a.dh0, ws + w.W, ws + w.dU);
        tr.mark("dstate_scan");
        if (cudaGetLastError() != cudaSuccess) return -1;
        n2 = gdn_backward_tiles(d, w, a, st, tr);
        if (n2 > 0) n2 += 1;
    } else {
        n2 = d.io_bf16 ? backward_lin_t<__nv_bfloat16>(d, w, a, st, tr) : backward_lin_t<float>(d, w, a, st, tr);
    }
    if (n2 < 0) return -1;
    float *ws = a.ws;
    long n_tok = (long)d.B * d.T;
    int hp = 1;
    while (hp < d.H) hp <<= 1;
    const float *Gq = ws + w.Gq, *Gk = ws + w.Gk, *dGq = ws + w.dGq, *dGk = ws + w.dGk;
    switch (hp) {
        case 1: launch_gate_bwd<1>(Gq, Gk, dGq, dGk, a.dlq, a.dlk, n_tok, d.H, st); break;
        case 2: launch_gate_bwd<2>(Gq, Gk, dGq, dGk, a.dlq, a.dlk, n_tok, d.H, st); break;
        case 4: launch_gate_bwd<4>(Gq, Gk, dGq, dGk, a.dlq, a.dlk, n_tok, d.H, st); break;
        case 8: launch_gate_bwd<8>(Gq, Gk, dGq, dGk, a.dlq, a.dlk, n_tok, d.H, st); break;
        case 16: launch_gate_bwd<16>(Gq, Gk, dGq, dGk, a.dlq, a.dlk, n_tok, d.H, st); break;
        default: launch_gate_bwd<32>(Gq, Gk, dGq, dGk, a.dlq, a.dlk, n_tok, d.H, st); break;
    }
    tr.mark("gate_bwd");
    if (cudaGetLastError() != cudaSuccess) return -1;
    return n1 + n2 + 1;
}

}  // namespace sla
