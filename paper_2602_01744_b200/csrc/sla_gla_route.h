// Which form a call of the tensor-core Softmax-GLA / -RetNet kernels takes: one 64-wide head a CTA or two, long sequences of a packed batch whole or in
// segments.  Host rules on sizes alone, so that a test can ask them without a GPU.
#pragma once
#include "sla_internal.h"

#include <algorithm>
#include <cmath>

namespace sla {

// A pair's chunk takes 1.04 to 1.13 times as long as one head's (8 x 4096 tokens x 32 heads, forward and step: Softmax-GLA 381 and 1167 us one head
// a CTA, 198 and 620 in pairs, half the CTAs; Softmax-RetNet 346 and 863, 196 and 481), so pairs gain where single heads do not all
// run at once.  Where one long sequence of a packed batch is what a call lasts they would lose: a sequence of 4000 tokens beside 17 of 256, 32 heads,
// step 567 us single, 585 in pairs.  Both are estimated in chunk times: the longest sequence, or what an SM gets where there are more
// CTAs than SMs (equal sequences: whole waves of them).
constexpr double PAIR_CHUNK = 1.1;
inline bool pairs_of_heads(const Dims &d, const Varlen *vl, double sms) {
    if (d.dk != 64 || d.dv != 64 || d.H % 2) return false;
    if (vl && vl->n_of && vl->fwd) return vl->pairs;        // (what the cut was chosen for)
    if (vl && vl->n_of) vl = vl->whole;                     // (the form in which the forward pass leaves the state images)
    auto lasts = [&](long heads) {
        if (!(vl && vl->n_seq)) return std::ceil(d.B * heads / sms) * d.NT;
        long chunks = 0, longest = 0;
        for (const SeqInfo &s : vl->seqs) {
            chunks += s.NT;
            longest = std::max<long>(longest, s.NT);
        }
        return std::max<double>(longest, chunks * heads / sms);
    };
    return PAIR_CHUNK * lasts(d.H / 2) < lasts(d.H);
}

// A packed batch lasts as long as its longest sequence's chain of chunks, or what an SM gets.  Cut into segments the chain gets shorter, for a
// pass over the cut sequences' k, v and decay beside the forward pass (the state every segment starts from) and one over q, dO and decay beside
// the backward pass, each with a fold over its results.  Estimated in chunk times of the pass (2.1 us forward, 6.6 backward, one CTA an SM): an SM that gets
// work all the time takes 1.2 times as long a chunk as a chain by itself, a chunk of the first pass 0.8 of a forward one, of the second 0.33 of a backward
// one, launches and first loads 7 and 4, a segment's states 2.5 and 0.8 in what all SMs together move.  Against measured calls (T x heads of 128, longest
// sequence; forward, and backward with gates: before -> cut, us): 8192 x 8, 4880 tokens 161 -> 56, 449 -> 100; 4096 x 16, 1695 64.5 -> 60.3, 173 -> 108;
// 32768 x 16, 11120 372 -> 303, 1013 -> 635; 16384 x 16, 3167 119 -> 136 (not taken), 323 -> 269.  The length aimed at is at least 8
// chunks (a sequence's segments are equal but for the last, and may then be shorter).  The host's share is not estimated: on new tensors a call encodes 14 maps
// for every entry of the table, 20 to 38 us a step whose buffers change each time, cut or not (17 sequences uncut 19 to 33).
inline void cut_sequences(const Dims &d, const Varlen &vl, Varlen &cut, double sms) {
    const double size = d.dk * d.dv / (128.0 * 128);
    long longest = 0;
    for (const SeqInfo &s : vl.seqs) longest = std::max<long>(longest, s.NT);
    if (longest < 16) return;
    const int whole_hpc = pairs_of_heads(d, &vl, sms) ? 2 : 1;
    auto lasts = [&](long L, int hpc, double pass, double fixed, double edge) {     // sequences longer than L in equal segments, hpc heads a CTA
        double chunks = 0, cut_chunks = 0, top = 0, cut_top = 0, segs = 0;
        const double heads = (double)d.H / hpc;
        for (const SeqInfo &s : vl.seqs) {
            const long n = (s.NT + L - 1) / L, len = (s.NT + n - 1) / n;
            chunks += s.NT;
            top = std::max<double>(top, len);
            if (n > 1) { cut_chunks += s.NT; cut_top = std::max<double>(cut_top, len); segs += n; }
        }
        const double all = std::max(top, 1.2 * chunks * heads / sms), chunk = hpc == 2 ? PAIR_CHUNK : 1;
        return segs > 0 ? chunk * (all + pass * std::max(cut_top, 1.2 * cut_chunks * heads / sms)) + fixed + edge * size * segs * d.H / sms : chunk * all;
    };
    const double whole = lasts(longest, whole_hpc, 0, 0, 0);
    double best = 0.95 * whole;
    long best_L = 0;
    for (int hpc = whole_hpc; hpc <= (d.dk == 64 && d.dv == 64 && d.H % 2 == 0 ? 2 : 1); ++hpc)
        for (long P = 2; P <= 64 && (longest + P - 1) / P >= 8; ++P) {
            const long L = (longest + P - 1) / P;
            const bool fwd = lasts(L, hpc, 0.8, 7, 2.5) < whole;
            const double t = lasts(L, hpc, 0.33, 4, 0.8);
            if (t < best && (fwd || hpc == whole_hpc)) { best = t; best_L = L; cut.fwd = fwd; cut.pairs = hpc == 2; }     // (a whole forward pass decides on the pairs)
        }
    if (!best_L) return;
    std::vector<SeqInfo> by_id(vl.seqs);
    std::sort(by_id.begin(), by_id.end(), [](const SeqInfo &a, const SeqInfo &b) { return a.id < b.id; });
    for (const SeqInfo &s : by_id) {
        cut.cut.push_back((int)cut.seqs.size());
        const int n = (int)((s.NT + best_L - 1) / best_L), len = (s.NT + n - 1) / n;
        for (int t0 = 0; t0 < s.T; t0 += len * d.C) {
            const int T = std::min(len * d.C, s.T - t0), id = (int)cut.seqs.size();
            cut.seqs.push_back({s.t0 + t0, T, (T + d.C - 1) / d.C, s.slot0, id, t0 + T == s.T ? s.id : -1, t0 == 0 ? s.id : -1, s.NT, t0 / d.C});
        }
    }
    cut.cut.push_back((int)cut.seqs.size());
    std::stable_sort(cut.seqs.begin(), cut.seqs.end(), [](const SeqInfo &a, const SeqInfo &b) { return a.NT > b.NT; });
    cut.slots = vl.slots;
    cut.n_of = (int)by_id.size();
    cut.n_seq = (int)cut.seqs.size();
    for (int i = 0; i < cut.n_seq; ++i)
        if (cut.seqs[i].ht_id < 0) { cut.cut.push_back(i); ++cut.n_left; }
    for (int i = 0; i < cut.n_seq; ++i)
        if (cut.seqs[i].dh0_id < 0) { cut.cut.push_back(i); ++cut.n_right; }
}

}  // namespace sla
