// Which of the two Softmax-GatedDeltaNet kernel families a call runs on: one CTA per sequence (sla_gdn_tc.cu, sla_gdn_tc_bwd.cu) or
// chunk-parallel (sla_gdn_chunk.cu).  Host arithmetic only, nothing of CUDA, so that the rules are tested without a GPU.
#pragma once

namespace sla {
namespace gdn {

struct Load {
    long longest;       // chunks of the longest sequence
    long chunks, seqs;  // over all (sequence, head) pairs
    long sms;           // SMs that a cooperative grid of one CTA each can fill; 0: no such grid here
    bool wide = true;   // values of 128 columns (two scan items a sequence and head; one at 64)
};

// The chunk-parallel form needs records in memory and a grid-wide barrier; its serial chain is a seventh of the one-CTA kernels' (1.1
// against 7 us a chunk of the longest sequence).  Above the line, one-CTA against chunk-parallel, 128-wide heads, B x T x H: forward
// 1 x 1088 x 4 123 / 39 us, 4 x 512 x 16 64 / 39, 1 x 2048 x 4 223 / 57; training step 382 / 84, 221 / 106, 698 / 127.  Below it lie the
// forward passes that callers have always made without a workspace (1 x 1024 x 4: 111 us, 4 x 256 x 16: 35).  Training steps, which bring
// one anyway, take the same line, but for chunk_parallel_step, so that a step's forward and a forward alone mostly run the same kernels; the
// longer ones below it would gain from the chunk-parallel form.
inline bool chunk_parallel(const Load &l) { return l.sms > 0 && (l.longest > 16 || l.chunks > 256); }

// The sequences, one CTA each, fill the SMs by themselves: to four fifths of a whole number of waves or more.
inline bool filled(const Load &l) {
    const long waves = (l.seqs + l.sms - 1) / l.sms;
    return 5 * l.seqs >= 4 * waves * l.sms;
}

// A training step, whose forward leaves records for its backward.  Sequences of one chunk have no chain to shorten, and writing and reading
// their records costs more than it saves where the sequences fill the SMs and values are 128 wide; two chunks in a single wave alike.
// One-CTA against chunk-parallel, 128-wide heads: 17 x 64 x 16 80 / 99 us, 64 x 64 x 16 260 / 283, 512 x 64 x 16 1675 / 1868, 9 x 128 x 16
// 68 / 74; but 10 x 128 x 16 113 / 99, 18 x 128 x 16 144 / 129, 9 x 256 x 16 131 / 115, and with 64-wide values 64 x 64 x 16 249 / 206,
// 9 x 128 x 16 65 / 52.  (20 x 64 x 16, which does not fill the SMs, keeps the form of a forward alone although it loses: 105 / 114.)
inline bool chunk_parallel_step(const Load &l) {
    if (!chunk_parallel(l)) return false;
    return !l.wide || !filled(l) || !(l.longest == 1 || (l.longest == 2 && l.seqs <= l.sms));
}

// A forward pass that keeps no records gains nothing from the chunk-parallel form where every sequence is short (up to 8 chunks) and
// the sequences fill the SMs.  One-CTA against chunk-parallel:
// 8 x 512 x 16 63.6 / 67.8 us, 18 x 512 x 16 127.4 / 131.7, 64 x 128 x 16 146 / 162; but 12 x 512 x 16 (two waves, 65 % filled)
// 123.5 / 96.1 and 8 x 1024 x 16 121.2 / 110.9.
inline bool chunk_parallel_forward(const Load &l) {
    return chunk_parallel(l) && (l.longest > 8 || !filled(l));
}

// What a launch of the chunk-parallel kernels answers when the context has no room for its cooperative grid (a part of the GPU, say):
// nothing has run, and the one-CTA kernels, which need no such grid, serve the call.  chunked: the form that ran.
constexpr int REFUSED = -3;
template <class Chunked, class OneCta>
int run(bool &chunked, Chunked chunk_form, OneCta one_cta_form) {
    if (chunked) {
        const int n = chunk_form();
        if (n != REFUSED) return n;
        chunked = false;
    }
    return one_cta_form();
}

}  // namespace gdn
}  // namespace sla
