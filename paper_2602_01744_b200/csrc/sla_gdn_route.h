// Which of the two Softmax-GatedDeltaNet kernel families a call runs on: one CTA per sequence (sla_gdn_tc.cu, sla_gdn_tc_bwd.cu) or
// chunk-parallel (sla_gdn_chunk.cu).  Host arithmetic only, nothing of CUDA, so that the rules are tested without a GPU.
#pragma once

namespace sla {
namespace gdn {

struct Load {
    long longest;       // chunks of the longest sequence
    long chunks, seqs;  // over all (sequence, head) pairs
    long sms;           // SMs that a cooperative grid of one CTA each can fill; 0: no such grid here
};

// The chunk-parallel form needs records in memory and a grid-wide barrier; its serial chain is a seventh of the one-CTA kernels' (1.1
// against 7 us a chunk of the longest sequence).  Above the line, one-CTA against chunk-parallel, 128-wide heads, B x T x H: forward
// 1 x 1088 x 4 123 / 39 us, 4 x 512 x 16 64 / 39, 1 x 2048 x 4 223 / 57; training step 382 / 84, 221 / 106, 698 / 127.  Below it lie the
// forward passes that callers have always made without a workspace (1 x 1024 x 4: 111 us, 4 x 256 x 16: 35).  Training steps, which bring
// one anyway, take the same line so that a step's forward and a forward alone mostly run the same kernels; the longer ones
// below it would gain from the chunk-parallel form.
inline bool chunk_parallel(const Load &l) { return l.sms > 0 && (l.longest > 16 || l.chunks > 256); }

// A forward pass that keeps no records gains nothing from the chunk-parallel form where every sequence is short (up to 8 chunks) and
// the sequences fill the SMs by themselves, to four fifths of a whole number of waves or more.  One-CTA against chunk-parallel:
// 8 x 512 x 16 63.6 / 67.8 us, 18 x 512 x 16 127.4 / 131.7, 64 x 128 x 16 146 / 162; but 12 x 512 x 16 (two waves, 65 % filled)
// 123.5 / 96.1 and 8 x 1024 x 16 121.2 / 110.9.
inline bool chunk_parallel_forward(const Load &l) {
    if (!chunk_parallel(l)) return false;
    const long waves = (l.seqs + l.sms - 1) / l.sms;
    return l.longest > 8 || 5 * l.seqs < 4 * waves * l.sms;
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
