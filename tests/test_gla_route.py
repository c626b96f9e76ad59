"""Which form a packed batch takes on the Softmax-GLA / -RetNet kernels (csrc/sla_gla_route.h), on the host."""
import ctypes
import random
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
SRC = r"""
#include "sla_gla_route.h"
using namespace sla;
static Dims dims(int H, int d) { Dims x{}; x.B = 1; x.H = H; x.dk = x.dv = d; x.C = 64; return x; }
static Varlen table(const int *tokens, int n) {
    Varlen v;
    int t = 0, slots = 0;
    for (int i = 0; i < n; ++i) {
        v.seqs.push_back({t, tokens[i], (tokens[i] + 63) / 64, slots, i});
        t += tokens[i];
        slots += v.seqs.back().NT + 1;
    }
    v.slots = slots;
    v.n_seq = n;
    return v;
}
// segs: five ints a segment (first token, tokens, final state's number or -1, initial state's, first chunk in its sequence), in the caller's order.
// Returns the segments (0: not cut); *form: 1 the forward pass is cut, too, + 2 chosen for pairs, + 4 run in pairs, + 8 the uncut table runs in pairs
extern "C" int cut(int H, int d, int sms, const int *tokens, int n, int *segs, int *form) {
    const Dims x = dims(H, d);
    Varlen v = table(tokens, n), c;
    cut_sequences(x, v, c, sms);
    c.whole = &v;
    *form = c.fwd + 2 * c.pairs + 4 * pairs_of_heads(x, c.n_seq ? &c : &v, sms) + 8 * pairs_of_heads(x, &v, sms);
    for (const SeqInfo &s : c.seqs) {
        int *o = segs + 5 * s.id;
        o[0] = s.t0; o[1] = s.T; o[2] = s.ht_id; o[3] = s.dh0_id; o[4] = s.img_n0;
    }
    return c.n_seq;
}
"""


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    d = tmp_path_factory.mktemp("gla_route")
    (d / "route.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{ROOT / 'paper_2602_01744_b200' / 'csrc'}", f"-I{ROOT / 'include'}",
                    "-I/usr/local/cuda/include", "-o", str(d / "route.so"), str(d / "route.cpp")], check=True)
    L = ctypes.CDLL(str(d / "route.so"))

    def call(H, d, tokens, sms=148):
        segs, form = (ctypes.c_int * (5 * (sum(tokens) // 64 + 2 * len(tokens))))(), ctypes.c_int()
        n = L.cut(H, d, sms, (ctypes.c_int * len(tokens))(*tokens), len(tokens), segs, ctypes.byref(form))
        return [tuple(segs[5 * i:5 * i + 5]) for i in range(n)], form.value

    return call


def test_segments_cover_their_sequences(cut):
    rng, seen = random.Random(7), 0
    for _ in range(400):
        H, d = rng.choice([(1, 128), (4, 64), (8, 128), (16, 64), (32, 64)])
        tokens = [max(1, int(rng.expovariate(1 / 900))) for _ in range(rng.randint(1, 24))]
        segs, _ = cut(H, d, tokens)
        if not segs:
            continue
        seen += 1
        at, i = 0, 0
        for s, n in enumerate(tokens):
            first = at
            while at < first + n:
                t0, T, ht, dh0, chunk = segs[i]
                assert t0 == at and T > 0 and (t0 - first) == 64 * chunk
                assert dh0 == (s if at == first else -1) and ht == (s if at + T == first + n else -1)
                assert T % 64 == 0 or at + T == first + n
                at, i = at + T, i + 1
            assert at == first + n
        assert i == len(segs)
    assert seen > 100


# 64-wide heads: among them batches whose cut table, asked by itself, would have answered single heads where the cut was chosen for pairs
@pytest.mark.parametrize("H,chunks", [(4, (232, 47, 10, 4)), (8, (55, 40, 24, 21, 14, 5)), (16, (47, 19, 3, 3)), (4, (129, 83, 59, 29)), (32, (40, *[1] * 30)),
                                      (16, (27, 12, 6, 6, 5, 4, 4, 3, 2, 2, 2, 1, 1, 1))])
def test_a_cut_batch_runs_in_the_form_it_was_cut_for(cut, H, chunks):
    segs, form = cut(H, 64, [64 * c for c in chunks])
    fwd, chosen, run, whole = (bool(form & b) for b in (1, 2, 4, 8))
    assert segs and run == (chosen if fwd else whole) and (fwd or chosen == whole)
