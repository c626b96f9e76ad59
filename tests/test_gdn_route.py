"""Which kernels a Softmax-GatedDeltaNet call runs on (csrc/sla_gdn_route.h): the rules, and what happens when the cooperative launch is refused,
on the host, with the launches replaced by fakes."""
import ctypes
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2602_01744_b200" / "csrc"
SRC = r"""
#include "sla_gdn_route.h"
using namespace sla::gdn;
extern "C" int train(long longest, long chunks, long seqs, long sms) { return chunk_parallel({longest, chunks, seqs, sms}); }
extern "C" int step(long longest, long chunks, long seqs, long sms, int wide) { return chunk_parallel_step({longest, chunks, seqs, sms, wide != 0}); }
extern "C" int forward(long longest, long chunks, long seqs, long sms) { return chunk_parallel_forward({longest, chunks, seqs, sms}); }
// the answers of the two forms' launches; returns the call's, and in *form 1 if the chunk-parallel form ran, in *calls how many were tried
extern "C" int call(int chunked, int chunk_answer, int one_cta_answer, int *form, int *calls) {
    bool c = chunked;
    *calls = 0;
    const int n = run(c, [&] { ++*calls; return chunk_answer; }, [&] { ++*calls; return one_cta_answer; });
    *form = c;
    return n;
}
extern "C" int refused() { return REFUSED; }
"""


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    d = tmp_path_factory.mktemp("route")
    (d / "route.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(d / "route.so"), str(d / "route.cpp")], check=True)
    L = ctypes.CDLL(str(d / "route.so"))
    for f in (L.train, L.forward):
        f.argtypes = [ctypes.c_long] * 4
    L.step.argtypes = [ctypes.c_long] * 4 + [ctypes.c_int]
    return L


@pytest.mark.parametrize("longest,chunks,seqs", [(1, 1, 1), (8, 2304, 288), (16, 256, 16), (17, 17, 1), (1024, 16384, 16)])
def test_without_a_cooperative_grid_every_call_stays_on_the_one_cta_kernels(route, longest, chunks, seqs):
    assert not route.train(longest, chunks, seqs, 0) and not route.forward(longest, chunks, seqs, 0)


# (longest, chunks, sequences) on 148 SMs: training, forward alone
@pytest.mark.parametrize("load,train,forward", [((16, 256, 16), 0, 0), ((17, 17, 1), 1, 1), ((16, 257, 17), 1, 1),
                                                ((8, 1152, 144), 1, 0), ((8, 1536, 192), 1, 1), ((9, 1152, 128), 1, 1), ((2, 320, 160), 1, 1),
                                                ((2, 288, 144), 1, 0), ((1, 65535, 65535), 1, 0)])
def test_the_rules_lines(route, load, train, forward):
    assert (route.train(*load, 148), route.forward(*load, 148)) == (train, forward)


# a step of one chunk a sequence, or of two in one wave, where the sequences fill the SMs: 128-wide values, 64-wide ones
@pytest.mark.parametrize("load,wide,narrow", [((1, 257, 257), 0, 1), ((1, 8192, 8192), 0, 1), ((1, 320, 320), 1, 1), ((2, 288, 144), 0, 1), ((2, 320, 160), 1, 1),
                                              ((2, 576, 288), 1, 1), ((3, 432, 144), 1, 1), ((1, 256, 256), 0, 0), ((17, 17, 1), 1, 1)])
def test_steps_over_sequences_of_a_chunk_or_two(route, load, wide, narrow):
    assert (route.step(*load, 148, 1), route.step(*load, 148, 0)) == (wide, narrow)
    assert not route.step(*load, 0, 1)


def test_a_refused_cooperative_launch_leaves_the_call_to_the_one_cta_kernels(route):
    form, calls = ctypes.c_int(), ctypes.c_int()

    def call(chunked, chunk_answer, one_cta_answer):
        n = route.call(chunked, chunk_answer, one_cta_answer, ctypes.byref(form), ctypes.byref(calls))
        return n, form.value, calls.value

    refused = route.refused()
    assert refused < 0 and refused not in (-1, -2)       # (-1: a CUDA error, -2: unsupported)
    assert call(1, 2, 3) == (2, 1, 1)
    assert call(1, refused, 3) == (3, 0, 2)              # refused: served, and known as the other form's
    assert call(1, -1, 3) == (-1, 1, 1)                  # any other error is the caller's to know
    assert call(1, refused, -1) == (-1, 0, 2)
    assert call(0, 2, 3) == (3, 0, 1)
