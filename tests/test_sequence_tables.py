"""The device side of a plan's sequence tables (csrc/sla_tables.h) on the host, with fakes of the CUDA calls of which one after the other fails."""
import ctypes
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
SRC = r"""
#include "sla_tables.h"
#include <set>
#include <stdlib.h>
static int calls, fail_at, errors;
static std::set<void *> held;
static bool fails() { ++calls; if (fail_at < 0 ? calls < -fail_at : calls != fail_at) return false; ++errors; return true; }
static cudaError_t take(void **p, size_t n) {
    *p = nullptr;
    if (fails()) return cudaErrorMemoryAllocation;
    held.insert(*p = malloc(n));
    return cudaSuccess;
}
static cudaError_t give(void *p) { if (p && held.erase(p)) free(p); else if (p) abort(); return cudaSuccess; }
extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return take(p, n); }
cudaError_t cudaMallocHost(void **p, size_t n) { return take(p, n); }
cudaError_t cudaFree(void *p) { return give(p); }
cudaError_t cudaFreeHost(void *p) { return give(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { if (fails()) return cudaErrorUnknown; memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return take((void **)e, 1); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return give((void *)e); }
cudaError_t cudaGetLastError() { errors = 0; return cudaSuccess; }
}
static sla::Varlen table(int n, bool cut) {
    sla::Varlen v;
    for (int i = 0; i < n; ++i) v.seqs.push_back({64 * i, 64, 1, 2 * i, i});
    v.n_seq = n;
    if (cut) { v.n_of = 1; v.cut.assign(n + 1, 7); }
    return v;
}
// A plan that holds tables of 2 and 3 entries takes ones of 5 and (with_cut) 9 while the fail-th CUDA call fails, or (-fail) all from it on; 0: none.  Returns
// 10000 * answer + 1000 * (an error is left behind) + 100 * entries of the table + entries of the cut one; -1: what they hold does not fit;
// *most: CUDA calls that could fail; *leaked: allocations left after the release of everything
extern "C" int replace(int with_cut, int fail, int *most, int *leaked) {
    sla::Varlen varlen, cut;
    fail_at = 0;
    errors = 0;
    sla::replace_tables(varlen, cut, table(2, false), table(3, true));
    calls = 0;
    fail_at = fail;
    const bool ok = sla::replace_tables(varlen, cut, table(5, false), with_cut ? table(9, true) : sla::Varlen());
    *most = calls;
    int r = 10000 * ok + 1000 * (errors > 0) + 100 * varlen.n_seq + cut.n_seq;
    if ((int)varlen.seqs.size() != varlen.n_seq || memcmp(varlen.d_seqs, varlen.seqs.data(), sizeof(sla::SeqInfo) * varlen.n_seq)) r = -1;
    if (cut.n_seq ? cut.whole != &varlen || memcmp(cut.d_seqs, cut.seqs.data(), sizeof(sla::SeqInfo) * cut.n_seq) || memcmp(cut.d_cut, cut.cut.data(), 4 * cut.cut.size())
                  : cut.whole || cut.d_seqs || !cut.seqs.empty()) r = -1;
    sla::varlen_release(varlen);
    sla::varlen_release(cut);
    *leaked = (int)held.size();
    return r;
}
"""


@pytest.fixture(scope="module")
def replace(tmp_path_factory):
    d = tmp_path_factory.mktemp("tables")
    (d / "tables.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", f"-I{ROOT / 'paper_2602_01744_b200' / 'csrc'}", f"-I{ROOT / 'include'}",
                    "-I/usr/local/cuda/include", "-o", str(d / "tables.so"), str(d / "tables.cpp")], check=True)
    L = ctypes.CDLL(str(d / "tables.so"))

    def call(with_cut, fail):
        most, leaked = ctypes.c_int(), ctypes.c_int()
        r = L.replace(with_cut, fail, ctypes.byref(most), ctypes.byref(leaked))
        assert leaked.value == 0
        return r, most.value

    return call


def test_tables_are_replaced(replace):
    assert replace(1, 0)[0] == 10000 + 500 + 9
    assert replace(0, 0)[0] == 10000 + 500


def test_without_room_for_the_table_nothing_changes(replace):
    for with_cut in (0, 1):
        _, n = replace(with_cut, 0)
        for first in range(1, n + 1):
            assert replace(with_cut, -first)[0] == 1000 + 200 + 3         # (the caller takes the error back)
            assert with_cut or replace(0, first)[0] == 1000 + 200 + 3


def test_without_room_for_the_cut_table_the_batch_runs_uncut(replace):
    _, n = replace(1, 0)
    for fail in range(1, n + 1):
        assert replace(1, fail)[0] == 10000 + 500                         # and no error is left for the next call
