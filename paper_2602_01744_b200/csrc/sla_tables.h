// Device side of a plan's sequence tables (struct Varlen): host code only, so that a test can run it on fakes of the CUDA calls.
#pragma once
#include "sla_internal.h"

namespace sla {

inline void varlen_release(Varlen &v) {
    if (v.d_seqs) cudaFree(v.d_seqs);
    if (v.d_cut) cudaFree(v.d_cut);
    for (auto &g : v.reg) {
        if (g.dev) cudaFree(g.dev);
        if (g.host) cudaFreeHost(g.host);
        if (g.uploaded) cudaEventDestroy(g.uploaded);
        g = Varlen::Region();
    }
    v = Varlen();
}

// The table itself and, per kernel kind, room for the sequences' tensor maps.  Nothing is left of it where one of the calls fails.
inline bool varlen_to_device(Varlen &v) {
    const int n_seq = v.n_seq;
    bool ok = cudaMalloc((void **)&v.d_seqs, sizeof(SeqInfo) * n_seq) == cudaSuccess &&
              cudaMemcpy(v.d_seqs, v.seqs.data(), sizeof(SeqInfo) * n_seq, cudaMemcpyHostToDevice) == cudaSuccess;
    if (!v.cut.empty())
        ok = ok && cudaMalloc((void **)&v.d_cut, sizeof(int) * v.cut.size()) == cudaSuccess &&
             cudaMemcpy(v.d_cut, v.cut.data(), sizeof(int) * v.cut.size(), cudaMemcpyHostToDevice) == cudaSuccess;
    const size_t mb = (size_t)n_seq * Varlen::MAPS_PER_SEQ * sizeof(CUtensorMap);
    for (auto &g : v.reg)
        ok = ok && cudaMalloc((void **)&g.dev, mb) == cudaSuccess && cudaMallocHost((void **)&g.host, mb) == cudaSuccess &&
             cudaEventCreateWithFlags(&g.uploaded, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) varlen_release(v);
    return ok;
}

// Puts a packed batch's table, and the one with its long sequences cut where there is one, in the place of a plan's.  Without room for the
// cut one the batch runs uncut; without room for the table itself nothing changes and the answer is no.
inline bool replace_tables(Varlen &varlen, Varlen &cut, Varlen &&v, Varlen &&c) {
    if (!varlen_to_device(v)) return false;
    if (c.n_seq && !varlen_to_device(c)) cudaGetLastError();        // (taken back: the next call must not find it)
    varlen_release(varlen);
    varlen_release(cut);
    varlen = std::move(v);
    cut = std::move(c);
    cut.whole = cut.n_seq ? &varlen : nullptr;
    return true;
}

}  // namespace sla
