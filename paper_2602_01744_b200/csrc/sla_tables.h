// Device side of a plan's sequence tables (struct Varlen): host code only, so that a test can run it on fakes of the CUDA calls.
#pragma once
#include "sla_internal.h"

#include <string.h>

namespace sla {

inline void varlen_release(Varlen &v) {
    if (v.block) cudaFree(v.block);
    if (v.mirror) cudaFreeHost(v.mirror);
    for (auto &g : v.reg)
        if (g.uploaded) cudaEventDestroy(g.uploaded);
    v = Varlen();
}

// The table itself and, per kernel kind, room for the sequences' tensor maps; with `c`, that table's, too (in v's memory).  One allocation on the
// device, one of the mirror, one copy, because a packed batch sets its tables for every step: 46 us with eight allocations, three events and
// two copies a table, 95 for two such tables, 30 to 41 for either so.  No memory is left where one of the calls fails.
inline bool varlen_to_device(Varlen &v, Varlen *c = nullptr) {
    constexpr size_t regions = sizeof(v.reg) / sizeof(v.reg[0]);
    static_assert(sizeof(SeqInfo) % sizeof(int) == 0 && sizeof(CUtensorMap) % alignof(SeqInfo) == 0, "maps, then entries, then places lie side by side");
    Varlen *const tables[2] = {&v, c};
    size_t maps = 0, seqs = 0, cuts = 0;
    for (const Varlen *t : tables)
        if (t) {
            maps += regions * t->n_seq * Varlen::MAPS_PER_SEQ;
            seqs += t->n_seq;
            cuts += t->cut.size();
        }
    const size_t m = maps * sizeof(CUtensorMap), s = seqs * sizeof(SeqInfo), bytes = m + s + cuts * sizeof(int);
    auto failed = [&] {
        if (v.block) cudaFree(v.block);
        if (v.mirror) cudaFreeHost(v.mirror);
        v.block = v.mirror = nullptr;
        return false;
    };
    if (cudaMalloc(&v.block, bytes) != cudaSuccess || cudaMallocHost(&v.mirror, bytes) != cudaSuccess) return failed();
    char *const host = (char *)v.mirror, *const dev = (char *)v.block;
    size_t at_m = 0, at_s = m, at_c = m + s;
    for (Varlen *t : tables) {
        if (!t) continue;
        t->d_seqs = (SeqInfo *)(dev + at_s);
        t->d_cut = (int *)(dev + at_c);
        memcpy(host + at_s, t->seqs.data(), t->n_seq * sizeof(SeqInfo));
        if (!t->cut.empty()) memcpy(host + at_c, t->cut.data(), t->cut.size() * sizeof(int));
        at_s += t->n_seq * sizeof(SeqInfo);
        at_c += t->cut.size() * sizeof(int);
        for (auto &g : t->reg) {
            g.dev = (CUtensorMap *)(dev + at_m);
            g.host = (CUtensorMap *)(host + at_m);
            at_m += (size_t)t->n_seq * Varlen::MAPS_PER_SEQ * sizeof(CUtensorMap);
        }
    }
    return cudaMemcpy(dev + m, host + m, bytes - m, cudaMemcpyHostToDevice) == cudaSuccess || failed();
}

// Puts a packed batch's table, and the one with its long sequences cut where there is one, in the place of a plan's.  Without room for the
// cut one the batch runs uncut; without room for the table itself nothing changes and the answer is no.
inline bool replace_tables(Varlen &varlen, Varlen &cut, Varlen &&v, Varlen &&c) {
    if (c.n_seq && !varlen_to_device(v, &c)) {
        cudaGetLastError();             // (taken back: the next call must not find it)
        c = Varlen();
    }
    if (!c.n_seq && !varlen_to_device(v)) return false;
    varlen_release(cut);
    varlen_release(varlen);
    varlen = std::move(v);
    cut = std::move(c);
    cut.whole = cut.n_seq ? &varlen : nullptr;
    return true;
}

}  // namespace sla
