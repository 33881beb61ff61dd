// Anchor classes of the 4-cycle enumeration and the kernels of its light
// anchors (tg_c4_light.cu), used by tg_cycles.cu.
#pragma once

#include "tg_internal.cuh"

// An anchor's class by its walk cost c (sum of d_u over its neighbours u ranked
// below it): one warp, a CTA with a small table, a CTA with a large one, its
// own counter slot, or split over the grid.  Anchors of cost 0 close no cycle.
enum { kC4Warp = 0, kC4Cta, kC4CtaLarge, kC4Slot, kC4Split, kC4Classes };

struct C4HeavyInfo {
    unsigned long long cost;
    int64_t degree;
    uint32_t a, type;
};

struct C4Lists {
    DevBuf<unsigned long long> cost;      // per node
    DevBuf<uint32_t> list;                // class k's anchors at list + k n, in no order
    DevBuf<unsigned long long> queue;     // class sizes, then one queue per class
    int64_t n = 0, size[kC4Classes] = {};
    int lg[3] = {0, 0, 0};                // log2 of the table slots of the light classes
};

// Costs and classes of the part's anchors; t.unroll 1 splits none, 4 all of
// them, t.hash_slots caps the warp tables.
int tg_c4_classify(const tg_graph *g, const tg_tune &t, const tg_part &part, bool global,
                   C4Lists &out, cudaStream_t s);

// The light classes (kC4Warp, kC4Cta, kC4CtaLarge): their cycles added to the
// type-multiset totals g4, or (g4 = NULL) to the per-edge counters c4e.
int tg_c4_light(const tg_graph *g, const C4Lists &cls, unsigned long long *c4e,
                unsigned long long *g4, unsigned long long *work, cudaStream_t s);

// The split anchors, ascending, with their costs and degrees.
int tg_c4_heavy(const tg_graph *g, const C4Lists &cls, C4HeavyInfo *host, cudaStream_t s);

// 4-cliques whose lowest node's up list has at most *bits_max entries
// (tg_k4.cu), to the type-multiset totals g4 or (g4 = NULL) the per-edge
// counters k4e.  *nlong and *longest: the lists left out, the longest of them.
int tg_k4_bits(const tg_graph *g, const tg_lists &up, unsigned long long *k4e, unsigned long long *g4,
               unsigned long long *work, const tg_part &part, int64_t *nlong, int64_t *longest,
               int64_t *bits_max, cudaStream_t s);
