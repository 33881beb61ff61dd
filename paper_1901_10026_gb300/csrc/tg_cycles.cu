// Per-edge counts of Alg. 2-3 from two whole-graph enumerations.
//
// The identities in tg_reuse.cu express every enumerated orbit of Alg. 2-3
// through Alg. 1's typed triangle counts tau, per-node sums of tau and of the
// typed degrees, sums over the triangle nodes T_ij, and two more per-edge
// quantities that the paper obtains by walking the neighbour lists of
// S_i u S_j u T_ij:
//   C4_ij[a][b] = ordered pairs (x in Gamma_i^a \ {j}, w in Gamma_j^b \ {i})
//                 with x ~ w, i.e. the non-induced 4-cycles i-j-w-x through
//                 the edge; the 4-cycle term of the identities is
//                 S6 = C4 - B + [b = phi_i] |T^a|
//                 (the x in T part of C4 is sum over y in T^a of tau_jy[b],
//                 less i itself);
//   Q_ij[a][b]  = ordered adjacent pairs (y in T^a, z in T^b), i.e. the
//                 4-cliques through the edge.
// Here both are accumulated per edge from enumerations of the whole graph in
// degree order (a node ranks higher when its new id is smaller):
//   4-cycles: each non-induced 4-cycle a-u-b-u' is met once, at its
//     highest-ranked node a, as two wedges a-u-b and a-u'-b whose other nodes
//     rank below a.  Per anchor a, pass 1 counts the middles u of the wedges
//     ending at each b by type (c_t(b)); pass 2 adds, for every wedge, the
//     cycles it closes with the other middles to its two edges (per-edge
//     mode); the far ends then add C(c_t, 2) and c_t c_t' (global mode) and
//     clear the counters.  Light anchors keep their counters in shared memory
//     (tg_c4_light.cu); global mode walks costly ones in warp units over binned
//     waves and waves of counter slots.
//   4-cliques (tg_k4.cu; lists beyond its rows: k_k4, k_k4_global): each 4-clique x0 < v < w < x (by rank) is met once from
//     its lowest node along "up" lists (neighbours of higher rank) and adds one
//     to each of its six edges, keyed by the unordered types of the two nodes
//     off the edge.
// The enumeration work is the number of degree-ordered wedges plus the
// 4-clique search, instead of sum over w in S_i u S_j u T_ij of d_w per edge.
// Whole-graph sums (tg_sums.cu) need only the totals; the per-edge pass
// (tg_edges.cu) needs only Gamma_i n Gamma_j (the T
// sums) and O(L^2) identity and closed-form arithmetic.
#include <algorithm>
#include <new>
#include <vector>

#include "tg_cycles.cuh"
#include "tg_device.cuh"

using namespace tgd;

namespace {

// Inclusive block scan of a packed (count << 52 | length) word; returns the
// inclusive value of this thread and leaves the block total in wsum[32].
__device__ __forceinline__ uint64_t block_scan_packed(uint64_t v, uint64_t *wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
    uint64_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint64_t y = lane < W ? wsum[lane] : 0ull;
        const uint64_t y0 = y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t z = __shfl_up_sync(kFull, y, o);
            if (lane >= o) y += z;
        }
        if (lane < W) wsum[lane] = y - y0;
        if (lane == W - 1) wsum[32] = y;
    }
    __syncthreads();
    return incl + wsum[warp];
}

constexpr uint64_t kLenMask = ((uint64_t)1 << 41) - 1;

// ------------------------------------------------------------ 4-cycles ----
struct C4Params {
    const int64_t *rowptr;
    const uint32_t *adj;
    const uint32_t *eid;
    const uint8_t *ntype;
    int64_t n;
    int32_t L;
    int32_t tile;              // members staged per tile (<= blockDim.x)
    int32_t acc_l2;            // L * L in per-edge mode, 0 in global mode
    uint32_t *scratch;         // slots of n * L counters (per far end, per type), an
                               // n-entry list of the far ends met and a bitmap of them
                               // (n bits); counters and bitmap zero on entry and on exit
    int64_t slot_words;
    unsigned long long *queue;
    unsigned long long *c4e;   // per-edge mode: M * L * L, [type next to i][type next to j]
    unsigned long long *g4;    // global mode: C(L+3,4) non-induced 4-cycles by type multiset
    int64_t n4;
    const int4 *units;         // split kernel: (slot, anchor, first member, end member)
    const struct C4Unit *wunits;  // walk kernel: position ranges of the split anchors
    int64_t n_units;
    int32_t phase;             // split kernel: the pass of this launch
    unsigned long long *work;  // [4]: wedges
    // dense waves (global mode): the costly anchors heavy[q], their walk
    // positions (member costs d_u, exclusive prefix per anchor at pbase[q]),
    // and the first anchor index of the wave (slot = q - q0)
    const uint32_t *heavy;
    const int64_t *mprefix;
    const int64_t *pbase;
    int64_t q0;
    // slot layout: 32-bit counts at b L + t (half = 0) or 16-bit counts at
    // b Lp + t, Lp = L rounded up to even, two to a word (half = 1); the
    // far-end bitmap starts at word bits_off of the slot
    int32_t half;
    int64_t bits_off;
};

// A warp unit of k_c4_walk: positions [lo, hi) of the walk of split anchor
// q, starting in the list of its member m.
struct C4Unit {
    int64_t lo, hi;
    int32_t q, m;
};

constexpr int kC4Threads = 256;
constexpr int64_t kWaveMax = 128;       // costly anchors of one wave (global mode), at most
constexpr int64_t kWalkUnitMin = 512;    // walk positions of a warp unit, at least

struct C4Smem {
    int64_t *m_end, *m_org;
    uint64_t *wsum;
    unsigned long long *acc;
    uint32_t *m_u, *m_e;
    unsigned long long *s_item, *h4;
    unsigned int *s_nb;
};

__device__ __forceinline__ C4Smem c4_smem(unsigned char *smem, int TM, int acc_l2) {
    C4Smem m;
    m.m_end = reinterpret_cast<int64_t *>(smem);
    m.m_org = m.m_end + TM;
    m.wsum = reinterpret_cast<uint64_t *>(m.m_org + TM);
    m.acc = reinterpret_cast<unsigned long long *>(m.wsum + 34);
    m.m_u = reinterpret_cast<uint32_t *>(m.acc + (size_t)TM * acc_l2);
    m.m_e = m.m_u + TM;
    m.s_item = reinterpret_cast<unsigned long long *>(m.m_e + TM + (TM & 1));
    m.s_nb = reinterpret_cast<unsigned int *>(m.s_item + 1);
    m.h4 = m.s_item + 2;  // global mode: n4 entries
    return m;
}

// One pass over one tile of anchor a's list (list positions [tile, tile_end),
// at most p.tile of them): the members u (neighbours ranked below a) of the
// tile and, for each, the entries b of u's list ranked below a.  The members'
// lists are walked as one sequence of positions.  Pass 0 counts the middles per
// (b, type), and lists each b the first time it is met (in `list`, count in *nb)
// or, without a list, marks it in the slot's bitmap; pass 1 (per-edge mode only)
// adds the cycles each wedge closes to its two edges.  Called by every thread of
// the CTA (it holds barriers).
__device__ void c4_tile(const C4Params &p, const C4Smem &sm, uint32_t a, int ta, int64_t ba,
                        int tile, int tile_end, int phase, uint32_t *cnt, uint32_t *list,
                        unsigned int *nb, unsigned long long &wk) {
    const int tid = threadIdx.x;
    const int L = p.L, L2 = L * L, TM = p.tile;
    const int x = tile + tid;
    bool mem = false;
    uint32_t wu = 0;
    int64_t bu = 0;
    int du = 0;
    if (tid < TM && x < tile_end) {
        wu = __ldg(p.adj + ba + x);
        const uint32_t u = wu & TG_IDMASK;
        if (u > a) {
            bu = p.rowptr[u];
            du = (int)(p.rowptr[u + 1] - bu);
            mem = du > 1;
        }
    }
    const uint64_t incl = block_scan_packed(((uint64_t)mem << 52) | (uint64_t)(mem ? du : 0), sm.wsum);
    const uint64_t tot = sm.wsum[32];
    const int nmem = (int)(tot >> 52);
    const int64_t total = (int64_t)(tot & kLenMask);
    if (mem) {
        const int r = (int)((incl >> 52) - 1);
        const int64_t end = (int64_t)(incl & kLenMask);
        sm.m_end[r] = end;
        sm.m_org[r] = bu - (end - du);
        sm.m_u[r] = wu;
        sm.m_e[r] = __ldg(p.eid + ba + x);
    }
    if (phase == 1)
        for (int q = tid; q < nmem * L2; q += blockDim.x) sm.acc[q] = 0ull;
    __syncthreads();
    // the CTA's threads make the same number of steps: a loop over each thread's own
    // positions took 3.01 and not 2.78 ms for K_{64,20000}
    for (int64_t base = 0; base < total; base += blockDim.x) {
        const int64_t pos = base + tid;
        if (pos >= total) continue;
        int lo = 0, hi = nmem - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (sm.m_end[mid] > pos)
                hi = mid;
            else
                lo = mid + 1;
        }
        const int64_t at = sm.m_org[lo] + pos;
        const uint32_t wb = __ldg(p.adj + at);
        const uint32_t b = wb & TG_IDMASK;
        if (b <= a) continue;  // b must rank below a (and differ from it)
        const uint32_t wmu = sm.m_u[lo];
        const int tu = (int)(wmu >> TG_TSHIFT);
        uint32_t *cb = cnt + (int64_t)b * L;
        if (phase == 0) {
            atomicAdd(cb + tu, 1u);  // result unused: no round trip
            uint32_t *bw = cnt + p.n * (L + 1) + (b >> 5);
            const uint32_t bit = 1u << (b & 31u);
            if (list) {
                // the first wedge to reach b lists it
                if (!(atomicOr(bw, bit) & bit)) list[atomicAdd(nb, 1u)] = b;
            } else {
                atomicOr(bw, bit);  // marks b for the scan of k_c4_pairs
            }
            ++wk;
            continue;
        }
        uint32_t c[TG_MAX_TYPES];
        uint32_t sum = 0;
#pragma unroll
        for (int t = 0; t < TG_MAX_TYPES; ++t) {
            c[t] = t < L ? __ldcg(cb + t) : 0u;
            sum += c[t];
        }
        if (sum < 2u) continue;  // no other middle: no cycle
        const int tb = (int)(wb >> TG_TSHIFT);
        const uint32_t u = wmu & TG_IDMASK;
        unsigned long long *row_ub = p.c4e + (int64_t)__ldg(p.eid + at) * L2;
        unsigned long long *row_au = sm.acc + (int64_t)lo * L2 + tb * L;
#pragma unroll
        for (int t = 0; t < TG_MAX_TYPES; ++t) {
            if (t < L) {
                const uint32_t v = c[t] - (t == tu ? 1u : 0u);
                if (v) {
                    // edge (u, b): u's cycle neighbour a, b's is u' (type t);
                    // the row is keyed from its larger-id end
                    atomicAdd(row_ub + (u > b ? ta * L + t : t * L + ta), (unsigned long long)v);
                    // edge (a, u): u (the larger id) sees b, a sees u'
                    atomicAdd(row_au + t, (unsigned long long)v);
                }
            }
        }
    }
    __syncthreads();
    if (phase == 1) {
        for (int q = tid; q < nmem * L2; q += blockDim.x) {
            const unsigned long long v = sm.acc[q];
            if (v) atomicAdd(p.c4e + (int64_t)sm.m_e[q / L2] * L2 + (q % L2), v);
        }
        __syncthreads();
    }
}

// The cycles of one far end b (type tb) of an anchor of type ta, from its
// middle counts c[t] (t < L): C(c_t, 2) for t = t' and c_t c_t' for t < t',
// each under the multiset {ta, tb, t, t'}, into the shared histogram h4.  Only
// the types with a non-zero count are visited.
__device__ __forceinline__ void c4_add(unsigned long long *h4, int L, int ta, int tb,
                                       const uint32_t *c) {
    uint32_t mask = 0;
    for (int t = 0; t < L; ++t)
        if (c[t]) mask |= 1u << t;
    int s0 = ta, s1 = tb;
    sort2(s0, s1);
    for (uint32_t mt = mask; mt; mt &= mt - 1u) {
        const int t = __ffs(mt) - 1;
        const unsigned long long ct = c[t];
        if (ct > 1) {
            int q0 = s0, q1 = s1, q2 = t, q3 = t;
            sort2(q0, q2);
            sort2(q1, q3);
            sort2(q1, q2);
            atomicAdd(h4 + colex4(q0, q1, q2, q3), ct * (ct - 1) / 2);
        }
        for (uint32_t mu = mt & (mt - 1u); mu; mu &= mu - 1u) {
            const int u = __ffs(mu) - 1;
            int q0 = s0, q1 = s1, q2 = t, q3 = u;
            sort2(q0, q2);
            sort2(q1, q3);
            sort2(q1, q2);
            atomicAdd(h4 + colex4(q0, q1, q2, q3), ct * c[u]);
        }
    }
}

// Far end b of anchor a (counters cb, per type): global mode adds its cycles; both
// modes then clear b's counters.
__device__ __forceinline__ void c4_one(const C4Params &p, unsigned long long *h4, int ta,
                                       uint32_t *cb, uint32_t b) {
    const int L = p.L;
    uint32_t c[TG_MAX_TYPES];
    uint32_t sum = 0;
    for (int t = 0; t < L; ++t) {
        c[t] = __ldcg(cb + t);
        sum += c[t];
    }
    if (p.g4 && sum > 1) c4_add(h4, L, ta, p.ntype[b], c);  // one middle closes no cycle
    for (int t = 0; t < L; ++t)
        if (c[t]) cb[t] = 0u;
}

// c4_one for a 16-bit slot: b's counts are the halves of its (L + 1) / 2
// words at cw (low half the even type), words no other far end shares.
__device__ __forceinline__ void c4_one16(const C4Params &p, unsigned long long *h4, int ta,
                                         uint32_t *cw, uint32_t b) {
    const int L = p.L, nw = (L + 1) >> 1;
    uint32_t c[TG_MAX_TYPES];
    uint32_t sum = 0;
    for (int q = 0; q < nw; ++q) {
        const uint32_t w = __ldcg(cw + q);
        c[2 * q] = w & 0xffffu;
        if (2 * q + 1 < L) c[2 * q + 1] = w >> 16;
        sum += (w & 0xffffu) + (w >> 16);
        if (w) cw[q] = 0u;
    }
    if (p.g4 && sum > 1) c4_add(h4, L, ta, p.ntype[b], c);  // one middle closes no cycle
}

// Position of the j-th (from 0) set bit of m; m has more than j set bits.
__device__ __forceinline__ int select_bit(uint32_t m, int j) {
    int pos = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int c = __popc(m & ((1u << w) - 1u));
        if (j >= c) {
            j -= c;
            m >>= w;
            pos += w;
        }
    }
    return pos;
}

// The listed far ends of anchor a (entries q0, q0 + step, ... < nb).
__device__ __forceinline__ void c4_pairs(const C4Params &p, const C4Smem &sm, int ta,
                                         uint32_t *cnt, const uint32_t *list, unsigned int nb,
                                         unsigned int q0, unsigned int step) {
    for (unsigned int q = q0; q < nb; q += step) {
        const uint32_t b = __ldcg(list + q);  // written by other threads this anchor
        c4_one(p, sm.h4, ta, cnt + (int64_t)b * p.L, b);
        cnt[p.n * (p.L + 1) + (b >> 5)] = 0u;  // every set bit of the word is listed
    }
}

__device__ __forceinline__ void c4_finish(const C4Params &p, const C4Smem &sm,
                                          unsigned long long wk) {
    if (p.g4) {
        __syncthreads();
        for (int64_t q = threadIdx.x; q < p.n4; q += blockDim.x)
            if (sm.h4[q]) atomicAdd(p.g4 + q, sm.h4[q]);
    }
    if (p.work && wk) atomicAdd(p.work + 4, wk);
}

// The anchors of alist: one CTA per anchor, the passes in turn over the CTA's
// own counter slot.
__global__ void __launch_bounds__(kC4Threads) k_c4(C4Params p, const uint32_t *alist, int64_t na) {
    extern __shared__ __align__(16) unsigned char smem[];
    const C4Smem sm = c4_smem(smem, p.tile, p.acc_l2);
    const int tid = threadIdx.x;
    if (p.g4)
        for (int64_t q = tid; q < p.n4; q += blockDim.x) sm.h4[q] = 0ull;
    uint32_t *cnt = p.scratch + (int64_t)blockIdx.x * p.slot_words;
    uint32_t *list = cnt + p.n * p.L;
    unsigned long long wk = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) *sm.s_item = atomicAdd(p.queue, 1ull);
        __syncthreads();
        const unsigned long long item = *sm.s_item;
        if (item >= (unsigned long long)na) break;
        const uint32_t a = alist[item];
        const int64_t ba = p.rowptr[a];
        const int da = (int)(p.rowptr[a + 1] - ba);
        if (da < 2) continue;  // a cycle through a needs two of its neighbours
        const int ta = p.ntype[a];
        if (tid == 0) *sm.s_nb = 0u;
        __syncthreads();
        for (int tile = 0; tile < da; tile += p.tile)
            c4_tile(p, sm, a, ta, ba, tile, min(da, tile + p.tile), 0, cnt, list, sm.s_nb, wk);
        if (!p.g4)
            for (int tile = 0; tile < da; tile += p.tile)
                c4_tile(p, sm, a, ta, ba, tile, min(da, tile + p.tile), 1, cnt, list, sm.s_nb, wk);
        __syncthreads();
        c4_pairs(p, sm, ta, cnt, list, *sm.s_nb, tid, blockDim.x);
    }
    c4_finish(p, sm, wk);
}

// Marked (costly) anchors: their tiles are units spread over the whole grid,
// each anchor on a counter slot of its own; one launch per pass, so a pass
// sees every count of the pass before it.
__global__ void __launch_bounds__(kC4Threads) k_c4_split(C4Params p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const C4Smem sm = c4_smem(smem, p.tile, p.acc_l2);
    const int tid = threadIdx.x;
    if (p.g4)
        for (int64_t q = tid; q < p.n4; q += blockDim.x) sm.h4[q] = 0ull;
    unsigned long long wk = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) *sm.s_item = atomicAdd(p.queue, 1ull);
        __syncthreads();
        const unsigned long long item = *sm.s_item;
        if (item >= (unsigned long long)p.n_units) break;
        const int4 un = p.units[item];
        const uint32_t a = (uint32_t)un.y;
        const int64_t ba = p.rowptr[a];
        uint32_t *cnt = p.scratch + (int64_t)un.x * p.slot_words;
        c4_tile(p, sm, a, p.ntype[a], ba, un.z, un.w, p.phase, cnt, nullptr, nullptr, wk);
    }
    c4_finish(p, sm, wk);
}

// The far ends of the wave's split anchors (na slots, anchors[slot] the
// anchor of a slot), from the slots' bitmaps: each warp takes 32 bitmap words
// at a time, lists their set bits across the lanes (a scan of the words'
// popcounts) and treats 32 far ends per step, one per lane.  Clears the bitmap
// words it reads.  Shared memory: the type-multiset histogram, one copy per
// warp when `priv` (else one per CTA).
__global__ void __launch_bounds__(kC4Threads) k_c4_pairs(C4Params p, const uint32_t *anchors,
                                                         int na, int priv) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long *h4all = reinterpret_cast<unsigned long long *>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int copies = priv ? (int)(blockDim.x >> 5) : 1;
    if (p.g4) {
        for (int64_t q = threadIdx.x; q < p.n4 * copies; q += blockDim.x) h4all[q] = 0ull;
        __syncthreads();
    }
    unsigned long long *h4 = h4all + (priv ? (int64_t)warp * p.n4 : 0);
    const int L = p.L;
    const int64_t words = (p.n + 31) >> 5;
    const int64_t cps = (words + 31) >> 5;  // chunks of 32 words per slot
    const int64_t total = (int64_t)na * cps;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < total; c += nw) {
        const int64_t slot = c / cps, wc = c - slot * cps;
        uint32_t *cnt = p.scratch + slot * p.slot_words;
        uint32_t *bw = cnt + p.bits_off;
        const int64_t wi = wc * 32 + lane;
        uint32_t m = 0;
        if (wi < words) {
            m = __ldcg(bw + wi);
            if (m) bw[wi] = 0u;
        }
        const int k = __popc(m);
        int incl = k;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        const int tot = __shfl_sync(kFull, incl, 31);
        if (tot == 0) continue;
        const int ta = p.ntype[anchors[slot]];
        for (int base = 0; base < tot; base += 32) {
            const int kk = base + lane;
            int r = 0;  // the lane whose word holds far end kk
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
                const int v = __shfl_sync(kFull, incl, r + st - 1);
                if (v <= kk) r += st;
            }
            const uint32_t mr = __shfl_sync(kFull, m, r);
            const int er = __shfl_sync(kFull, incl - k, r);
            if (kk < tot) {
                const uint32_t b = (uint32_t)((wc * 32 + r) * 32 + select_bit(mr, kk - er));
                if (p.half)
                    c4_one16(p, h4, ta, cnt + (int64_t)b * ((L + 1) >> 1), b);
                else
                    c4_one(p, h4, ta, cnt + (int64_t)b * L, b);
            }
        }
    }
    if (p.g4) {
        __syncthreads();
        for (int64_t q = threadIdx.x; q < p.n4; q += blockDim.x) {
            unsigned long long v = 0;
            for (int cpy = 0; cpy < copies; ++cpy) v += h4all[cpy * p.n4 + q];
            if (v) atomicAdd(p.g4 + q, v);
        }
    }
}

// ------------------------------------------------- dense waves (global) ----
// Costly anchors when a few counter slots of n L words fit in L2: a wave of
// anchors counts into its slots with fire-and-forget adds only (no far-end
// bitmap), and k_c4_dense_pairs then scans the slots densely.  Work units cut
// each anchor's walk (its members' lists in order) into position ranges of
// about equal length, so one hub member's long list spreads over many CTAs.

// Walk positions of the costly anchors: member x of heavy[q] costs d_u when it
// is a member (u ranked below the anchor, d_u > 1), else 0; mprefix holds the
// exclusive prefix from pbase[q], totals[q] the sum.  One CTA per anchor.
__global__ void k_c4_prefix(const uint32_t *heavy, const int64_t *pbase, const int64_t *rowptr,
                            const uint32_t *adj, int64_t *mprefix, unsigned long long *totals) {
    __shared__ uint64_t wsum[34];
    const int64_t q = blockIdx.x;
    const uint32_t a = heavy[q];
    const int64_t ba = rowptr[a];
    const int da = (int)(rowptr[a + 1] - ba);
    int64_t *out = mprefix + pbase[q];
    uint64_t run = 0;
    for (int c = 0; c < da; c += blockDim.x) {
        const int x = c + threadIdx.x;
        uint64_t v = 0;
        if (x < da) {
            const uint32_t u = __ldg(adj + ba + x) & TG_IDMASK;
            if (u > a) {
                const int64_t du = rowptr[u + 1] - rowptr[u];
                v = du > 1 ? (uint64_t)du : 0ull;
            }
        }
        const uint64_t incl = block_scan_packed(v, wsum);
        if (x < da) out[x] = (int64_t)(run + incl - v);
        run += wsum[32];
        __syncthreads();  // wsum is rewritten by the next chunk's scan
    }
    if (threadIdx.x == 0) totals[q] = run;
}

// Units of the walk waves: unit u belongs to anchor q with ustart[q] <= u <
// ustart[q + 1], covers positions [k tgt[q], min((k + 1) tgt[q], totals[q]))
// for k = u - ustart[q], and starts at the member holding its first position.
__global__ void k_c4_units(const int64_t *ustart, int64_t nq, const int64_t *tgt,
                           const unsigned long long *totals, const int64_t *mprefix,
                           const int64_t *pbase, const uint32_t *heavy, const int64_t *rowptr,
                           C4Unit *units) {
    const int64_t nu = ustart[nq];
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < nu;
         u += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = nq - 1;  // last q with ustart[q] <= u
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (ustart[mid] <= u)
                lo = mid;
            else
                hi = mid - 1;
        }
        const int64_t q = lo;
        const int64_t f_lo = (u - ustart[q]) * tgt[q];
        const int64_t f_hi = min(f_lo + tgt[q], (int64_t)totals[q]);
        const uint32_t a = heavy[q];
        const int da = (int)(rowptr[a + 1] - rowptr[a]);
        const int64_t *pre = mprefix + pbase[q];
        int m0 = 0, m1 = da - 1;  // last member m with pre[m] <= f_lo
        while (m0 < m1) {
            const int mid = (m0 + m1 + 1) >> 1;
            if (pre[mid] <= f_lo)
                m0 = mid;
            else
                m1 = mid - 1;
        }
        C4Unit un;
        un.lo = f_lo;
        un.hi = f_hi;
        un.q = (int32_t)q;
        un.m = m0;
        units[u] = un;
    }
}

// Positions [f_lo, f_hi) of one chunk of 32 members (lane values len, bu, tu;
// the chunk's first position `at`) for k_c4_walk: the members' list lengths are
// scanned across the lanes (running sums in IT, int when every list is short
// enough), and each position is mapped to its member by a 5-step search over
// the lanes' running sums.  kWalkUnroll batches of 32 positions are in flight
// per step (their list loads, then their counter adds, then the bitmap marks),
// so each lane keeps several returning adds outstanding.  Returns the chunk's
// length.
constexpr int kWalkUnroll = 4;

template <class IT>
__device__ __forceinline__ int64_t c4_chunk_count(const C4Params &p, uint32_t a, int64_t len64,
                                                  int64_t bu, int tu, int64_t at, int64_t f_lo,
                                                  int64_t f_hi, uint32_t *cnt, uint32_t *bits,
                                                  unsigned long long &wk) {
    const int lane = threadIdx.x & 31;
    const int L = p.L;
    const IT len = (IT)len64;
    IT incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const IT y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const IT total = __shfl_sync(kFull, incl, 31);
    const IT lo = (IT)(f_lo > at ? (f_lo - at < (int64_t)total ? f_lo - at : (int64_t)total) : 0);
    const IT hi = (IT)(f_hi - at < (int64_t)total ? f_hi - at : (int64_t)total);
    const int Lp = L + (L & 1);
    for (IT b0 = lo; b0 < hi; b0 += 32 * kWalkUnroll) {
        uint32_t bv[kWalkUnroll];
        uint32_t *ca[kWalkUnroll];
        int sh[kWalkUnroll];
        bool ok[kWalkUnroll];
#pragma unroll
        for (int q = 0; q < kWalkUnroll; ++q) {
            const IT pos = b0 + 32 * q + lane;
            int r = 0;  // the first member whose running sum exceeds pos
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
                const IT v = __shfl_sync(kFull, incl, r + st - 1);
                if (v <= pos) r += st;
            }
            const int64_t bur = __shfl_sync(kFull, bu, r);
            const IT str = __shfl_sync(kFull, incl - len, r);
            const int tur = __shfl_sync(kFull, tu, r);
            ok[q] = false;
            bv[q] = 0;
            ca[q] = cnt;
            sh[q] = 0;
            if (pos < hi) {
                const uint32_t b = __ldg(p.adj + bur + (int64_t)(pos - str)) & TG_IDMASK;
                if (b > a) {
                    ok[q] = true;
                    bv[q] = b;
                    if (p.half) {
                        const int64_t k = (int64_t)b * Lp + tur;
                        ca[q] = cnt + (k >> 1);
                        sh[q] = (int)(k & 1) * 16;
                    } else {
                        ca[q] = cnt + (int64_t)b * L + tur;
                    }
                }
            }
        }
        uint32_t old[kWalkUnroll];
#pragma unroll
        for (int q = 0; q < kWalkUnroll; ++q) old[q] = ok[q] ? atomicAdd(ca[q], 1u << sh[q]) : 0xffffffffu;
#pragma unroll
        for (int q = 0; q < kWalkUnroll; ++q) {
            if (!ok[q]) continue;
            ++wk;
            // the first middle of a type at b marks b
            if (!((old[q] >> sh[q]) & (p.half ? 0xffffu : 0xffffffffu)))
                atomicOr(bits + (bv[q] >> 5), 1u << (bv[q] & 31u));
        }
    }
    return (int64_t)total;
}

// Pass 0 of a wave of costly anchors (global mode): one warp per unit, adding
// to the counters of its anchor's slot and marking a far end in the slot's
// bitmap when a count of it leaves zero; k_c4_pairs then takes the marked ends.
constexpr int kC4WalkWarps = 8;

__global__ void __launch_bounds__(kC4WalkWarps * 32) k_c4_walk(C4Params p) {
    const int lane = threadIdx.x & 31;
    unsigned long long wk = 0;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= (unsigned long long)p.n_units) break;
        const C4Unit un = p.wunits[item];
        const uint32_t a = p.heavy[un.q];
        const int64_t ba = p.rowptr[a];
        const int da = (int)(p.rowptr[a + 1] - ba);
        uint32_t *cnt = p.scratch + (un.q - p.q0) * p.slot_words;
        uint32_t *bits = cnt + p.bits_off;
        int64_t at = p.mprefix[p.pbase[un.q] + un.m];
        for (int m = un.m; m < da && at < un.hi; m += 32) {
            const int x = m + lane;
            int64_t len = 0, bu = 0;
            int tu = 0;
            if (x < da) {
                const uint32_t wu = __ldg(p.adj + ba + x);
                const uint32_t u = wu & TG_IDMASK;
                if (u > a) {
                    bu = p.rowptr[u];
                    const int64_t du = p.rowptr[u + 1] - bu;
                    if (du > 1) {
                        len = du;
                        tu = (int)(wu >> TG_TSHIFT);
                    }
                }
            }
            if (__all_sync(kFull, len < ((int64_t)1 << 26)))
                at += c4_chunk_count<int>(p, a, len, bu, tu, at, un.lo, un.hi, cnt, bits, wk);
            else
                at += c4_chunk_count<int64_t>(p, a, len, bu, tu, at, un.lo, un.hi, cnt, bits, wk);
        }
    }
    if (p.work) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wk += __shfl_xor_sync(kFull, wk, o);
        if (lane == 0 && wk) atomicAdd(p.work + 4, wk);
    }
}

// Pass 1 of a wave in per-edge mode: one warp per unit, for every wedge a-u-b
// of it whose far end has another middle the cycles closed with those, added
// to the rows of its two edges.  A member's list of 32 entries or more is taken
// by the whole warp: its entries are sorted by type, so the part of edge (a, u)
// is summed over the warp per type of b and kept in registers, one add per
// (type of b, type of the other middle); only the row of (u, b) takes an add
// per wedge.  Shorter lists are taken 32 positions at a time across members,
// both rows by adds.  Before, a CTA's threads added every wedge of a member to
// one shared-memory accumulator, up to 32 lanes on one address (13.4 ms for
// the 5.5e7 wedges of CL-125K, L = 5, against 1.8 ms here).  Bound by the adds
// to the rows of (u, b), one per wedge and type of middle.
constexpr int kWedgeLong = 32;

template <int LP>
__device__ __forceinline__ uint32_t wedge_counts(const C4Params &p, const uint32_t *cnt, uint32_t b,
                                                 bool ok, uint32_t (&c)[LP]) {
    uint32_t sum = 0;
#pragma unroll
    for (int t = 0; t < LP; ++t) {
        c[t] = ok && t < p.L ? __ldg(cnt + (int64_t)b * p.L + t) : 0u;
        sum += c[t];
    }
    return sum;
}

template <int LP>
__global__ void __launch_bounds__(kC4WalkWarps * 32) k_c4_wedges(C4Params p) {
    const int lane = threadIdx.x & 31, L = p.L, L2 = L * L;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= (unsigned long long)p.n_units) break;
        const C4Unit un = p.wunits[item];
        const uint32_t a = p.heavy[un.q];
        const int ta = p.ntype[a];
        const int64_t ba = p.rowptr[a];
        const int da = (int)(p.rowptr[a + 1] - ba);
        const uint32_t *cnt = p.scratch + (un.q - p.q0) * p.slot_words;
        int64_t at = p.mprefix[p.pbase[un.q] + un.m];
        for (int m = un.m; m < da && at < un.hi; m += 32) {
            const int x = m + lane;
            int64_t len = 0, bu = 0;
            uint32_t wu = 0;
            if (x < da) {
                wu = __ldg(p.adj + ba + x);
                const uint32_t u = wu & TG_IDMASK;
                if (u > a) {
                    bu = p.rowptr[u];
                    const int64_t du = p.rowptr[u + 1] - bu;
                    if (du > 1) len = du;
                }
            }
            int64_t incl = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            const int64_t first = at + incl - len;  // walk position of this member's list
            at += __shfl_sync(kFull, incl, 31);
            // long lists, the part inside the unit
            unsigned todo = __ballot_sync(kFull, len >= kWedgeLong && first < un.hi && first + len > un.lo);
            for (; todo; todo &= todo - 1u) {
                const int src = __ffs(todo) - 1;
                const int64_t lbu = __shfl_sync(kFull, bu, src), lf = __shfl_sync(kFull, first, src);
                const int64_t ll = __shfl_sync(kFull, len, src);
                const uint32_t lw = __shfl_sync(kFull, wu, src);
                const uint32_t u = lw & TG_IDMASK;
                const int tu = (int)(lw >> TG_TSHIFT);
                const int64_t p0 = un.lo > lf ? un.lo - lf : 0, p1 = un.hi - lf < ll ? un.hi - lf : ll;
                unsigned long long *row_au = p.c4e + (int64_t)__ldg(p.eid + ba + m + src) * L2;
                unsigned long long acc = 0;  // lane t: cycles with b of type cur, the other middle of type t
                int cur = 0;
                for (int64_t c0 = p0; c0 < p1; c0 += 32) {
                    const int64_t pos = lbu + c0 + lane;
                    const uint32_t wb = c0 + lane < p1 ? __ldg(p.adj + pos) : 0u;
                    const uint32_t b = wb & TG_IDMASK;
                    bool ok = c0 + lane < p1 && b > a;
                    if (!__any_sync(kFull, ok)) continue;
                    uint32_t c[LP];
                    ok = wedge_counts<LP>(p, cnt, b, ok, c) >= 2u;
                    unsigned left = __ballot_sync(kFull, ok);
                    if (!left) continue;
                    const int tb = (int)(wb >> TG_TSHIFT);
                    const bool ub = u > b;
                    unsigned long long *row_ub =
                        ok ? p.c4e + (int64_t)__ldg(p.eid + pos) * L2 + (ub ? ta * L : ta) : nullptr;
#pragma unroll
                    for (int t = 0; t < LP; ++t) {
                        c[t] = ok ? c[t] - (t == tu ? 1u : 0u) : 0u;
                        if (c[t]) atomicAdd(row_ub + (ub ? t : t * L), (unsigned long long)c[t]);
                    }
                    while (left) {
                        const int g = __shfl_sync(kFull, tb, __ffs(left) - 1);
                        left &= ~__ballot_sync(kFull, tb == g);
                        if (g != cur) {
                            if (lane < L && acc) atomicAdd(row_au + cur * L + lane, acc);
                            acc = 0;
                            cur = g;
                        }
#pragma unroll
                        for (int t = 0; t < LP; ++t) {
                            if (t >= L) continue;
                            const unsigned sum = __reduce_add_sync(kFull, tb == g ? c[t] : 0u);
                            if (lane == t) acc += sum;
                        }
                    }
                }
                if (lane < L && acc) atomicAdd(row_au + cur * L + lane, acc);
            }
            // short lists that begin inside the unit, as one sequence
            const int ls = len < kWedgeLong && first >= un.lo && first < un.hi ? (int)len : 0;
            int si = ls;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, si, o);
                if (lane >= o) si += y;
            }
            const int total = __shfl_sync(kFull, si, 31);
            const int64_t org = bu - (si - ls);
            for (int c0 = 0; c0 < total; c0 += 32) {
                const int pos = c0 + lane;
                int r = 0;  // the member whose list holds pos
#pragma unroll
                for (int st = 16; st > 0; st >>= 1) {
                    const int v = __shfl_sync(kFull, si, r + st - 1);
                    if (v <= pos) r += st;
                }
                const int64_t e = __shfl_sync(kFull, org, r) + pos;
                const uint32_t wr = __shfl_sync(kFull, wu, r);
                const uint32_t wb = pos < total ? __ldg(p.adj + e) : 0u;
                const uint32_t b = wb & TG_IDMASK;
                uint32_t c[LP];
                if (wedge_counts<LP>(p, cnt, b, pos < total && b > a, c) < 2u) continue;
                const int tu = (int)(wr >> TG_TSHIFT);
                const bool ub = (wr & TG_IDMASK) > b;
                unsigned long long *row_ub = p.c4e + (int64_t)__ldg(p.eid + e) * L2 + (ub ? ta * L : ta);
                unsigned long long *row_au =
                    p.c4e + (int64_t)__ldg(p.eid + ba + m + r) * L2 + (int)(wb >> TG_TSHIFT) * L;
#pragma unroll
                for (int t = 0; t < LP; ++t) {
                    const uint32_t v = c[t] ? c[t] - (t == tu ? 1u : 0u) : 0u;
                    if (!v) continue;
                    atomicAdd(row_ub + (ub ? t : t * L), (unsigned long long)v);
                    atomicAdd(row_au + t, (unsigned long long)v);
                }
            }
        }
    }
}

// One count into the histogram under the sorted multiset {a, b, c, d}.
__device__ __forceinline__ void k4_hist_add(unsigned long long *h4, int a, int b, int c, int d,
                                            unsigned long long v) {
    sort2(a, b);
    sort2(c, d);
    sort2(a, c);
    sort2(b, d);
    sort2(b, c);
    atomicAdd(h4 + colex4(a, b, c, d), v);
}

// ------------------------------------------------- binned waves (global) --
// Anchors whose walk is long against the number of far-end windows it spans
// (hubs): the counters stay on chip.  Far ends are numbered type by type, in
// id order inside a type, each type padded to whole windows of 2^wlg, so a window
// holds far ends of one type and a list sorted by (type, id) runs through the
// windows in order.  Every wedge a-u-b of a wave's walks becomes the 16-bit entry
// (b mod 2^wlg) << tlg | type of u in the bucket of (anchor, window).  A count
// pass sizes the buckets and a fill pass writes them, each with one counter add
// per run of consecutive lanes in one bucket.  k_c4_bin_gram then counts each
// bucket's entries by (b, t) in a dense shared-memory table of the window's far
// ends and sums c_t c_t' over the far ends in registers, for runs of anchors of
// one type in one window, whose sums all go to the multisets {ta, tb, t, t'}.
// DRAM sees the walk twice and 2 bytes per wedge written and read once, instead
// of a counter read and write per wedge.
//
// With windows over the node ids (types mixed) a far end's pairs went, one 64-bit
// shared add each, to a table by (type of b, pair).  4-cycle phase, before -> now:
// R-MAT-21 (1.43e10 wedges, L = 8) 316 -> 166 ms, CL-1M (9.1e8, L = 5) 33.5 -> 19.0
// ms, CL-100K (5.8e7) 4.1 -> 2.5 ms.
struct C4Bin {
    const int64_t *rowptr;
    const uint32_t *adj;
    const uint32_t *badj;      // adjacency entries with the far-end number for the id
    const uint32_t *thr;       // per binned anchor and type: far ends from here rank below it
    int32_t L, wlg, tlg, half;
    const uint32_t *heavy;     // the binned anchors
    const uint8_t *htype;      // their types
    const int64_t *mprefix;    // walk positions of their members (k_c4_prefix)
    const int64_t *pbase;
    const C4Unit *units;       // warp units of the wave
    int64_t n_units;
    int64_t q0;                // first anchor of the wave (bucket row = q - q0)
    int64_t W;                 // far-end windows
    uint32_t tbase[TG_MAX_TYPES + 1];  // first far-end number of each type (whole windows)
    uint32_t *cnt;             // K W bucket sizes (count pass), write cursors (fill pass)
    uint16_t *bins;            // the wave's entries, bucket after bucket
    const uint32_t *offs;      // K W + 1 bucket offsets
    const int2 *runs;          // anchors [x, y) of one type, at most kBinRun
    int64_t nitems;            // runs x windows
    unsigned long long *queue;
    unsigned long long *g4;
    int64_t n4;
    unsigned long long *work;  // [4]: wedges
};

// Numbering of the far ends: nodes [0, n) (the non-isolated ones) in blocks of
// kRankBlock; per type the blocks' counts (cnt[t nblk + block], then scanned).
constexpr int kRankBlock = 1024;

__global__ void __launch_bounds__(kRankBlock) k_bin_hist(const uint8_t *ntype, int64_t n, int64_t nblk,
                                                         int L, uint32_t *cnt) {
    __shared__ uint32_t c[TG_MAX_TYPES];
    if (threadIdx.x < TG_MAX_TYPES) c[threadIdx.x] = 0u;
    __syncthreads();
    const int64_t v = blockIdx.x * (int64_t)kRankBlock + threadIdx.x;
    const int t = v < n ? (int)ntype[v] : -1;
    for (int k = 0; k < L; ++k) {
        const unsigned m = __ballot_sync(kFull, t == k);
        if ((threadIdx.x & 31) == 0 && m) atomicAdd(&c[k], (uint32_t)__popc(m));
    }
    __syncthreads();
    if (threadIdx.x < L) cnt[threadIdx.x * nblk + blockIdx.x] = c[threadIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0) cnt[L * nblk] = 0u;
}

// base[t]: first far-end number of type t, padded to multiples of 2^lg; one warp
__global__ void k_bin_bases(const uint32_t *scan, int64_t nblk, int L, int lg, uint32_t *base) {
    if (threadIdx.x != 0) return;
    uint32_t at = 0;
    for (int t = 0; t < L; ++t) {
        base[t] = at;
        const uint32_t c = scan[(t + 1) * nblk] - scan[t * nblk];
        at += ((c + (1u << lg) - 1u) >> lg) << lg;
    }
    base[L] = at;
}

__global__ void __launch_bounds__(kRankBlock) k_bin_numbers(const uint8_t *ntype, int64_t n, int64_t nblk,
                                                            int L, const uint32_t *scan,
                                                            const uint32_t *base, uint32_t *num) {
    __shared__ uint32_t c[kRankBlock / 32][TG_MAX_TYPES];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t v = blockIdx.x * (int64_t)kRankBlock + threadIdx.x;
    const int t = v < n ? (int)ntype[v] : -1;
    uint32_t rank = 0;
    for (int k = 0; k < L; ++k) {
        const unsigned m = __ballot_sync(kFull, t == k);
        if (t == k) rank = (uint32_t)__popc(m & ((1u << lane) - 1u));
        if (lane == 0) c[warp][k] = (uint32_t)__popc(m);
    }
    __syncthreads();
    if (t < 0) return;
    for (int w = 0; w < warp; ++w) rank += c[w][t];
    num[v] = base[t] + (scan[t * nblk + blockIdx.x] - scan[t * nblk]) + rank;
}

__global__ void k_bin_entries(const uint32_t *adj, int64_t entries, const uint32_t *num, uint32_t *badj) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < entries;
         x += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t w = __ldg(adj + x);
        badj[x] = (w & ~TG_IDMASK) | __ldg(num + (w & TG_IDMASK));
    }
}

// thr[q L + t]: base[t] plus the nodes of type t with ids up to anchor q's; one
// warp per anchor.
__global__ void k_bin_thresholds(const uint32_t *heavy, int64_t na, const uint8_t *ntype, int64_t nblk,
                                 int L, const uint32_t *scan, const uint32_t *base, uint32_t *thr,
                                 uint8_t *htype) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; q < na; q += nw) {
        const int64_t a = heavy[q], blk = a / kRankBlock;
        uint32_t c = lane < L ? base[lane] + (scan[lane * nblk + blk] - scan[lane * nblk]) : 0u;
        for (int64_t v0 = blk * kRankBlock; v0 <= a; v0 += 32) {
            const int t = v0 + lane <= a ? (int)ntype[v0 + lane] : -1;
            for (int k = 0; k < L; ++k) {
                const unsigned m = __ballot_sync(kFull, t == k);
                if (lane == k) c += (uint32_t)__popc(m);
            }
        }
        if (lane < L) thr[q * L + lane] = c;
        if (lane == 0) htype[q] = ntype[a];
    }
}

constexpr int kBinUnroll = 4;              // batches of 32 positions in flight
constexpr int kBinFill = 32;            // default: binned when a walk averages this many wedges per window
constexpr size_t kBinTable = 64 * 1024;  // bytes of the dense far-end table
constexpr int kBinRun = 16;              // anchors of one type taken together, at most

// 32 consecutive positions of a walk, one per lane (entry w of a list in far-end
// numbers; in: the position belongs to the unit; tu: the type of its member): the
// entries ranked below the anchor (from their type's threshold on; lane t holds
// type t's) go to their buckets cb[window].  Runs of one bucket among consecutive
// lanes take their places with one add; the fill pass writes the entries.
template <bool kFill>
__device__ __forceinline__ void bin_put(const C4Bin &p, uint32_t *cb, uint32_t thr, uint32_t w, bool in,
                                        int tu, unsigned long long &wk) {
    const int lane = threadIdx.x & 31;
    const uint32_t from = __shfl_sync(kFull, thr, (int)(w >> TG_TSHIFT));
    const uint32_t b = w & TG_IDMASK;
    const bool ok = in && b >= from;
    const int key = ok ? (int)(b >> p.wlg) : -1;
    const int prev = __shfl_up_sync(kFull, key, 1);
    const bool head = lane == 0 || key != prev;
    const unsigned heads = __ballot_sync(kFull, head);
    const unsigned upto = (2u << lane) - 1u;
    uint32_t base = 0;
    if (head && ok) {
        const unsigned above = heads & ~upto;
        const uint32_t len = (uint32_t)((above ? __ffs(above) - 1 : 32) - lane);
        if (kFill)
            base = atomicAdd(cb + key, len);
        else
            atomicAdd(cb + key, len);
        if (!kFill) wk += len;
    }
    if (kFill) {
        const int rs = 31 - __clz(heads & upto);  // the run's first lane
        base = __shfl_sync(kFull, base, rs);
        if (ok)
            p.bins[base + (uint32_t)(lane - rs)] =
                (uint16_t)(((b & ((1u << p.wlg) - 1u)) << p.tlg) | (uint32_t)tu);
    }
}

// The count (kFill = false) or fill pass of a binned wave: one warp per unit.  A
// member's list of kBinLong entries or more is taken by the whole warp, kBinUnroll
// batches of 32 in flight, without the search that maps positions to members;
// shorter lists are taken as one sequence by the unit in which they begin.
constexpr int kBinLong = 64;

template <bool kFill>
__global__ void __launch_bounds__(kC4WalkWarps * 32) k_c4_bin_walk(C4Bin p) {
    const int lane = threadIdx.x & 31;
    unsigned long long wk = 0;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= (unsigned long long)p.n_units) break;
        const C4Unit un = p.units[item];
        const uint32_t a = p.heavy[un.q];
        const int64_t ba = p.rowptr[a];
        const int da = (int)(p.rowptr[a + 1] - ba);
        uint32_t *cb = p.cnt + (un.q - p.q0) * p.W;
        const uint32_t thr = lane < p.L ? p.thr[(int64_t)un.q * p.L + lane] : 0u;
        int64_t at = p.mprefix[p.pbase[un.q] + un.m];
        for (int m = un.m; m < da && at < un.hi; m += 32) {
            const int x = m + lane;
            int64_t bu = 0;
            int len = 0, tu = 0;
            if (x < da) {
                const uint32_t wu = __ldg(p.adj + ba + x);
                const uint32_t u = wu & TG_IDMASK;
                if (u > a) {
                    bu = p.rowptr[u];
                    const int64_t du = p.rowptr[u + 1] - bu;
                    if (du > 1) {
                        len = (int)du;
                        tu = (int)(wu >> TG_TSHIFT);
                    }
                }
            }
            int64_t incl = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            const int64_t first = at + incl - len;  // walk position of this member's list
            at += __shfl_sync(kFull, incl, 31);
            // long lists, the part [q0, q1) inside the unit
            const int64_t q0 = un.lo > first ? un.lo - first : 0;
            const int64_t q1 = un.hi - first < len ? un.hi - first : len;
            for (unsigned todo = __ballot_sync(kFull, len >= kBinLong && q0 < q1); todo; todo &= todo - 1u) {
                const int src = __ffs(todo) - 1;
                const uint32_t *list = p.badj + __shfl_sync(kFull, bu + q0, src);
                const int cnt = (int)__shfl_sync(kFull, q1 - q0, src), t = __shfl_sync(kFull, tu, src);
                for (int c = lane; c - lane < cnt; c += 32 * kBinUnroll) {
                    uint32_t w[kBinUnroll];
#pragma unroll
                    for (int z = 0; z < kBinUnroll; ++z) w[z] = c + 32 * z < cnt ? __ldg(list + c + 32 * z) : 0u;
#pragma unroll
                    for (int z = 0; z < kBinUnroll; ++z) bin_put<kFill>(p, cb, thr, w[z], c + 32 * z < cnt, t, wk);
                }
            }
            // short lists that begin inside the unit
            const int ls = len < kBinLong && first >= un.lo && first < un.hi ? len : 0;
            int si = ls;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, si, o);
                if (lane >= o) si += y;
            }
            const int total = __shfl_sync(kFull, si, 31);
            const int64_t org = bu - (si - ls);
            for (int c = 0; c < total; c += 32 * kBinUnroll) {
                uint32_t w[kBinUnroll];
                int t[kBinUnroll];
#pragma unroll
                for (int z = 0; z < kBinUnroll; ++z) {
                    const int pos = c + 32 * z + lane;
                    int r = 0;  // the member whose list holds pos
#pragma unroll
                    for (int st = 16; st > 0; st >>= 1) {
                        const int v = __shfl_sync(kFull, si, r + st - 1);
                        if (v <= pos) r += st;
                    }
                    const int64_t e = __shfl_sync(kFull, org, r) + pos;
                    t[z] = __shfl_sync(kFull, tu, r);
                    w[z] = pos < total ? __ldg(p.badj + e) : 0u;
                }
#pragma unroll
                for (int z = 0; z < kBinUnroll; ++z)
                    bin_put<kFill>(p, cb, thr, w[z], c + 32 * z + lane < total, t[z], wk);
            }
        }
    }
    if (!kFill && p.work) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wk += __shfl_xor_sync(kFull, wk, o);
        if (lane == 0 && wk) atomicAdd(p.work + 4, wk);
    }
}

// Counts of a far-end row of k_c4_bin_gram (a power of two from L on; L <= 8), 0
// for more types (k_c4_bin_pairs).  Counts of a power law of 100K nodes and 1M edges
// (hub 36K) take 4.8, 4.1, 3.9 ms with 2, 3, 4 types, 3.4 to 3.8 with 5 to 8 and 9.0
// with 9.  Rows of eight counts for 2 to 4 types, on the tensor cores, would take 3.8,
// 3.5, 3.4 ms.  A row of 9 to 16 counts spans two matrices of eight: its products are not
// written, and k_c4_bin_pairs is what there was (18.4 ms in all before the windows had
// one type).
__host__ __device__ constexpr int bin_lanes(int L) { return L <= 2 ? 2 : L <= 4 ? 4 : L <= 8 ? 8 : 0; }

// Type of window w.
__device__ __forceinline__ int bin_type(const C4Bin &p, int64_t w) {
    int t = 0;
    while (t + 1 < p.L && (int64_t)(p.tbase[t + 1] >> p.wlg) <= w) ++t;
    return t;
}

constexpr int kGramThreads = 512;

__device__ __forceinline__ void ldsm_t4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// d[0..1] += x^T y over 16 far ends: x0, y0 hold the counts of far ends 0..7 in the
// transposed ldmatrix layout (lane: type lane / 4, far ends 2 (lane % 4) and the
// next), x1, y1 those of far ends 8..15; d[0..1]: types (lane / 4, 2 (lane % 4) and
// the next).  Row 8 of A is `row8` (lanes 0..3): with ones there, d[2..3] of lanes
// 0..3 are the sums of y.
__device__ __forceinline__ void gram16(float (&d)[4], uint32_t x0, uint32_t x1, uint32_t row8, uint32_t y0,
                                       uint32_t y1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %5}, {%7, %8}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(x0), "r"(row8), "r"(x1), "r"(y0), "r"(y1));
}

// A count c below 1024 read as an fp16 value is the subnormal c 2^-24, so products
// of two counts are exact multiples of 2^-48 and sums of counts of 2^-24.
constexpr float kGramScale = 281474976710656.f, kSumScale = 16777216.f;

// Buckets of a binned wave, L <= 8 types.  A CTA takes an item (anchors of one
// type, one window): bucket after bucket it counts the entries in the table (a row
// of counts per far end), then sums c_t c_t' over the far ends and clears it.  With
// eight 16-bit counts a row (5 to 8 types) the sums are X^T X of the table X on the
// tensor cores: a row is a row of an 8 x 8 matrix of 16-bit values, so one ldmatrix
// gives 32 far ends in the layout of both operands, and the counts are used as they
// stand, as fp16 subnormals.  The fp32 sums hold integers below 2^24 (times a power
// of two) and are exact: a warp adds them to its 64-bit sums before the blocks of 128
// far ends since then could pass it (33 blocks of counts up to 63, or one of counts
// up to 255 and 16 of those).  Where a count is larger its high and low bytes take
// its place: 65536 H^T H + 256 (H^T L + L^T H) + L^T L.  On R-MAT-18 the kernel takes
// 2.5 ms (5.7 with the sums in integer registers, 3.0 with the counts converted and a
// second product for sum c); the reads and clears of the 64 KB table (1,024 shared
// wavefronts a bucket) and the two barriers a bucket bound it.  Two CTAs per SM: three
// need spills (R-MAT-21 174 against 166 ms).  The other row widths sum the rows
// with two middles or more in groups of G lanes, lane a holding sum c_a c_b for every
// b.  No add to shared memory is made until the item's end.
template <int G, bool kHalf>
__global__ void __launch_bounds__(kGramThreads, 2) k_c4_bin_gram(C4Bin p) {
    constexpr int RW = kHalf ? G / 2 : G;  // words of a row
    constexpr bool kMma = kHalf && G == 8;
    constexpr int kSums = kMma ? 2 : G;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long s_item;
    __shared__ uint32_t s_off[2 * kBinRun];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nfar = 1 << p.wlg;
    uint32_t *tab = reinterpret_cast<uint32_t *>(smem);
    unsigned long long *h4 = reinterpret_cast<unsigned long long *>(smem + (size_t)nfar * RW * 4);
    for (int q = tid; q < nfar * RW; q += kGramThreads) tab[q] = 0u;
    for (int64_t q = tid; q < p.n4; q += kGramThreads) h4[q] = 0ull;
    // this lane's type and its group (or first column)
    const int ga = kMma ? lane / 4 : lane % G, gg = kMma ? lane % 4 : lane / G;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(p.queue, 1ull);
        __syncthreads();
        if (s_item >= (unsigned long long)p.nitems) break;
        const int64_t w = (int64_t)s_item % p.W;
        const int2 run = p.runs[(int64_t)s_item / p.W];
        const int nr = run.y - run.x;
        if (tid < nr) {
            const int64_t b = (run.x + tid - p.q0) * p.W + w;
            s_off[2 * tid] = p.offs[b];
            s_off[2 * tid + 1] = p.offs[b + 1];
        }
        __syncthreads();
        unsigned long long acc[kSums], one[2] = {0ull, 0ull};
#pragma unroll
        for (int b = 0; b < kSums; ++b) acc[b] = 0ull;
        // kMma: the fp32 sums since the last settling (row 8, lanes 0..3: sums of the
        // counts of types 2 gg and the next), and the blocks in them by weight
        float ll[4] = {0.f, 0.f, 0.f, 0.f};
        int spent = 0;
        const uint32_t row8 = lane < 4 ? 0x3c003c00u : 0u;  // 1.0, 1.0
        auto settle = [&]() {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                acc[b % kSums] += (uint32_t)(ll[b] * kGramScale);
                one[b] += (uint32_t)(ll[2 + b] * kSumScale);
                ll[b] = ll[2 + b] = 0.f;
            }
            spent = 0;
        };
        // four entries at 8-byte boundaries; those outside the bucket are left out
        auto fetch = [&](uint32_t k, uint32_t c1) -> uint2 {
            return k < c1 ? *reinterpret_cast<const uint2 *>(p.bins + k) : make_uint2(0u, 0u);
        };
        auto count = [&](uint2 e, uint32_t k, uint32_t c0, uint32_t c1) {
            if (k >= c1) return;
            const bool whole = k >= c0 && k + 4 <= c1;
#pragma unroll
            for (int z = 0; z < 4; ++z) {
                const uint32_t x = ((z < 2 ? e.x : e.y) >> (16 * (z & 1))) & 0xffffu;
                if (!whole && (k + z < c0 || k + z >= c1)) continue;
                if (kHalf)
                    atomicAdd(tab + (x >> 1), 1u << (16 * (x & 1u)));
                else
                    atomicAdd(tab + x, 1u);
            }
        };
        uint32_t k0 = (s_off[0] & ~3u) + 4u * tid;
        uint2 ahead = fetch(k0, s_off[1]);
        for (int r = 0; r < nr; ++r) {
            const uint32_t c0 = s_off[2 * r], c1 = s_off[2 * r + 1];
            for (uint32_t k = k0; k < c1; k += 4 * kGramThreads) {
                const uint2 e = ahead;
                ahead = fetch(k + 4 * kGramThreads, c1);
                count(e, k, c0, c1);
            }
            if (r + 1 < nr) {  // the next bucket's first entries, before the rows are taken
                k0 = (s_off[2 * r + 2] & ~3u) + 4u * tid;
                ahead = fetch(k0, s_off[2 * r + 3]);
            }
            if (c0 == c1) continue;  // uniform across the CTA
            __syncthreads();
            if (kMma) {
                // a warp takes 128 rows at a time
                for (int r0 = 128 * warp; r0 < nfar; r0 += 128 * (kGramThreads / 32)) {
                    uint32_t x[4][4], big = 0;
                    const uint32_t base = (uint32_t)__cvta_generic_to_shared(tab + (r0 + lane) * RW);
#pragma unroll
                    for (int z = 0; z < 4; ++z) {
                        ldsm_t4(base + z * 32 * RW * 4, x[z]);
                        big |= x[z][0] | x[z][1] | x[z][2] | x[z][3];
                    }
                    big = __reduce_or_sync(kFull, big);
                    if (big == 0u) continue;
                    uint4 *row = reinterpret_cast<uint4 *>(tab) + r0 + lane;
#pragma unroll
                    for (int z = 0; z < 4; ++z) row[32 * z] = make_uint4(0u, 0u, 0u, 0u);
                    if (!(big & 0xff00ff00u)) {
                        const int weight = big & 0xffc0ffc0u ? 17 : 1;
                        if (spent + weight > 33) settle();
                        spent += weight;
#pragma unroll
                        for (int z = 0; z < 4; ++z) {
                            gram16(ll, x[z][0], x[z][1], row8, x[z][0], x[z][1]);
                            gram16(ll, x[z][2], x[z][3], row8, x[z][2], x[z][3]);
                        }
                    } else {
                        settle();
                        float lh[4] = {0.f, 0.f, 0.f, 0.f}, hh[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int z = 0; z < 4; ++z)
#pragma unroll
                            for (int h = 0; h < 4; h += 2) {
                                const uint32_t l0 = x[z][h] & 0x00ff00ffu, l1 = x[z][h + 1] & 0x00ff00ffu;
                                const uint32_t h0 = (x[z][h] >> 8) & 0x00ff00ffu;
                                const uint32_t h1 = (x[z][h + 1] >> 8) & 0x00ff00ffu;
                                gram16(ll, l0, l1, row8, l0, l1);
                                gram16(lh, l0, l1, 0u, h0, h1);
                                gram16(lh, h0, h1, 0u, l0, l1);
                                gram16(hh, h0, h1, row8, h0, h1);
                            }
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            acc[b % kSums] += 256ull * (uint32_t)(lh[b] * kGramScale) +
                                              65536ull * (uint32_t)(hh[b] * kGramScale);
                            one[b] += 256ull * (uint32_t)(hh[2 + b] * kSumScale);
                        }
                        settle();
                    }
                }
            } else {
                for (int row = tid; row < nfar; row += kGramThreads) {
                    uint32_t v[RW], any = 0, sum = 0;
                    uint32_t *tr = tab + row * RW;
#pragma unroll
                    for (int z = 0; z < RW; ++z) {
                        v[z] = tr[z];
                        any |= v[z];
                        sum += kHalf ? (v[z] & 0xffffu) + (v[z] >> 16) : v[z];
                    }
                    if (any) {
#pragma unroll
                        for (int z = 0; z < RW; ++z) tr[z] = 0u;
                    }
                    // one middle closes no cycle
                    for (unsigned m = __ballot_sync(kFull, sum > 1u); m;) {
                        unsigned mine = m;  // this group's row: the gg-th set bit
#pragma unroll
                        for (int z = 0; z < 32 / G; ++z) {
                            if (z < gg) mine &= mine - 1u;
                            m &= m - 1u;
                        }
                        const int src = mine ? __ffs(mine) - 1 : 0;
                        uint32_t c[G], ca = 0;
#pragma unroll
                        for (int z = 0; z < RW; ++z) {
                            const uint32_t y = __shfl_sync(kFull, v[z], src);
                            if (kHalf) {
                                c[2 * z] = y & 0xffffu;
                                c[2 * z + 1] = y >> 16;
                            } else {
                                c[z] = y;
                            }
                        }
#pragma unroll
                        for (int b = 0; b < G; ++b)
                            if (b == ga) ca = c[b];
                        if (!mine) ca = 0u;
                        one[0] += ca;
#pragma unroll
                        for (int b = 0; b < kSums; ++b) acc[b] += (unsigned long long)ca * c[b];
                    }
                }
            }
            __syncthreads();
        }
        // the item's sums over the groups of a warp, then into the histogram; `own`:
        // the sum of the counts of this lane's type
        unsigned long long own = one[0];
        if (kMma) {
            settle();
            const unsigned long long s0 = __shfl_sync(kFull, one[0], ga / 2), s1 = __shfl_sync(kFull, one[1], ga / 2);
            own = ga & 1 ? s1 : s0;
        } else {
#pragma unroll
            for (int o = G; o < 32; o <<= 1) {
                own += __shfl_xor_sync(kFull, own, o);
#pragma unroll
                for (int b = 0; b < kSums; ++b) acc[b] += __shfl_xor_sync(kFull, acc[b], o);
            }
        }
        if ((kMma || gg == 0) && own) {
            const int ta = p.htype[run.x], tb = bin_type(p, w);
#pragma unroll
            for (int b = 0; b < kSums; ++b) {
                const int t = kMma ? 2 * gg + b : b;
                if (t < ga) continue;
                const unsigned long long x = t == ga ? (acc[b] - own) / 2 : acc[b];
                if (x) k4_hist_add(h4, ta, tb, ga, t, x);
            }
        }
    }
    __syncthreads();
    for (int64_t q = tid; q < p.n4; q += kGramThreads)
        if (h4[q]) atomicAdd(p.g4 + q, h4[q]);
}

// The same for more than 8 types: a far end's first entry puts it on a list; then
// one thread per listed far end adds its pairs to a shared histogram (c4_add).
constexpr int kBinPairThreads = 1024;

__global__ void __launch_bounds__(kBinPairThreads) k_c4_bin_pairs(C4Bin p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x;
    const int L = p.L, Lp = L + (L & 1);
    const int nfar = 1 << p.wlg;
    unsigned long long *h4 = reinterpret_cast<unsigned long long *>(smem);
    uint32_t *tab = reinterpret_cast<uint32_t *>(smem + (((size_t)p.n4 * 8 + 15) & ~(size_t)15));
    const int twords = p.half ? nfar * (Lp >> 1) : nfar * L;
    uint32_t *tbits = tab + twords;                                      // nfar / 32 words
    uint16_t *flist = reinterpret_cast<uint16_t *>(tbits + nfar / 32);  // touched far ends
    const volatile uint32_t *vtab = tab;
    __shared__ unsigned long long s_item;
    __shared__ uint32_t s_nl;
    for (int64_t q = tid; q < p.n4; q += blockDim.x) h4[q] = 0ull;
    for (int q = tid; q < twords + nfar / 32; q += blockDim.x) tab[q] = 0u;
    if (tid == 0) s_nl = 0u;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(p.queue, 1ull);
        __syncthreads();
        if (s_item >= (unsigned long long)p.nitems) break;
        const int64_t w = (int64_t)s_item % p.W;
        const int2 run = p.runs[(int64_t)s_item / p.W];
        const int ta = p.htype[run.x], tb = bin_type(p, w);
        for (int r = run.x; r < run.y; ++r) {
            const int64_t bucket = (r - p.q0) * p.W + w;
            const uint32_t c0 = p.offs[bucket], c1 = p.offs[bucket + 1];
            if (c0 == c1) continue;  // uniform across the CTA
            for (uint32_t k = c0 + tid; k < c1; k += blockDim.x) {
                const uint32_t ev = p.bins[k];
                const uint32_t bl = ev >> p.tlg, t = ev & ((1u << p.tlg) - 1u);
                bool first;
                if (p.half) {
                    const uint32_t idx = bl * (uint32_t)Lp + t;
                    const int sh = (int)(idx & 1u) * 16;
                    first = ((atomicAdd(tab + (idx >> 1), 1u << sh) >> sh) & 0xffffu) == 0u;
                } else {
                    first = atomicAdd(tab + bl * (uint32_t)L + t, 1u) == 0u;
                }
                if (first) {
                    const uint32_t bit = 1u << (bl & 31u);
                    if (!(atomicOr(tbits + (bl >> 5), bit) & bit)) flist[atomicAdd(&s_nl, 1u)] = (uint16_t)bl;
                }
            }
            __syncthreads();
            const uint32_t nl = s_nl;
            for (uint32_t x = tid; x < nl; x += blockDim.x) {
                const uint32_t bl = flist[x];
                uint32_t c[TG_MAX_TYPES];
                uint32_t sum = 0;
                for (int t = 0; t < L; ++t) {
                    const uint32_t at = p.half ? (bl * (uint32_t)Lp + t) >> 1 : bl * (uint32_t)L + t;
                    c[t] = p.half ? (vtab[at] >> (16 * (t & 1))) & 0xffffu : vtab[at];
                    sum += c[t];
                }
                const int row = p.half ? Lp >> 1 : L;
                for (int q = 0; q < row; ++q) tab[bl * (uint32_t)row + q] = 0u;
                if (sum >= 2) c4_add(h4, L, ta, tb, c);
            }
            __syncthreads();
            for (int q = tid; q < nfar / 32; q += blockDim.x) tbits[q] = 0u;
            if (tid == 0) s_nl = 0u;
            __syncthreads();
        }
    }
    for (int64_t q = tid; q < p.n4; q += blockDim.x)
        if (h4[q]) atomicAdd(p.g4 + q, h4[q]);
}

// ----------------------------------------------------------- 4-cliques ----
struct K4Params {
    const int64_t *uoff;       // up lists (tg_lists)
    const uint32_t *uadj;
    const uint32_t *ueid;
    const int32_t *utoff;
    const uint8_t *ntype;
    int64_t n;
    int32_t L, P;
    int32_t cap;               // W entries per warp in shared memory
    unsigned long long *queue;
    unsigned long long *k4e;   // M * P, 4-cliques by the types of the two other nodes
    unsigned long long *work;  // [5]: candidate tests, [6]: 4-cliques
    int64_t min_d0;            // only x0 with up lists longer than this
};

constexpr int kK4Warps = 8;

__device__ __forceinline__ void k4_add(unsigned long long *k4e, int64_t e, int P, int L, int a,
                                       int b, unsigned long long v) {
    atomicAdd(k4e + e * P + pair_index(L, a, b), v);
}

// 4-cliques per edge, one warp per lowest node x0.
__global__ void __launch_bounds__(kK4Warps * 32) k_k4(K4Params p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = p.L, P = p.P, cap = p.cap;
    uint32_t *w_ent = reinterpret_cast<uint32_t *>(smem) + (size_t)warp * cap * (3 + L);
    int32_t *w_p0 = reinterpret_cast<int32_t *>(w_ent + cap);  // position in x0's list
    int32_t *w_pv = w_p0 + cap;                                  // position in v's list
    uint32_t *xacc = reinterpret_cast<uint32_t *>(w_pv + cap);  // cap * L
    const uint32_t below = (1u << lane) - 1u;
    unsigned long long wk_cand = 0, wk_k4 = 0;

    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= (unsigned long long)p.n) break;
        const uint32_t x0 = (uint32_t)item;
        const int64_t b0 = p.uoff[x0];
        const int d0 = (int)(p.uoff[x0 + 1] - b0);
        if (d0 < 3 || d0 <= p.min_d0) continue;  // x0 is the lowest node: three more above it
        const int t0 = p.ntype[x0];
        const int32_t *to0 = p.utoff + (int64_t)x0 * (L + 1);
        for (int c0 = 0; c0 < d0; c0 += 32) {
            const int xx = c0 + lane;
            uint32_t ev = 0;
            bool isup = false;
            if (xx < d0) {
                ev = __ldg(p.uadj + b0 + xx);
                isup = true;
            }
            unsigned upm = __ballot_sync(kFull, isup);
            while (upm) {
                const int src = __ffs(upm) - 1;
                upm &= upm - 1;
                const uint32_t vent = __shfl_sync(kFull, ev, src);
                const uint32_t v = vent & TG_IDMASK;
                const int tv = (int)(vent >> TG_TSHIFT);
                const int64_t bv = p.uoff[v];
                const int dv = (int)(p.uoff[v + 1] - bv);
                const int32_t *tov = p.utoff + (int64_t)v * (L + 1);
                const int64_t e0v = __ldg(p.ueid + b0 + c0 + src);
                // W = up(v) n up(x0) (= up(v) n Gamma(x0)), in the order of up(v)
                int nw = 0;
                for (int c1 = 0; c1 < dv; c1 += 32) {
                    const int q = c1 + lane;
                    bool ok = false;
                    uint32_t wq = 0;
                    int pos0 = -1;
                    if (q < dv) {
                        wq = __ldg(p.uadj + bv + q);
                        pos0 = find_pos(p.uadj, b0, to0, wq);
                        ok = pos0 >= 0;
                    }
                    const unsigned m = __ballot_sync(kFull, ok);
                    const int r = nw + __popc(m & below);
                    if (ok && r < cap) {
                        w_ent[r] = wq;
                        w_p0[r] = pos0;
                        w_pv[r] = q;
                    }
                    nw += __popc(m);
                }
                if (nw < 2) {
                    __syncwarp();
                    continue;
                }
                const bool staged = nw <= cap;
                if (staged)
                    for (int q = lane; q < nw * L; q += 32) xacc[q] = 0u;
                __syncwarp();
                // every w of W (staged: from shared memory; else re-derived)
                for (int c1 = 0, k = 0; staged ? k < nw : c1 < dv;) {
                    unsigned wm;
                    uint32_t wlane = 0;
                    int p0lane = -1;
                    if (staged) {
                        wm = 1u;
                    } else {
                        const int q = c1 + lane;
                        bool ok = false;
                        if (q < dv) {
                            wlane = __ldg(p.uadj + bv + q);
                            p0lane = find_pos(p.uadj, b0, to0, wlane);
                            ok = p0lane >= 0;
                        }
                        wm = __ballot_sync(kFull, ok);
                    }
                    while (wm) {
                        const int sl = __ffs(wm) - 1;
                        wm &= wm - 1;
                        uint32_t went;
                        int wp0, wpv;
                        if (staged) {
                            went = w_ent[k];
                            wp0 = w_p0[k];
                            wpv = w_pv[k];
                        } else {
                            went = __shfl_sync(kFull, wlane, sl);
                            wp0 = __shfl_sync(kFull, p0lane, sl);
                            wpv = c1 + sl;
                        }
                        const uint32_t w = went & TG_IDMASK;
                        const int tw = (int)(went >> TG_TSHIFT);
                        const int64_t bw = p.uoff[w];
                        const int dw = (int)(p.uoff[w + 1] - bw);
                        const int64_t e0w = __ldg(p.ueid + b0 + wp0);
                        const int64_t evw = __ldg(p.ueid + bv + wpv);
                        for (int c2 = 0; c2 < dw; c2 += 32) {
                            const int r = c2 + lane;
                            int key = -1;
                            if (r < dw) {
                                const uint32_t xe = __ldg(p.uadj + bw + r);
                                {
                                    ++wk_cand;
                                    int64_t e0x = -1;
                                    if (staged) {
                                        int lo = 0, hi = nw;
                                        while (lo < hi) {
                                            const int mid = (lo + hi) >> 1;
                                            if (w_ent[mid] < xe)
                                                lo = mid + 1;
                                            else
                                                hi = mid;
                                        }
                                        if (lo < nw && w_ent[lo] == xe) {
                                            // (x0,x) and (v,x) are summed per x below
                                            atomicAdd(xacc + lo * L + tw, 1u);
                                            e0x = 0;
                                        }
                                    } else {
                                        const int px0 = find_pos(p.uadj, b0, to0, xe);
                                        if (px0 >= 0) {
                                            const int pxv = find_pos(p.uadj, bv, tov, xe);
                                            if (pxv >= 0) {
                                                e0x = 0;
                                                k4_add(p.k4e, __ldg(p.ueid + b0 + px0), P, L, tv, tw, 1ull);
                                                k4_add(p.k4e, __ldg(p.ueid + bv + pxv), P, L, t0, tw, 1ull);
                                            }
                                        }
                                    }
                                    if (e0x >= 0) {
                                        key = (int)(xe >> TG_TSHIFT);
                                        k4_add(p.k4e, __ldg(p.ueid + bw + r), P, L, t0, tv, 1ull);
                                        ++wk_k4;
                                    }
                                }
                            }
                            // edges (x0,v), (x0,w), (v,w), summed over x of one type
                            const unsigned mm = __match_any_sync(kFull, key);
                            if (key >= 0 && lane == __ffs(mm) - 1) {
                                const unsigned long long c = (unsigned long long)__popc(mm);
                                k4_add(p.k4e, e0v, P, L, tw, key, c);
                                k4_add(p.k4e, e0w, P, L, tv, key, c);
                                k4_add(p.k4e, evw, P, L, t0, key, c);
                            }
                        }
                        if (staged) ++k;
                    }
                    if (!staged) c1 += 32;
                }
                if (staged) {
                    __syncwarp();
                    for (int q = lane; q < nw * L; q += 32) {
                        const uint32_t c = xacc[q];
                        if (c) {
                            const int kx = q / L, tw = q % L;
                            k4_add(p.k4e, __ldg(p.ueid + b0 + w_p0[kx]), P, L, tv, tw, c);
                            k4_add(p.k4e, __ldg(p.ueid + bv + w_pv[kx]), P, L, t0, tw, c);
                        }
                    }
                }
                __syncwarp();
            }
        }
    }
    if (p.work) {
        if (wk_cand) atomicAdd(p.work + 5, wk_cand);
        if (wk_k4) atomicAdd(p.work + 6, wk_k4);
    }
}

// 4-cliques by type multiset only (global mode).  As k_k4, each clique is met
// from its lowest node x0 and the next one v; here a warp's work item is a
// run of kK4GChunk oriented edges (x0, v) of the up lists, so the edges of a
// costly x0 spread over many warps.  Membership in up(x0) and in
// W = up(v) n up(x0) is a probe of a per-warp hash set when the set fits (cap
// entries), else a search of the sorted up lists.
struct K4GParams {
    const int64_t *uoff;
    const uint32_t *uadj;
    const int32_t *utoff;
    const uint8_t *ntype;
    int64_t n;
    int64_t m;  // entries of the up lists (edges)
    int32_t L;
    int32_t cap;  // set entries per warp (tables of 2^hlg >= 2 cap slots)
    int32_t hlg;
    int32_t min_d0;  // k_k4_global: only x0 with up lists longer than this
    unsigned long long *queue;
    unsigned long long *g4;
    int64_t n4;
    unsigned long long *work;
    int32_t pidx, pcnt;   // only lowest nodes x0 with x0 mod pcnt == pidx
};

constexpr int kK4GWarps = 8;
constexpr int kK4GChunk = 8;  // oriented edges (x0, v) per work item

__global__ void __launch_bounds__(kK4GWarps * 32) k_k4_global(K4GParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = p.L, cap = p.cap, tsz = 1 << p.hlg;
    unsigned long long *h4 = reinterpret_cast<unsigned long long *>(smem);
    const size_t h4b = ((size_t)p.n4 * 8 + 15) & ~(size_t)15;
    uint32_t *went = reinterpret_cast<uint32_t *>(smem + h4b) + (size_t)warp * (cap + 2 * tsz);
    uint32_t *hx = went + cap;
    uint32_t *hw = hx + tsz;
    for (int64_t q = threadIdx.x; q < p.n4; q += blockDim.x) h4[q] = 0ull;
    __syncthreads();
    const uint32_t below = (1u << lane) - 1u;
    unsigned long long wk_cand = 0, wk_k4 = 0;
    const int64_t nchunks = (p.m + kK4GChunk - 1) / kK4GChunk;
    int64_t cur = -1;  // x0 whose up list the hash set hx holds
    int lgx = 5;
    bool xh = false;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= (unsigned long long)nchunks) break;
        // the chunk's oriented edges (x0, v): positions q of the up lists
        const int64_t q0 = (int64_t)item * kK4GChunk;
        const int64_t q1 = min(p.m, q0 + kK4GChunk);
        int64_t x0 = 0;
        {
            int64_t lo = 0, hi = p.n - 1;  // last x0 with uoff[x0] <= q0
            while (lo < hi) {
                const int64_t mid = (lo + hi + 1) >> 1;
                if (__ldg(p.uoff + mid) <= q0)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            x0 = lo;
        }
        for (int64_t qq = q0; qq < q1; ++qq) {
        while (__ldg(p.uoff + x0 + 1) <= qq) ++x0;
        const int64_t b0 = __ldg(p.uoff + x0);
        const int d0 = (int)(__ldg(p.uoff + x0 + 1) - b0);
        if (d0 < 3 || d0 <= p.min_d0 || x0 % p.pcnt != p.pidx) continue;  // three more above
                                                  // x0; or a bitmap kernel's; or another part's
        const int t0 = p.ntype[x0];
        const int32_t *to0 = p.utoff + x0 * (L + 1);
        if (x0 != cur) {
            cur = x0;
            xh = d0 <= cap;
            lgx = 5;
            while ((1 << lgx) < 2 * d0 && lgx < p.hlg) ++lgx;
            __syncwarp();
            if (xh) {
                for (int q = lane; q < (1 << lgx); q += 32) hx[q] = 0u;
                __syncwarp();
                for (int q = lane; q < d0; q += 32) hset_put(hx, lgx, __ldg(p.uadj + b0 + q) & TG_IDMASK);
                __syncwarp();
            }
        }
        {
            {
                const uint32_t vent = __ldg(p.uadj + qq);
                const uint32_t v = vent & TG_IDMASK;
                const int tv = (int)(vent >> TG_TSHIFT);
                const int64_t bv = p.uoff[v];
                const int dv = (int)(p.uoff[v + 1] - bv);
                const int32_t *tov = p.utoff + (int64_t)v * (L + 1);
                // W = up(v) n up(x0)
                int nw = 0;
                for (int c1 = 0; c1 < dv; c1 += 32) {
                    const int q = c1 + lane;
                    bool ok = false;
                    uint32_t wq = 0;
                    if (q < dv) {
                        wq = __ldg(p.uadj + bv + q);
                        ok = xh ? hset_has(hx, lgx, wq & TG_IDMASK) : find_pos(p.uadj, b0, to0, wq) >= 0;
                    }
                    const unsigned m = __ballot_sync(kFull, ok);
                    const int r = nw + __popc(m & below);
                    if (ok && r < cap) went[r] = wq;
                    nw += __popc(m);
                }
                if (nw < 2) {
                    __syncwarp();
                    continue;
                }
                const bool staged = nw <= cap;
                int lgw = 5;
                while ((1 << lgw) < 2 * nw && lgw < p.hlg) ++lgw;
                if (staged) {
                    for (int q = lane; q < (1 << lgw); q += 32) hw[q] = 0u;
                    __syncwarp();
                    for (int q = lane; q < nw; q += 32) hset_put(hw, lgw, went[q] & TG_IDMASK);
                }
                __syncwarp();
                for (int c1 = 0, k = 0; staged ? k < nw : c1 < dv;) {
                    unsigned wm;
                    uint32_t wlane = 0;
                    if (staged) {
                        wm = 1u;
                    } else {
                        const int q = c1 + lane;
                        bool ok = false;
                        if (q < dv) {
                            wlane = __ldg(p.uadj + bv + q);
                            ok = xh ? hset_has(hx, lgx, wlane & TG_IDMASK)
                                    : find_pos(p.uadj, b0, to0, wlane) >= 0;
                        }
                        wm = __ballot_sync(kFull, ok);
                    }
                    while (wm) {
                        const int sl = __ffs(wm) - 1;
                        wm &= wm - 1;
                        const uint32_t went_k = staged ? went[k] : __shfl_sync(kFull, wlane, sl);
                        const uint32_t w = went_k & TG_IDMASK;
                        const int tw = (int)(went_k >> TG_TSHIFT);
                        const int64_t bw = p.uoff[w];
                        const int dw = (int)(p.uoff[w + 1] - bw);
                        int s0 = t0, s1 = tv, s2 = tw;
                        sort2(s0, s1);
                        sort2(s1, s2);
                        sort2(s0, s1);
                        for (int c2 = 0; c2 < dw; c2 += 32) {
                            const int r = c2 + lane;
                            int key = -1;
                            if (r < dw) {
                                const uint32_t xe = __ldg(p.uadj + bw + r);
                                ++wk_cand;
                                bool in;
                                if (staged) {
                                    in = hset_has(hw, lgw, xe & TG_IDMASK);
                                } else {
                                    in = (xh ? hset_has(hx, lgx, xe & TG_IDMASK)
                                             : find_pos(p.uadj, b0, to0, xe) >= 0) &&
                                         find_pos(p.uadj, bv, tov, xe) >= 0;
                                }
                                if (in) {
                                    key = (int)(xe >> TG_TSHIFT);
                                    ++wk_k4;
                                }
                            }
                            const unsigned mm = __match_any_sync(kFull, key);
                            if (key >= 0 && lane == __ffs(mm) - 1) {
                                int q0 = s0, q1 = s1, q2 = s2, q3 = key;
                                sort2(q2, q3);
                                sort2(q1, q2);
                                sort2(q0, q1);
                                atomicAdd(h4 + colex4(q0, q1, q2, q3), (unsigned long long)__popc(mm));
                            }
                        }
                        if (staged) ++k;
                    }
                    if (!staged) c1 += 32;
                }
                __syncwarp();
            }
        }
        }
    }
    __syncthreads();
    for (int64_t q = threadIdx.x; q < p.n4; q += blockDim.x)
        if (h4[q]) atomicAdd(p.g4 + q, h4[q]);
    if (p.work) {
        if (wk_cand) atomicAdd(p.work + 5, wk_cand);
        if (wk_k4) atomicAdd(p.work + 6, wk_k4);
    }
}

// The longest up list.
__global__ void k_max_up(const int64_t *uoff, int64_t n, unsigned long long *mx) {
    unsigned long long m = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, (unsigned long long)(uoff[i + 1] - uoff[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
    if ((threadIdx.x & 31) == 0 && m) atomicMax(mx, m);
}

// Global mode: the per-edge pass ran with Q = C4 = 0.  Summed over the edges,
// Q and C4 enter the graphlet sums (each identity is linear in them) only
// through the type-multiset totals of 4-cliques K4 and of non-induced
// 4-cycles N_C4; added here to the undivided sums of h3..h8:
//   h3 -12 N_C4 - 36 K4, h4 -12 K4, h5 +4 N_C4 + 12 K4, h6 +48 K4,
//   h7 -30 K4, h8 +6 K4.   (c4 = N_C4, k4 = K4; arithmetic mod 2^64.)
__global__ void k_cyc_correct(unsigned long long *hist, int64_t off4, int64_t n4,
                              const unsigned long long *c4, const unsigned long long *k4) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n4;
         r += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long w = c4[r], k = k4[r];
        hist[off4 + 0 * n4 + r] += (unsigned long long)(-12ll) * w + (unsigned long long)(-36ll) * k;
        hist[off4 + 1 * n4 + r] += (unsigned long long)(-12ll) * k;
        hist[off4 + 2 * n4 + r] += 4ull * w + 12ull * k;
        hist[off4 + 3 * n4 + r] += 48ull * k;
        hist[off4 + 4 * n4 + r] += (unsigned long long)(-30ll) * k;
        hist[off4 + 5 * n4 + r] += 6ull * k;
    }
}



// Launch shape of k_c4_pairs: per-warp histogram copies when they fit in 64 KB.
struct PairsConf {
    size_t smem;
    int priv;
    int64_t grid;
};
int c4_pairs_conf(int64_t n4, PairsConf &c) {
    const size_t one = (size_t)n4 * 8;
    c.priv = one * (kC4Threads / 32) <= (size_t)64 * 1024 ? 1 : 0;
    c.smem = c.priv ? one * (kC4Threads / 32) : one;
    TG_TRY(tg_allow_max_smem((const void *)k_c4_pairs));
    int per = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_c4_pairs, kC4Threads, c.smem));
    c.grid = (int64_t)tg_num_sms() * (per > 0 ? per : 1);
    return TG_OK;
}

// Waves of the split anchors list[0 .. nheavy) (degrees hdeg): walk positions
// per anchor (k_c4_prefix), warp units of about a quarter of a warp's share of
// each wave (k_c4_units), then per wave of K anchors (K = slots of p.scratch)
// k_c4_walk, in per-edge mode k_c4_wedges, and k_c4_pairs.
int c4_walk_waves(const C4Params &p, const tg_graph *g, const uint32_t *list, int64_t nheavy,
                  const std::vector<int64_t> &hdeg, int64_t K, cudaStream_t s) {
    PairsConf pc;
    TG_TRY(c4_pairs_conf(p.n4, pc));
    const int64_t pgrid = pc.grid;
    const size_t psmem = pc.smem;
    const int ppriv = pc.priv;
    std::vector<int64_t> pb((size_t)nheavy + 1, 0);
    for (int64_t q = 0; q < nheavy; ++q) pb[q + 1] = pb[q] + hdeg[q];
    DevBuf<int64_t> dpb, dmp;
    DevBuf<unsigned long long> dtot;
    if (!dpb.alloc(nheavy + 1, s) || !dmp.alloc(pb[nheavy], s) || !dtot.alloc(nheavy, s))
        return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemcpyAsync(dpb.p, pb.data(), (nheavy + 1) * 8, cudaMemcpyHostToDevice, s));
    k_c4_prefix<<<(unsigned)nheavy, 256, 0, s>>>(list, dpb.p, g->rowptr, g->adj, dmp.p, dtot.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    std::vector<unsigned long long> tot_h((size_t)nheavy);
    TG_TRY_CUDA(cudaMemcpyAsync(tot_h.data(), dtot.p, nheavy * 8, cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    int wper = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&wper, k_c4_walk, kC4WalkWarps * 32, 0));
    if (wper < 1) wper = 1;
    void (*const wedges)(C4Params) = g->L <= 4 ? k_c4_wedges<4> : g->L <= 8 ? k_c4_wedges<8> : k_c4_wedges<16>;
    int eper = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&eper, wedges, kC4WalkWarps * 32, 0));
    if (eper < 1) eper = 1;
    const int64_t walk_grid = (int64_t)tg_num_sms() * wper;
    const int64_t warps = walk_grid * kC4WalkWarps;
    // waves: runs of at most K consecutive anchors of one counter width; an
    // anchor with fewer than 2^16 neighbours counts in 16-bit halves (no
    // count can reach 2^16), the others and per-edge mode in 32-bit words
    const int64_t half_max = p.g4 ? 65536 : 0;
    std::vector<int64_t> wq0, wq1;
    std::vector<int> whalf;
    for (int64_t q = 0; q < nheavy;) {
        const int half = hdeg[q] < half_max ? 1 : 0;
        int64_t e = q + 1;
        while (e < nheavy && e - q < K && (hdeg[e] < half_max ? 1 : 0) == half) ++e;
        wq0.push_back(q);
        wq1.push_back(e);
        whalf.push_back(half);
        q = e;
    }
    const int64_t nwaves = (int64_t)wq0.size();
    std::vector<int64_t> us((size_t)nheavy + 1, 0), tg((size_t)nheavy, 1);
    for (int64_t w = 0; w < nwaves; ++w) {
        const int64_t q0 = wq0[w], q1 = wq1[w];
        unsigned long long wt = 0;
        for (int64_t q = q0; q < q1; ++q) wt += tot_h[q];
        const int64_t tgt =
            std::max<int64_t>(kWalkUnitMin, (int64_t)((wt + 4 * warps - 1) / (4 * warps)));
        for (int64_t q = q0; q < q1; ++q) {
            tg[q] = tgt;
            us[q + 1] = us[q] + (int64_t)((tot_h[q] + tgt - 1) / tgt);
        }
    }
    const int64_t nunits = us[nheavy];
    DevBuf<int64_t> dus, dtg;
    DevBuf<C4Unit> dun;
    DevBuf<unsigned long long> dq;
    if (!dus.alloc(nheavy + 1, s) || !dtg.alloc(nheavy, s) || !dun.alloc(nunits ? nunits : 1, s) ||
        !dq.alloc(2 * nwaves, s))
        return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemcpyAsync(dus.p, us.data(), (nheavy + 1) * 8, cudaMemcpyHostToDevice, s));
    TG_TRY_CUDA(cudaMemcpyAsync(dtg.p, tg.data(), nheavy * 8, cudaMemcpyHostToDevice, s));
    TG_TRY_CUDA(cudaMemsetAsync(dq.p, 0, 2 * nwaves * 8, s));
    if (nunits > 0) {
        const unsigned ug = (unsigned)std::min<int64_t>((nunits + 255) / 256, 65535LL * 16);
        k_c4_units<<<ug, 256, 0, s>>>(dus.p, nheavy, dtg.p, dtot.p, dmp.p, dpb.p, list, g->rowptr,
                                      dun.p); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    C4Params pd = p;
    pd.phase = 0;
    pd.heavy = list;
    pd.mprefix = dmp.p;
    pd.pbase = dpb.p;
    const int L = p.L;
    for (int64_t w = 0; w < nwaves; ++w) {
        const int64_t q0 = wq0[w], q1 = wq1[w];
        pd.q0 = q0;
        pd.half = whalf[w];
        pd.bits_off = whalf[w] ? p.n * ((L + 1) >> 1) : p.n * (L + 1);
        pd.wunits = dun.p + us[q0];
        pd.n_units = us[q1] - us[q0];
        pd.queue = dq.p + w;
        if (pd.n_units > 0) {
            const int64_t need = (pd.n_units + kC4WalkWarps - 1) / kC4WalkWarps;
            const int64_t grid = std::min<int64_t>(walk_grid, need);
            k_c4_walk<<<(unsigned)grid, kC4WalkWarps * 32, 0, s>>>(pd); tg_note_launch();
            TG_TRY_CUDA(cudaGetLastError());
            if (!p.g4) {
                pd.queue = dq.p + nwaves + w;
                wedges<<<(unsigned)std::min<int64_t>((int64_t)tg_num_sms() * eper, need), kC4WalkWarps * 32,
                         0, s>>>(pd); tg_note_launch();
                TG_TRY_CUDA(cudaGetLastError());
            }
        }
        k_c4_pairs<<<(unsigned)pgrid, kC4Threads, psmem, s>>>(pd, list + q0, (int)(q1 - q0), ppriv); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    // the host vectors are read by the copies above before they go out of scope
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return TG_OK;
}

// Bits of the type in a bucket entry: an entry is the index of its count in a table
// of 2^tlg counts a row.
int bin_tlg(int L) { return L <= 2 ? 1 : L <= 4 ? 2 : L <= 8 ? 3 : 4; }

// Window bits of the binned waves: the largest window whose dense table (16-bit
// counts when half, else 32-bit) fits kBinTable bytes, with room for the type in
// a 16-bit entry.
int c4_bin_wlg(int L, int half) {
    const int G = bin_lanes(L), Lp = L + (L & 1);
    const size_t per = G ? (size_t)G * (half ? 2 : 4) : half ? (size_t)Lp * 2 : (size_t)L * 4;
    const int tbits = bin_tlg(L);
    int wlg = 5;
    while (wlg < 16 - tbits && ((size_t)1 << (wlg + 1)) * per <= kBinTable) ++wlg;
    return wlg;
}

// Global-mode binned waves of the anchors list[0 .. na) (degrees hdeg): walk
// positions per anchor (k_c4_prefix), warp units (k_c4_units), the far ends'
// numbers, then per wave (anchors of one counter width, at most `ecap` walk
// positions in all) the count pass, the bucket offsets, the fill pass and the
// bucket pairs.  list is sorted by (counter width, type), types in ltype.
int c4_bin_waves(const tg_graph *g, const uint32_t *list, int64_t na,
                 const std::vector<int64_t> &hdeg, const std::vector<uint8_t> &ltype, int64_t n4, unsigned long long *g4,
                 unsigned long long *work, int64_t ecap, cudaStream_t s) {
    const int L = g->L;
    const int64_t n = g->n_nonisolated;
    std::vector<int64_t> pb((size_t)na + 1, 0);
    for (int64_t q = 0; q < na; ++q) pb[q + 1] = pb[q] + hdeg[q];
    DevBuf<int64_t> dpb, dmp;
    DevBuf<unsigned long long> dtot;
    if (!dpb.alloc(na + 1, s) || !dmp.alloc(pb[na], s) || !dtot.alloc(na, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemcpyAsync(dpb.p, pb.data(), (na + 1) * 8, cudaMemcpyHostToDevice, s));
    k_c4_prefix<<<(unsigned)na, 256, 0, s>>>(list, dpb.p, g->rowptr, g->adj, dmp.p, dtot.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    // far-end numbers, types padded to the windows of the 16-bit waves (those of
    // the 32-bit ones divide them)
    const int64_t nblk = (n + kRankBlock - 1) / kRankBlock;
    DevBuf<uint32_t> tcnt, tbase, num, badj, thr;
    DevBuf<uint8_t> htype;
    if (!tcnt.alloc(L * nblk + 1, s) || !tbase.alloc(L + 1, s) || !num.alloc(n, s) ||
        !badj.alloc(2 * g->M, s) || !thr.alloc(na * L, s) || !htype.alloc(na, s))
        return TG_ENOMEM;
    k_bin_hist<<<(unsigned)nblk, kRankBlock, 0, s>>>(g->ntype, n, nblk, L, tcnt.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    TG_TRY(tg_scan_u32(tcnt.p, tcnt.p, L * nblk + 1, s));
    k_bin_bases<<<1, 32, 0, s>>>(tcnt.p, nblk, L, c4_bin_wlg(L, 1), tbase.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    k_bin_numbers<<<(unsigned)nblk, kRankBlock, 0, s>>>(g->ntype, n, nblk, L, tcnt.p, tbase.p, num.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    k_bin_entries<<<(unsigned)std::min<int64_t>((2 * g->M + 255) / 256, 65535LL * 16), 256, 0, s>>>(
        g->adj, 2 * g->M, num.p, badj.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    k_bin_thresholds<<<(unsigned)std::min<int64_t>((na + 7) / 8, 65535), 256, 0, s>>>(
        list, na, g->ntype, nblk, L, tcnt.p, tbase.p, thr.p, htype.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    C4Bin pb0{};
    TG_TRY_CUDA(cudaMemcpyAsync(pb0.tbase, tbase.p, (L + 1) * 4, cudaMemcpyDeviceToHost, s));
    std::vector<unsigned long long> tot_h((size_t)na);
    TG_TRY_CUDA(cudaMemcpyAsync(tot_h.data(), dtot.p, na * 8, cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    int wper = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&wper, k_c4_bin_walk<false>,
                                                              kC4WalkWarps * 32, 0));
    if (wper < 1) wper = 1;
    const int64_t walk_grid = (int64_t)tg_num_sms() * wper;
    const int64_t warps = walk_grid * kC4WalkWarps;
    // waves: consecutive anchors of one counter width, within ecap positions
    // and 2^22 buckets
    std::vector<int64_t> wq0, wq1;
    std::vector<int> whalf;
    int64_t wmax = 0;
    for (int64_t q = 0; q < na;) {
        const int half = hdeg[q] < 65536 ? 1 : 0;
        const int64_t W = (int64_t)pb0.tbase[L] >> c4_bin_wlg(L, half);
        int64_t e = q + 1;
        unsigned long long tot = tot_h[q];
        while (e < na && (hdeg[e] < 65536 ? 1 : 0) == half && tot + tot_h[e] <= (unsigned long long)ecap &&
               (e - q + 1) * W <= ((int64_t)1 << 22)) {
            tot += tot_h[e];
            ++e;
        }
        wq0.push_back(q);
        wq1.push_back(e);
        whalf.push_back(half);
        wmax = std::max<int64_t>(wmax, (e - q) * W);
        q = e;
    }
    const int64_t nwaves = (int64_t)wq0.size();
    std::vector<int64_t> us((size_t)na + 1, 0), tg((size_t)na, 1);
    unsigned long long wtmax = 0;
    for (int64_t w = 0; w < nwaves; ++w) {
        unsigned long long wt = 0;
        for (int64_t q = wq0[w]; q < wq1[w]; ++q) wt += tot_h[q];
        wtmax = std::max(wtmax, wt);
        const int64_t tgt =
            std::max<int64_t>(kWalkUnitMin, (int64_t)((wt + 4 * warps - 1) / (4 * warps)));
        for (int64_t q = wq0[w]; q < wq1[w]; ++q) {
            tg[q] = tgt;
            us[q + 1] = us[q] + (int64_t)((tot_h[q] + tgt - 1) / tgt);
        }
    }
    // runs of anchors of one type inside a wave
    std::vector<int2> runs;
    std::vector<int64_t> wr((size_t)nwaves + 1, 0);
    for (int64_t w = 0; w < nwaves; ++w) {
        for (int64_t q = wq0[w]; q < wq1[w];) {
            int64_t e = q + 1;
            while (e < wq1[w] && e - q < kBinRun && ltype[e] == ltype[q]) ++e;
            runs.push_back(make_int2((int)q, (int)e));
            q = e;
        }
        wr[w + 1] = (int64_t)runs.size();
    }
    const int64_t nunits = us[na];
    DevBuf<int2> druns;
    DevBuf<int64_t> dus, dtg;
    DevBuf<C4Unit> dun;
    DevBuf<unsigned long long> dq;
    DevBuf<uint32_t> cnt, offs;
    DevBuf<uint16_t> bins;
    if (!dus.alloc(na + 1, s) || !dtg.alloc(na, s) || !dun.alloc(nunits ? nunits : 1, s) ||
        !dq.alloc(3 * nwaves, s) || !cnt.alloc(wmax + 1, s) || !offs.alloc(wmax + 1, s) ||
        !bins.alloc(wtmax + 4, s) || !druns.alloc(runs.size(), s))
        return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemcpyAsync(druns.p, runs.data(), runs.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
    TG_TRY_CUDA(cudaMemcpyAsync(dus.p, us.data(), (na + 1) * 8, cudaMemcpyHostToDevice, s));
    TG_TRY_CUDA(cudaMemcpyAsync(dtg.p, tg.data(), na * 8, cudaMemcpyHostToDevice, s));
    TG_TRY_CUDA(cudaMemsetAsync(dq.p, 0, 3 * nwaves * 8, s));
    if (nunits > 0) {
        const unsigned ug = (unsigned)std::min<int64_t>((nunits + 255) / 256, 65535LL * 16);
        k_c4_units<<<ug, 256, 0, s>>>(dus.p, na, dtg.p, dtot.p, dmp.p, dpb.p, list, g->rowptr,
                                      dun.p); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    pb0.rowptr = g->rowptr;
    pb0.adj = g->adj;
    pb0.badj = badj.p;
    pb0.thr = thr.p;
    pb0.htype = htype.p;
    pb0.L = L;
    pb0.heavy = list;
    pb0.mprefix = dmp.p;
    pb0.pbase = dpb.p;
    pb0.cnt = cnt.p;
    pb0.bins = bins.p;
    pb0.offs = offs.p;
    pb0.g4 = g4;
    pb0.n4 = n4;
    pb0.work = work;
    for (int64_t w = 0; w < nwaves; ++w) {
        const int64_t q0 = wq0[w], q1 = wq1[w];
        C4Bin pw = pb0;
        pw.half = whalf[w];
        pw.wlg = c4_bin_wlg(L, pw.half);
        pw.tlg = bin_tlg(L);
        pw.W = (int64_t)pw.tbase[L] >> pw.wlg;
        pw.q0 = q0;
        const int64_t nb = (q1 - q0) * pw.W;
        pw.units = dun.p + us[q0];
        pw.n_units = us[q1] - us[q0];
        if (pw.n_units == 0) continue;
        const int64_t need = (pw.n_units + kC4WalkWarps - 1) / kC4WalkWarps;
        const int64_t grid = std::min<int64_t>(walk_grid, need);
        // bucket sizes, then offsets (one more entry, zero, takes the total)
        TG_TRY_CUDA(cudaMemsetAsync(cnt.p, 0, (nb + 1) * 4, s));
        pw.queue = dq.p + 3 * w;
        k_c4_bin_walk<false><<<(unsigned)grid, kC4WalkWarps * 32, 0, s>>>(pw); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
        TG_TRY(tg_scan_u32(cnt.p, offs.p, nb + 1, s));
        TG_TRY_CUDA(cudaMemcpyAsync(cnt.p, offs.p, nb * 4, cudaMemcpyDeviceToDevice, s));
        pw.queue = dq.p + 3 * w + 1;
        k_c4_bin_walk<true><<<(unsigned)grid, kC4WalkWarps * 32, 0, s>>>(pw); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
        pw.runs = druns.p + wr[w];
        pw.nitems = (wr[w + 1] - wr[w]) * pw.W;
        const int G = bin_lanes(L), Lp = L + (L & 1);
        const size_t nfar = (size_t)1 << pw.wlg, h4b = ((size_t)n4 * 8 + 15) & ~(size_t)15;
        void (*const fn)(C4Bin) = G == 2   ? (pw.half ? k_c4_bin_gram<2, true> : k_c4_bin_gram<2, false>)
                                  : G == 4 ? (pw.half ? k_c4_bin_gram<4, true> : k_c4_bin_gram<4, false>)
                                  : G == 8 ? (pw.half ? k_c4_bin_gram<8, true> : k_c4_bin_gram<8, false>)
                                           : k_c4_bin_pairs;
        const int threads = G ? kGramThreads : kBinPairThreads;
        const size_t psmem = h4b + (G ? nfar * G * (pw.half ? 2 : 4)
                                      : (pw.half ? nfar * (Lp >> 1) : nfar * L) * 4 + nfar / 32 * 4 + nfar * 2);
        TG_TRY(tg_allow_max_smem((const void *)fn));
        int pper = 0;
        TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pper, fn, threads, psmem));
        if (pper < 1) pper = 1;
        const int64_t pgrid = std::min<int64_t>((int64_t)tg_num_sms() * pper, pw.nitems);
        pw.queue = dq.p + 3 * w + 2;
        fn<<<(unsigned)pgrid, threads, psmem, s>>>(pw); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    // the host vectors are read by the copies above before they go out of scope
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return TG_OK;
}

}  // namespace

int tg_cyc_cycles(const tg_graph *g, unsigned long long *c4e, unsigned long long *g4,
                  unsigned long long *work, const tg_tune &t, const tg_part &part, cudaStream_t s) {
    if (g->M == 0) return TG_OK;
    const int L = g->L, L2 = L * L;
    const int64_t n = g->n;
    const bool global = g4 != nullptr;
    const int64_t n4 = tg_binom(L + 3, 4);
    const size_t avail = (size_t)tg_smem_optin() - 1024;
    // staged members per tile: their lists, ids and (a, u) accumulators
    const size_t per_member = 8 + 8 + 4 + 4 + (global ? 0 : (size_t)L2 * 8);
    const size_t fixed = 34 * 8 + 16 + 8 + (global ? (size_t)n4 * 8 : 0);
    if (fixed + 32 * per_member > avail) return TG_EINVAL;
    int TM = (int)std::min<size_t>(kC4Threads, (avail - fixed) / per_member);
    TM &= ~31;
    if (TM < 32) return TG_EINVAL;
    const size_t smem = (size_t)TM * per_member + fixed;
    TG_TRY(tg_allow_max_smem((const void *)k_c4));
    TG_TRY(tg_allow_max_smem((const void *)k_c4_split));
    TG_TRY(tg_allow_max_smem((const void *)k_c4_pairs));
    int per_sm = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_c4, kC4Threads, smem));
    if (per_sm < 1) per_sm = 1;
    const int64_t full_grid = (int64_t)tg_num_sms() * per_sm;

    // Anchors by walk cost: light ones count in shared memory (tg_c4_light.cu),
    // costlier ones are split over the grid (unroll 1 splits none, 4 every
    // anchor), the rest of them take one CTA and a counter slot each.
    C4Lists cls;
    TG_TRY(tg_c4_classify(g, t, part, global, cls, s));
    const int64_t nheavy = cls.size[kC4Split];
    std::vector<C4HeavyInfo> info((size_t)nheavy);
    TG_TRY(tg_c4_heavy(g, cls, info.data(), s));
    std::vector<uint32_t> heavy((size_t)nheavy);
    std::vector<int64_t> hdeg((size_t)nheavy);
    for (int64_t q = 0; q < nheavy; ++q) {
        heavy[q] = info[q].a;
        hdeg[q] = info[q].degree;
    }

    // counter slots: one per CTA of k_c4, one per split anchor of a wave; all
    // within a quarter of free memory
    const bool walk_waves = t.hash_slots >= 64;
    // Per-edge waves: kWaveMax costly anchors have about 2^20 walk positions or more; of
    // cheaper ones (unroll 4 alone splits them) a wave takes as many as have that many, a
    // wave being three launches.  With kWaveMax throughout, rows with unroll 4 took 63 ms
    // and not 23 on a cycle of 300,000 nodes, 11.7 and not 4.8 on ER 50K/400K.
    int64_t wave_max = kWaveMax;
    if (!global && nheavy > 0) {
        unsigned long long walk = 0;
        for (const C4HeavyInfo &x : info) walk += x.cost;
        const unsigned long long mean = std::max<unsigned long long>(1, walk / (unsigned long long)nheavy);
        wave_max = std::max(kWaveMax, std::min(full_grid, (int64_t)((1ull << 20) / mean)));
    }
    const int64_t slot_words = n * (L + 1) + (n + 31) / 32;
    const size_t slot_bytes = (size_t)slot_words * 4;
    int64_t want = 0;
    if (cls.size[kC4Slot] > 0) want = std::min<int64_t>(full_grid, cls.size[kC4Slot]);
    if (nheavy > 0)
        want = std::max<int64_t>(want, std::min<int64_t>(walk_waves ? wave_max : full_grid, nheavy));
    size_t free_b = 0, total_b = 0;
    TG_TRY_CUDA(cudaMemGetInfo(&free_b, &total_b));
    int64_t slots = std::min<int64_t>(want, (int64_t)(free_b / 4 / (slot_bytes ? slot_bytes : 1)));
    if (want > 0 && slots < 1) {
        if (slot_bytes > free_b / 2) return TG_ENOMEM;
        slots = 1;
    }
    DevBuf<uint32_t> scratch;
    if (slots > 0) {
        if (!scratch.alloc((size_t)slots * slot_words, s)) return TG_ENOMEM;
        TG_TRY_CUDA(cudaMemsetAsync(scratch.p, 0, (size_t)slots * slot_bytes, s));
    }
    C4Params p{};
    p.rowptr = g->rowptr;
    p.adj = g->adj;
    p.eid = g->eid;
    p.ntype = g->ntype;
    p.n = n;
    p.L = L;
    p.tile = TM;
    p.acc_l2 = global ? 0 : L2;
    p.scratch = scratch.p;
    p.slot_words = slot_words;
    p.c4e = c4e;
    p.g4 = g4;
    p.n4 = n4;
    p.work = work;
    p.half = 0;
    p.bits_off = n * (L + 1);

    if (nheavy > 0 && walk_waves) {
        // each split anchor's walk is cut into position ranges of about equal
        // length (warp units); in global mode anchors whose walk averages
        // bin_fill wedges per far-end window they span go to the binned waves;
        // the others to waves of `slots` anchors counting in global memory,
        // whose far ends k_c4_pairs takes
        const int64_t bin_fill = t.c4_bin_fill > 0 ? t.c4_bin_fill : kBinFill;
        size_t fb = 0, tb = 0;
        TG_TRY_CUDA(cudaMemGetInfo(&fb, &tb));
        // bucket entries of one wave: 2 bytes each, within an eighth of free memory
        const int64_t ecap = std::min<int64_t>((int64_t)1 << 31, (int64_t)(fb / 16));
        std::vector<uint32_t> lb, ls;
        // far-end numbers, types padded to whole windows, have to fit an entry's id
        const bool numbered = g->n_nonisolated + ((int64_t)L << c4_bin_wlg(L, 1)) <= (int64_t)TG_IDMASK;
        std::vector<int64_t> db, ds;
        std::vector<uint8_t> tyb;
        std::vector<C4HeavyInfo> ib;
        for (int64_t q = 0; q < nheavy; ++q) {
            const int half = hdeg[q] < 65536 ? 1 : 0;
            const int wlg = c4_bin_wlg(L, half);
            const int64_t span = ((g->n_nonisolated - 1) >> wlg) - ((int64_t)heavy[q] >> wlg) + 1;
            const bool bin = global && numbered && t.unroll != 1 && info[q].cost >= (unsigned long long)bin_fill * span &&
                             info[q].cost <= (unsigned long long)ecap;
            if (bin) {
                ib.push_back(info[q]);
                continue;
            }
            ls.push_back(heavy[q]);
            ds.push_back(hdeg[q]);
        }
        // binned anchors by counter width, then type
        std::stable_sort(ib.begin(), ib.end(), [](const C4HeavyInfo &x, const C4HeavyInfo &y) {
            const bool xw = x.degree < 65536, yw = y.degree < 65536;
            return xw != yw ? yw : x.type < y.type;
        });
        for (const C4HeavyInfo &x : ib) {
            lb.push_back(x.a);
            db.push_back(x.degree);
            tyb.push_back((uint8_t)x.type);
        }
        DevBuf<uint32_t> dlb, dls;
        if (!dlb.alloc(lb.size() + 1, s) || !dls.alloc(ls.size() + 1, s)) return TG_ENOMEM;
        if (!lb.empty()) {
            TG_TRY_CUDA(cudaMemcpyAsync(dlb.p, lb.data(), lb.size() * 4, cudaMemcpyHostToDevice, s));
            TG_TRY(c4_bin_waves(g, dlb.p, (int64_t)lb.size(), db, tyb, n4, g4, work, ecap, s));
        }
        if (!ls.empty()) {
            TG_TRY_CUDA(cudaMemcpyAsync(dls.p, ls.data(), ls.size() * 4, cudaMemcpyHostToDevice, s));
            TG_TRY(c4_walk_waves(p, g, dls.p, (int64_t)ls.size(), ds, slots, s));
        }
        TG_TRY_CUDA(cudaStreamSynchronize(s));
    } else if (nheavy > 0) {
        // member tiles of 'TM' members as units (both passes in per-edge mode)
        PairsConf pc;
        TG_TRY(c4_pairs_conf(n4, pc));
        const int64_t pgrid = pc.grid;
        const size_t psmem = pc.smem;
        const int ppriv = pc.priv;
        const int64_t wave = slots;
        std::vector<int4> units;
        std::vector<int64_t> wave_start;
        for (int64_t q0 = 0; q0 < nheavy; q0 += wave) {
            wave_start.push_back((int64_t)units.size());
            for (int64_t q = q0; q < std::min(nheavy, q0 + wave); ++q)
                for (int64_t tl = 0; tl < hdeg[q]; tl += TM)
                    units.push_back(make_int4((int)(q - q0), (int)heavy[q], (int)tl,
                                              (int)std::min<int64_t>(tl + TM, hdeg[q])));
        }
        wave_start.push_back((int64_t)units.size());
        DevBuf<int4> du;
        DevBuf<uint32_t> dl;
        if (!du.alloc(units.size(), s) || !dl.alloc(nheavy, s)) return TG_ENOMEM;
        TG_TRY_CUDA(cudaMemcpyAsync(dl.p, heavy.data(), nheavy * 4, cudaMemcpyHostToDevice, s));
        TG_TRY_CUDA(cudaMemcpyAsync(du.p, units.data(), units.size() * sizeof(int4),
                                    cudaMemcpyHostToDevice, s));
        DevBuf<unsigned long long> wq;
        if (!wq.alloc(2 * (wave_start.size() - 1), s)) return TG_ENOMEM;
        TG_TRY_CUDA(cudaMemsetAsync(wq.p, 0, 2 * (wave_start.size() - 1) * 8, s));
        C4Params ps = p;
        for (size_t w = 0; w + 1 < wave_start.size(); ++w) {
            const int64_t u0 = wave_start[w], nu = wave_start[w + 1] - u0;
            const int64_t a0 = (int64_t)w * wave, na = std::min<int64_t>(wave, nheavy - a0);
            ps.units = du.p + u0;
            ps.n_units = nu;
            const int64_t grid = std::min<int64_t>(full_grid, nu);
            for (int ph = 0; ph < (global ? 1 : 2); ++ph) {
                ps.phase = ph;
                ps.queue = wq.p + 2 * w + ph;
                k_c4_split<<<(unsigned)grid, kC4Threads, smem, s>>>(ps); tg_note_launch();
                TG_TRY_CUDA(cudaGetLastError());
            }
            k_c4_pairs<<<(unsigned)pgrid, kC4Threads, psmem, s>>>(ps, dl.p + a0, (int)na, ppriv); tg_note_launch();
            TG_TRY_CUDA(cudaGetLastError());
        }
        // the host vectors are read by the copies above before they go out of scope
        TG_TRY_CUDA(cudaStreamSynchronize(s));
    }
    TG_TRY(tg_c4_light(g, cls, c4e, g4, work, s));
    // the other anchors, one CTA and counter slot each
    if (cls.size[kC4Slot] > 0) {
        C4Params pl = p;
        pl.queue = cls.queue.p + kC4Classes + kC4Slot;
        pl.phase = 0;
        const int64_t grid = std::min<int64_t>(slots, cls.size[kC4Slot]);
        k_c4<<<(unsigned)grid, kC4Threads, smem, s>>>(pl, cls.list.p + (int64_t)kC4Slot * n,
                                                      cls.size[kC4Slot]); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    return TG_OK;
}

int tg_cyc_cliques(const tg_graph *g, unsigned long long *k4e, unsigned long long *g4,
                   unsigned long long *work, const tg_tune &t, const tg_part &part, cudaStream_t s) {
    if (g->M == 0) return TG_OK;
    const int L = g->L;
    const bool global = g4 != nullptr;
    const int64_t n4 = tg_binom(L + 3, 4);
    const size_t avail = (size_t)tg_smem_optin() - 1024;
    const int64_t n = g->n;
    const tg_lists *up = nullptr;
    TG_TRY(tg_graph_lists(g, &up, s));
    DevBuf<unsigned long long> queue;
    if (!queue.alloc(1, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(queue.p, 0, 8, s));
    // bitmap kernels (tg_k4.cu); up lists beyond them, or with a hash_slots cap
    // below 64 all of them, go to the hash-set kernels
    int64_t maxup = 0, bits_max = 0;
    if (t.hash_slots >= 64) {
        int64_t nlong = 0;
        TG_TRY(tg_k4_bits(g, *up, k4e, g4, work, part, &nlong, &maxup, &bits_max, s));
        if (nlong == 0) return TG_OK;
    } else if (global) {
        DevBuf<unsigned long long> mx;
        if (!mx.alloc(1, s)) return TG_ENOMEM;
        TG_TRY_CUDA(cudaMemsetAsync(mx.p, 0, 8, s));
        k_max_up<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, s>>>(up->uoff, n, mx.p); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
        TG_TRY_CUDA(cudaMemcpyAsync(&maxup, mx.p, 8, cudaMemcpyDeviceToHost, s));
        TG_TRY_CUDA(cudaStreamSynchronize(s));
    }
    if (global) {
        const size_t h4b = ((size_t)n4 * 8 + 15) & ~(size_t)15;
        K4GParams q{};
        q.uoff = up->uoff;
        q.uadj = up->uadj;
        q.utoff = up->utoff;
        q.ntype = g->ntype;
        q.n = n;
        q.m = g->M;
        q.L = L;
        q.queue = queue.p;
        q.g4 = g4;
        q.n4 = n4;
        q.work = work;
        q.pidx = part.index;
        q.pcnt = part.count;
        // hash sets sized to the largest up list, within the hash_slots cap
        int gcap = (int)std::min<int64_t>(std::min(1024, t.hash_slots), (maxup + 31) & ~(int64_t)31);
        if (gcap < 32) gcap = 32;
        int hlg = 5;
        while ((1 << hlg) < 2 * gcap) ++hlg;
        size_t gsmem = h4b + (size_t)kK4GWarps * (gcap + 2 * (1 << hlg)) * 4;
        while (gsmem > avail && gcap > 32) {
            gcap -= 32;
            hlg = 5;
            while ((1 << hlg) < 2 * gcap) ++hlg;
            gsmem = h4b + (size_t)kK4GWarps * (gcap + 2 * (1 << hlg)) * 4;
        }
        TG_TRY(tg_allow_max_smem((const void *)k_k4_global));
        int gper = 0;
        TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&gper, k_k4_global,
                                                                  kK4GWarps * 32, gsmem));
        if (gper < 1) gper = 1;
        int64_t ggrid = (int64_t)tg_num_sms() * gper;
        const int64_t gneed = (g->M / kK4GChunk + kK4GWarps) / kK4GWarps;
        if (ggrid > gneed) ggrid = gneed;
        if (ggrid < 1) ggrid = 1;
        q.cap = gcap;
        q.hlg = hlg;
        q.min_d0 = (int32_t)bits_max;
        k_k4_global<<<(unsigned)ggrid, kK4GWarps * 32, gsmem, s>>>(q); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
        return TG_OK;
    }
    const size_t per_entry = (size_t)(3 + L) * 4;
    // W entries staged per warp; hash_slots caps it (a small cap sends large W
    // sets down the path that tests membership in the global lists instead)
    int cap = (int)std::min<size_t>(std::min(512, t.hash_slots), avail / kK4Warps / per_entry);
    cap &= ~31;
    if (cap < 32) return TG_EINVAL;
    const size_t smem = (size_t)kK4Warps * cap * per_entry;
    TG_TRY(tg_allow_max_smem((const void *)k_k4));
    int per_sm = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_k4, kK4Warps * 32, smem));
    if (per_sm < 1) per_sm = 1;
    int64_t grid = (int64_t)tg_num_sms() * per_sm;
    const int64_t need = (g->n + kK4Warps - 1) / kK4Warps;
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    K4Params p{};
    p.uoff = up->uoff;
    p.uadj = up->uadj;
    p.ueid = up->ueid;
    p.utoff = up->utoff;
    p.ntype = g->ntype;
    p.n = g->n;
    p.L = L;
    p.P = L * (L + 1) / 2;
    p.cap = cap;
    p.queue = queue.p;
    p.k4e = k4e;
    p.work = work;
    p.min_d0 = bits_max;
    k_k4<<<(unsigned)grid, kK4Warps * 32, smem, s>>>(p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    return TG_OK;
}

// ---------------------------------------------- global shortcut ----
int tg_cyc_correct(unsigned long long *hist, int L, const unsigned long long *c4w,
                   const unsigned long long *k4, cudaStream_t s) {
    const int64_t n4 = tg_binom(L + 3, 4);
    const int64_t off4 = tg_binom(L + 1, 2) + 2 * tg_binom(L + 2, 3);
    k_cyc_correct<<<(unsigned)((n4 + 255) / 256), 256, 0, s>>>(hist, off4, n4, c4w, k4); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    return TG_OK;
}
