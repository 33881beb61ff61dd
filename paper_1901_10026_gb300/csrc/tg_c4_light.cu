// Light anchors of the 4-cycle enumeration (see tg_cycles.cu): anchors whose
// walk fits a table of far ends in shared memory, for global totals and for
// per-edge counters.
//
// A table slot holds a far end's id and its middle counts by type; the slots
// that were claimed go on a list, so the far ends are taken, and their slots
// cleared, without a scan of the table.  Up to 511 walk positions the table is
// one warp's and its counts are bytes (every member has a list of at least
// two, so no count exceeds half the cost); up to 2047 and 8191 it is a CTA's
// with 16-bit counts.  Per-edge mode walks a second time and adds, for every
// wedge whose far end has another middle, the cycles it closes to its two
// edges; most wedges of a sparse graph have none and cost two shared-memory
// reads.
//
// Measured (4-cycle phase, before -> now): ER 100K/1M (L = 5, 1.2e7 wedges) 2.48
// -> 0.67 ms, ER-1000 0.67 -> 0.07 ms; before, an 8192-slot table of 114 KB
// left one 256-thread CTA per SM, the whole table was scanned and cleared per
// anchor, and a warp claimed 32 anchors at a time.  The classes and their lists
// take one kernel (two with hubs) instead of twelve launches.  What bounds it
// now is the latency of the walk's gathers (list heads, then entries) and the
// shared-memory atomics.
#include <algorithm>

#include "tg_cycles.cuh"
#include "tg_device.cuh"

using namespace tgd;

namespace {

// ---------------------------------------------------------------- classes --
constexpr int kCostThreads = 256;
constexpr int kCostLane = 32;   // degree up to which one lane sums a node's list
constexpr int kCostHub = 256;   // degree from which a list is cut into chunks
constexpr int kCostChunk = 1024;

// Nodes of degree above kCostHub come first (ids are degree-ordered), so their
// lists are a prefix of adj: warps take chunks of it and add each owner's part.
// One warp per list took 37 ms on CL-1M's 230K-entry hubs.
__global__ void __launch_bounds__(kCostThreads) k_c4_hub_cost(const int64_t *rowptr,
                                                              const uint32_t *adj, int64_t n,
                                                              unsigned long long *cost) {
    const int lane = threadIdx.x & 31;
    int64_t lo = 0, hi = n;  // first node of degree <= kCostHub
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (__ldg(rowptr + mid + 1) - __ldg(rowptr + mid) > kCostHub)
            lo = mid + 1;
        else
            hi = mid;
    }
    const int64_t nh = lo, total = __ldg(rowptr + nh);
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c * kCostChunk < total;
         c += nw) {
        int64_t x0 = c * kCostChunk;
        const int64_t x1 = min(total, x0 + kCostChunk);
        int64_t a = 0, top = nh - 1;  // last node with rowptr[a] <= x0
        while (a < top) {
            const int64_t mid = (a + top + 1) >> 1;
            if (__ldg(rowptr + mid) <= x0)
                a = mid;
            else
                top = mid - 1;
        }
        for (; x0 < x1; ++a) {
            const int64_t e = min(x1, __ldg(rowptr + a + 1));
            unsigned long long v = 0;
#pragma unroll 4
            for (int64_t x = x0 + lane; x < e; x += 32) {
                const uint32_t u = __ldg(adj + x) & TG_IDMASK;
                if ((int64_t)u > a) v += (unsigned long long)(__ldg(rowptr + u + 1) - __ldg(rowptr + u));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
            if (lane == 0 && v) atomicAdd(cost + a, v);
            x0 = e;
        }
    }
}

// A warp takes 32 consecutive nodes: a lane sums the list of its node when it
// is short, the warp together the longer ones, one after the other (hubs have
// their cost from k_c4_hub_cost).  One add per class and warp claims the list
// positions.
__global__ void __launch_bounds__(kCostThreads) k_c4_classify(
    const int64_t *rowptr, const uint32_t *adj, int64_t n, unsigned long long lite,
    unsigned long long mid, unsigned long long large, unsigned long long thr, int pidx, int pcnt,
    unsigned long long *cost, uint32_t *list, unsigned long long *size) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c * 32 < n; c += nw) {
        const int64_t a = c * 32 + lane;
        int64_t b = 0;
        int d = 0;
        if (a < n && a % pcnt == pidx) {
            b = rowptr[a];
            d = (int)(rowptr[a + 1] - b);
        }
        unsigned long long v = 0;
        if (d >= 2 && d <= kCostLane)
            for (int x = 0; x < d; ++x) {
                const uint32_t u = __ldg(adj + b + x) & TG_IDMASK;
                if ((int64_t)u > a) v += (unsigned long long)(__ldg(rowptr + u + 1) - __ldg(rowptr + u));
            }
        if (d > kCostHub) v = cost[a];
        for (unsigned m = __ballot_sync(kFull, d > kCostLane && d <= kCostHub); m; m &= m - 1u) {
            const int src = __ffs(m) - 1;
            const int64_t as = c * 32 + src, bs = __shfl_sync(kFull, b, src);
            const int ds = __shfl_sync(kFull, d, src);
            unsigned long long w = 0;
#pragma unroll 4
            for (int x = lane; x < ds; x += 32) {
                const uint32_t u = __ldg(adj + bs + x) & TG_IDMASK;
                if ((int64_t)u > as) w += (unsigned long long)(__ldg(rowptr + u + 1) - __ldg(rowptr + u));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(kFull, w, o);
            if (lane == src) v = w;
        }
        if (a < n && d <= kCostHub) cost[a] = v;
        int cls = -1;
        if (v > thr)
            cls = kC4Split;
        else if (v > 0)
            cls = v <= lite ? kC4Warp : v <= mid ? kC4Cta : v <= large ? kC4CtaLarge : kC4Slot;
#pragma unroll
        for (int k = 0; k < kC4Classes; ++k) {
            const unsigned m = __ballot_sync(kFull, cls == k);
            if (!m) continue;
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(size + k, (unsigned long long)__popc(m));
            base = __shfl_sync(kFull, base, 0);
            if (cls == k) list[(int64_t)k * n + (int64_t)base + __popc(m & ((1u << lane) - 1u))] = (uint32_t)a;
        }
    }
}

// Up to so many split anchors are sorted on the host, more on the device.  1,024 take 33
// us there and the two launches and the sort 20 here; but the 300,000 of a cycle
// (unroll 4) took 6 ms there, while a hub's few hundred, sorted here, made counts of
// power laws 20 us longer (4.46 ms) and seven unions of a batch 180 (12.6 ms).
constexpr int64_t kHostSort = 1024;

__global__ void k_c4_heavy_keys(const uint32_t *list, int64_t count, uint64_t *keys) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < count;
         q += (int64_t)gridDim.x * blockDim.x)
        keys[q] = list[q];
}

template <class Id>
__global__ void k_c4_heavy_info(const Id *list, int64_t count, const int64_t *rowptr,
                                const uint8_t *ntype, const unsigned long long *cost,
                                C4HeavyInfo *out) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < count;
         q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = (uint32_t)list[q];
        out[q] = C4HeavyInfo{cost[a], rowptr[a + 1] - rowptr[a], a, ntype[a]};
    }
}

// ----------------------------------------------------------- light anchors --
struct LightParams {
    const int64_t *rowptr;
    const uint32_t *adj;
    const uint32_t *eid;
    const uint8_t *ntype;
    const uint32_t *list;
    int64_t count;
    const unsigned long long *cost;
    int32_t L, lg_max, grab;
    unsigned long long *queue;
    unsigned long long *c4e;  // per-edge mode: M x L x L
    unsigned long long *g4;   // global mode: C(L+3,4)
    int64_t n4;
    unsigned long long *work;  // [4]: wedges
};

// One warp's share (chunks of 32 members m0, m0 + stride, ...) of the walk of
// anchor a: op(ok, entry b of u's list, its position, member x of Gamma_a,
// entry u), called by all lanes, ok where b ranks below a; kWalkBatch batches
// of 32 positions in flight.
constexpr int kWalkBatch = 4;

template <class Op>
__device__ __forceinline__ void light_walk(const LightParams &p, uint32_t a, int64_t ba, int da,
                                           int m0, int stride, int step, Op op) {
    const int lane = threadIdx.x & 31;
    for (int m = m0; m < da; m += stride) {
        const int x = m + lane;
        uint32_t wu = 0;
        int64_t bu = 0;
        int len = 0;
        if (lane < step && x < da) {
            wu = __ldg(p.adj + ba + x);
            const uint32_t u = wu & TG_IDMASK;
            if (u > a) {
                bu = __ldg(p.rowptr + u);
                const int du = (int)(__ldg(p.rowptr + u + 1) - bu);
                if (du > 1) len = du;
            }
        }
        int incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        const int total = __shfl_sync(kFull, incl, 31);
        const int64_t org = bu - (incl - len);
        for (int b0 = 0; b0 < total; b0 += 32 * kWalkBatch) {
            uint32_t wb[kWalkBatch], wr[kWalkBatch];
            int64_t at[kWalkBatch];
            int rr[kWalkBatch];
#pragma unroll
            for (int q = 0; q < kWalkBatch; ++q) {
                const int pos = b0 + 32 * q + lane;
                int r = 0;  // the first member whose running sum exceeds pos
#pragma unroll
                for (int st = 16; st > 0; st >>= 1) {
                    const int v = __shfl_sync(kFull, incl, r + st - 1);
                    if (v <= pos) r += st;
                }
                rr[q] = r;
                at[q] = __shfl_sync(kFull, org, r) + pos;
                wr[q] = __shfl_sync(kFull, wu, r);
                wb[q] = pos < total ? __ldg(p.adj + at[q]) : 0u;
            }
#pragma unroll
            for (int q = 0; q < kWalkBatch; ++q)
                op(b0 + 32 * q + lane < total && (wb[q] & TG_IDMASK) > a, wb[q], at[q], m + rr[q], wr[q]);
        }
    }
}

// The table: keys (id + 1, 0 empty), counts by type (kBits each, packed into
// the slot's kW words), the list of claimed slots.
template <int kBits>
struct FarTable {
    uint32_t *keys, *cnt;
    uint16_t *claimed;
    int words;  // count words of a slot

    static __host__ __device__ int slot_words(int L) { return (L * kBits + 31) / 32; }
    static __host__ __device__ size_t bytes(int L, int lg) {
        return ((size_t)1 << lg) * (4 + 4 * slot_words(L) + 2);
    }
    __device__ void place(unsigned char *base, int L, int lg) {
        words = slot_words(L);
        keys = reinterpret_cast<uint32_t *>(base);
        cnt = keys + (1 << lg);
        claimed = reinterpret_cast<uint16_t *>(cnt + ((size_t)words << lg));
    }
    // slot of id, claimed when absent (isnew); at most 2^lg - 1 ids are put in
    __device__ int claim(int lg, uint32_t id, bool &isnew) const {
        const uint32_t mask = (1u << lg) - 1u;
        uint32_t h = hset_slot(id, lg);
        isnew = false;
        const volatile uint32_t *k = keys;  // slots claimed by other lanes while this one probes
        for (int probe = 0; probe < (1 << lg); ++probe) {
            uint32_t old = k[h];  // most wedges meet a far end already there: no exchange
            if (old == 0u) {
                old = atomicCAS(keys + h, 0u, id + 1u);
                isnew = old == 0u;
                if (isnew) return (int)h;
            }
            if (old == id + 1u) return (int)h;
            h = (h + 1u) & mask;
        }
        return 0;  // not reached: the table is never full
    }
    __device__ int find(int lg, uint32_t id) const {
        const uint32_t mask = (1u << lg) - 1u;
        uint32_t h = hset_slot(id, lg);
        for (int probe = 0; probe < (1 << lg); ++probe) {
            const uint32_t k = keys[h];
            if (k == id + 1u) return (int)h;
            if (k == 0u) return -1;
            h = (h + 1u) & mask;
        }
        return -1;
    }
    __device__ void add(int slot, int t) const {
        const int bit = t * kBits;
        atomicAdd(cnt + slot * words + (bit >> 5), 1u << (bit & 31));
    }
    __device__ uint32_t get(int slot, int t) const {
        const int bit = t * kBits;
        return (cnt[slot * words + (bit >> 5)] >> (bit & 31)) & ((1u << kBits) - 1u);
    }
    __device__ uint32_t sum(int slot) const {
        uint32_t s = 0;
        for (int w = 0; w < words; ++w) {
            const uint32_t v = cnt[slot * words + w];
            s += kBits == 8 ? __dp4a(v, 0x01010101u, 0u) : (v & 0xffffu) + (v >> 16);
        }
        return s;
    }
    __device__ void clear(int slot) const {
        keys[slot] = 0u;
        for (int w = 0; w < words; ++w) cnt[slot * words + w] = 0u;
    }
};

// Far end in `slot` of an anchor of type ta: C(c_t, 2) and c_t c_t' per pair of
// middle types, into the histogram h4.
template <class Table>
__device__ __forceinline__ void far_end(const LightParams &p, const Table &tab, int slot, int ta,
                                        unsigned long long *h4) {
    if (tab.sum(slot) < 2u) return;  // one middle closes no cycle
    int s0 = ta, s1 = p.ntype[tab.keys[slot] - 1u];
    sort2(s0, s1);
    for (int t = 0; t < p.L; ++t) {
        const unsigned long long ct = tab.get(slot, t);
        if (!ct) continue;
        for (int u = t; u < p.L; ++u) {
            const unsigned long long cu = tab.get(slot, u);
            const unsigned long long v = u == t ? ct * (ct - 1) / 2 : ct * cu;
            if (!v) continue;
            int q0 = s0, q1 = s1, q2 = t, q3 = u;
            sort2(q0, q2);
            sort2(q1, q3);
            sort2(q1, q2);
            atomicAdd(h4 + colex4(q0, q1, q2, q3), v);
        }
    }
}

// Per-edge mode: the cycles that the wedge a-u-b (entry wb at list position
// `at`, member x of Gamma_a) closes with the other middles of b.
template <class Table>
__device__ __forceinline__ void wedge_edges(const LightParams &p, const Table &tab, int lg, int ta,
                                            int64_t ba, uint32_t wb, int64_t at, int x, uint32_t wu) {
    const int slot = tab.find(lg, wb & TG_IDMASK);
    if (slot < 0 || tab.sum(slot) < 2u) return;
    const int L = p.L, L2 = L * L;
    const int tu = (int)(wu >> TG_TSHIFT), tb = (int)(wb >> TG_TSHIFT);
    // rows are keyed from the larger-id end: (u, b) sees a and u', (a, u) sees b and u'
    const bool ub = (wu & TG_IDMASK) > (wb & TG_IDMASK);
    unsigned long long *row_ub = p.c4e + (int64_t)__ldg(p.eid + at) * L2 + (ub ? ta * L : ta);
    unsigned long long *row_au = p.c4e + (int64_t)__ldg(p.eid + ba + x) * L2 + tb * L;
    const int step = ub ? 1 : L;
    for (int t = 0; t < L; ++t) {
        const uint32_t v = tab.get(slot, t) - (t == tu ? 1u : 0u);
        if (!v) continue;
        atomicAdd(row_ub + t * step, (unsigned long long)v);
        atomicAdd(row_au + t, (unsigned long long)v);
    }
}

constexpr int kLightWarps = 8;

template <bool kEdge>
__global__ void __launch_bounds__(kLightWarps * 32) k_c4_warp(LightParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = p.L, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long *h4 = reinterpret_cast<unsigned long long *>(smem);
    if (!kEdge)
        for (int64_t q = threadIdx.x; q < p.n4; q += blockDim.x) h4[q] = 0ull;
    FarTable<8> tab;
    const size_t tbytes = (FarTable<8>::bytes(L, p.lg_max) + 15) & ~(size_t)15;
    tab.place(smem + (kEdge ? 0 : ((size_t)p.n4 * 8 + 15) & ~(size_t)15) + warp * tbytes, L, p.lg_max);
    for (int q = lane; q < (1 + tab.words) << p.lg_max; q += 32) tab.keys[q] = 0u;
    __syncthreads();
    unsigned long long wk = 0;
    for (;;) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(p.queue, (unsigned long long)p.grab);
        base = __shfl_sync(kFull, base, 0);
        if (base >= (unsigned long long)p.count) break;
        const int64_t stop = min((int64_t)base + p.grab, p.count);
        for (int64_t i = (int64_t)base; i < stop; ++i) {
            const uint32_t a = p.list[i];
            const int64_t ba = p.rowptr[a];
            const int da = (int)(p.rowptr[a + 1] - ba);
            const int ta = p.ntype[a];
            const unsigned long long ca = p.cost[a];
            int lg = 5;
            while ((1ull << lg) <= ca) ++lg;  // at most lg_max: cost < 2^lg_max
            int nl = 0;  // claimed slots
            light_walk(p, a, ba, da, 0, 32, 32, [&](bool ok, uint32_t wb, int64_t, int, uint32_t wu) {
                bool isnew = false;
                int h = 0;
                if (ok) {
                    h = tab.claim(lg, wb & TG_IDMASK, isnew);
                    tab.add(h, (int)(wu >> TG_TSHIFT));
                    ++wk;
                }
                const unsigned nm = __ballot_sync(kFull, isnew);
                if (isnew) tab.claimed[nl + __popc(nm & ((1u << lane) - 1u))] = (uint16_t)h;
                nl += __popc(nm);
            });
            __syncwarp();
            if (kEdge) {
                light_walk(p, a, ba, da, 0, 32, 32, [&](bool ok, uint32_t wb, int64_t at, int x, uint32_t wu) {
                    if (ok) wedge_edges(p, tab, lg, ta, ba, wb, at, x, wu);
                });
                __syncwarp();
            }
            for (int q = lane; q < nl; q += 32) {
                const int slot = tab.claimed[q];
                if (!kEdge) far_end(p, tab, slot, ta, h4);
                tab.clear(slot);
            }
            __syncwarp();
        }
    }
    if (!kEdge) {
        __syncthreads();
        for (int64_t q = threadIdx.x; q < p.n4; q += blockDim.x)
            if (h4[q]) atomicAdd(p.g4 + q, h4[q]);
    }
    if (p.work) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wk += __shfl_xor_sync(kFull, wk, o);
        if (lane == 0 && wk) atomicAdd(p.work + 4, wk);
    }
}

template <bool kEdge>
__global__ void __launch_bounds__(1024) k_c4_cta(LightParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long s_item;
    __shared__ int s_nl;
    const int L = p.L, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long *h4 = reinterpret_cast<unsigned long long *>(smem);
    if (!kEdge)
        for (int64_t q = tid; q < p.n4; q += blockDim.x) h4[q] = 0ull;
    FarTable<16> tab;
    tab.place(smem + (kEdge ? 0 : ((size_t)p.n4 * 8 + 15) & ~(size_t)15), L, p.lg_max);
    for (int q = tid; q < (1 + tab.words) << p.lg_max; q += blockDim.x) tab.keys[q] = 0u;
    unsigned long long wk = 0;
    const int nwarps = blockDim.x >> 5;
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_item = atomicAdd(p.queue, 1ull);
            s_nl = 0;
        }
        __syncthreads();
        const unsigned long long item = s_item;
        if (item >= (unsigned long long)p.count) break;
        const uint32_t a = p.list[item];
        const int64_t ba = p.rowptr[a];
        const int da = (int)(p.rowptr[a + 1] - ba);
        const int ta = p.ntype[a];
        const unsigned long long ca = p.cost[a];
        const int step = max(4, min(32, (da + nwarps - 1) / nwarps));  // members a warp takes at once
        int lg = 5;
        while ((1ull << lg) <= ca) ++lg;
        light_walk(p, a, ba, da, step * warp, step * nwarps, step, [&](bool ok, uint32_t wb, int64_t, int, uint32_t wu) {
            bool isnew = false;
            int h = 0;
            if (ok) {
                h = tab.claim(lg, wb & TG_IDMASK, isnew);
                tab.add(h, (int)(wu >> TG_TSHIFT));
                ++wk;
            }
            const unsigned nm = __ballot_sync(kFull, isnew);
            if (!nm) return;
            int base = 0;
            if (lane == 0) base = atomicAdd(&s_nl, __popc(nm));
            base = __shfl_sync(kFull, base, 0);
            if (isnew) tab.claimed[base + __popc(nm & ((1u << lane) - 1u))] = (uint16_t)h;
        });
        __syncthreads();
        if (kEdge) {
            light_walk(p, a, ba, da, step * warp, step * nwarps, step,
                       [&](bool ok, uint32_t wb, int64_t at, int x, uint32_t wu) {
                           if (ok) wedge_edges(p, tab, lg, ta, ba, wb, at, x, wu);
                       });
            __syncthreads();
        }
        const int nl = s_nl;
        for (int q = tid; q < nl; q += blockDim.x) {
            const int slot = tab.claimed[q];
            if (!kEdge) far_end(p, tab, slot, ta, h4);
            tab.clear(slot);
        }
    }
    if (!kEdge) {
        __syncthreads();
        for (int64_t q = tid; q < p.n4; q += blockDim.x)
            if (h4[q]) atomicAdd(p.g4 + q, h4[q]);
    }
    if (p.work) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wk += __shfl_xor_sync(kFull, wk, o);
        if (lane == 0 && wk) atomicAdd(p.work + 4, wk);
    }
}

// Threads of a CTA class, and the shared memory of a light class's launch.
constexpr int kCtaThreads[2] = {256, 1024};
constexpr int kLgMax[3] = {9, 11, 13};

size_t light_smem(int cls, int L, int64_t n4, bool global, int lg) {
    const size_t hist = global ? ((size_t)n4 * 8 + 15) & ~(size_t)15 : 0;
    if (cls == kC4Warp) return hist + kLightWarps * ((FarTable<8>::bytes(L, lg) + 15) & ~(size_t)15);
    return hist + FarTable<16>::bytes(L, lg);
}

template <bool kEdge>
int launch_light(const tg_graph *g, const C4Lists &cls, LightParams p, cudaStream_t s) {
    for (int k = kC4Warp; k <= kC4CtaLarge; ++k) {
        if (cls.size[k] == 0) continue;
        const void *fn = k == kC4Warp ? (const void *)k_c4_warp<kEdge> : (const void *)k_c4_cta<kEdge>;
        const int threads = k == kC4Warp ? kLightWarps * 32 : kCtaThreads[k - kC4Cta];
        const size_t smem = light_smem(k, g->L, p.n4, !kEdge, cls.lg[k]);
        TG_TRY(tg_allow_max_smem(fn));
        int per = 0;
        TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem));
        if (per < 1) return TG_EINVAL;
        int64_t grid = (int64_t)tg_num_sms() * per;
        p.list = cls.list.p + (int64_t)k * cls.n;
        p.count = cls.size[k];
        p.lg_max = cls.lg[k];
        p.queue = cls.queue.p + kC4Classes + k;
        if (k == kC4Warp) {
            grid = std::min<int64_t>(grid, (p.count + kLightWarps - 1) / kLightWarps);
            // anchors per queue access: about eight accesses a warp
            p.grab = (int)std::max<int64_t>(1, std::min<int64_t>(8, p.count / (grid * kLightWarps * 8)));
            k_c4_warp<kEdge><<<(unsigned)grid, threads, smem, s>>>(p);
        } else {
            grid = std::min<int64_t>(grid, p.count);
            k_c4_cta<kEdge><<<(unsigned)grid, threads, smem, s>>>(p);
        }
        tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    return TG_OK;
}

}  // namespace

int tg_c4_classify(const tg_graph *g, const tg_tune &t, const tg_part &part, bool global,
                   C4Lists &out, cudaStream_t s) {
    const int64_t n = g->n, n4 = tg_binom(g->L + 3, 4);
    out.n = n;
    if (!out.cost.alloc(n, s) || !out.list.alloc((size_t)kC4Classes * n, s) ||
        !out.queue.alloc(2 * kC4Classes, s))
        return TG_ENOMEM;
    const size_t avail = (size_t)tg_smem_optin() - 1024;
    for (int k = kC4Warp; k <= kC4CtaLarge; ++k) {
        int lg = kLgMax[k];
        while (lg > 5 && (light_smem(k, g->L, n4, global, lg) > avail ||
                          (k == kC4Warp && (1 << lg) > t.hash_slots)))
            --lg;
        out.lg[k] = lg;
    }
    const unsigned long long lite = (1ull << out.lg[0]) - 1, mid = (1ull << out.lg[1]) - 1,
                             large = (1ull << out.lg[2]) - 1;
    const unsigned long long thr = t.unroll == 1 ? ~0ull : t.unroll == 4 ? 0ull : large;
    TG_TRY_CUDA(cudaMemsetAsync(out.queue.p, 0, 2 * kC4Classes * 8, s));
    if (g->max_degree > kCostHub) {
        TG_TRY_CUDA(cudaMemsetAsync(out.cost.p, 0, n * 8, s));
        k_c4_hub_cost<<<tg_num_sms() * 8, kCostThreads, 0, s>>>(g->rowptr, g->adj, n, out.cost.p);
        tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    const int64_t grid = std::min<int64_t>((n + kCostThreads - 1) / kCostThreads, (int64_t)tg_num_sms() * 8);
    k_c4_classify<<<(unsigned)grid, kCostThreads, 0, s>>>(g->rowptr, g->adj, n, lite, mid, large, thr,
                                                          part.index, part.count, out.cost.p,
                                                          out.list.p, out.queue.p);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    unsigned long long size[kC4Classes];
    TG_TRY_CUDA(cudaMemcpyAsync(size, out.queue.p, sizeof(size), cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    for (int k = 0; k < kC4Classes; ++k) out.size[k] = (int64_t)size[k];
    return TG_OK;
}

int tg_c4_heavy(const tg_graph *g, const C4Lists &cls, C4HeavyInfo *host, cudaStream_t s) {
    const int64_t count = cls.size[kC4Split];
    if (count == 0) return TG_OK;
    const uint32_t *list = cls.list.p + (int64_t)kC4Split * cls.n;
    const unsigned grid = (unsigned)std::min<int64_t>((count + 255) / 256, 4096);
    DevBuf<C4HeavyInfo> info;
    DevBuf<uint64_t> k1, k2;
    if (!info.alloc(count, s)) return TG_ENOMEM;
    if (count <= kHostSort) {
        k_c4_heavy_info<<<grid, 256, 0, s>>>(list, count, g->rowptr, g->ntype, cls.cost.p, info.p); tg_note_launch();
    } else {
        if (!k1.alloc(count, s) || !k2.alloc(count, s)) return TG_ENOMEM;
        k_c4_heavy_keys<<<grid, 256, 0, s>>>(list, count, k1.p); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
        uint64_t *sorted = nullptr;
        TG_TRY(tg_radix_sort_u64(k1.p, k2.p, count, tg_bitlen((uint64_t)(g->n - 1)), s, &sorted));
        k_c4_heavy_info<<<grid, 256, 0, s>>>(sorted, count, g->rowptr, g->ntype, cls.cost.p, info.p); tg_note_launch();
    }
    TG_TRY_CUDA(cudaGetLastError());
    TG_TRY_CUDA(cudaMemcpyAsync(host, info.p, count * sizeof(C4HeavyInfo), cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    if (count <= kHostSort)
        std::sort(host, host + count, [](const C4HeavyInfo &x, const C4HeavyInfo &y) { return x.a < y.a; });
    return TG_OK;
}

int tg_c4_light(const tg_graph *g, const C4Lists &cls, unsigned long long *c4e,
                unsigned long long *g4, unsigned long long *work, cudaStream_t s) {
    LightParams p{};
    p.rowptr = g->rowptr;
    p.adj = g->adj;
    p.eid = g->eid;
    p.ntype = g->ntype;
    p.cost = cls.cost.p;
    p.L = g->L;
    p.c4e = c4e;
    p.g4 = g4;
    p.n4 = tg_binom(g->L + 3, 4);
    p.work = work;
    return g4 ? launch_light<false>(g, cls, p, s) : launch_light<true>(g, cls, p, s);
}
