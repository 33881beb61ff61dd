// 4-cliques from bitmaps of the up lists, for type-multiset totals and for
// per-edge counters.
//
// Each 4-clique x0 < v < w < x (by rank) is met from its lowest node x0 as a
// triangle of the graph G0 that the nodes of up(x0) (its higher-ranked
// neighbours) form among themselves.  Row v of G0 is a bitmap over the positions
// of up(x0).  Positions are laid out type by type, each type padded to whole
// words when more than one word is needed, so that a word has one type and
// popc(row_v & row_w) counts the x of that type.
//   global mode: rows hold the higher-ranked neighbours; every pair (v, w in
//     row_v) adds its popcounts to the histogram under {t0, tv, tw, type}.
//   per-edge mode: rows hold all neighbours, so T_vw[t] = popc over type t is
//     the number of cliques {x0, v, w, x} with x of type t.  Edge (v, w) gets
//     T_vw[t] under {t0, t}; edge (x0, v) gets sum over w of type a of
//     T_vw[b] under {a, b} (halved for a = b, where both orders are met).
//     No clique is visited by itself: an edge of G0 costs L adds.
//
// Building the rows dominates: the up lists of up(x0)'s members are scanned
// (about 2.5e9 entries on R-MAT-18 for 7e7 edges of G0) and a quarter of the
// entries are hits.  A bit per hashed id sorts out the misses with one shared
// read, and the rest wait until they fill a warp, so the hash probes run with
// all lanes; the kernel issues on 85 % of cycles.  Measured (clique phase, before
// -> now): R-MAT-21 global 90 -> 63 ms, CL-1M 7.2 -> 5.4 ms; per-edge rows of
// CL-125K 8.9 -> 1.4 ms (there each clique was found by a search and added to its
// six edges one by one).
#include <algorithm>

#include "tg_cycles.cuh"
#include "tg_device.cuh"

using namespace tgd;

namespace {

constexpr int kWords = 128;  // most words of a row

// Classes of x0 by the length of up(x0): one warp and one word a row, then a
// CTA with rows in shared memory (three sizes of CTA) or in its slice of
// global memory, then the lists left to the callers' hash-set kernels.
enum { kUpWarp = 0, kUpS, kUpM, kUpL, kUpXL, kUpLong, kUpClasses };
constexpr int kUpMin = 2, kUpWarpMax = 32, kUpSMax = 160, kUpMMax = 512;  // list lengths
constexpr int kUpThreads[kUpClasses] = {256, 128, 512, 1024, 512, 0};

__host__ __device__ inline int up_words(int d, int L) { return (d + 31 * L) / 32; }

// Lists the x0 of every class (no order); size[k] its length, size[kUpClasses
// + k] its longest list.
__global__ void k_up_classes(const int64_t *uoff, int64_t n, int L, int pidx, int pcnt,
                             uint32_t *list, unsigned long long *size) {
    const int lane = threadIdx.x & 31;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; c < n; c += nthreads) {
        const int64_t x = c + lane;
        int64_t d = 0;
        if (x < n && x % pcnt == pidx) d = uoff[x + 1] - uoff[x];
        int cls = -1;
        if (d > kUpMin) {
            cls = d <= kUpWarpMax ? kUpWarp : d <= kUpSMax ? kUpS : d <= kUpMMax ? kUpM : kUpLong;
            if (cls == kUpLong && d <= 32 * kWords)
                cls = up_words((int)d, L) <= 64 ? kUpL : up_words((int)d, L) <= kWords ? kUpXL : kUpLong;
        }
        for (int k = 0; k < kUpClasses; ++k) {
            const unsigned m = __ballot_sync(kFull, cls == k);
            if (!m) continue;
            const unsigned top = __reduce_max_sync(kFull, cls == k ? (unsigned)d : 0u);
            unsigned long long base = 0;
            if (lane == 0) {
                base = atomicAdd(size + k, (unsigned long long)__popc(m));
                atomicMax(size + kUpClasses + k, (unsigned long long)top);
            }
            base = __shfl_sync(kFull, base, 0);
            if (cls == k) list[(int64_t)k * n + (int64_t)base + __popc(m & ((1u << lane) - 1u))] = (uint32_t)x;
        }
    }
}

struct CliqueParams {
    const int64_t *uoff;
    const uint32_t *uadj;
    const uint32_t *ueid;
    const int32_t *utoff;
    const uint8_t *ntype;
    const uint32_t *list;  // the x0 of this class
    int64_t count;
    int32_t L, P, hlg;
    unsigned long long *queue;
    unsigned long long *k4e;  // per-edge mode: M x P
    unsigned long long *g4;   // global mode: C(L+3,4)
    int64_t n4;
    uint32_t *rows;  // rows in global memory: rows_stride words per CTA
    int64_t rows_stride;
    unsigned long long *work;  // [5]: pairs (v, w), [6]: 4-cliques
};

__device__ __forceinline__ void hist_add(unsigned long long *h4, int a, int b, int c, int d,
                                         unsigned long long v) {
    sort2(a, b);
    sort2(c, d);
    sort2(a, c);
    sort2(b, d);
    sort2(b, c);
    atomicAdd(h4 + colex4(a, b, c, d), v);
}

__device__ __forceinline__ uint32_t bit_range(int lo, int hi) {  // bits [lo, hi), 0 <= lo <= hi <= 32
    const uint32_t h = hi >= 32 ? 0xffffffffu : (1u << hi) - 1u;
    const uint32_t l = lo >= 32 ? 0xffffffffu : (1u << lo) - 1u;
    return h & ~l;
}

// Per-edge mode counts every clique at its three upper edges: the sum over all
// warps is divided by 3 mod 2^64, each part times the inverse of 3.
constexpr unsigned long long kThird = 0xAAAAAAAAAAAAAAABull;

__device__ __forceinline__ void add_work(unsigned long long *work, int slot, unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(work + slot, v);
}

// ------------------------------------------------------------- one word ----
constexpr int kBitWarps = 8;
constexpr int kBitHits = 32 * 31 / 2;  // edges of G0, at most
constexpr int kBitBatch = 2;           // chunks of 32 entries in flight
// Lists of d0 members are searched, pair by pair, where scanning them would read more
// than kSearchCost d0^2 entries.  Clique phase by scans alone, and with a cost of 4, 2
// and 1: CL-1M 4.58, 4.05, 3.75, 3.66 ms, CL-100K 0.72, 0.69, 0.69, 0.62; R-MAT-21
// 60.4 -> 56.0, per-edge rows of CL-125K 1.26 -> 1.15.
constexpr int kSearchCost = 1;

struct BitWarp {
    uint32_t hk[64], hv[64], row[32], tmask[TG_MAX_TYPES];
};
struct BitHits {
    uint32_t eid[kBitHits];
    uint16_t vw[kBitHits];
};

template <bool kEdge>
__global__ void __launch_bounds__(kBitWarps * 32) k_k4_warp(CliqueParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, L = p.L;
    unsigned long long *h4 = reinterpret_cast<unsigned long long *>(smem);
    const size_t off = kEdge ? 0 : ((size_t)p.n4 * 8 + 15) & ~(size_t)15;
    BitWarp &sm = reinterpret_cast<BitWarp *>(smem + off)[warp];
    BitHits &hits = reinterpret_cast<BitHits *>(smem + off + kBitWarps * sizeof(BitWarp))[kEdge ? warp : 0];
    if (!kEdge)
        for (int64_t q = threadIdx.x; q < p.n4; q += blockDim.x) h4[q] = 0ull;
    __syncthreads();
    unsigned long long wk = 0, wpairs = 0;
    for (;;) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(p.queue, 4ull);
        base = __shfl_sync(kFull, base, 0);
        if (base >= (unsigned long long)p.count) break;
        const int64_t stop = min((int64_t)base + 4, p.count);
        for (int64_t it = (int64_t)base; it < stop; ++it) {
            const uint32_t x0 = p.list[it];
            const int64_t b0 = __ldg(p.uoff + x0);
            const int d0 = (int)(__ldg(p.uoff + x0 + 1) - b0);
            const int t0 = p.ntype[x0];
            const int32_t *to0 = p.utoff + (int64_t)x0 * (L + 1);
            sm.hk[lane] = sm.hk[lane + 32] = 0u;
            sm.row[lane] = 0u;
            if (lane < L) sm.tmask[lane] = bit_range(__ldg(to0 + lane), __ldg(to0 + lane + 1));
            __syncwarp();
            uint32_t ve = 0;
            int64_t bv = 0;
            int dv = 0;
            if (lane < d0) {
                ve = __ldg(p.uadj + b0 + lane);
                hmap_put(sm.hk, sm.hv, 6, ve & TG_IDMASK, (uint32_t)lane);
                bv = __ldg(p.uoff + (ve & TG_IDMASK));
                dv = (int)(__ldg(p.uoff + (ve & TG_IDMASK) + 1) - bv);
            }
            __syncwarp();
            // the members' up lists as one sequence, 32 entries at a time
            int incl = dv;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            const int total = __shfl_sync(kFull, incl, 31);
            const int64_t org = bv - (incl - dv);
            int nh = 0;
            // member w found in member v's list at position `at`, in any lanes
            auto found = [&](bool hit, int v, uint32_t w, int64_t at) {
                if (hit) atomicOr(&sm.row[v], 1u << w);
                if (kEdge) {
                    if (hit) atomicOr(&sm.row[w], 1u << v);
                    const unsigned m = __ballot_sync(kFull, hit);
                    if (hit) {
                        const int k = nh + __popc(m & ((1u << lane) - 1u));
                        hits.eid[k] = __ldg(p.ueid + at);
                        hits.vw[k] = (uint16_t)((v << 5) | w);
                    }
                    nh += __popc(m);
                }
            };
            if (total > kSearchCost * d0 * d0) {
                // a lane per pair of members (x, x + o mod d0)
                const int half = d0 >> 1, pairs = d0 * half;
                for (int c = 0; c < pairs; c += 32) {
                    const int k = c + lane, o = 1 + k / d0;
                    int x = k - (o - 1) * d0, y = x + o;
                    if (y >= d0) y -= d0;
                    const bool in = k < pairs && !(2 * o == d0 && x >= half);
                    if (!in) x = y = 0;
                    const uint32_t ex = __shfl_sync(kFull, ve, x), ey = __shfl_sync(kFull, ve, y);
                    const bool swap = (ex & TG_IDMASK) < (ey & TG_IDMASK);
                    const int v = swap ? y : x, w = swap ? x : y;  // w ranks above v
                    const uint32_t ev = swap ? ey : ex, ew = swap ? ex : ey;
                    const int64_t b = __shfl_sync(kFull, bv, v);
                    int lo = 0, end = 0;
                    if (in) {
                        const int32_t *to = p.utoff + (int64_t)(ev & TG_IDMASK) * (L + 1) + (ew >> TG_TSHIFT);
                        lo = __ldg(to);
                        end = __ldg(to + 1);
                    }
                    int hi = end;
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (__ldg(p.uadj + b + mid) < ew)
                            lo = mid + 1;
                        else
                            hi = mid;
                    }
                    __syncwarp();
                    found(lo < end && __ldg(p.uadj + b + lo) == ew, v, (uint32_t)w, b + lo);
                }
            } else {
                for (int c = 0; c < total; c += 32 * kBitBatch) {
                    int64_t at[kBitBatch];
                    uint32_t e[kBitBatch];
                    int of[kBitBatch];
#pragma unroll
                    for (int z = 0; z < kBitBatch; ++z) {
                        const int pos = c + 32 * z + lane;
                        int r = 0;  // the member whose list holds pos
#pragma unroll
                        for (int st = 16; st > 0; st >>= 1) {
                            const int v = __shfl_sync(kFull, incl, r + st - 1);
                            if (v <= pos) r += st;
                        }
                        of[z] = r;
                        at[z] = __shfl_sync(kFull, org, r) + pos;
                        e[z] = pos < total ? __ldg(p.uadj + at[z]) : 0u;
                    }
#pragma unroll
                    for (int z = 0; z < kBitBatch; ++z) {
                        uint32_t w = 0xffffffffu;
                        if (c + 32 * z + lane < total) w = hmap_get(sm.hk, sm.hv, 6, e[z] & TG_IDMASK);
                        found(w != 0xffffffffu, of[z], w, at[z]);
                    }
                }
            }
            __syncwarp();
            const uint32_t mine = sm.row[lane];
            const int tv = (int)(ve >> TG_TSHIFT);
            if (!kEdge) {
                // lane v takes the members w of its bitmap in turn
                uint32_t m = mine;
                while (m) {
                    const int q = __ffs(m) - 1;
                    m &= m - 1u;
                    ++wpairs;
                    const uint32_t both = mine & sm.row[q];
                    if (!both) continue;
                    int tw = 0;
                    while (!((sm.tmask[tw] >> q) & 1u)) ++tw;
                    wk += __popc(both);
                    for (int t = 0; t < L; ++t) {
                        const int c = __popc(both & sm.tmask[t]);
                        if (c) hist_add(h4, t0, tv, tw, t, (unsigned long long)c);
                    }
                }
            } else {
                for (int k = lane; k < nh; k += 32) {  // edges (v, w)
                    const int v = hits.vw[k] >> 5, w = hits.vw[k] & 31;
                    const uint32_t both = sm.row[v] & sm.row[w];
                    ++wpairs;
                    if (!both) continue;
                    wk += __popc(both);
                    unsigned long long *row = p.k4e + (int64_t)hits.eid[k] * p.P;
                    for (int t = 0; t < L; ++t) {
                        const int c = __popc(both & sm.tmask[t]);
                        if (c) atomicAdd(row + pair_index(L, t0, t), (unsigned long long)c);
                    }
                }
                if (mine) {  // edges (x0, v)
                    unsigned long long *row = p.k4e + (int64_t)__ldg(p.ueid + b0 + lane) * p.P;
                    for (int a = 0; a < L; ++a) {
                        const uint32_t ma = mine & sm.tmask[a];
                        if (!ma) continue;
                        for (int b = a; b < L; ++b) {
                            const uint32_t mb = mine & sm.tmask[b];
                            if (!mb) continue;
                            unsigned c = 0;
                            for (uint32_t m = ma; m; m &= m - 1u) c += __popc(sm.row[__ffs(m) - 1] & mb);
                            if (a == b) c >>= 1;
                            if (c) atomicAdd(row + pair_index(L, a, b), (unsigned long long)c);
                        }
                    }
                }
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
        add_work(p.work, 5, wpairs);
        add_work(p.work, 6, kEdge ? wk * kThird : wk);
    }
}

// --------------------------------------------------------------- rows ----
// One CTA per x0.  Rows of up to 64 words are kept in shared memory when they
// fit (a pair (v, w) then costs one conflict-free read per word), else in the
// CTA's slice of global memory.  In global mode a warp takes a run of
// consecutive v, so of few types, and keeps the counts per (type of w, word)
// in columns of shared memory that only their lane touches; they go to the
// histogram, summed over the words of a type, when the type of v changes.
// Adding them per v put up to 32 lanes on a few 64-bit shared counters (214 ms
// of R-MAT-21's count against 165 with the columns, before the scan was changed).
constexpr int kPend = 64;  // entries a warp keeps waiting
constexpr int kScan = 4;   // chunks of 32 entries in flight

template <int WPL, bool kEdge, bool kSmem>
__global__ void __launch_bounds__(WPL == 2 ? 1024 : 512) k_k4_rows(CliqueParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long s_item;
    __shared__ int wt[kWords], ws[TG_MAX_TYPES + 1], to[TG_MAX_TYPES + 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
    const int L = p.L;
    unsigned long long *h4 = reinterpret_cast<unsigned long long *>(smem);
    const size_t off = kEdge ? 0 : ((size_t)p.n4 * 8 + 15) & ~(size_t)15;
    uint32_t *hk = reinterpret_cast<uint32_t *>(smem + off);
    uint32_t *hv = hk + (1 << p.hlg);
    uint32_t *seen = hv + (1 << p.hlg);  // 2^(hlg + 3) bits
    uint2 *pend = reinterpret_cast<uint2 *>(seen + (1 << p.hlg) / 4) + warp * kPend;
    // global mode: this warp's counts per (type of w, word)
    uint32_t *cols = seen + (1 << p.hlg) / 4 + W * kPend * 2;
    uint32_t *rows = kSmem ? cols + (kEdge ? 0 : W * L * 32 * WPL)
                           : p.rows + (size_t)blockIdx.x * (size_t)p.rows_stride;
    if (!kEdge) cols += warp * L * 32 * WPL;
    auto get = [&](size_t x) -> uint32_t { return kSmem ? rows[x] : __ldcg(rows + x); };
    if (!kEdge)
        for (int64_t q = tid; q < p.n4; q += blockDim.x) h4[q] = 0ull;
    if (!kEdge)
        for (int q = lane; q < L * 32 * WPL; q += 32) cols[q] = 0u;
    unsigned long long wk = 0, wpairs = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(p.queue, 1ull);
        __syncthreads();
        if (s_item >= (unsigned long long)p.count) break;
        const uint32_t x0 = p.list[s_item];
        const int64_t b0 = __ldg(p.uoff + x0);
        const int d0 = (int)(__ldg(p.uoff + x0 + 1) - b0);
        const int t0 = p.ntype[x0];
        const int32_t *to0 = p.utoff + (int64_t)x0 * (L + 1);
        int lg = 5;
        while ((1 << lg) < 2 * d0) ++lg;  // at most p.hlg
        if (tid <= L) to[tid] = __ldg(to0 + tid);
        for (int q = tid; q < (1 << lg); q += blockDim.x) hk[q] = 0u;
        for (int q = tid; q < (1 << lg) / 4; q += blockDim.x) seen[q] = 0u;
        __syncthreads();
        if (tid == 0) {
            int w = 0;
            for (int t = 0; t < L; ++t) {
                ws[t] = w;
                w += (to[t + 1] - to[t] + 31) >> 5;
            }
            ws[L] = w;
        }
        __syncthreads();
        const int words = ws[L];
        for (int k = tid; k < words; k += blockDim.x) {
            int t = 0;
            while (t + 1 < L && ws[t + 1] <= k) ++t;
            wt[k] = t;
        }
        for (int q = tid; q < d0; q += blockDim.x) {
            const uint32_t e = __ldg(p.uadj + b0 + q);
            const int t = (int)(e >> TG_TSHIFT);
            hmap_put(hk, hv, lg, e & TG_IDMASK, (uint32_t)(32 * ws[t] + (q - to[t])));
            const uint32_t h = hset_slot(e & TG_IDMASK, lg + 3);
            atomicOr(seen + (h >> 5), 1u << (h & 31u));
        }
        for (int q = tid; q < d0 * words; q += blockDim.x) rows[q] = 0u;
        __syncthreads();
        // rows: warp per member v.  An entry of up(v) is looked up only when its
        // bit of `seen` is set; these wait until 32 of them fill a warp.
        int np = 0;
        auto settle = [&](int count) {
            if (lane >= count) return;
            const uint2 yq = pend[lane];
            const uint32_t pp = hmap_get(hk, hv, lg, yq.x & TG_IDMASK);
            if (pp == 0xffffffffu) return;
            atomicOr(rows + (size_t)yq.y * words + (pp >> 5), 1u << (pp & 31u));
            if (kEdge) {
                const int ty = (int)(yq.x >> TG_TSHIFT);
                const int qy = to[ty] + (int)pp - 32 * ws[ty];
                int tq = 0;
                while (to[tq + 1] <= (int)yq.y) ++tq;
                const int pv = 32 * ws[tq] + ((int)yq.y - to[tq]);
                atomicOr(rows + (size_t)qy * words + (pv >> 5), 1u << (pv & 31));
            }
        };
        for (int q = warp; q < d0; q += W) {
            const uint32_t ve = __ldg(p.uadj + b0 + q);
            const int64_t bv = __ldg(p.uoff + (ve & TG_IDMASK));
            const int dv = (int)(__ldg(p.uoff + (ve & TG_IDMASK) + 1) - bv);
            for (int c = 0; c < dv; c += 32 * kScan) {
                uint32_t y[kScan];
#pragma unroll
                for (int z = 0; z < kScan; ++z)
                    y[z] = c + 32 * z + lane < dv ? __ldg(p.uadj + bv + c + 32 * z + lane) : 0xffffffffu;
#pragma unroll
                for (int z = 0; z < kScan; ++z) {
                    const uint32_t h = hset_slot(y[z] & TG_IDMASK, lg + 3);
                    const bool maybe = y[z] != 0xffffffffu && ((seen[h >> 5] >> (h & 31u)) & 1u);
                    const unsigned m = __ballot_sync(kFull, maybe);
                    if (maybe) pend[np + __popc(m & ((1u << lane) - 1u))] = make_uint2(y[z], (uint32_t)q);
                    np += __popc(m);
                    if (np >= 32) {
                        __syncwarp();
                        settle(32);
                        np -= 32;
                        __syncwarp();
                        if (lane < np) pend[lane] = pend[lane + 32];
                        __syncwarp();
                    }
                }
            }
        }
        __syncwarp();
        settle(np);
        __syncthreads();
        int ty[WPL];
#pragma unroll
        for (int i = 0; i < WPL; ++i) ty[i] = lane + 32 * i < words ? wt[lane + 32 * i] : -1;
        // the columns of the v of type tv so far into the histogram
        auto drain = [&](int tv) {
            if (kEdge || tv < 0) return;
            for (int w = 0; w < L; ++w) {
                uint32_t c[WPL];
                unsigned all = 0;
#pragma unroll
                for (int i = 0; i < WPL; ++i) {
                    c[i] = cols[w * 32 * WPL + lane + 32 * i];
                    all |= c[i];
                }
                if (!__any_sync(kFull, all != 0u)) continue;
                unsigned mine = 0;
                for (int t = 0; t < L; ++t) {
                    unsigned sum = 0;
#pragma unroll
                    for (int i = 0; i < WPL; ++i) sum += ty[i] == t ? c[i] : 0u;
                    sum = __reduce_add_sync(kFull, sum);
                    if (lane == t) mine = sum;
                }
#pragma unroll
                for (int i = 0; i < WPL; ++i) cols[w * 32 * WPL + lane + 32 * i] = 0u;
                if (mine) hist_add(h4, t0, tv, w, lane, (unsigned long long)mine);
                wk += mine;
            }
        };
        const int run = kEdge ? 1 : (d0 + W - 1) / W;  // consecutive v of a warp
        int tvc = -1;
        for (int q = kEdge ? warp : warp * run; q < (kEdge ? d0 : min(d0, (warp + 1) * run)); q += kEdge ? W : 1) {
            const uint32_t ve = __ldg(p.uadj + b0 + q);
            const int tv = (int)(ve >> TG_TSHIFT);
            if (tv != tvc) {
                drain(tvc);
                tvc = tv;
            }
            uint32_t rv[WPL], acc[WPL];
#pragma unroll
            for (int i = 0; i < WPL; ++i) {
                const int kk = lane + 32 * i;
                rv[i] = kk < words ? get((size_t)q * words + kk) : 0u;
                acc[i] = 0u;
            }
            unsigned any = rv[0];
#pragma unroll
            for (int i = 1; i < WPL; ++i) any |= rv[i];
            if (!__any_sync(kFull, any != 0u)) continue;
            const int64_t e0 = kEdge ? (int64_t)__ldg(p.ueid + b0 + q) : 0;
            // counts of the pairs (v, w of type cur) so far, per word: into the
            // columns, or the row of (x0, v)
            auto flush = [&](int cur) {
                if (cur < 0) return;
                if (!kEdge) {
#pragma unroll
                    for (int i = 0; i < WPL; ++i)
                        if (acc[i]) cols[cur * 32 * WPL + lane + 32 * i] += acc[i];
                } else {
                    unsigned c = 0;
#pragma unroll
                    for (int i = 0; i < WPL; ++i) {
                        c += ty[i] == cur ? acc[i] : 0u;
                        if (ty[i] > cur && acc[i])
                            atomicAdd(p.k4e + e0 * p.P + pair_index(L, cur, ty[i]), (unsigned long long)acc[i]);
                    }
                    c = __reduce_add_sync(kFull, c);  // every pair of one type was met twice
                    if (lane == 0 && c) atomicAdd(p.k4e + e0 * p.P + pair_index(L, cur, cur), (unsigned long long)(c >> 1));
                }
#pragma unroll
                for (int i = 0; i < WPL; ++i) acc[i] = 0u;
            };
            int cur = -1;
#pragma unroll
            for (int i = 0; i < WPL; ++i) {
                for (unsigned nz = __ballot_sync(kFull, rv[i] != 0u); nz; nz &= nz - 1u) {
                    const int k = 32 * i + __ffs(nz) - 1;
                    uint32_t x = __shfl_sync(kFull, rv[i], k & 31);
                    const int tw = wt[k];
                    if (tw != cur) {
                        flush(cur);
                        cur = tw;
                    }
                    const int qb = to[tw] + 32 * (k - ws[tw]);  // member index of the word's bit 0
                    wpairs += lane == 0 ? __popc(x) : 0;
                    while (x) {
                        // four rows in flight
                        size_t rw[4];
                        int nr = 0;
#pragma unroll
                        for (int z = 0; z < 4; ++z) {
                            rw[z] = 0;
                            if (x) {
                                rw[z] = (size_t)(qb + __ffs(x) - 1) * words;
                                x &= x - 1u;
                                ++nr;
                            }
                        }
#pragma unroll
                        for (int j = 0; j < WPL; ++j) {
                            const int kk = lane + 32 * j;
                            uint32_t v[4];
#pragma unroll
                            for (int z = 0; z < 4; ++z) v[z] = z < nr && kk < words ? get(rw[z] + kk) : 0u;
#pragma unroll
                            for (int z = 0; z < 4; ++z) acc[j] += (uint32_t)__popc(rv[j] & v[z]);
                        }
                    }
                }
            }
            flush(cur);
            if (!kEdge) continue;
            // edges (v, w), w in up(v): T_vw by type.  With rows of at most 16 (8)
            // words two (four) groups of lanes take an edge each.
            const int gsz = WPL > 1 || words > 16 ? 32 : words > 8 ? 16 : 8;
            const int nsub = 32 / gsz, sub = lane / gsz, kl = lane % gsz;
            uint32_t rg[WPL];
            int tg[WPL];
#pragma unroll
            for (int j = 0; j < WPL; ++j) {
                rg[j] = __shfl_sync(kFull, rv[j], kl);
                tg[j] = __shfl_sync(kFull, ty[j], kl);
            }
            const int64_t bv = __ldg(p.uoff + (ve & TG_IDMASK));
            const int dv = (int)(__ldg(p.uoff + (ve & TG_IDMASK) + 1) - bv);
            for (int c = 0; c < dv; c += 32) {
                uint32_t pp = 0xffffffffu, eid = 0;
                int qy = 0;
                if (c + lane < dv) {
                    const uint32_t y = __ldg(p.uadj + bv + c + lane);
                    pp = hmap_get(hk, hv, lg, y & TG_IDMASK);
                    if (pp != 0xffffffffu) {
                        const int t = (int)(y >> TG_TSHIFT);
                        qy = to[t] + (int)pp - 32 * ws[t];
                        eid = __ldg(p.ueid + bv + c + lane);
                    }
                }
                for (unsigned m = __ballot_sync(kFull, pp != 0xffffffffu); m;) {
                    unsigned mine = m;  // this group's edge: the sub-th set bit
                    for (int i = 0; i < sub; ++i) mine &= mine - 1u;
                    for (int i = 0; i < nsub; ++i) m &= m - 1u;
                    const int src = mine ? __ffs(mine) - 1 : 32;
                    const size_t rw = (size_t)__shfl_sync(kFull, qy, src & 31) * words;
                    const int64_t e = __shfl_sync(kFull, eid, src & 31);
#pragma unroll
                    for (int j = 0; j < WPL; ++j) {
                        const int kk = kl + 32 * j;
                        const uint32_t c = src < 32 && kk < words ? (uint32_t)__popc(rg[j] & get(rw + kk)) : 0u;
                        if (!c) continue;
                        wk += c;
                        atomicAdd(p.k4e + e * p.P + pair_index(L, t0, tg[j]), (unsigned long long)c);
                    }
                }
            }
        }
        drain(tvc);
    }
    if (!kEdge) {
        __syncthreads();
        for (int64_t q = tid; q < p.n4; q += blockDim.x)
            if (h4[q]) atomicAdd(p.g4 + q, h4[q]);
    }
    if (p.work) {
        add_work(p.work, 5, wpairs);
        add_work(p.work, 6, kEdge ? wk * kThird : wk);
    }
}

template <bool kEdge>
int launch_cliques(const unsigned long long (&size)[2 * kUpClasses], CliqueParams p, const uint32_t *list,
                   unsigned long long *queue, int64_t n, cudaStream_t s) {
    const size_t h4b = kEdge ? 0 : ((size_t)p.n4 * 8 + 15) & ~(size_t)15;
    const size_t avail = (size_t)tg_smem_optin() - 2048;
    DevBuf<uint32_t> rows[2];
    for (int k = kUpWarp; k <= kUpXL; ++k) {
        if (size[k] == 0) continue;
        p.list = list + (int64_t)k * n;
        p.count = (int64_t)size[k];
        p.queue = queue + k;
        if (k == kUpWarp) {
            const size_t smem = h4b + kBitWarps * (sizeof(BitWarp) + (kEdge ? sizeof(BitHits) : 0));
            const void *fn = (const void *)k_k4_warp<kEdge>;
            TG_TRY(tg_allow_max_smem(fn));
            int per = 0;
            TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kBitWarps * 32, smem));
            const int64_t grid = std::min<int64_t>((int64_t)tg_num_sms() * std::max(per, 1),
                                                   (p.count + kBitWarps - 1) / kBitWarps);
            k_k4_warp<kEdge><<<(unsigned)grid, kBitWarps * 32, smem, s>>>(p);
            tg_note_launch();
            TG_TRY_CUDA(cudaGetLastError());
            continue;
        }
        const int dmax = (int)size[kUpClasses + k];
        p.hlg = 5;
        while ((1 << p.hlg) < 2 * dmax) ++p.hlg;
        const int wpl = k == kUpXL ? 4 : k == kUpL ? 2 : 1;
        const size_t rbytes = (size_t)dmax * up_words(dmax, p.L) * 4;
        auto fixed = [&](int th) {  // shared memory besides the rows
            return h4b + (size_t)9 * ((size_t)1 << p.hlg) + (size_t)(th / 32) * kPend * 8 +
                   (kEdge ? 0 : (size_t)(th / 32) * p.L * 32 * wpl * 4);
        };
        // Rows in shared memory where a quarter of the class's threads or more leaves
        // room for them, else in global memory with CTAs of up to 512.  The cliques of
        // R-MAT-23, whose longest rows do not fit, take 725 ms when the threads are cut to
        // 64 in vain, 410 with 1024, 382 with 512, 413 with 256; those of R-MAT-21, whose
        // rows fit, 56 with 1024 and 60 with 512.
        int threads = kUpThreads[k];
        while (threads > std::max(64, kUpThreads[k] / 4) && fixed(threads) + rbytes > avail) threads /= 2;
        const bool sm = k != kUpXL && fixed(threads) + rbytes <= avail;
        if (!sm) {
            threads = std::min(kUpThreads[k], 512);
            while (threads > 64 && fixed(threads) > avail) threads /= 2;
        }
        const size_t base = fixed(threads);
        const size_t smem = base + (sm ? rbytes : 0);
        if (smem > avail) return TG_EINVAL;
        void (*fn)(CliqueParams) = k == kUpXL ? k_k4_rows<4, kEdge, false>
                                   : k == kUpL ? (sm ? k_k4_rows<2, kEdge, true> : k_k4_rows<2, kEdge, false>)
                                   : sm ? k_k4_rows<1, kEdge, true> : k_k4_rows<1, kEdge, false>;
        TG_TRY(tg_allow_max_smem((const void *)fn));
        int per = 0;
        TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem));
        const int64_t grid = std::min<int64_t>((int64_t)tg_num_sms() * std::max(per, 1), p.count);
        if (!sm) {
            DevBuf<uint32_t> &r = rows[k == kUpXL];
            p.rows_stride = (int64_t)(rbytes / 4);
            if (!r.alloc((size_t)grid * (size_t)p.rows_stride, s)) return TG_ENOMEM;
            p.rows = r.p;
        }
        fn<<<(unsigned)grid, threads, smem, s>>>(p);
        tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    return TG_OK;
}

}  // namespace

int tg_k4_bits(const tg_graph *g, const tg_lists &up, unsigned long long *k4e, unsigned long long *g4,
               unsigned long long *work, const tg_part &part, int64_t *nlong, int64_t *longest,
               int64_t *bits_max, cudaStream_t s) {
    const int64_t n = g->n;
    const int L = g->L;
    DevBuf<uint32_t> list;
    DevBuf<unsigned long long> size;
    if (!list.alloc((size_t)kUpClasses * n, s) || !size.alloc(3 * kUpClasses, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(size.p, 0, 3 * kUpClasses * 8, s));
    k_up_classes<<<(unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)tg_num_sms() * 8), 256, 0, s>>>(
        up.uoff, n, L, part.index, part.count, list.p, size.p);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    unsigned long long h[2 * kUpClasses];
    TG_TRY_CUDA(cudaMemcpyAsync(h, size.p, sizeof(h), cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    CliqueParams p{};
    p.uoff = up.uoff;
    p.uadj = up.uadj;
    p.ueid = up.ueid;
    p.utoff = up.utoff;
    p.ntype = g->ntype;
    p.L = L;
    p.P = L * (L + 1) / 2;
    p.k4e = k4e;
    p.g4 = g4;
    p.n4 = tg_binom(L + 3, 4);
    p.work = work;
    *nlong = (int64_t)h[kUpLong];
    *longest = (int64_t)h[kUpClasses + kUpLong];
    int d = 32 * kWords;
    while (up_words(d, L) > kWords) --d;
    *bits_max = d;
    return g4 ? launch_cliques<false>(h, p, list.p, size.p + 2 * kUpClasses, n, s)
              : launch_cliques<true>(h, p, list.p, size.p + 2 * kUpClasses, n, s);
}
