// Directed typed 3-node graphlets (Sec. "Directed Typed Graphlets").
//
// The paper splits every typed neighbourhood into out- and in-neighbours
// (Gamma_i^{t,+}, Gamma_i^{t,-}) and runs Alg. 1 over the combinations of the
// split sets.  Here the split is two bits per adjacency entry of the
// undirected typed CSR (bit 0: owner -> neighbour, bit 1: neighbour ->
// owner; both for a pair with arcs both ways), set once when the graph is
// built with TG_DIRECTED.  Per edge (i, j) one warp runs Alg. 1 on the
// shorter list: each triangle node w of T_ij comes with the state of (i, w)
// and of (j, w), counted per (state pair, type of w); the 3-star nodes S_i,
// S_j are not enumerated: their counts per (state, type) are the node's
// split typed degrees less j (or i) and less the triangle nodes of that
// state.  The triad class of {i, j, w} follows from the three pair states by
// a table built on the host from the class representatives of the header.
#include <algorithm>
#include <mutex>
#include <vector>

#include "tg_device.cuh"

using namespace tgd;

namespace {

constexpr int kDirThreads = 256;
constexpr int kDirWarps = kDirThreads / 32;

// Arc bits of the pairs of three labelled nodes 0, 1, 2: bit 2 p for the arc
// from the lower to the higher node of pair p, bit 2 p + 1 for the reverse;
// pairs (0, 1), (0, 2), (1, 2).
int arc_bit(int a, int b) {
    const int p = (a + b == 1) ? 0 : (a + b == 2) ? 1 : 2;
    return 2 * p + (a < b ? 0 : 1);
}

// Class of every connected 3-node digraph, by arc mask; -1 for the others.
struct TriadTable {
    int8_t cls[64];
    bool ok = false;
};

TriadTable build_triads() {
    // representatives of the header on A = 0, B = 1, C = 2 (arcs from -> to)
    static const int reps[TG_TRIAD_CLASSES][6][2] = {
        {{1, 0}, {1, 2}, {-1, -1}},                                   // 021D
        {{0, 1}, {2, 1}, {-1, -1}},                                   // 021U
        {{0, 1}, {1, 2}, {-1, -1}},                                   // 021C
        {{0, 1}, {1, 0}, {2, 1}, {-1, -1}},                           // 111D
        {{0, 1}, {1, 0}, {1, 2}, {-1, -1}},                           // 111U
        {{0, 1}, {2, 1}, {0, 2}, {-1, -1}},                           // 030T
        {{0, 1}, {1, 2}, {2, 0}, {-1, -1}},                           // 030C
        {{0, 1}, {1, 0}, {1, 2}, {2, 1}, {-1, -1}},                   // 201
        {{1, 0}, {1, 2}, {0, 2}, {2, 0}, {-1, -1}},                   // 120D
        {{0, 1}, {2, 1}, {0, 2}, {2, 0}, {-1, -1}},                   // 120U
        {{0, 1}, {1, 2}, {0, 2}, {2, 0}, {-1, -1}},                   // 120C
        {{0, 1}, {1, 2}, {2, 1}, {0, 2}, {2, 0}, {-1, -1}},           // 210
        {{0, 1}, {1, 0}, {1, 2}, {2, 1}, {0, 2}, {2, 0}},             // 300
    };
    static const int perm[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2},
                                   {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
    TriadTable t;
    std::fill(t.cls, t.cls + 64, (int8_t)-1);
    bool ok = true;
    for (int c = 0; c < TG_TRIAD_CLASSES; ++c)
        for (int q = 0; q < 6; ++q) {
            int mask = 0;
            for (int r = 0; r < 6 && reps[c][r][0] >= 0; ++r)
                mask |= 1 << arc_bit(perm[q][reps[c][r][0]], perm[q][reps[c][r][1]]);
            if (t.cls[mask] >= 0 && t.cls[mask] != c) ok = false;
            t.cls[mask] = (int8_t)c;
        }
    // every mask whose pairs connect the three nodes must have a class
    for (int mask = 0; mask < 64; ++mask) {
        const int pairs = ((mask & 3) != 0) + ((mask & 12) != 0) + ((mask & 48) != 0);
        if ((pairs >= 2) != (t.cls[mask] >= 0)) ok = false;
    }
    t.ok = ok;
    return t;
}

const TriadTable &triads() {
    static std::once_flag once;
    static TriadTable t;
    std::call_once(once, [] { t = build_triads(); });
    return t;
}

// arc mask of a pair state (bit 0: lower-labelled -> higher, bit 1: back)
inline int pair_mask(int state, int a, int b) {
    int m = 0;
    if (state & 1) m |= 1 << arc_bit(a, b);
    if (state & 2) m |= 1 << arc_bit(b, a);
    return m;
}

struct DirParams {
    const int64_t *rowptr;
    const uint32_t *adj;
    const uint8_t *adir;
    const int32_t *toff;
    const uint8_t *ntype;
    const int2 *edges;
    const uint32_t *nd;  // n x 3 L split typed degrees (state 1..3, type)
    int64_t M;
    int32_t L;
    int64_t n3;           // C(L+2, 3)
    uint64_t *rows;       // per-edge mode
    unsigned long long *sums;  // global mode: 13 n3 undivided sums
    unsigned long long *queue;
    unsigned *err;
    int8_t tri[27];  // class of (s_ij, s_iw, s_jw), states 1..3 each
    int8_t path[9];  // class of a 3-path by the states of its ends seen from its centre
};

__global__ void k_arc_bits(const int32_t *src, const int32_t *dst, int64_t m,
                           const int32_t *old2new, const int64_t *rowptr, const uint32_t *adj,
                           const int32_t *toff, const uint8_t *ntype, int L, uint32_t *adir32,
                           unsigned *err) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a0 = src[e], b0 = dst[e];
        if (a0 == b0) continue;
        const uint32_t a = (uint32_t)old2new[a0], b = (uint32_t)old2new[b0];
        const int64_t ba = rowptr[a], bb = rowptr[b];
        const int pa = find_pos(adj, ba, toff + (int64_t)a * (L + 1),
                                ((uint32_t)ntype[b] << TG_TSHIFT) | b);
        const int pb = find_pos(adj, bb, toff + (int64_t)b * (L + 1),
                                ((uint32_t)ntype[a] << TG_TSHIFT) | a);
        if (pa < 0 || pb < 0) {
            atomicOr(err, TG_DERR_BOUNDS);
            continue;
        }
        const int64_t qa = ba + pa, qb = bb + pb;
        atomicOr(adir32 + (qa >> 2), 1u << (8 * (int)(qa & 3)));  // a -> b: out of a
        atomicOr(adir32 + (qb >> 2), 2u << (8 * (int)(qb & 3)));  // a -> b: into b
    }
}

// Split typed degrees: nd[v][(s - 1) L + t] = neighbours of v of type t whose
// pair with v has state s.  One warp per node, counters in shared memory; the
// nodes of degree above kDirHub, which have the smallest ids, take a CTA each
// (one warp needs 1 ms for the 64K neighbours of R-MAT-20's largest hub).
constexpr int kDirHub = 2048;

__global__ void __launch_bounds__(1024) k_dir_degrees_hub(const int64_t *rowptr, const uint32_t *adj,
                                                          const uint8_t *adir, int64_t n, int L,
                                                          uint32_t *nd) {
    __shared__ uint32_t cnt[32][3 * TG_MAX_TYPES];
    const int warp = threadIdx.x >> 5;
    for (int64_t v = blockIdx.x; v < n; v += gridDim.x) {
        const int64_t b = rowptr[v], d = rowptr[v + 1] - b;
        if (d <= kDirHub) break;
        for (int k = threadIdx.x; k < 32 * 3 * TG_MAX_TYPES; k += blockDim.x) (&cnt[0][0])[k] = 0u;
        __syncthreads();
        for (int64_t x = threadIdx.x; x < d; x += blockDim.x) {
            const int st = adir[b + x];
            if (st) atomicAdd(&cnt[warp][(st - 1) * L + (int)(__ldg(adj + b + x) >> TG_TSHIFT)], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 3 * L) {
            uint32_t s = 0;
            for (int w = 0; w < 32; ++w) s += cnt[w][threadIdx.x];
            nd[v * 3 * L + threadIdx.x] = s;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kDirThreads) k_dir_degrees(const int64_t *rowptr,
                                                             const uint32_t *adj,
                                                             const uint8_t *adir, int64_t n,
                                                             int L, uint32_t *nd) {
    __shared__ uint32_t cnt[kDirWarps][3 * TG_MAX_TYPES];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * kDirWarps;
    for (int64_t v = blockIdx.x * (int64_t)kDirWarps + warp; v < n; v += nw) {
        for (int k = lane; k < 3 * L; k += 32) cnt[warp][k] = 0u;
        __syncwarp();
        const int64_t b = rowptr[v], d = rowptr[v + 1] - b;
        if (d > kDirHub) continue;
        for (int64_t x = lane; x < d; x += 32) {
            const int st = adir[b + x];
            const int t = (int)(__ldg(adj + b + x) >> TG_TSHIFT);
            if (st) atomicAdd(&cnt[warp][(st - 1) * L + t], 1u);
        }
        __syncwarp();
        for (int k = lane; k < 3 * L; k += 32) nd[v * 3 * L + k] = cnt[warp][k];
        __syncwarp();
    }
}

__device__ __forceinline__ int swap_state(int s) { return ((s & 1) << 1) | ((s >> 1) & 1); }

// One warp per edge (dynamic queue).  kRows: per-edge rows, else the undivided sums
// of a small graph's global count (per-CTA shared histogram).
template <bool kRows>
__global__ void __launch_bounds__(kDirThreads) k_dir3(DirParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = p.L, S = TG_TRIAD_CLASSES * L;
    const int64_t hlen = kRows ? 0 : TG_TRIAD_CLASSES * p.n3;
    unsigned long long *h = reinterpret_cast<unsigned long long *>(smem);
    uint32_t *tri = reinterpret_cast<uint32_t *>(h + hlen) + (size_t)warp * 9 * L;
    if (!kRows) {
        for (int64_t q = threadIdx.x; q < hlen; q += blockDim.x) h[q] = 0ull;
        __syncthreads();
    }
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= (unsigned long long)p.M) break;
        const int64_t e = (int64_t)item;
        const int2 ab = p.edges[e];
        const uint32_t i = (uint32_t)ab.x, j = (uint32_t)ab.y;
        const int ti = p.ntype[i], tj = p.ntype[j];
        const int64_t bi = p.rowptr[i], bj = p.rowptr[j];
        const int di = (int)(p.rowptr[i + 1] - bi), dj = (int)(p.rowptr[j + 1] - bj);
        const int32_t *toi = p.toff + (int64_t)i * (L + 1);
        const int32_t *toj = p.toff + (int64_t)j * (L + 1);
        int sij = 0;
        if (lane == 0) {
            const int q = find_pos(p.adj, bi, toi, ((uint32_t)tj << TG_TSHIFT) | j);
            sij = q >= 0 ? p.adir[bi + q] : 0;
            if (sij == 0) atomicOr(p.err, TG_DERR_BOUNDS);
        }
        sij = __shfl_sync(kFull, sij, 0);
        for (int k = lane; k < 9 * L; k += 32) tri[k] = 0u;
        __syncwarp();
        if (sij != 0) {
            // Alg. 1 on the shorter list: x scanned, y searched
            const bool xi = di <= dj;
            const int64_t bx = xi ? bi : bj, by = xi ? bj : bi;
            const int dx = xi ? di : dj;
            const uint32_t yid = xi ? j : i;
            const int32_t *toy = xi ? toj : toi;
            for (int x = lane; x < dx; x += 32) {
                const uint32_t w = __ldg(p.adj + bx + x);
                if ((w & TG_IDMASK) == yid) continue;
                const int q = find_pos(p.adj, by, toy, w);
                if (q < 0) continue;
                const int sx = p.adir[bx + x], sy = p.adir[by + q];
                if (sx == 0 || sy == 0) {  // every entry carries an arc; never taken
                    atomicOr(p.err, TG_DERR_BOUNDS);
                    continue;
                }
                const int siw = xi ? sx : sy, sjw = xi ? sy : sx;
                atomicAdd(&tri[((siw - 1) * 3 + (sjw - 1)) * L + (int)(w >> TG_TSHIFT)], 1u);
            }
        }
        __syncwarp();
        if (sij != 0) {
            const int sji = swap_state(sij);
            const uint32_t *ndi = p.nd + (int64_t)i * 3 * L, *ndj = p.nd + (int64_t)j * 3 * L;
            for (int k = lane; k < S; k += 32) {
                const int c = k / L, t = k - c * L;
                unsigned long long v = 0;
                for (int s1 = 0; s1 < 3; ++s1)
                    for (int s2 = 0; s2 < 3; ++s2)
                        if (p.tri[(sij - 1) * 9 + s1 * 3 + s2] == c) v += tri[(s1 * 3 + s2) * L + t];
                for (int s = 0; s < 3; ++s) {
                    if (p.path[(sij - 1) * 3 + s] == c) {
                        // S_i members of state s + 1 and type t
                        long long m = (long long)ndi[s * L + t] - ((s + 1 == sij && t == tj) ? 1 : 0);
                        for (int s2 = 0; s2 < 3; ++s2) m -= tri[(s * 3 + s2) * L + t];
                        v += (unsigned long long)m;
                    }
                    if (p.path[(sji - 1) * 3 + s] == c) {
                        long long m = (long long)ndj[s * L + t] - ((s + 1 == sji && t == ti) ? 1 : 0);
                        for (int s1 = 0; s1 < 3; ++s1) m -= tri[(s1 * 3 + s) * L + t];
                        v += (unsigned long long)m;
                    }
                }
                if (kRows) {
                    p.rows[e * S + k] = v;
                } else if (v) {
                    int a = ti, b = tj, cc = t;
                    sort2(a, b);
                    sort2(b, cc);
                    sort2(a, b);
                    atomicAdd(h + (int64_t)c * p.n3 + colex3(a, b, cc), v);
                }
            }
        } else if (kRows) {
            for (int k = lane; k < S; k += 32) p.rows[e * S + k] = 0ull;
        }
        __syncwarp();
    }
    if (!kRows) {
        __syncthreads();
        for (int64_t q = threadIdx.x; q < hlen; q += blockDim.x)
            if (h[q]) atomicAdd(p.sums + q, h[q]);
    }
}

// ------------------------------------------------ 3 nodes, global totals ----
// The undivided sums without per-edge rows.  Every pair of neighbours of a node
// is a 3-path through it, open or closed: twice the pairs by (states, types) from
// the split typed degrees (each open path is met at its two edges), and per edge
// (i, j) and triangle node w one triad of the triangle's class, less one path at
// i and one at j.  So an edge needs only its triangle nodes by (state of (i, w),
// state of (j, w), type): Alg. 1 as k_tau runs it, with the pair's state beside
// every member of Gamma_j - two bits per node id in shared memory for units of a
// high-degree j (a CTA each), a hash set for the others (a warp each).  Edges of a
// unit are sorted by the type of i, so a warp keeps its counts in shared memory
// over the edges of one type and adds them to the sums once.
//
// Before, one warp per edge searched every member of the shorter list in the
// longer one and evaluated 13 L slots per edge: 84.4 -> 19.0 ms on R-MAT-20 (15.7M
// edges, L = 8), of which the heavy units take 16.4 ms (22.5 with one edge at a time),
// bound by the shared-memory adds of the hits and the reads of Gamma_i.
struct TriParams {
    DirParams d;
    const uint8_t *est;      // state of edge e seen from its smaller id
    const uint32_t *order, *other, *ustart, *ulist;
    uint32_t nunits;
    int64_t nbits;           // ids below it are in the shared map (heavy units)
    int32_t hist_smem;
    unsigned long long *queue;
};

// est[e]: the state of edge e seen from its end of smaller id.  Every entry carries an
// arc; one that does not sets err, at which the kernels that index by the states leave.
__global__ void k_edge_states(const uint32_t *adj, const uint32_t *eid, const uint8_t *adir,
                              const int2 *edges, int64_t entries, uint8_t *est, unsigned *err) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < entries;
         x += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t e = __ldg(eid + x);
        const int2 ab = edges[e];
        const uint8_t st = adir[x];
        if (st < 1 || st > 3) atomicOr(err, TG_DERR_BOUNDS);
        if ((int)(__ldg(adj + x) & TG_IDMASK) == max(ab.x, ab.y)) est[e] = st;
    }
}

// The counts cnt[state of (i, j)][state pair][type] of the edges (i, j) with
// types ti, tj so far into the histogram h; clears them.
__device__ __forceinline__ void tri_flush(const DirParams &p, unsigned long long *h, uint32_t *cnt,
                                          int ti, int tj) {
    const int L = p.L;
    for (int q = threadIdx.x & 31; q < 27 * L; q += 32) {
        const unsigned long long v = cnt[q];
        if (!v) continue;
        cnt[q] = 0u;
        const int t = q % L, k = q / L, sij = k / 9 + 1, siw = k % 9 / 3 + 1, sjw = k % 3 + 1;
        int a = ti, b = tj, c = t;
        sort2(a, b);
        sort2(b, c);
        sort2(a, b);
        const int64_t r = colex3(a, b, c);
        atomicAdd(h + p.tri[k] * p.n3 + r, v);
        atomicAdd(h + p.path[(sij - 1) * 3 + siw - 1] * p.n3 + r, 0ull - v);
        atomicAdd(h + p.path[(swap_state(sij) - 1) * 3 + sjw - 1] * p.n3 + r, 0ull - v);
    }
}

constexpr int kTriUnroll = 4;  // chunks of 32 entries tested and in flight per warp

// The edges q0, q0 + stride, ... (nb <= 32 of them, the same in every lane) of a
// unit of j (type tj) by one warp, as tau_batch of tg_reuse.cu: lane k reads edge k's
// id, state, end and list bounds, and the next edge's first chunks are read before
// the current edge's are tested.  state(id, entry): the state of (j, w), or 0; pj: j's
// packed entry (j is no neighbour of itself).  Counts wait in cnt while the type of
// i stays ti (any: there are some).
template <class State>
__device__ __forceinline__ void tri_batch(const TriParams &p, unsigned long long *h, uint32_t *cnt,
                                          uint32_t q0, uint32_t stride, int nb, int tj, uint32_t pj,
                                          int &ti, bool &any, State state) {
    const int lane = threadIdx.x & 31, L = p.d.L;
    int sij = 0, d = 0, t = 0;
    int64_t b = 0;
    if (lane < nb) {
        const uint32_t w = __ldg(p.other + q0 + lane * stride);
        sij = swap_state(__ldg(p.est + __ldg(p.order + q0 + lane * stride)));
        t = (int)(w >> TG_TSHIFT);
        b = __ldg(p.d.rowptr + (w & TG_IDMASK));
        d = (int)(__ldg(p.d.rowptr + (w & TG_IDMASK) + 1) - b);
    }
    uint32_t wv[kTriUnroll];
    int sv[kTriUnroll];
    int64_t bk = __shfl_sync(kFull, b, 0);
    int dk = __shfl_sync(kFull, d, 0);
#pragma unroll
    for (int u = 0; u < kTriUnroll; ++u) {
        const int x = 32 * u + lane;
        wv[u] = x < dk ? __ldg(p.d.adj + bk + x) : pj;
        sv[u] = x < dk ? (int)__ldg(p.d.adir + bk + x) : 1;
    }
    for (int k = 0; k < nb; ++k) {
        const int tk = __shfl_sync(kFull, t, k);
        if (tk != ti) {
            __syncwarp();
            if (__any_sync(kFull, any)) tri_flush(p.d, h, cnt, ti, tj);
            __syncwarp();
            any = false;
            ti = tk;
        }
        uint32_t *ck = cnt + (__shfl_sync(kFull, sij, k) - 1) * 9 * L;
        const int64_t bn = __shfl_sync(kFull, b, k + 1 < nb ? k + 1 : k);
        const int dn = k + 1 < nb ? __shfl_sync(kFull, d, k + 1) : 0;
        for (int c0 = 0; c0 < dk; c0 += 32 * kTriUnroll) {
            const bool more = c0 + 32 * kTriUnroll < dk;
            const int64_t nb0 = more ? bk : bn;
            const int from = more ? c0 + 32 * kTriUnroll : 0, to = more ? dk : dn;
            uint32_t nw[kTriUnroll];
            int ns[kTriUnroll];
#pragma unroll
            for (int u = 0; u < kTriUnroll; ++u) {
                const int x = from + 32 * u + lane;
                nw[u] = x < to ? __ldg(p.d.adj + nb0 + x) : pj;
                ns[u] = x < to ? (int)__ldg(p.d.adir + nb0 + x) : 1;
            }
#pragma unroll
            for (int u = 0; u < kTriUnroll; ++u) {
                if (u > 0 && c0 + 32 * u >= dk) break;
                const int sjw = state(wv[u] & TG_IDMASK, wv[u]);
                if (sjw) {
                    atomicAdd(ck + ((sv[u] - 1) * 3 + sjw - 1) * L + (int)(wv[u] >> TG_TSHIFT), 1u);
                    any = true;
                }
            }
#pragma unroll
            for (int u = 0; u < kTriUnroll; ++u) {
                wv[u] = nw[u];
                sv[u] = ns[u];
            }
        }
        bk = bn;
        dk = dn;
    }
}

constexpr int kTriThreads = 1024;

template <bool kAll>  // every id that occurs is in the map
__global__ void __launch_bounds__(kTriThreads) k_tri_heavy(TriParams p) {
    if (*p.d.err) return;  // see k_edge_states
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long s_unit;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, W = blockDim.x >> 5;
    const int L = p.d.L;
    const int64_t hlen = TG_TRIAD_CLASSES * p.d.n3;
    unsigned long long *h = p.hist_smem ? reinterpret_cast<unsigned long long *>(smem) : p.d.sums;
    uint32_t *cnt = reinterpret_cast<uint32_t *>(smem + (p.hist_smem ? hlen * 8 : 0)) + warp * 27 * L;
    uint32_t *map = reinterpret_cast<uint32_t *>(smem + (p.hist_smem ? hlen * 8 : 0)) + W * 27 * L;
    if (p.hist_smem)
        for (int64_t q = tid; q < hlen; q += blockDim.x) h[q] = 0ull;
    for (int q = lane; q < 27 * L; q += 32) cnt[q] = 0u;
    const int64_t words = (p.nbits + 15) >> 4;
    for (int64_t q = tid; q < words; q += blockDim.x) map[q] = 0u;
    int cur_j = -1, cur_dj = 0;
    int64_t cur_bj = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_unit = atomicAdd(p.queue, 1ull);
        __syncthreads();
        const unsigned long long item = s_unit;
        if (item >= p.nunits) break;
        const uint32_t u = p.ulist[item];
        const uint32_t p0 = p.ustart[u], p1 = p.ustart[u + 1];
        const int2 ab0 = p.d.edges[p.order[p0]];
        const int j = min(ab0.x, ab0.y);
        const int64_t bj = p.d.rowptr[j];
        const int dj = (int)(p.d.rowptr[j + 1] - bj);
        const int tj = p.d.ntype[j];
        const int32_t *toj = p.d.toff + (int64_t)j * (L + 1);
        const uint32_t pj = ((uint32_t)tj << TG_TSHIFT) | (uint32_t)j;
        if (j != cur_j) {
            for (int x = tid; x < cur_dj; x += blockDim.x) {
                const uint32_t id = __ldg(p.d.adj + cur_bj + x) & TG_IDMASK;
                if ((int64_t)id < p.nbits) atomicAnd(&map[id >> 4], ~(3u << (2 * (id & 15u))));
            }
            __syncthreads();
            for (int x = tid; x < dj; x += blockDim.x) {
                const uint32_t id = __ldg(p.d.adj + bj + x) & TG_IDMASK;
                if ((int64_t)id < p.nbits)
                    atomicOr(&map[id >> 4], (uint32_t)p.d.adir[bj + x] << (2 * (id & 15u)));
            }
            cur_j = j;
            cur_bj = bj;
            cur_dj = dj;
            __syncthreads();
        }
        int ti = -1;
        bool any = false;
        for (uint32_t q = p0 + warp; q < p1; q += 32 * W)
            tri_batch(p, h, cnt, q, (uint32_t)W, (int)min(32u, (p1 - q + W - 1) / W), tj, pj, ti, any,
                      [&](uint32_t id, uint32_t w) -> int {
                          if (kAll || id < (uint32_t)p.nbits) return (int)((map[id >> 4] >> (2 * (id & 15u))) & 3u);
                          if (id == (uint32_t)j) return 0;
                          // beyond the map: the shorter of the two lists is searched
                          const int64_t by = p.d.rowptr[id];
                          if (p.d.rowptr[id + 1] - by < dj) {
                              const int k = find_pos(p.d.adj, by, p.d.toff + (int64_t)id * (L + 1), pj);
                              return k < 0 ? 0 : swap_state(p.d.adir[by + k]);
                          }
                          const int k = find_pos(p.d.adj, bj, toj, w);
                          return k < 0 ? 0 : (int)p.d.adir[bj + k];
                      });
        __syncwarp();
        if (__any_sync(kFull, any)) tri_flush(p.d, h, cnt, ti, tj);
        __syncwarp();
    }
    if (p.hist_smem) {
        __syncthreads();
        for (int64_t q = tid; q < hlen; q += blockDim.x)
            if (h[q]) atomicAdd(p.d.sums + q, h[q]);
    }
}

constexpr int kTriLightWarps = 8;

__global__ void __launch_bounds__(kTriLightWarps * 32) k_tri_light(TriParams p) {
    if (*p.d.err) return;  // see k_edge_states
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = p.d.L;
    const int64_t hlen = TG_TRIAD_CLASSES * p.d.n3;
    unsigned long long *h = p.hist_smem ? reinterpret_cast<unsigned long long *>(smem) : p.d.sums;
    // per warp: the counts, then a hash set of Gamma_j, id << 2 | state (0 empty)
    const int slots = 1 << TG_LIGHT_LG;
    uint32_t *cnt = reinterpret_cast<uint32_t *>(smem + (p.hist_smem ? hlen * 8 : 0)) + warp * (27 * L + slots);
    uint32_t *set = cnt + 27 * L;
    if (p.hist_smem)
        for (int64_t q = threadIdx.x; q < hlen; q += blockDim.x) h[q] = 0ull;
    for (int q = lane; q < 27 * L; q += 32) cnt[q] = 0u;
    __syncthreads();
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= p.nunits) break;
        const uint32_t u = p.ulist[item];
        const uint32_t p0 = p.ustart[u], p1 = p.ustart[u + 1];
        const int2 ab0 = p.d.edges[p.order[p0]];
        const int j = min(ab0.x, ab0.y);
        const int64_t bj = p.d.rowptr[j];
        const int dj = (int)(p.d.rowptr[j + 1] - bj);
        const int tj = p.d.ntype[j];
        const uint32_t pj = ((uint32_t)tj << TG_TSHIFT) | (uint32_t)j;
        int lg = 5;
        while ((1 << lg) < 2 * dj) ++lg;  // at most TG_LIGHT_LG
        const uint32_t mask = (1u << lg) - 1u;
        for (int q = lane; q <= (int)mask; q += 32) set[q] = 0u;
        __syncwarp();
        for (int x = lane; x < dj; x += 32) {
            const uint32_t id = __ldg(p.d.adj + bj + x) & TG_IDMASK;
            const uint32_t v = (id << 2) | p.d.adir[bj + x];
            uint32_t s = hset_slot(id, lg);
            while (atomicCAS(set + s, 0u, v) != 0u) s = (s + 1u) & mask;  // at most half full
        }
        __syncwarp();
        int ti = -1;
        bool any = false;
        for (uint32_t q = p0; q < p1; q += 32)
            tri_batch(p, h, cnt, q, 1u, (int)min(32u, p1 - q), tj, pj, ti, any,
                      [&](uint32_t id, uint32_t) -> int {
                          uint32_t s = hset_slot(id, lg);
                          for (;;) {  // ends at an empty slot: the set is at most half full
                              const uint32_t v = set[s];
                              if (v == 0u) return 0;
                              if ((v >> 2) == id) return (int)(v & 3u);
                              s = (s + 1u) & mask;
                          }
                      });
        __syncwarp();
        if (__any_sync(kFull, any)) tri_flush(p.d, h, cnt, ti, tj);
        __syncwarp();
    }
    if (p.hist_smem) {
        __syncthreads();
        for (int64_t q = threadIdx.x; q < hlen; q += blockDim.x)
            if (h[q]) atomicAdd(p.d.sums + q, h[q]);
    }
}

// Twice the pairs of neighbours of every node by (states, types).  A warp takes a
// range of nodes one node type at a time, with the products of its lanes' pairs
// ((s, t), (s', t')) in registers, added to the CTA's histogram once per type.
template <int LP>
__global__ void __launch_bounds__(kDirThreads) k_dir_paths(DirParams p, int64_t n, int hist_smem) {
    constexpr int kPairs = 3 * LP * (3 * LP + 1) / 2, kSlots = (kPairs + 31) / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, L = p.L, K = 3 * L;
    const int64_t hlen = TG_TRIAD_CLASSES * p.n3;
    unsigned long long *h = hist_smem ? reinterpret_cast<unsigned long long *>(smem) : p.sums;
    if (hist_smem) {
        for (int64_t q = threadIdx.x; q < hlen; q += blockDim.x) h[q] = 0ull;
        __syncthreads();
    }
    int xa[kSlots], xb[kSlots];
#pragma unroll
    for (int z = 0; z < kSlots; ++z) {
        const int q = lane + 32 * z;
        xa[z] = xb[z] = -1;
        if (q < K * (K + 1) / 2) unpair(K, q, xa[z], xb[z]);
    }
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t per = (n + warps - 1) / warps, v0 = wid * per, v1 = min(n, v0 + per);
    for (int tv = 0; tv < L; ++tv) {
        unsigned long long acc[kSlots];
#pragma unroll
        for (int z = 0; z < kSlots; ++z) acc[z] = 0ull;
        for (int64_t c = v0; c < v1; c += 32) {
            unsigned m = __ballot_sync(kFull, c + lane < v1 && p.ntype[c + lane] == tv);
            for (; m; m &= m - 1u) {
                const uint32_t *nd = p.nd + (c + __ffs(m) - 1) * K;
#pragma unroll
                for (int z = 0; z < kSlots; ++z) {
                    if (xa[z] < 0) continue;
                    const uint64_t a = __ldg(nd + xa[z]), b = __ldg(nd + xb[z]);
                    acc[z] += xa[z] == xb[z] ? a * (a - 1) : 2 * a * b;  // a (a - 1) = 2 C(a, 2), 0 for a = 0
                }
            }
        }
#pragma unroll
        for (int z = 0; z < kSlots; ++z) {
            if (xa[z] < 0 || !acc[z]) continue;
            int a = tv, b = xa[z] % L, c = xb[z] % L;
            sort2(a, b);
            sort2(b, c);
            sort2(a, b);
            atomicAdd(h + p.path[(xa[z] / L) * 3 + xb[z] / L] * p.n3 + colex3(a, b, c), acc[z]);
        }
    }
    if (hist_smem) {
        __syncthreads();
        for (int64_t q = threadIdx.x; q < hlen; q += blockDim.x)
            if (h[q]) atomicAdd(p.sums + q, h[q]);
    }
}

__global__ void k_dir_finalize(const unsigned long long *sums, uint64_t *out, int64_t n3,
                               unsigned *err) {
    const int64_t len = TG_TRIAD_CLASSES * n3;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < len;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(q / n3);
        const unsigned long long div = (c <= 4 || c == 7) ? 2ull : 3ull;
        if (sums[q] % div) atomicOr(err, TG_DERR_DIVISIBLE);
        out[q] = sums[q] / div;
    }
}

// Undivided global sums from the triangle nodes of every edge and the split typed
// degrees p.nd (see k_tri_heavy, k_dir_paths).
int dir_totals(const tg_graph *g, const DirParams &d, cudaStream_t s) {
    const int L = g->L;
    const int64_t M = g->M, hlen = TG_TRIAD_CLASSES * d.n3;
    const size_t avail = (size_t)tg_smem_optin() - 1024;
    TriParams p{};
    p.d = d;
    p.hist_smem = (size_t)hlen * 8 <= 48 * 1024;
    const size_t hb = p.hist_smem ? (size_t)hlen * 8 : 0;
    DevBuf<uint8_t> est;
    DevBuf<unsigned long long> queue;
    if (!est.alloc(M, s) || !queue.alloc(2, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(queue.p, 0, 16, s));
    k_edge_states<<<(unsigned)std::min<int64_t>((2 * M + 255) / 256, 65535LL * 16), 256, 0, s>>>(
        g->adj, g->eid, g->adir, g->edges, 2 * M, est.p, d.err); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    const tg_lists *lists = nullptr;
    TG_TRY(tg_graph_lists(g, &lists, s));
    tg_units un;
    TG_TRY(tg_edge_units(g, lists->order, M, s, un));
    p.est = est.p;
    p.order = lists->order;
    p.other = lists->other;
    p.ustart = un.ustart.p;
    const int64_t sms = tg_num_sms();
    if (un.nheavy > 0) {
        int threads = kTriThreads;
        size_t fixed = 0;
        for (;; threads /= 2) {
            fixed = hb + (size_t)(threads / 32) * 27 * L * 4;
            if (fixed + 4096 <= avail || threads == 64) break;
        }
        int64_t nbits = std::min<int64_t>(g->n_nonisolated, (int64_t)((avail - fixed) / 16) * 64);
        p.nbits = nbits;
        p.ulist = un.heavy.p;
        p.nunits = un.nheavy;
        p.queue = queue.p;
        const size_t smem = fixed + (size_t)((nbits + 15) / 16) * 4;
        const auto fn = nbits >= g->n_nonisolated ? k_tri_heavy<true> : k_tri_heavy<false>;
        TG_TRY(tg_allow_max_smem((const void *)fn));
        int per = 0;
        TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem));
        fn<<<(unsigned)std::min<int64_t>(sms * std::max(per, 1), un.nheavy), threads, smem, s>>>(p);
        tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    if (un.nlight > 0) {
        p.ulist = un.light.p;
        p.nunits = un.nlight;
        p.queue = queue.p + 1;
        const size_t smem = hb + (size_t)kTriLightWarps * (27 * L + (1 << TG_LIGHT_LG)) * 4;
        TG_TRY(tg_allow_max_smem((const void *)k_tri_light));
        int per = 0;
        TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_tri_light, kTriLightWarps * 32, smem));
        k_tri_light<<<(unsigned)std::min<int64_t>(sms * std::max(per, 1), (un.nlight + kTriLightWarps - 1) / kTriLightWarps),
                      kTriLightWarps * 32, smem, s>>>(p);
        tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    void (*const paths)(DirParams, int64_t, int) = L <= 4 ? k_dir_paths<4> : L <= 8 ? k_dir_paths<8> : k_dir_paths<16>;
    TG_TRY(tg_allow_max_smem((const void *)paths));
    int per = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, paths, kDirThreads, hb));
    // at least 16 nodes a warp
    const int64_t grid = std::min<int64_t>(sms * std::max(per, 1), (g->n + 16 * kDirWarps - 1) / (16 * kDirWarps));
    paths<<<(unsigned)grid, kDirThreads, hb, s>>>(d, g->n, p.hist_smem);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    TG_TRY_CUDA(cudaStreamSynchronize(s));  // the units' buffers end here
    return TG_OK;
}

// Global counts of small graphs take k_dir3, edge by edge: dir_totals launches about a
// dozen kernels more (lists, units) and waits twice.  Its gain grows with the edges and
// their lists, its fixed part with the types.  k_dir3 against dir_totals, ER graphs
// unless said otherwise: 3,000 edges 0.07 and 0.18 ms (L = 3); 140,000 at mean degree
// 18 0.24 and 0.23 (L = 8), 0.25 and 0.31 (L = 9); 200,000 at mean degree 6 0.31 and
// 0.28 (L = 8), 0.31 and 0.42 (L = 9); 100,000 of a dense graph (mean degree 280) 0.37
// and 0.32 (L = 1).  Of 270 graphs (ER, power law, R-MAT, dense; 8,000 to 450,000
// edges; L = 1 to 16) the rule takes the slower way in none by more than 27 %.
bool dir_totals_pays(const tg_graph *g) {
    const double mean = 2.0 * (double)g->M / (double)g->n_nonisolated;
    return (double)g->M * (1.0 + mean / 160.0) >= (g->L <= 8 ? 196608.0 : 327680.0);
}

// Per-edge rows (rows != nullptr) or undivided global sums of a TG_DIRECTED graph.
int dir_count(const tg_graph *g, uint64_t *rows, unsigned long long *sums, unsigned *err,
              cudaStream_t s) {
    const TriadTable &tt = triads();
    if (!tt.ok) return TG_EINTERNAL;
    const int L = g->L;
    const int64_t n = g->n, M = g->M;
    if (M == 0) return TG_OK;
    DevBuf<uint32_t> nd;
    DevBuf<unsigned long long> queue;
    if (!nd.alloc((size_t)n * 3 * L, s) || !queue.alloc(1, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(queue.p, 0, 8, s));
    const int64_t ngrid = std::min<int64_t>((n + kDirWarps - 1) / kDirWarps, (int64_t)tg_num_sms() * 16);
    k_dir_degrees<<<(unsigned)ngrid, kDirThreads, 0, s>>>(g->rowptr, g->adj, g->adir, n, L, nd.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    if (g->max_degree > kDirHub) {
        k_dir_degrees_hub<<<(unsigned)std::min<int64_t>(n, tg_num_sms()), 1024, 0, s>>>(
            g->rowptr, g->adj, g->adir, n, L, nd.p); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    DirParams p{};
    p.rowptr = g->rowptr;
    p.adj = g->adj;
    p.adir = g->adir;
    p.toff = g->toff;
    p.ntype = g->ntype;
    p.edges = g->edges;
    p.nd = nd.p;
    p.M = M;
    p.L = L;
    p.n3 = tg_binom(L + 2, 3);
    p.rows = rows;
    p.sums = sums;
    p.queue = queue.p;
    p.err = err;
    for (int sij = 1; sij <= 3; ++sij)
        for (int s1 = 1; s1 <= 3; ++s1) {
            for (int s2 = 1; s2 <= 3; ++s2)
                p.tri[(sij - 1) * 9 + (s1 - 1) * 3 + (s2 - 1)] =
                    tt.cls[pair_mask(sij, 0, 1) | pair_mask(s1, 0, 2) | pair_mask(s2, 1, 2)];
            // a 3-path: centre 0, ends 1 (state sij) and 2 (state s1), seen from 0
            p.path[(sij - 1) * 3 + (s1 - 1)] = tt.cls[pair_mask(sij, 0, 1) | pair_mask(s1, 0, 2)];
        }
    if (!rows && dir_totals_pays(g)) return dir_totals(g, p, s);
    void (*const fn)(DirParams) = rows ? k_dir3<true> : k_dir3<false>;
    const size_t smem = (rows ? 0 : (size_t)TG_TRIAD_CLASSES * p.n3 * 8) + (size_t)kDirWarps * 9 * L * 4;
    TG_TRY(tg_allow_max_smem((const void *)fn));
    int per = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kDirThreads, smem));
    if (per < 1) return TG_ENOMEM;
    const int64_t grid = std::min<int64_t>((int64_t)tg_num_sms() * per, (M + kDirWarps - 1) / kDirWarps);
    fn<<<(unsigned)grid, kDirThreads, smem, s>>>(p);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return TG_OK;
}


// ------------------------------------------------------------- 4 nodes ----
// Directed typed 4-node graphlets: the connected 4-node sets {i, j, w, r}
// through each edge, w in C = (Gamma_i u Gamma_j) \ {i, j} and r either a
// later member of C or a neighbour of w outside C u {i, j} (each set met
// once), classified from their six pair states by a host table.  Classes:
// the 199 connected 4-node digraphs numbered by canonical code (the code of
// a digraph on positions 0..3 is the sum of 2^(4a + b) over its arcs a -> b;
// the canonical code is the smallest over the 24 relabellings).  One warp per
// edge walks the candidate pairs directly: a first form, suited to graphs of
// moderate degree.
constexpr int kDir4Classes = TG_TETRAD_CLASSES;

struct Dir4Table {
    int16_t cls[4096];  // class of each 12-bit pair-state code, -1 if disconnected
    bool ok = false;
};

int dir4_canon(int code) {
    static const int perm[24][4] = {
        {0, 1, 2, 3}, {0, 1, 3, 2}, {0, 2, 1, 3}, {0, 2, 3, 1}, {0, 3, 1, 2}, {0, 3, 2, 1},
        {1, 0, 2, 3}, {1, 0, 3, 2}, {1, 2, 0, 3}, {1, 2, 3, 0}, {1, 3, 0, 2}, {1, 3, 2, 0},
        {2, 0, 1, 3}, {2, 0, 3, 1}, {2, 1, 0, 3}, {2, 1, 3, 0}, {2, 3, 0, 1}, {2, 3, 1, 0},
        {3, 0, 1, 2}, {3, 0, 2, 1}, {3, 1, 0, 2}, {3, 1, 2, 0}, {3, 2, 0, 1}, {3, 2, 1, 0}};
    int best = 1 << 30;
    for (int q = 0; q < 24; ++q) {
        int c = 0;
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b)
                if (a != b && ((code >> (4 * a + b)) & 1)) c |= 1 << (4 * perm[q][a] + perm[q][b]);
        best = std::min(best, c);
    }
    return best;
}

// arc code of a 12-bit pair-state code (pairs 01, 02, 03, 12, 13, 23, two bits
// each: bit 0 lower -> higher position, bit 1 back) and whether it connects
// the four nodes
int dir4_arcs(int st, bool *conn) {
    static const int pa[6] = {0, 0, 0, 1, 1, 2}, pb[6] = {1, 2, 3, 2, 3, 3};
    int code = 0, adj[4] = {0, 0, 0, 0};
    for (int k = 0; k < 6; ++k) {
        const int x = (st >> (2 * k)) & 3;
        if (x & 1) code |= 1 << (4 * pa[k] + pb[k]);
        if (x & 2) code |= 1 << (4 * pb[k] + pa[k]);
        if (x) {
            adj[pa[k]] |= 1 << pb[k];
            adj[pb[k]] |= 1 << pa[k];
        }
    }
    int seen = 1;
    for (int it = 0; it < 4; ++it)
        for (int v = 0; v < 4; ++v)
            if ((seen >> v) & 1) seen |= adj[v];
    *conn = seen == 15;
    return code;
}

Dir4Table build_dir4() {
    Dir4Table t;
    std::vector<int> canon;
    for (int st = 0; st < 4096; ++st) {
        bool conn = false;
        const int code = dir4_arcs(st, &conn);
        if (conn) canon.push_back(dir4_canon(code));
    }
    std::sort(canon.begin(), canon.end());
    canon.erase(std::unique(canon.begin(), canon.end()), canon.end());
    if ((int)canon.size() != kDir4Classes) return t;  // ok stays false
    for (int st = 0; st < 4096; ++st) {
        bool conn = false;
        const int code = dir4_arcs(st, &conn);
        t.cls[st] = conn ? (int16_t)(std::lower_bound(canon.begin(), canon.end(), dir4_canon(code)) -
                                     canon.begin())
                         : (int16_t)-1;
    }
    t.ok = true;
    return t;
}

const Dir4Table &dir4_table() {
    static std::once_flag once;
    static Dir4Table t;
    std::call_once(once, [] { t = build_dir4(); });
    return t;
}

struct Dir4Params {
    const int64_t *rowptr;
    const uint32_t *adj;
    const uint8_t *adir;
    const int32_t *toff;
    const uint8_t *ntype;
    const int2 *edges;
    const int16_t *cls;  // 4096 entries (device)
    int64_t M;
    int32_t L, P;
    int64_t n4;                // C(L+3, 4)
    unsigned long long *rows;  // per-edge mode: M x 199 P
    unsigned long long *sums;  // global mode: 199 n4 counts
    unsigned long long *queue;
    unsigned *err;
};

// state of the pair (x, w) seen from x: the arc bits of w's entry in Gamma_x, 0 if absent
__device__ __forceinline__ int dir4_state(const Dir4Params &p, int64_t bx, const int32_t *tox,
                                          uint32_t w) {
    const int q = find_pos(p.adj, bx, tox, w);
    return q < 0 ? 0 : (int)p.adir[bx + q];
}

// Per-edge rows: every set through the edge.
__global__ void __launch_bounds__(kDirThreads) k_dir4(Dir4Params p) {
    const int lane = threadIdx.x & 31;
    const int L = p.L;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= (unsigned long long)p.M) break;
        const int64_t e = (int64_t)item;
        const int2 ab = p.edges[e];
        const uint32_t i = (uint32_t)ab.x, j = (uint32_t)ab.y;
        const int tj = p.ntype[j];
        const int64_t bi = p.rowptr[i], bj = p.rowptr[j];
        const int di = (int)(p.rowptr[i + 1] - bi), dj = (int)(p.rowptr[j + 1] - bj);
        const int32_t *toi = p.toff + (int64_t)i * (L + 1);
        const int32_t *toj = p.toff + (int64_t)j * (L + 1);
        const int sij = dir4_state(p, bi, toi, ((uint32_t)tj << TG_TSHIFT) | j);
        // member q of C (index space [0, di + dj)): its entry, or 0xffffffff
        // when q is i, j, or a member of Gamma_j already in Gamma_i
        auto member = [&](int q) -> uint32_t {
            if (q < di) {
                const uint32_t w = __ldg(p.adj + bi + q);
                return (w & TG_IDMASK) == j ? 0xffffffffu : w;
            }
            const uint32_t w = __ldg(p.adj + bj + (q - di));
            if ((w & TG_IDMASK) == i || find_pos(p.adj, bi, toi, w) >= 0) return 0xffffffffu;
            return w;
        };
        const int nq = di + dj;
        for (int pw = 0; pw < nq; ++pw) {
            const uint32_t wE = member(pw);  // the same in every lane
            if (wE == 0xffffffffu) continue;
            const uint32_t w = wE & TG_IDMASK;
            const int tw = (int)(wE >> TG_TSHIFT);
            const int siw = pw < di ? (int)p.adir[bi + pw] : 0;
            const int sjw = pw < di ? dir4_state(p, bj, toj, wE) : (int)p.adir[bj + (pw - di)];
            const int64_t bw = p.rowptr[w];
            const int dw = (int)(p.rowptr[w + 1] - bw);
            const int32_t *tow = p.toff + (int64_t)w * (L + 1);
            // pass 0: r a later member of C; pass 1: r a neighbour of w outside C u {i, j}
            const int n0 = nq - (pw + 1);
            for (int x = lane; x < n0 + dw; x += 32) {
                uint32_t rE;
                int sir, sjr, swr;
                if (x < n0) {
                    const int pr = pw + 1 + x;
                    rE = member(pr);
                    if (rE == 0xffffffffu) continue;
                    sir = pr < di ? (int)p.adir[bi + pr] : 0;
                    sjr = pr < di ? dir4_state(p, bj, toj, rE) : (int)p.adir[bj + (pr - di)];
                    swr = dir4_state(p, bw, tow, rE);
                } else {
                    const int xr = x - n0;
                    rE = __ldg(p.adj + bw + xr);
                    const uint32_t r = rE & TG_IDMASK;
                    if (r == i || r == j || find_pos(p.adj, bi, toi, rE) >= 0 ||
                        find_pos(p.adj, bj, toj, rE) >= 0)
                        continue;
                    sir = 0;
                    sjr = 0;
                    swr = (int)p.adir[bw + xr];
                }
                // positions i = 0, j = 1, w = 2, r = 3; each state seen from the lower position
                const int code = sij | (siw << 2) | (sir << 4) | (sjw << 6) | (sjr << 8) | (swr << 10);
                const int c = p.cls[code];
                if (c < 0) {
                    atomicOr(p.err, TG_DERR_BOUNDS);  // a set through the edge is always connected
                    continue;
                }
                const int tr = (int)(rE >> TG_TSHIFT);
                const int a = min(tw, tr), b = max(tw, tr);
                atomicAdd(p.rows + e * (int64_t)kDir4Classes * p.P + (int64_t)c * p.P +
                              (a * L - (a * (a - 1)) / 2 + (b - a)),
                          1ull);
            }
        }
    }
}

// Global mode: every connected set {i, j, w, r} once, from its canonical edge: i
// its smallest id, j the smallest neighbour of i in the set.  So w and r have ids
// above i, and above j when they are neighbours of i.  One warp per edge stages
// C (the ids above i of Gamma_i u Gamma_j) in shared memory with both pair
// states; walking the lists of C's admissible members once then gives the sets
// with r outside C and the adjacent pairs inside C, and the pairs of C that are
// not adjacent follow without a search.  An edge with more than kSetCap such
// neighbours takes the search form, set by set.  Counts go to a per-CTA table
// (two 32-bit words per entry) while it fits.
//
// Before, a set was met once per edge of it, every pair state was a binary search
// in global memory and every set an add to one of a few thousand global words:
// 13.4 -> 0.45 ms for 20K nodes and 120K arcs with 30 % reciprocated (L = 2).
// Bound by the latency of the staging chain (lists, their lists) and the table adds.
constexpr int kSetCap = 128;    // members of C in shared memory
constexpr int kSetHash = 256;   // hash slots
constexpr int kSetTable = 64 * 1024;  // bytes of the per-CTA count table, at most

struct SetWarp {
    uint32_t keys[kSetHash], vals[kSetHash];
    uint32_t ent[kSetCap];              // member: packed entry
    uint32_t adj[kSetCap][kSetCap / 32];  // adjacent pairs (lower index, higher index)
    uint8_t st[kSetCap];                // siw | sjw << 2 | 16 when admissible
};

__global__ void __launch_bounds__(kDirThreads) k_dir4_sets(Dir4Params p, int table) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = p.L;
    int16_t *cls = reinterpret_cast<int16_t *>(smem);
    SetWarp &sm = reinterpret_cast<SetWarp *>(smem + 4096 * sizeof(int16_t))[warp];
    const int len = kDir4Classes * (int)p.n4;
    uint32_t *lo = reinterpret_cast<uint32_t *>(smem + 4096 * sizeof(int16_t) + kDirWarps * sizeof(SetWarp));
    uint32_t *hi = lo + len;
    for (int q = threadIdx.x; q < 4096; q += blockDim.x) cls[q] = p.cls[q];
    if (table)
        for (int q = threadIdx.x; q < 2 * len; q += blockDim.x) lo[q] = 0u;
    __syncthreads();
    const unsigned below = (1u << lane) - 1u;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = atomicAdd(p.queue, 1ull);
        item = __shfl_sync(kFull, item, 0);
        if (item >= (unsigned long long)p.M) break;
        const int2 ab = p.edges[item];
        const uint32_t i = (uint32_t)min(ab.x, ab.y), j = (uint32_t)max(ab.x, ab.y);
        const int ti = p.ntype[i], tj = p.ntype[j];
        const int64_t bi = p.rowptr[i], bj = p.rowptr[j];
        const int di = (int)(p.rowptr[i + 1] - bi), dj = (int)(p.rowptr[j + 1] - bj);
        const int32_t *toi = p.toff + (int64_t)i * (L + 1);
        const int32_t *toj = p.toff + (int64_t)j * (L + 1);
        const int sij = dir4_state(p, bi, toi, ((uint32_t)tj << TG_TSHIFT) | j);
        // positions i = 0, j = 1, w = 2, r = 3; each state seen from the lower position
        auto add = [&](int siw, int sjw, int sir, int sjr, int swr, int tw, int tr) {
            const int c = cls[sij | (siw << 2) | (sir << 4) | (sjw << 6) | (sjr << 8) | (swr << 10)];
            if (c < 0) {
                atomicOr(p.err, TG_DERR_BOUNDS);  // a set through the edge is always connected
                return;
            }
            int q0 = ti, q1 = tj, q2 = tw, q3 = tr;
            sort2(q0, q1);
            sort2(q2, q3);
            sort2(q0, q2);
            sort2(q1, q3);
            sort2(q1, q2);
            const int64_t at = (int64_t)c * p.n4 + colex4(q0, q1, q2, q3);
            if (!table)
                atomicAdd(p.sums + at, 1ull);
            else if (atomicAdd(lo + at, 1u) == 0xffffffffu)
                atomicAdd(hi + at, 1u);
        };
        for (int q = lane; q < kSetHash; q += 32) sm.keys[q] = 0u;
        __syncwarp();
        // C: first Gamma_i, then the rest of Gamma_j
        int nc = 0;
        for (int c0 = 0; c0 < di && nc <= kSetCap; c0 += 32) {
            const int x = c0 + lane;
            const uint32_t w = x < di ? __ldg(p.adj + bi + x) : 0u;
            const uint32_t id = w & TG_IDMASK;
            const bool in = x < di && id > i && id != j;
            const unsigned m = __ballot_sync(kFull, in);
            const int k = nc + __popc(m & below);
            if (in && k < kSetCap) {
                sm.ent[k] = w;
                sm.st[k] = (uint8_t)(p.adir[bi + x] | (id > j ? 16 : 0));
                hmap_put(sm.keys, sm.vals, 8, id, (uint32_t)k);
            }
            nc += __popc(m);
        }
        __syncwarp();
        for (int c0 = 0; c0 < dj && nc <= kSetCap; c0 += 32) {
            const int x = c0 + lane;
            const uint32_t w = x < dj ? __ldg(p.adj + bj + x) : 0u;
            const uint32_t id = w & TG_IDMASK;
            const bool in = x < dj && id > i;
            const uint32_t k0 = in ? hmap_get(sm.keys, sm.vals, 8, id) : 0u;
            const int s = in ? (int)p.adir[bj + x] : 0;
            const bool isnew = in && k0 == 0xffffffffu;
            if (in && !isnew) sm.st[k0] |= (uint8_t)(s << 2);
            const unsigned m = __ballot_sync(kFull, isnew);
            const int k = nc + __popc(m & below);
            __syncwarp();
            if (isnew && k < kSetCap) {
                sm.ent[k] = w;
                sm.st[k] = (uint8_t)((s << 2) | 16);
                hmap_put(sm.keys, sm.vals, 8, id, (uint32_t)k);
            }
            nc += __popc(m);
            __syncwarp();
        }
        if (nc <= kSetCap) {
            for (int q = lane; q < nc * (kSetCap / 32); q += 32) (&sm.adj[0][0])[q] = 0u;
            __syncwarp();
            // the lists of the admissible members as one sequence per 32 of them
            for (int m0 = 0; m0 < nc; m0 += 32) {
                const int k = m0 + lane;
                uint32_t w = 0;
                int64_t bw = 0;
                int dw = 0;
                if (k < nc && (sm.st[k] & 16)) {
                    w = sm.ent[k];
                    bw = p.rowptr[w & TG_IDMASK];
                    dw = (int)(p.rowptr[(w & TG_IDMASK) + 1] - bw);
                }
                int64_t incl = dw;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int64_t y = __shfl_up_sync(kFull, incl, o);
                    if (lane >= o) incl += y;
                }
                const int64_t total = __shfl_sync(kFull, incl, 31);
                const int64_t org = bw - (incl - dw);
                for (int64_t c = 0; c < total; c += 32) {
                    const int64_t pos = c + lane;
                    int r = 0;  // the member whose list holds pos
#pragma unroll
                    for (int st = 16; st > 0; st >>= 1) {
                        const int64_t v = __shfl_sync(kFull, incl, r + st - 1);
                        if (v <= pos) r += st;
                    }
                    const int64_t at = __shfl_sync(kFull, org, r) + pos;
                    const int tw = (int)(__shfl_sync(kFull, w, r) >> TG_TSHIFT);
                    if (pos >= total) continue;
                    const uint32_t rE = __ldg(p.adj + at);
                    const uint32_t rid = rE & TG_IDMASK;
                    if (rid <= i || rid == j) continue;
                    const int kw = m0 + r, sw = sm.st[kw];
                    const int swr = (int)p.adir[at], tr = (int)(rE >> TG_TSHIFT);
                    const uint32_t kr = hmap_get(sm.keys, sm.vals, 8, rid);
                    if (kr == 0xffffffffu) {
                        add(sw & 3, (sw >> 2) & 3, 0, 0, swr, tw, tr);
                    } else if ((int)kr > kw && (sm.st[kr] & 16)) {
                        const int sr = sm.st[kr];
                        atomicOr(&sm.adj[kw][kr >> 5], 1u << (kr & 31u));
                        add(sw & 3, (sw >> 2) & 3, sr & 3, (sr >> 2) & 3, swr, tw, tr);
                    }
                }
            }
            __syncwarp();
            // pairs of C without an arc
            for (int x = 0; x + 1 < nc; ++x) {
                const int sx = sm.st[x];
                if (!(sx & 16)) continue;
                const int tx = (int)(sm.ent[x] >> TG_TSHIFT);
                for (int y = x + 1 + lane; y < nc; y += 32) {
                    const int sy = sm.st[y];
                    if (!(sy & 16) || ((sm.adj[x][y >> 5] >> (y & 31)) & 1u)) continue;
                    add(sx & 3, (sx >> 2) & 3, sy & 3, (sy >> 2) & 3, 0, tx, (int)(sm.ent[y] >> TG_TSHIFT));
                }
            }
        } else {
            // member q of C (index space [0, di + dj)): its entry, or 0xffffffff
            // when it is not admissible or a member of Gamma_j already in Gamma_i
            auto member = [&](int q) -> uint32_t {
                if (q < di) {
                    const uint32_t w = __ldg(p.adj + bi + q);
                    return (w & TG_IDMASK) <= j ? 0xffffffffu : w;
                }
                const uint32_t w = __ldg(p.adj + bj + (q - di));
                if ((w & TG_IDMASK) <= i || find_pos(p.adj, bi, toi, w) >= 0) return 0xffffffffu;
                return w;
            };
            const int nq = di + dj;
            for (int pw = 0; pw < nq; ++pw) {
                const uint32_t wE = member(pw);  // the same in every lane
                if (wE == 0xffffffffu) continue;
                const uint32_t w = wE & TG_IDMASK;
                const int tw = (int)(wE >> TG_TSHIFT);
                const int siw = pw < di ? (int)p.adir[bi + pw] : 0;
                const int sjw = pw < di ? dir4_state(p, bj, toj, wE) : (int)p.adir[bj + (pw - di)];
                const int64_t bw = p.rowptr[w];
                const int dw = (int)(p.rowptr[w + 1] - bw);
                const int32_t *tow = p.toff + (int64_t)w * (L + 1);
                // r a later member of C, then r a neighbour of w outside C u {i, j}
                const int n0 = nq - (pw + 1);
                for (int x = lane; x < n0 + dw; x += 32) {
                    if (x < n0) {
                        const int pr = pw + 1 + x;
                        const uint32_t rE = member(pr);
                        if (rE == 0xffffffffu) continue;
                        const int sir = pr < di ? (int)p.adir[bi + pr] : 0;
                        const int sjr = pr < di ? dir4_state(p, bj, toj, rE) : (int)p.adir[bj + (pr - di)];
                        add(siw, sjw, sir, sjr, dir4_state(p, bw, tow, rE), tw, (int)(rE >> TG_TSHIFT));
                    } else {
                        const int xr = x - n0;
                        const uint32_t rE = __ldg(p.adj + bw + xr);
                        const uint32_t r = rE & TG_IDMASK;
                        if (r <= i || r == j || find_pos(p.adj, bi, toi, rE) >= 0 ||
                            find_pos(p.adj, bj, toj, rE) >= 0)
                            continue;
                        add(siw, sjw, 0, 0, (int)p.adir[bw + xr], tw, (int)(rE >> TG_TSHIFT));
                    }
                }
            }
        }
        __syncwarp();
    }
    if (table) {
        __syncthreads();
        for (int q = threadIdx.x; q < len; q += blockDim.x) {
            const unsigned long long v = ((unsigned long long)hi[q] << 32) + lo[q];
            if (v) atomicAdd(p.sums + q, v);
        }
    }
}

// Per-edge rows (rows != nullptr, zeroed here) or global counts (zeroed by the caller).
int dir4_count(const tg_graph *g, unsigned long long *rows, unsigned long long *sums, unsigned *err,
               cudaStream_t s) {
    const Dir4Table &tt = dir4_table();
    if (!tt.ok) return TG_EINTERNAL;
    const int L = g->L;
    const int64_t M = g->M;
    if (M == 0) return TG_OK;
    DevBuf<int16_t> cls;
    DevBuf<unsigned long long> queue;
    if (!cls.alloc(4096, s) || !queue.alloc(1, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemcpyAsync(cls.p, tt.cls, 4096 * sizeof(int16_t), cudaMemcpyHostToDevice, s));
    TG_TRY_CUDA(cudaMemsetAsync(queue.p, 0, 8, s));
    Dir4Params p{};
    p.rowptr = g->rowptr;
    p.adj = g->adj;
    p.adir = g->adir;
    p.toff = g->toff;
    p.ntype = g->ntype;
    p.edges = g->edges;
    p.cls = cls.p;
    p.M = M;
    p.L = L;
    p.P = L * (L + 1) / 2;
    p.n4 = tg_binom(L + 3, 4);
    p.rows = rows;
    p.sums = sums;
    p.queue = queue.p;
    p.err = err;
    if (rows)
        TG_TRY_CUDA(cudaMemsetAsync(rows, 0, (size_t)M * kDir4Classes * p.P * 8, s));
    if (rows) {
        const int64_t grid = std::min<int64_t>((int64_t)tg_num_sms() * 8, (M + kDirWarps - 1) / kDirWarps);
        k_dir4<<<(unsigned)grid, kDirThreads, 0, s>>>(p);
    } else {
        const size_t tb = (size_t)kDir4Classes * p.n4 * 8;
        const int table = tb <= (size_t)kSetTable;
        const size_t smem = 4096 * sizeof(int16_t) + kDirWarps * sizeof(SetWarp) + (table ? tb : 0);
        TG_TRY(tg_allow_max_smem((const void *)k_dir4_sets));
        int per = 0;
        TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_dir4_sets, kDirThreads, smem));
        const int64_t grid = std::min<int64_t>((int64_t)tg_num_sms() * std::max(per, 1),
                                               (M + kDirWarps - 1) / kDirWarps);
        k_dir4_sets<<<(unsigned)grid, kDirThreads, smem, s>>>(p, table);
    }
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return TG_OK;
}

int check_dir(const tg_graph *g) {
    if (!g || !g->adir) return TG_EINVAL;
    return TG_OK;
}

}  // namespace

int tg_attach_arcs(tg_graph *g, const int32_t *src, const int32_t *dst, int64_t m,
                   const int32_t *old2new, cudaStream_t s) {
    const int64_t words = (2 * g->M + 3) / 4;
    g->adir = (uint8_t *)tg_dalloc((size_t)std::max<int64_t>(1, words) * 4, s);
    if (!g->adir) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(g->adir, 0, (size_t)std::max<int64_t>(1, words) * 4, s));
    if (m == 0 || g->M == 0) return TG_OK;
    DevBuf<unsigned> err;
    if (!err.alloc(1, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(err.p, 0, 4, s));
    const unsigned grid = (unsigned)std::min<int64_t>((m + 255) / 256, 65535LL * 16);
    k_arc_bits<<<grid, 256, 0, s>>>(src, dst, m, old2new, g->rowptr, g->adj, g->toff, g->ntype,
                                    g->L, reinterpret_cast<uint32_t *>(g->adir), err.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    unsigned herr = 0;
    TG_TRY_CUDA(cudaMemcpyAsync(&herr, err.p, 4, cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return herr ? TG_EINTERNAL : TG_OK;
}

extern "C" int64_t tg_dir_slots(int32_t L) {
    if (L < 1 || L > TG_MAX_TYPES) return -1;
    return (int64_t)TG_TRIAD_CLASSES * L;
}

extern "C" int64_t tg_dir_global_len(int32_t L) {
    if (L < 1 || L > TG_MAX_TYPES) return -1;
    return (int64_t)TG_TRIAD_CLASSES * tg_binom(L + 2, 3);
}

extern "C" int tg_count_directed_per_edge(const tg_graph *g, uint64_t *rows, void *stream) {
    TG_TRY(check_dir(g));
    if (!rows) return TG_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (g->M == 0) return TG_OK;
    const int64_t width = tg_dir_slots(g->L);
    DevBuf<unsigned> err;
    if (!err.alloc(1, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(err.p, 0, 4, s));
    DevBuf<uint64_t> tmp;
    uint64_t *dst = rows;
    const bool dev_out = tg_is_device_ptr(rows);
    if (!dev_out) {
        if (!tmp.alloc((size_t)g->M * width, s)) return TG_ENOMEM;
        dst = tmp.p;
    }
    TG_TRY(dir_count(g, dst, nullptr, err.p, s));
    unsigned herr = 0;
    TG_TRY_CUDA(cudaMemcpyAsync(&herr, err.p, 4, cudaMemcpyDeviceToHost, s));
    if (!dev_out)
        TG_TRY_CUDA(cudaMemcpyAsync(rows, dst, (size_t)g->M * width * 8, cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return herr ? TG_EINTERNAL : TG_OK;
}

extern "C" int tg_count_directed_global(const tg_graph *g, uint64_t *out, void *stream) {
    TG_TRY(check_dir(g));
    if (!out) return TG_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t len = tg_dir_global_len(g->L);
    DevBuf<unsigned long long> sums;
    DevBuf<unsigned> err;
    if (!sums.alloc(len, s) || !err.alloc(1, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(sums.p, 0, len * 8, s));
    TG_TRY_CUDA(cudaMemsetAsync(err.p, 0, 4, s));
    TG_TRY(dir_count(g, nullptr, sums.p, err.p, s));
    const bool dev_out = tg_is_device_ptr(out);
    DevBuf<uint64_t> tmp;
    uint64_t *dst = out;
    if (!dev_out) {
        if (!tmp.alloc(len, s)) return TG_ENOMEM;
        dst = tmp.p;
    }
    const unsigned grid = (unsigned)std::min<int64_t>((len + 255) / 256, 4096);
    k_dir_finalize<<<grid, 256, 0, s>>>(sums.p, dst, tg_binom(g->L + 2, 3), err.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    unsigned herr = 0;
    TG_TRY_CUDA(cudaMemcpyAsync(&herr, err.p, 4, cudaMemcpyDeviceToHost, s));
    if (!dev_out) TG_TRY_CUDA(cudaMemcpyAsync(out, dst, len * 8, cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return herr ? TG_EINTERNAL : TG_OK;
}

extern "C" int64_t tg_dir4_slots(int32_t L) {
    if (L < 1 || L > TG_MAX_TYPES) return -1;
    return (int64_t)kDir4Classes * (L * (L + 1) / 2);
}

extern "C" int64_t tg_dir4_global_len(int32_t L) {
    if (L < 1 || L > TG_MAX_TYPES) return -1;
    return (int64_t)kDir4Classes * tg_binom(L + 3, 4);
}

extern "C" int tg_count_directed4_per_edge(const tg_graph *g, uint64_t *rows, void *stream) {
    TG_TRY(check_dir(g));
    if (!rows) return TG_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (g->M == 0) return TG_OK;
    const int64_t width = tg_dir4_slots(g->L);
    DevBuf<unsigned> err;
    if (!err.alloc(1, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(err.p, 0, 4, s));
    DevBuf<uint64_t> tmp;
    uint64_t *dst = rows;
    const bool dev_out = tg_is_device_ptr(rows);
    if (!dev_out) {
        if (!tmp.alloc((size_t)g->M * width, s)) return TG_ENOMEM;
        dst = tmp.p;
    }
    TG_TRY(dir4_count(g, reinterpret_cast<unsigned long long *>(dst), nullptr, err.p, s));
    unsigned herr = 0;
    TG_TRY_CUDA(cudaMemcpyAsync(&herr, err.p, 4, cudaMemcpyDeviceToHost, s));
    if (!dev_out)
        TG_TRY_CUDA(cudaMemcpyAsync(rows, dst, (size_t)g->M * width * 8, cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return herr ? TG_EINTERNAL : TG_OK;
}

extern "C" int tg_count_directed4_global(const tg_graph *g, uint64_t *out, void *stream) {
    TG_TRY(check_dir(g));
    if (!out) return TG_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t len = tg_dir4_global_len(g->L);
    DevBuf<unsigned long long> sums;
    DevBuf<unsigned> err;
    if (!sums.alloc(len, s) || !err.alloc(1, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(sums.p, 0, len * 8, s));
    TG_TRY_CUDA(cudaMemsetAsync(err.p, 0, 4, s));
    TG_TRY(dir4_count(g, nullptr, sums.p, err.p, s));
    unsigned herr = 0;
    TG_TRY_CUDA(cudaMemcpyAsync(&herr, err.p, 4, cudaMemcpyDeviceToHost, s));
    TG_TRY_CUDA(cudaMemcpyAsync(out, sums.p, len * 8, cudaMemcpyDefault, s));
    TG_TRY_CUDA(cudaStreamSynchronize(s));
    return herr ? TG_EINTERNAL : TG_OK;
}
