// Whole-graph global sums from node-level and edge-level totals.
//
// For a global count the per-edge rows are never needed, only their sums by
// type multiset.  Every orbit of Alg. 2-3 summed over all edges is a fixed
// combination of the non-induced copies N of each 4-node pattern (the
// containment inversion of the induced counts), and apart from the 4-cycles W
// and the 4-cliques K (enumerated by tg_cycles.cu) these need no pass over
// the triangle nodes of an edge:
//   N_S4 (stars)            per node v:  products of three typed degrees
//   N_TT (tailed triangles) per node v:  Theta_v[b][c] / 2 triangles of types
//                           {b, c} at v, times the remaining typed degree
//   N_P4 (4-paths)          per node v:  sum over its neighbours w > v of
//                           d_w^a - [a = phi_v], times d_v^b - [b = phi_w],
//                           less tau_vw[a] for the closed ones (a = b)
//   N_D  (diamonds)         per edge:    tau_a tau_b (a < b), C(tau_a, 2)
//   P3, triangles, edges    per node / per edge
// so that the undivided sums (per-edge counts summed over the edges, |E(H)| per
// copy) are, mod 2^64,
//   h1 = 2 N_P3 - 2 H2                       H2 = sum of tau (3 per triangle)
//   h3 = 3 (N_P4 - 2 N_TT + 6 N_D - 4 W - 12 K)
//   h4 = 3 (N_S4 - N_TT + 2 N_D - 4 K)       h5 = 4 (W - N_D + 3 K)
//   h6 = 4 (N_TT - 4 N_D + 12 K)             h7 = 5 (N_D - 6 K)   h8 = 6 K
// Every N is summed as a count of copies (no division of a wrapped sum), so
// the sums equal those of the per-edge pass (tg_edges.cu) mod 2^64.
//
// The factors |E(H)| are put in here, so their division afterwards tells nothing of the
// totals (but for triangles).  What the totals say of one another is checked instead:
//   per node       Theta_v[b][c] = Theta_v[c][b], and Theta_v[b][b] is even (both count
//                  triangles at v, from the tau of different edges);
//   per type pair  the triangles at the nodes by the types of the other two (Theta) are
//                  those of the edges between the types (tau);
//   per type       sum of D[.][a] = sum over w of u_w d_w^a, less the edges whose end of
//                  smaller id has type a (u_w: neighbours of smaller id);
//   per multiset   no induced count is negative (3-paths, 4-paths, 4-cycles, tailed
//                  triangles, diamonds: below 2^60 while 2M < 2^31; stars may wrap).
// A wrong tau, Theta or D, or 4-cycle and 4-clique totals that do not fit them, set
// TG_DERR_TOTALS.
//
// The per-edge pass gathers three rows per triangle node and holds 3 L^2
// 64-bit sums per edge; here an edge costs its tau row and a node its Theta
// and D rows, read once.
//
// Measured (whole build + count, per-edge pass before -> totals): R-MAT-21
// (L = 8, 31.8M edges) 800 -> 505 ms, CL-1M 87.0 -> 60.1 ms, CL 100K/1M
// 12.2 -> 8.6 ms, ER 100K/1M 6.1 -> 4.5 ms; k = 3 on ER 1M/5M 18.9 -> 4.6 ms.
// The replaced phase alone: 303 -> 7 ms on R-MAT-21, 28.8 -> 1.9 ms on CL-1M.
// The two kernels read tau, Theta and D once (3.4 GB on R-MAT-21, 0.5 ms at the
// copy rate) and are bound by their integer arithmetic.
#include <algorithm>

#include "tg_device.cuh"

using namespace tgd;

namespace {

__device__ __forceinline__ int64_t key4(int a, int b, int c, int d) {
    sort2(a, b);
    sort2(c, d);
    sort2(a, c);
    sort2(b, d);
    sort2(b, c);
    return colex4(a, b, c, d);
}
__device__ __forceinline__ int64_t key3(int a, int b, int c) {
    sort2(a, b);
    sort2(b, c);
    sort2(a, b);
    return colex3(a, b, c);
}

// sums (zeroed): [edges: E2][P3: n3][H2: n3][P4: n4][S4: n4][TT: n4][D: n4], then (k = 4)
// the triangles of the nodes and of the edges by type pair [P] [P], the defects of D [L]
struct SumParams {
    const int32_t *toff;
    const uint8_t *ntype;
    const int2 *edges;
    const uint32_t *tau;
    const uint32_t *theta;  // k = 4
    const uint32_t *dlow;   // k = 4: sum over w in Gamma_v^s, w > v, of d_w^a - [a = phi_v]
    const int32_t *utoff;   // typed offsets of the up lists
    unsigned *err;
    int64_t n, M;
    int32_t L, P, k;
    int64_t e2, n3, n4;
    int64_t eblocks;  // CTAs of the edge totals; those after them make the checks
    unsigned long long *sums;
};

__device__ __forceinline__ void flush_nonzero(unsigned long long *dst, unsigned long long v) {
    if (v) atomicAdd(dst, v);
}

// ----------------------------------------------------------------- checks --
// What Theta and D say of tau, of one another and of the degrees (see the head).  A
// thread per entry of a row, the same entry of every row it takes, so its sums stay in
// registers.  One more pass over the rows, by further CTAs of the edge totals' launch
// (CTA `block` of `blocks`): counts of ER 100K/1M and of a power law of 8M edges take as
// long as without it (1,518 us and 30.8 ms), 25 and 110 us longer with a launch of its
// own, 45 and 500 us with the same sums inside k_sum_nodes, in its registers.
// part: P + L words.
constexpr int kCheckThreads = 256;
constexpr int kCheckBatch = 4;  // rows in flight

__device__ __forceinline__ void sum_checks(const SumParams &p, int64_t block, int64_t blocks,
                                           unsigned long long *part) {
    const int L = p.L, L2 = L * L, P = p.P, R = kCheckThreads / L2;
    for (int x = threadIdx.x; x < P + L; x += kCheckThreads) part[x] = 0ull;
    __syncthreads();
    if (threadIdx.x < R * L2) {
        const int q = threadIdx.x % L2, s = q / L, a = q % L;
        unsigned long long tri = 0, dsum = 0;  // triangles of (s, a), D of column a
        bool bad = false;
        const int64_t step = blocks * R;
        for (int64_t v0 = block * R + threadIdx.x / L2; v0 < p.n; v0 += step * kCheckBatch) {
            uint32_t t[kCheckBatch], m[kCheckBatch], x[kCheckBatch];
#pragma unroll
            for (int y = 0; y < kCheckBatch; ++y) {
                const int64_t v = v0 + y * step;
                const bool in = v < p.n;
                t[y] = in ? __ldg(p.theta + v * L2 + q) : 0u;
                m[y] = in ? __ldg(p.theta + v * L2 + a * L + s) : 0u;
                x[y] = in ? __ldg(p.dlow + v * L2 + q) : 0u;
            }
#pragma unroll
            for (int y = 0; y < kCheckBatch; ++y) {
                bad |= t[y] != m[y] || (s == a && (t[y] & 1u));
                tri += s == a ? t[y] >> 1 : t[y];
                dsum += x[y];
            }
        }
        if (s <= a) flush_nonzero(part + pair_index(L, s, a), tri);
        flush_nonzero(part + P + a, 0ull - dsum);
        if (bad && p.err) atomicOr(p.err, TG_DERR_TOTALS);
    }
    // the other side of D: a thread per type of a node
    const int R2 = kCheckThreads / L, b = threadIdx.x % L;
    if (threadIdx.x < R2 * L) {
        unsigned long long sum = 0;
        const int64_t step = blocks * R2;
        for (int64_t v0 = block * R2 + threadIdx.x / L; v0 < p.n; v0 += step * 2) {
            uint32_t up[2], d[2], all[2];
            int tv[2];
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const int64_t v = v0 + y * step;
                const bool in = v < p.n;
                const int32_t *to = p.toff + v * (L + 1);
                up[y] = in ? (uint32_t)__ldg(p.utoff + v * (L + 1) + L) : 0u;
                d[y] = in ? (uint32_t)(__ldg(to + b + 1) - __ldg(to + b)) : 0u;
                all[y] = in ? (uint32_t)__ldg(to + L) : 0u;
                tv[y] = in ? (int)p.ntype[v] : -1;
            }
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                sum += (unsigned long long)up[y] * d[y];
                if (b == tv[y]) sum -= all[y] - up[y];
            }
        }
        flush_nonzero(part + P + b, sum);
    }
    __syncthreads();
    unsigned long long *out = p.sums + p.e2 + 2 * p.n3 + 4 * p.n4;  // [P] triangles, [P] the edges', [L]
    for (int x = threadIdx.x; x < P + L; x += kCheckThreads) flush_nonzero(out + (x < P ? x : x + P), part[x]);
}

// ------------------------------------------------------------ edge totals --
// Per unordered type pair of the endpoints: sum of tau_a, of tau_a tau_b
// (a < b) and of C(tau_a, 2), and the number of edges.  A warp takes 32 edges
// at a time (their tau rows are one contiguous read), stages the rows in
// shared memory, and goes through the edges of one type pair after the other:
// lane q holds the products of type pairs q, q + 32, ... in registers and adds
// them to the CTA's table once per type pair present, on distinct addresses.
constexpr int kSumWarps = 8;
static_assert(kSumWarps * 32 == kCheckThreads, "the checks run in the same launch");

// Five CTAs per SM: with the registers that the checks would take there are four, and
// the k = 3 count of an ER graph of 5M edges takes 1,862 and not 1,847 us.
template <int LP>
__global__ void __launch_bounds__(kSumWarps * 32, LP <= 8 ? 5 : 1) k_sum_edges(SumParams p) {
    constexpr int kPairs = LP * (LP + 1) / 2, kSlots = (kPairs + 31) / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = p.L, P = p.P, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool four = p.k == 4;
    // [P][L] sums of tau, [P] edges, (k = 4) [P][P] products, then the rows
    unsigned long long *ts = reinterpret_cast<unsigned long long *>(smem);
    if (blockIdx.x >= p.eblocks) {  // k = 4: P (L + 1 + P) words and more
        sum_checks(p, blockIdx.x - p.eblocks, gridDim.x - p.eblocks, ts);
        return;
    }
    unsigned long long *ne = ts + P * L;
    unsigned long long *tab = ne + P;
    const int words = P * L + P + (four ? P * P : 0);
    uint32_t *row = reinterpret_cast<uint32_t *>(ts + words) + warp * 32 * (LP + 1);
    for (int q = threadIdx.x; q < words; q += blockDim.x) ts[q] = 0ull;
    int pa[kSlots], pb[kSlots];
    uint32_t nec[kSlots];  // edges of the lane's type pairs, added to ne at the end
#pragma unroll
    for (int z = 0; z < kSlots; ++z) {
        const int q = lane + 32 * z;
        pa[z] = pb[z] = 0;
        nec[z] = 0u;
        if (q < P) unpair(L, q, pa[z], pb[z]);
    }
    __syncthreads();
    const int64_t nw = p.eblocks * kSumWarps;
    for (int64_t c = (int64_t)blockIdx.x * kSumWarps + warp; c * 32 < p.M; c += nw) {
        const int64_t e0 = c * 32;
        const int cnt = (int)min((int64_t)32, p.M - e0);
        int pt = -1;
        if (lane < cnt) {
            const int2 ab = p.edges[e0 + lane];
            pt = pair_index(L, p.ntype[ab.x], p.ntype[ab.y]);
        }
        bool any = false;
        for (int x = lane; x < cnt * L; x += 32) {
            const uint32_t v = __ldg(p.tau + e0 * L + x);
            any |= v != 0u;
            row[(x / L) * (LP + 1) + x % L] = v;
        }
        any = __any_sync(kFull, any);
        __syncwarp();
        unsigned todo = __ballot_sync(kFull, pt >= 0);
        while (todo) {
            const int g = __shfl_sync(kFull, pt, __ffs(todo) - 1);
            unsigned grp = __ballot_sync(kFull, pt == g);
            todo &= ~grp;
#pragma unroll
            for (int z = 0; z < kSlots; ++z)
                if (lane + 32 * z == g) nec[z] += (uint32_t)__popc(grp);
            if (!any) continue;
            unsigned long long acc[kSlots], st = 0;
#pragma unroll
            for (int z = 0; z < kSlots; ++z) acc[z] = 0ull;
            for (; grp; grp &= grp - 1u) {
                const uint32_t *r = row + (__ffs(grp) - 1) * (LP + 1);
                if (lane < L) st += r[lane];
                if (four) {
#pragma unroll
                    for (int z = 0; z < kSlots; ++z) {
                        const uint64_t a = r[pa[z]], b = r[pb[z]];
                        acc[z] += pa[z] == pb[z] ? c2(a) : a * b;
                    }
                }
            }
            if (lane < L) flush_nonzero(ts + g * L + lane, st);
            if (four) {
#pragma unroll
                for (int z = 0; z < kSlots; ++z)
                    if (lane + 32 * z < P) flush_nonzero(tab + g * P + lane + 32 * z, acc[z]);
            }
        }
        __syncwarp();  // the rows are rewritten by the next chunk
    }
#pragma unroll
    for (int z = 0; z < kSlots; ++z)
        if (nec[z]) atomicAdd(ne + lane + 32 * z, (unsigned long long)nec[z]);
    __syncthreads();
    unsigned long long *s_p3 = p.sums + p.e2, *s_h2 = s_p3 + p.n3, *s_p4 = s_h2 + p.n3;
    unsigned long long *s_d = s_p4 + 3 * p.n4;
    for (int q = threadIdx.x; q < words; q += blockDim.x) {
        const unsigned long long v = ts[q];
        if (!v) continue;
        int i, j;
        if (q < P * L) {
            const int a = q % L;
            unpair(L, q / L, i, j);
            atomicAdd(s_h2 + key3(i, j, a), v);
            if (four) atomicAdd(s_p4 + key4(i, j, a, a), 0ull - v);  // closed 4-paths
        } else if (q < P * L + P) {
            unpair(L, q - P * L, i, j);
            atomicAdd(p.sums + (int64_t)i + (int64_t)(j + 1) * j / 2, v);
        } else {
            int a, b;
            const int x = q - P * L - P;
            unpair(L, x / P, i, j);
            unpair(L, x % P, a, b);
            atomicAdd(s_d + key4(i, j, a, b), v);
        }
    }
    if (!four) return;
    for (int q = threadIdx.x; q < P; q += blockDim.x) {
        unsigned long long v = 0;
        for (int a = 0; a < L; ++a) v += ts[q * L + a];
        flush_nonzero(s_d + p.n4 + P + q, v);
    }
}

// ------------------------------------------------------------ node totals --
// A team of T = max(32, LP^2) lanes takes a contiguous range of nodes, one
// node type at a time, so that a lane's accumulators (its ordered pair (s, a)
// against every third type) stay in registers and are added to the CTA's
// histogram once per type.  Warps of a team share no state: each takes the
// pairs of its own lanes and reads the node's rows itself.
constexpr int kNodeThreads = 256;
constexpr int kNodeMin = 16;  // nodes of a team's range, at least
// nodes whose rows are read before they are used: of an 8M-edge power law's sums (L = 5)
// 1.88 ms become 1.63 with 2 and 1.67 with 4
constexpr int kNodeBatch = 2;

// C(x, 3), the factors 2 and 3 taken out before the product
__device__ __forceinline__ unsigned long long c3(uint32_t x) {
    const uint32_t m = x % 3u;
    uint32_t p = x, q = x - 1u, r = x - 2u;
    if (x < 3u) return 0ull;
    if (m == 0u) p /= 3u;
    if (m == 1u) q /= 3u;
    if (m == 2u) r /= 3u;
    if (x & 1u)
        q >>= 1;
    else
        p >>= 1;
    return (unsigned long long)p * q * r;
}

template <int LP>
__global__ void __launch_bounds__(kNodeThreads, LP <= 4 ? 4 : LP <= 8 ? 2 : 1) k_sum_nodes(SumParams p) {
    constexpr int kTeam = LP * LP < 32 ? 32 : LP * LP;
    constexpr int kTeams = kNodeThreads / kTeam;
    constexpr int kN4 = (LP + 2) * (LP + 1) * LP / 6;  // triples of types
    constexpr int kS4 = (kN4 + kTeam - 1) / kTeam;
    extern __shared__ __align__(16) unsigned char smem[];
    // [P3: n3] (k = 4: [P4: n4][S4: n4][TT: n4])
    unsigned long long *h3 = reinterpret_cast<unsigned long long *>(smem);
    unsigned long long *h4 = h3 + p.n3;
    const bool four = p.k == 4;
    const int64_t hlen = p.n3 + (four ? 3 * p.n4 : 0);
    for (int64_t q = threadIdx.x; q < hlen; q += blockDim.x) h3[q] = 0ull;
    __syncthreads();
    const int L = p.L, L2 = L * L, P = p.P, lane = threadIdx.x & 31;
    const int q = threadIdx.x % kTeam;  // this lane's pair
    const int s = q / L, a = q % L;     // ordered pair (s, a) when q < L2
    const bool pair = q < L2;
    int p3a = 0, p3b = 0;
    if (q < P) unpair(L, q, p3a, p3b);
    int ts[kS4], tt[kS4], tu[kS4];
    const int n_tri = (L + 2) * (L + 1) * L / 6;
#pragma unroll
    for (int z = 0; z < kS4; ++z) {
        int m = q + z * kTeam;
        ts[z] = -1;
        tt[z] = tu[z] = 0;
        if (m < n_tri) {  // colex decoding of s <= t <= u
            int u = 0;
            while ((u + 3) * (u + 2) * (u + 1) / 6 <= m) ++u;
            m -= (u + 2) * (u + 1) * u / 6;
            int t = 0;
            while ((t + 2) * (t + 1) / 2 <= m) ++t;
            ts[z] = m - (t + 1) * t / 2;
            tt[z] = t;
            tu[z] = u;
        }
    }
    const int64_t teams = (int64_t)gridDim.x * kTeams;
    const int64_t team = (int64_t)blockIdx.x * kTeams + threadIdx.x / kTeam;
    const int64_t per = (p.n + teams - 1) / teams;
    const int64_t v0 = team * per, v1 = min(p.n, v0 + per);
    for (int tv = 0; tv < L; ++tv) {
        unsigned long long acc3 = 0, accP[LP], accT[LP], accS[kS4];
#pragma unroll
        for (int b = 0; b < LP; ++b) accP[b] = accT[b] = 0ull;
#pragma unroll
        for (int z = 0; z < kS4; ++z) accS[z] = 0ull;
        for (int64_t c = v0; c < v1; c += 32) {
            unsigned m = __ballot_sync(kFull, c + lane < v1 && p.ntype[c + lane] == tv);
            while (m) {
                // kNodeBatch nodes' rows in flight; zero rows add nothing
                uint32_t dn[kNodeBatch], xn[kNodeBatch], tn[kNodeBatch];
#pragma unroll
                for (int y = 0; y < kNodeBatch; ++y) {
                    const bool in = m != 0u;
                    const int64_t v = c + (in ? __ffs(m) - 1 : 0);
                    m &= m - 1u;
                    const int32_t *to = p.toff + v * (L + 1);
                    dn[y] = in && lane < L ? (uint32_t)(__ldg(to + lane + 1) - __ldg(to + lane)) : 0u;
                    xn[y] = in && four && pair ? __ldg(p.dlow + v * L2 + q) : 0u;
                    tn[y] = in && four && pair && s <= a ? __ldg(p.theta + v * L2 + q) : 0u;
                }
#pragma unroll
                for (int y = 0; y < kNodeBatch; ++y) {
                    const uint32_t d = dn[y], x = xn[y];
                    uint32_t t = tn[y];
                    const uint32_t da = __shfl_sync(kFull, d, p3a), db = __shfl_sync(kFull, d, p3b);
                    if (q < P) acc3 += p3a == p3b ? c2(da) : (uint64_t)da * db;
                    if (!four) continue;
                    if (s == a) t >>= 1;
#pragma unroll
                    for (int b = 0; b < LP; ++b) {
                        if (b < L) {
                            const uint32_t dd = __shfl_sync(kFull, d, b);
                            // x > 0 has a neighbour of type s, t > 0 one of types s and a
                            accP[b] += x ? (uint64_t)x * (dd - (b == s)) : 0ull;
                            accT[b] += t ? (uint64_t)t * (dd - (b == s) - (b == a)) : 0ull;
                        }
                    }
#pragma unroll
                    for (int z = 0; z < kS4; ++z) {
                        const uint64_t x0 = __shfl_sync(kFull, d, ts[z] < 0 ? 0 : ts[z]);
                        const uint64_t x1 = __shfl_sync(kFull, d, tt[z]);
                        const uint64_t x2 = __shfl_sync(kFull, d, tu[z]);
                        uint64_t w = 0;
                        if (ts[z] < 0)
                            w = 0;
                        else if (ts[z] == tu[z])
                            w = c3((uint32_t)x0);
                        else if (ts[z] == tt[z])
                            w = c2(x0) * x2;
                        else if (tt[z] == tu[z])
                            w = x0 * c2(x1);
                        else
                            w = x0 * x1 * x2;
                        accS[z] += w;
                    }
                }
            }
        }
        if (q < P) flush_nonzero(h3 + key3(tv, p3a, p3b), acc3);
        if (!four) continue;
        if (pair) {
#pragma unroll
            for (int b = 0; b < LP; ++b)
                if (b < L) {
                    flush_nonzero(h4 + key4(tv, s, a, b), accP[b]);
                    flush_nonzero(h4 + 2 * p.n4 + key4(tv, s, a, b), accT[b]);
                }
        }
#pragma unroll
        for (int z = 0; z < kS4; ++z)
            if (ts[z] >= 0) flush_nonzero(h4 + p.n4 + key4(tv, ts[z], tt[z], tu[z]), accS[z]);
    }
    __syncthreads();
    unsigned long long *out3 = p.sums + p.e2, *out4 = out3 + 2 * p.n3;
    for (int64_t z = threadIdx.x; z < hlen; z += blockDim.x)
        flush_nonzero(z < p.n3 ? out3 + z : out4 + (z - p.n3), h3[z]);
}

// The undivided sums from the totals (and the 4-cycles W, 4-cliques K), and the checks
// of the totals.
__global__ void k_sum_combine(const unsigned long long *sums, int64_t e2, int64_t n3, int64_t n4, int L,
                              int k, const unsigned long long *w, const unsigned long long *k4,
                              unsigned long long *hist, unsigned *err) {
    const int64_t off2 = e2 + n3, off4 = off2 + n3, len = off4 + (k == 4 ? n4 : 0);
    const int P = L * (L + 1) / 2;
    const unsigned long long *tri = sums + off4 + 4 * n4, *etri = tri + P, *defect = etri + P;
    bool bad = false;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < len;
         x += (int64_t)gridDim.x * blockDim.x) {
        if (x < e2) {
            hist[x] = sums[x];
        } else if (x < off2) {
            const unsigned long long p3 = sums[x] - sums[x + n3];
            hist[x] = 2 * p3;
            bad |= (long long)p3 < 0;
        } else if (x < off4) {
            hist[x] = sums[x];
        } else {
            const int64_t r = x - off4;
            const unsigned long long p4 = sums[x], s4 = sums[x + n4], tt = sums[x + 2 * n4],
                                     d = sums[x + 3 * n4], c = w[r], q = k4[r];
            const unsigned long long h3 = p4 - 2 * tt + 6 * d - 4 * c - 12 * q, h5 = c - d + 3 * q,
                                     h6 = tt - 4 * d + 12 * q, h7 = d - 6 * q;
            hist[off4 + r] = 3 * h3;
            hist[off4 + n4 + r] = 3 * (s4 - tt + 2 * d - 4 * q);
            hist[off4 + 2 * n4 + r] = 4 * h5;
            hist[off4 + 3 * n4 + r] = 4 * h6;
            hist[off4 + 4 * n4 + r] = 5 * h7;
            hist[off4 + 5 * n4 + r] = 6 * q;
            bad |= (long long)(h3 | h5 | h6 | h7) < 0;
            if (r < P) bad |= tri[r] != etri[r];  // L <= P <= C(L + 3, 4)
            if (r < L) bad |= defect[r] != 0ull;
        }
    }
    if (bad && err) atomicOr(err, TG_DERR_TOTALS);
}

size_t edges_smem(const SumParams &p, int LP) {
    const size_t words = (size_t)p.P * p.L + p.P + (p.k == 4 ? (size_t)p.P * p.P : 0);
    return words * 8 + (size_t)kSumWarps * 32 * (LP + 1) * 4;
}

template <int LP>
int launch_sums(SumParams p, cudaStream_t s) {
    TG_TRY(tg_allow_max_smem((const void *)k_sum_edges<LP>));
    TG_TRY(tg_allow_max_smem((const void *)k_sum_nodes<LP>));
    const size_t es = edges_smem(p, LP);
    const size_t ns = (size_t)(p.n3 + (p.k == 4 ? 3 * p.n4 : 0)) * 8;
    int eper = 0, nper = 0;
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&eper, k_sum_edges<LP>, kSumWarps * 32, es));
    TG_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nper, k_sum_nodes<LP>, kNodeThreads, ns));
    if (eper < 1 || nper < 1) return TG_EINVAL;
    const int64_t sms = tg_num_sms();
    p.eblocks = std::max<int64_t>(1, std::min<int64_t>(sms * eper, (p.M + kSumWarps * 32 - 1) / (kSumWarps * 32)));
    int64_t checks = 0;
    if (p.k == 4) {
        const int64_t rows = (int64_t)(kCheckThreads / (p.L * p.L)) * kCheckBatch;
        checks = std::max<int64_t>(1, std::min<int64_t>(sms * eper, (p.n + rows - 1) / rows));
    }
    k_sum_edges<LP><<<(unsigned)(p.eblocks + checks), kSumWarps * 32, es, s>>>(p);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    constexpr int kTeams = kNodeThreads / (LP * LP < 32 ? 32 : LP * LP);
    const int64_t ng = std::min<int64_t>(sms * nper, (p.n + kNodeMin * kTeams - 1) / (kNodeMin * kTeams));
    k_sum_nodes<LP><<<(unsigned)std::max<int64_t>(1, ng), kNodeThreads, ns, s>>>(p);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    return TG_OK;
}

}  // namespace

int tg_sum_totals(const tg_graph *g, int k, const uint32_t *tau, const uint32_t *theta,
                  const uint32_t *dlow, const int32_t *utoff, const unsigned long long *c4w,
                  const unsigned long long *k4, unsigned long long *hist, unsigned *err, cudaStream_t s) {
    if (g->max_degree >= ((int64_t)1 << 27)) return TG_EOVERFLOW;  // as the per-edge pass
    SumParams p{};
    p.toff = g->toff;
    p.ntype = g->ntype;
    p.edges = g->edges;
    p.tau = tau;
    p.theta = theta;
    p.dlow = dlow;
    p.utoff = utoff;
    p.err = err;
    p.n = g->n;
    p.M = g->M;
    p.L = g->L;
    p.P = g->L * (g->L + 1) / 2;
    p.k = k;
    p.e2 = tg_binom(g->L + 1, 2);
    p.n3 = tg_binom(g->L + 2, 3);
    p.n4 = tg_binom(g->L + 3, 4);
    const int64_t len = p.e2 + 2 * p.n3 + (k == 4 ? 4 * p.n4 + 2 * p.P + p.L : 0);
    DevBuf<unsigned long long> sums;
    if (!sums.alloc(len, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(sums.p, 0, len * 8, s));
    p.sums = sums.p;
    if (g->L <= 4)
        TG_TRY(launch_sums<4>(p, s));
    else if (g->L <= 8)
        TG_TRY(launch_sums<8>(p, s));
    else
        TG_TRY(launch_sums<16>(p, s));
    k_sum_combine<<<(unsigned)((len + 255) / 256), 256, 0, s>>>(sums.p, p.e2, p.n3, p.n4, p.L, k, c4w, k4, hist,
                                                                err);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    return TG_OK;
}
