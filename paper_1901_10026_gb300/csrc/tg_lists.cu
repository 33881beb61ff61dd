// Oriented lists of a graph, made once per graph with its schedule: the up list
// of every node (its neighbours of higher rank, i.e. smaller id, with their
// edge ids and typed offsets) and the edges grouped by their higher-ranked end j.
//
// Both are compactions of the adjacency lists.  A list is sorted by (type, id),
// so the up neighbours are a prefix of every typed range and the others, whose
// edges belong to the group of the list's owner, a suffix; every entry's place
// follows from its position and the typed offsets alone.
//
// Measured (build + count): ER 1M/5M, k = 3, 4.6 -> 4.1 ms, ER 100K/1M 2.66 -> 2.45
// ms, CL-1M 54.5 -> 52.7 ms, ER-1000 849 -> 796 us.  Before, the groups came from a
// radix sort of all edges by (j, i) and the up lists from one warp per node, made
// again by every count.  The fill reads and writes each entry once (16 B) and is
// bound by the latency of its dependent reads.
#include <algorithm>

#include "tg_device.cuh"

using namespace tgd;

namespace {

// Typed offsets and sizes of the up lists: G lanes per node, lane t searching
// the end of type t's prefix.
template <int G>
__global__ void __launch_bounds__(256) k_up_count(const int64_t *rowptr, const uint32_t *adj,
                                                  const int32_t *toff, int64_t n, int L,
                                                  int32_t *utoff, int64_t *utot) {
    const int t = threadIdx.x % G;
    const int64_t ng = (int64_t)gridDim.x * (256 / G);
    // every lane of a warp makes the same number of steps
    for (int64_t v0 = (int64_t)blockIdx.x * (256 / G); v0 <= n; v0 += ng) {
        const int64_t v = v0 + threadIdx.x / G;
        int c = 0;
        if (v < n && t < L) {
            const int64_t b = __ldg(rowptr + v);
            const int32_t *to = toff + v * (L + 1);
            int lo = __ldg(to + t), hi = __ldg(to + t + 1);
            const int start = lo;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if ((int64_t)(__ldg(adj + b + mid) & TG_IDMASK) < v)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            c = lo - start;
        }
        int incl = c;
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o, G);
            if (t >= o) incl += y;
        }
        if (v < n) {
            if (t < L) utoff[v * (L + 1) + t + 1] = incl;
            if (t == 0) utoff[v * (L + 1)] = 0;
            if (t == L - 1) utot[v] = incl;
        } else if (v == n && t == 0) {
            utot[n] = 0;  // the scan's last entry takes the total
        }
    }
}

constexpr int kFillChunk = 1024;

// One warp per `chunk` consecutive adjacency entries (a multiple of 32), one lane per
// entry.  A chunk starts with a search for its node and is a chain of dependent reads
// after it, so it is made only as long as one wave of warps asks, up to kFillChunk:
// against chunks of kFillChunk throughout, 7.6 and not 49 us for 14,000 edges, 25 and
// not 56 for 1M, the same 122 for 5M.
// Nodes without neighbours have the largest ids, so 32 entries belong to at
// most 32 consecutive nodes.
__global__ void __launch_bounds__(256) k_oriented_fill(const int64_t *rowptr, const uint32_t *adj,
                                                       const uint32_t *eid, const int32_t *toff,
                                                       const int32_t *utoff, const int64_t *uoff,
                                                       int64_t n, int64_t total, int64_t chunk, int L,
                                                       uint32_t *uadj,
                                                       uint32_t *ueid, uint32_t *order, uint32_t *other) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c * chunk < total;
         c += nw) {
        const int64_t x0 = c * chunk, x1 = min(total, x0 + chunk);
        int64_t v = 0, top = n - 1;  // last node with rowptr[v] <= x0
        while (v < top) {
            const int64_t mid = (v + top + 1) >> 1;
            if (__ldg(rowptr + mid) <= x0)
                v = mid;
            else
                top = mid - 1;
        }
        for (int64_t b = x0; b < x1; b += 32) {
            const int64_t x = b + lane;
            // lists that end at or before x: lane k holds the end of node v + k
            const int64_t end = __ldg(rowptr + min(n, v + 1 + lane));
            int r = 0;
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
                const int64_t e = __shfl_sync(kFull, end, r + st - 1);
                if (e <= x) r += st;
            }
            const int64_t w = min(n - 1, v + r);
            // the node of the next 32 entries' first one
            v = __shfl_sync(kFull, min(n - 1, w + (__ldg(rowptr + w + 1) <= x + 1)), 31);
            if (x >= x1) continue;
            const uint32_t e = __ldg(adj + x);
            const uint32_t id = eid[x];
            const int t = (int)(e >> TG_TSHIFT);
            const int64_t rb = __ldg(rowptr + w), ub = __ldg(uoff + w);
            const int to = __ldg(toff + w * (L + 1) + t);
            const int u0 = __ldg(utoff + w * (L + 1) + t);
            const int in = (int)(x - rb) - to;  // place in the typed range
            if ((int64_t)(e & TG_IDMASK) < w) {
                uadj[ub + u0 + in] = e;
                ueid[ub + u0 + in] = id;
            } else {
                const int u1 = __ldg(utoff + w * (L + 1) + t + 1);
                const int64_t at = (rb - ub) + (to - u0) + in - (u1 - u0);
                order[at] = id;
                other[at] = e;
            }
        }
    }
}

}  // namespace

int tg_build_lists(const tg_graph *g, tg_lists &out, cudaStream_t s) {
    const int64_t n = g->n, M = g->M;
    const int L = g->L;
    DevBuf<int64_t> utot, uoff;
    DevBuf<int32_t> utoff;
    DevBuf<uint32_t> uadj, ueid, order, other;
    if (!utot.alloc(n + 1, s) || !uoff.alloc(n + 1, s) || !utoff.alloc((size_t)n * (L + 1), s) ||
        !uadj.alloc(M, s) || !ueid.alloc(M, s) || !order.alloc(M, s) || !other.alloc(M, s))
        return TG_ENOMEM;
    const int G = L <= 4 ? 4 : L <= 8 ? 8 : 16;
    const unsigned cg = (unsigned)std::min<int64_t>(n / (256 / G) + 1, (int64_t)tg_num_sms() * 64);
    (G == 4 ? k_up_count<4> : G == 8 ? k_up_count<8> : k_up_count<16>)<<<cg, 256, 0, s>>>(
        g->rowptr, g->adj, g->toff, n, L, utoff.p, utot.p);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    TG_TRY(tg_scan_i64(utot.p, uoff.p, n + 1, s));
    if (M > 0) {
        const int64_t wave = (int64_t)tg_num_sms() * 64;  // warps
        const int64_t chunk = std::min<int64_t>(kFillChunk, (2 * M / wave + 32) / 32 * 32);
        const unsigned fg = (unsigned)std::min<int64_t>((2 * M + 8 * chunk - 1) / (8 * chunk), wave);
        k_oriented_fill<<<fg, 256, 0, s>>>(g->rowptr, g->adj, g->eid, g->toff, utoff.p, uoff.p, n, 2 * M, chunk, L,
                                           uadj.p, ueid.p, order.p, other.p);
        tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
    }
    out.uoff = uoff.release();
    out.utoff = utoff.release();
    out.uadj = uadj.release();
    out.ueid = ueid.release();
    out.order = order.release();
    out.other = other.release();
    return TG_OK;
}
