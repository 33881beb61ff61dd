// Test access to the library's internals: planted mistakes in a graph's device
// arrays, and internal functions on a caller's data.  Linked against libtg.so.
#include <algorithm>
#include <vector>

#include "tg_internal.cuh"

// Clears the direction bits of `count` adjacency entries from `first` on.
extern "C" int tgi_clear_states(tg_graph *g, int64_t first, int64_t count) {
    if (!g || !g->adir || first < 0 || count < 0 || first + count > 2 * g->M) return -1;
    return (int)cudaMemset(g->adir + first, 0, (size_t)count);
}

namespace {

template <class T>
std::vector<T> down(const T *p, size_t count) {
    std::vector<T> v(count);
    cudaMemcpy(v.data(), p, count * sizeof(T), cudaMemcpyDeviceToHost);
    return v;
}

template <class T>
struct Up {
    T *p = nullptr;
    explicit Up(const std::vector<T> &v) {
        cudaMalloc(&p, std::max<size_t>(1, v.size()) * sizeof(T));
        cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
    }
    ~Up() { cudaFree(p); }
};

int64_t rank4(int a, int b, int c, int d) {
    int t[4] = {a, b, c, d};
    std::sort(t, t + 4);
    int64_t r = 0;
    for (int64_t i = 0; i < 4; ++i) r += tg_binom(t[i] + i, i + 1);
    return r;
}

}  // namespace

// What tg_sum_totals makes of the totals of a small graph, counted here from the
// definitions, with one mistake planted in them (0: none): 1 tau of edge `at` in type
// `type` one too large; 2 the same, and Theta made from it; 3 Theta of edge `at`'s first
// end, once more for the pair (type, type + 1 mod L) in both orders; 4 D of that end one
// too large; 5, 6 the 4-cycles of multiset `at` one less, one more; 7, 8 the 4-cliques.
extern "C" int tgi_sum_totals(const tg_graph *g, int k, int mistake, int64_t at, int type, uint64_t *hist,
                              unsigned *err) {
    const int64_t n = g->n, M = g->M;
    const int L = g->L, L2 = L * L;
    const auto rp = down(g->rowptr, n + 1);
    const auto adj = down(g->adj, 2 * M), eid = down(g->eid, 2 * M);
    const auto toff = down(g->toff, n * (L + 1));
    const auto ty = down(g->ntype, n);
    std::vector<uint8_t> a(n * n, 0);
    for (int64_t v = 0; v < n; ++v)
        for (int64_t x = rp[v]; x < rp[v + 1]; ++x) a[v * n + (adj[x] & TG_IDMASK)] = 1;
    std::vector<uint32_t> tau(M * L, 0), theta(n * L2, 0), dlow(n * L2, 0);
    for (int64_t v = 0; v < n; ++v)
        for (int64_t x = rp[v]; x < rp[v + 1]; ++x) {
            const int64_t w = adj[x] & TG_IDMASK;
            if (w < v) continue;
            for (int64_t u = 0; u < n; ++u) tau[eid[x] * (int64_t)L + ty[u]] += a[v * n + u] & a[w * n + u];
        }
    const std::vector<uint32_t> right = tau;
    if (mistake == 1 || mistake == 2) ++tau[at * L + type];
    const auto &from = mistake == 2 ? tau : right;
    int64_t end = 0;  // an end of edge `at`
    for (int64_t v = 0; v < n; ++v)
        for (int64_t x = rp[v]; x < rp[v + 1]; ++x) {
            const int64_t w = adj[x] & TG_IDMASK;
            if (eid[x] == at) end = v;
            for (int b = 0; b < L; ++b) {
                theta[v * L2 + ty[w] * L + b] += from[eid[x] * (int64_t)L + b];
                if (w > v)
                    dlow[v * L2 + ty[w] * L + b] +=
                        (uint32_t)(toff[w * (L + 1) + b + 1] - toff[w * (L + 1) + b]) - (b == ty[v]);
            }
        }
    if (mistake == 3) {
        const int b = (type + 1) % L;
        ++theta[end * L2 + type * L + b];
        ++theta[end * L2 + b * L + type];
    }
    if (mistake == 4) ++dlow[end * L2 + type];
    const int64_t n4 = tg_binom(L + 3, 4), len = tg_global_len(L, k);
    std::vector<unsigned long long> w4(n4, 0), k4(n4, 0);
    for (int64_t p = 0; p < n; ++p)
        for (int64_t q = p + 1; q < n; ++q)
            for (int64_t x = 0; x < n; ++x) {
                if (!a[p * n + x] || !a[q * n + x]) continue;
                for (int64_t y = x + 1; y < n; ++y) {
                    if (!a[p * n + y] || !a[q * n + y]) continue;
                    ++w4[rank4(ty[p], ty[q], ty[x], ty[y])];  // once per pair of opposite nodes
                    if (q < x && a[p * n + q] && a[x * n + y]) ++k4[rank4(ty[p], ty[q], ty[x], ty[y])];
                }
            }
    for (auto &x : w4) x /= 2;
    if (mistake == 5) --w4[at];
    if (mistake == 6) ++w4[at];
    if (mistake == 7) --k4[at];
    if (mistake == 8) ++k4[at];
    const tg_lists *lists = nullptr;
    int r = tg_graph_lists(g, &lists, nullptr);
    if (r != TG_OK) return r;
    const Up<uint32_t> dtau(tau), dtheta(theta), ddlow(dlow);
    const Up<unsigned long long> dw(w4), dk(k4), dh(std::vector<unsigned long long>(len, 0));
    const Up<unsigned> derr(std::vector<unsigned>(1, 0));
    r = tg_sum_totals(g, k, dtau.p, dtheta.p, ddlow.p, lists->utoff, dw.p, dk.p, dh.p, derr.p, nullptr);
    if (r != TG_OK) return r;
    if (cudaDeviceSynchronize() != cudaSuccess) return TG_ECUDA;
    const auto h = down(dh.p, len);
    std::copy(h.begin(), h.end(), hist);
    *err = down(derr.p, 1)[0];
    return TG_OK;
}

// The radix sort on host keys (and values, unless NULL), in place.
extern "C" int tgi_sort(int64_t n, int bits, int looks, uint64_t *keys, uint32_t *vals) {
    const std::vector<uint64_t> k(keys, keys + n);
    const std::vector<uint32_t> v(vals ? vals : (const uint32_t *)keys, vals ? vals + n : (const uint32_t *)keys + n);
    const Up<uint64_t> k1(k), k2(k);
    const Up<uint32_t> v1(v), v2(v);
    uint64_t *kr = nullptr;
    uint32_t *vr = nullptr;
    const int r = vals ? tg_radix_sort_kv(k1.p, k2.p, v1.p, v2.p, n, bits, nullptr, &kr, &vr, looks)
                       : tg_radix_sort_u64(k1.p, k2.p, n, bits, nullptr, &kr, looks);
    if (r != TG_OK) return r;
    if (cudaDeviceSynchronize() != cudaSuccess) return TG_ECUDA;
    cudaMemcpy(keys, kr, n * 8, cudaMemcpyDeviceToHost);
    if (vals) cudaMemcpy(vals, vr, n * 4, cudaMemcpyDeviceToHost);
    return TG_OK;
}
