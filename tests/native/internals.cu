// Test access to the library's internals: planted mistakes in a graph's device
// arrays, and internal functions on a caller's data.  Linked against libtg.so.
#include "tg_internal.cuh"

// Clears the direction bits of `count` adjacency entries from `first` on.
extern "C" int tgi_clear_states(tg_graph *g, int64_t first, int64_t count) {
    if (!g || !g->adir || first < 0 || count < 0 || first + count > 2 * g->M) return -1;
    return (int)cudaMemset(g->adir + first, 0, (size_t)count);
}
