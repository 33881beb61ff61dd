// Device primitives of the library: stream-ordered allocation with failure
// injection, exclusive scans and a stable LSD radix sort on uint64 keys.
// All kernels here are this library's own; no vendor sort or scan is used.
#include <algorithm>
#include <atomic>
#include <mutex>
#include <utility>
#include <vector>

#include "tg_internal.cuh"

// ------------------------------------------------------------ allocation --
static tg_alloc_fn g_alloc = nullptr;
static tg_free_fn g_free = nullptr;
static void *g_alloc_ctx = nullptr;
static std::atomic<int64_t> g_fail_countdown{0};
static std::atomic<uint64_t> g_launches{0};

void tg_note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

static thread_local int32_t g_cuda_error = 0;

void tg_note_cuda_error(cudaError_t e) { g_cuda_error = (int32_t)e; }

extern "C" int32_t tg_last_cuda_error(void) { return g_cuda_error; }

extern "C" uint64_t tg_launch_count(void) { return g_launches.load(); }

int tg_num_sms() {
    int dev = 0, sms = 0;
    (void)cudaGetDevice(&dev);
    (void)cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

int tg_smem_optin() {
    int dev = 0, v = 0;
    (void)cudaGetDevice(&dev);
    (void)cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v > 0 ? v : 48 * 1024;
}

// (device, kernel) pairs whose limit is already raised: the attribute is set
// once per kernel and device, not before every launch.
static std::mutex g_smem_mu;
static std::vector<std::pair<int, const void *>> g_smem_done;

int tg_allow_max_smem(const void *func) {
    int dev = 0, optin = 0;
    TG_TRY_CUDA(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lk(g_smem_mu);
        for (const auto &d : g_smem_done)
            if (d.first == dev && d.second == func) return TG_OK;
    }
    TG_TRY_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    cudaFuncAttributes fa{};
    TG_TRY_CUDA(cudaFuncGetAttributes(&fa, func));
    const int v = optin - (int)fa.sharedSizeBytes;
    if (v <= 0) return TG_EINVAL;
    TG_TRY_CUDA(cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, v));
    std::lock_guard<std::mutex> lk(g_smem_mu);
    g_smem_done.emplace_back(dev, func);
    return TG_OK;
}

extern "C" int tg_set_allocator(tg_alloc_fn alloc, tg_free_fn free_fn, void *ctx) {
    if ((alloc == nullptr) != (free_fn == nullptr)) return TG_EINVAL;
    g_alloc = alloc;
    g_free = free_fn;
    g_alloc_ctx = ctx;
    return TG_OK;
}

extern "C" int tg_debug_fail_alloc(int64_t n) {
    if (n < 0) return TG_EINVAL;
    g_fail_countdown.store(n);
    return TG_OK;
}

// Retained scratch: with a positive retention the library allocates from a
// pool of its own per device whose release threshold is that many bytes, so
// freed scratch stays mapped for the next call instead of going back to the
// device at each synchronisation.
constexpr int kMaxDevices = 64;
static std::mutex g_pool_mu;
static std::atomic<uint64_t> g_retain{0};
static cudaMemPool_t g_pools[kMaxDevices] = {};

static cudaMemPool_t lib_pool(int dev) {
    if (dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (!g_pools[dev]) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        uint64_t thr = g_retain.load();
        (void)cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
        g_pools[dev] = pool;
    }
    return g_pools[dev];
}

extern "C" int tg_set_memory_retention(uint64_t bytes) {
    g_retain.store(bytes);
    std::lock_guard<std::mutex> lk(g_pool_mu);
    for (int d = 0; d < kMaxDevices; ++d) {
        if (!g_pools[d]) continue;
        uint64_t thr = bytes;
        if (cudaMemPoolSetAttribute(g_pools[d], cudaMemPoolAttrReleaseThreshold, &thr) != cudaSuccess ||
            (bytes == 0 && cudaMemPoolTrimTo(g_pools[d], 0) != cudaSuccess)) {
            tg_note_cuda_error(cudaGetLastError());
            return TG_ECUDA;
        }
    }
    return TG_OK;
}

extern "C" int tg_trim_memory(void) {
    std::lock_guard<std::mutex> lk(g_pool_mu);
    for (int d = 0; d < kMaxDevices; ++d) {
        if (g_pools[d] && cudaMemPoolTrimTo(g_pools[d], 0) != cudaSuccess) {
            tg_note_cuda_error(cudaGetLastError());
            return TG_ECUDA;
        }
    }
    return TG_OK;
}

void *tg_dalloc(size_t bytes, cudaStream_t s) {
    int64_t c = g_fail_countdown.load();
    while (c > 0) {
        if (g_fail_countdown.compare_exchange_weak(c, c - 1)) {
            if (c == 1) return nullptr;  // the injected failure
            break;
        }
    }
    if (g_alloc) return g_alloc(bytes, s, g_alloc_ctx);
    void *p = nullptr;
    cudaMemPool_t pool = nullptr;
    if (g_retain.load() > 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) == cudaSuccess) pool = lib_pool(dev);
    }
    const cudaError_t e = pool ? cudaMallocFromPoolAsync(&p, bytes, pool, s) : cudaMallocAsync(&p, bytes, s);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    return p;
}

void tg_dfree(void *p, size_t bytes, cudaStream_t s) {
    if (!p) return;
    if (g_free) {
        g_free(p, bytes, s, g_alloc_ctx);
        return;
    }
    (void)cudaFreeAsync(p, s);
}

bool tg_is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

int tg_bitlen(uint64_t x) {
    int b = 0;
    while (x) {
        ++b;
        x >>= 1;
    }
    return b;
}

// ------------------------------------------------------------------ scans --
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

template <typename T>
__device__ T block_exclusive_scan(T v, T *warp_tot, T *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < (kScanThreads / 32) ? warp_tot[lane] : T(0);
        T wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < (kScanThreads / 32)) warp_tot[lane] = wi - w;
        if (lane == (kScanThreads / 32) - 1) *total = wi;
    }
    __syncthreads();
    T r = x - v + warp_tot[warp];
    __syncthreads();
    return r;
}

template <typename T>
__global__ void k_tile_reduce(const T *in, int64_t n, T *partial) {
    __shared__ T wt[kScanThreads / 32];
    __shared__ T tot;
    int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T s = 0;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q)
        if (base + q < n) s += in[base + q];
    (void)block_exclusive_scan<T>(s, wt, &tot);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

template <typename T>
__global__ void k_tile_scan(const T *in, T *out, int64_t n, const T *offsets) {
    __shared__ T wt[kScanThreads / 32];
    __shared__ T tot;
    int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T v[kScanItems];
    T s = 0;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        v[q] = (base + q < n) ? in[base + q] : T(0);
        s += v[q];
    }
    T run = block_exclusive_scan<T>(s, wt, &tot) + (offsets ? offsets[blockIdx.x] : T(0));
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        if (base + q < n) out[base + q] = run;
        run += v[q];
    }
}

template <typename T>
int scan_impl(const T *in, T *out, int64_t n, cudaStream_t s) {
    if (n <= 0) return TG_OK;
    int64_t blocks = (n + kScanTile - 1) / kScanTile;
    if (blocks == 1) {
        k_tile_scan<T><<<1, kScanThreads, 0, s>>>(in, out, n, nullptr); tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
        return TG_OK;
    }
    DevBuf<T> part;
    if (!part.alloc(blocks, s)) return TG_ENOMEM;
    k_tile_reduce<T><<<(unsigned)blocks, kScanThreads, 0, s>>>(in, n, part.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    TG_TRY(scan_impl<T>(part.p, part.p, blocks, s));
    k_tile_scan<T><<<(unsigned)blocks, kScanThreads, 0, s>>>(in, out, n, part.p); tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    return TG_OK;
}

}  // namespace

int tg_scan_u32(const uint32_t *in, uint32_t *out, int64_t n, cudaStream_t s) {
    return scan_impl<uint32_t>(in, out, n, s);
}
int tg_scan_i64(const int64_t *in, int64_t *out, int64_t n, cudaStream_t s) {
    return scan_impl<int64_t>(in, out, n, s);
}

// ------------------------------------------------------------- radix sort --
// LSD radix sort, 8-bit digits, one kernel per digit.  One pass over the keys
// counts the digits of every position; then each digit's kernel takes tiles of
// keys in order (a ticket per tile), ranks a tile's keys by their digit, learns
// the number of equal digits in the tiles before it from those tiles' published
// counts, and writes the tile in digit order, so the keys of one digit leave a
// tile as one run.  Stable.  Before, a digit took a histogram pass over the keys,
// a three-kernel scan of 256 counts per tile and a scatter of single keys.
//
// A tile's counts per digit are published in two steps, its own count and the
// sum over all tiles up to it, each a word with its state in the top bits.  A tile
// waits only for tiles of smaller tickets, which are running or done, and for at
// most TG_SORT_LOOKS idle looks at their words: then it counts the keys before it itself.
// Up to kSmallKeys keys one CTA makes all passes in shared memory.
//
// Measured (CSR build, before -> now): R-MAT-21 (33.6M draws) 14.6 -> 8.8 ms, ER
// 1M/5M 2.4 -> 1.75 ms, ER 100K/1M 0.79 -> 0.58 ms, ER-1000 0.34 -> 0.23 ms (33
// launches fewer).  A pass reads and writes every key once (16 or 24 B); the ranks
// of equal digits (one match per 32 keys) bound it.
namespace {

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr unsigned long long kSortOwn = 1ull << 62, kSortSum = 2ull << 62, kSortMask = kSortOwn - 1ull;
constexpr int kSmallThreads = 1024, kSmallItems = 12, kSmallKeys = kSmallThreads * kSmallItems;

// counts[pass][digit] over all keys
__global__ void __launch_bounds__(kSortThreads) k_sort_digits(const uint64_t *in, int64_t n, int passes,
                                                              uint32_t *counts) {
    extern __shared__ uint32_t h[];  // [passes][256]
    for (int q = threadIdx.x; q < passes * 256; q += blockDim.x) h[q] = 0u;
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += step) {
        const uint64_t k = in[i];
        const unsigned act = __activemask();
        for (int p = 0; p < passes; ++p) {
            const int d = (int)((k >> (8 * p)) & 255u);
            int same;  // high digits are often one value: one add for the warp
            __match_all_sync(act, d, &same);
            if (!same)
                atomicAdd(&h[p * 256 + d], 1u);
            else if ((threadIdx.x & 31) == __ffs(act) - 1)
                atomicAdd(&h[p * 256 + d], (uint32_t)__popc(act));
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < passes * 256; q += blockDim.x)
        if (h[q]) atomicAdd(&counts[q], h[q]);
}

// Ranks of a warp's keys among its equal digits, in order; cnt: the warp's 256
// counts, zero on entry.  `left`: keys of the warp's run that are inside n.
template <int kItems>
__device__ __forceinline__ void warp_ranks(const uint64_t (&key)[kItems], int64_t left, int shift,
                                           uint32_t *cnt, uint32_t (&rank)[kItems]) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int c = 0; c < kItems; ++c) {
        const bool valid = c * 32 + lane < left;
        const uint32_t d = valid ? (uint32_t)((key[c] >> shift) & 255u) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = valid ? cnt[d] : 0u;
        __syncwarp();
        rank[c] = before + __popc(peers & lt);
        if (valid && lane == 31 - __clz(peers)) cnt[d] = before + __popc(peers);
        __syncwarp();
    }
}

// Exclusive sum of one value per thread over the first 256 threads.  wsum: 8
// words; called by all threads of the CTA.
__device__ __forceinline__ uint32_t scan256(uint32_t v, uint32_t *wsum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (tid < 256 && lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t add = 0;
    if (tid < 256)
        for (int w = 0; w < warp; ++w) add += wsum[w];
    __syncthreads();
    return incl - v + add;
}

// Thread d < 256: the warps' counts of digit d become their first places among
// the tile's keys of digit d; returns the tile's count.
template <int kWarps>
__device__ __forceinline__ uint32_t digit_total(uint32_t (*cnt)[256]) {
    uint32_t own = 0;
    if (threadIdx.x < 256) {
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = cnt[w][threadIdx.x];
            cnt[w][threadIdx.x] = own;
            own += c;
        }
    }
    return own;
}

template <bool kVals>
struct SortSmem {
    uint64_t key[kSortTile];
    uint32_t val[kVals ? kSortTile : 1];
    uint32_t cnt[kSortWarps][256];
    uint32_t start[256];  // first slot of a digit in the tile
    uint32_t dest[256];   // output place of a digit's slots, less the slot
    uint32_t wsum[8];
    uint32_t tile, late;
};

// One digit: tile t's word of digit d is state[t 256 + d].
template <bool kVals>
__global__ void __launch_bounds__(kSortThreads) k_sort_digit(const uint64_t *in, uint64_t *out,
                                                             const uint32_t *vin, uint32_t *vout,
                                                             int64_t n, int shift, const uint32_t *counts,
                                                             unsigned long long *state, uint32_t *ticket,
                                                             int looks) {
    extern __shared__ __align__(16) unsigned char smem[];
    SortSmem<kVals> &sm = *reinterpret_cast<SortSmem<kVals> *>(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        sm.tile = atomicAdd(ticket, 1u);
        sm.late = 0u;
    }
    for (int q = tid; q < kSortWarps * 256; q += kSortThreads) (&sm.cnt[0][0])[q] = 0u;
    __syncthreads();
    const uint32_t tile = sm.tile;
    const int64_t t0 = (int64_t)tile * kSortTile;
    const int64_t w0 = t0 + (int64_t)warp * 32 * kSortItems;  // this warp's run of keys
    const int count = (int)min((int64_t)kSortTile, n - t0);
    uint64_t key[kSortItems];
    uint32_t val[kSortItems], rank[kSortItems];
#pragma unroll
    for (int c = 0; c < kSortItems; ++c) {
        const int64_t i = w0 + c * 32 + lane;
        key[c] = i < n ? in[i] : 0ull;
        val[c] = kVals && i < n ? vin[i] : 0u;
    }
    warp_ranks<kSortItems>(key, n - w0, shift, sm.cnt[warp], rank);
    __syncthreads();
    const uint32_t own = digit_total<kSortWarps>(sm.cnt);
    volatile unsigned long long *word = state + (size_t)tile * 256 + (tid & 255);
    if (tid < 256) *word = own | (tile == 0 ? kSortSum : kSortOwn);
    const uint32_t first = scan256(own, sm.wsum);
    const uint32_t base = scan256(tid < 256 ? counts[tid] : 0u, sm.wsum);
    unsigned long long sum = 0;  // equal digits of the tiles before this one
    if (tid < 256) {
        int spin = 0;
        for (int64_t t = (int64_t)tile - 1; t >= 0;) {
            const unsigned long long w = *(volatile unsigned long long *)(state + (size_t)t * 256 + tid);
            if (!(w & ~kSortMask) || looks < 0) {
                if (++spin > looks) {
                    sm.late = 1u;
                    break;
                }
                continue;
            }
            sum += w & kSortMask;
            if ((w & ~kSortMask) == kSortSum) break;
            --t;
        }
    }
    __syncthreads();
    if (sm.late) {  // a tile before this one is late: count its digits and all others'
        if (tid < 256) sm.dest[tid] = 0u;
        __syncthreads();
        for (int64_t i = tid; i < t0; i += kSortThreads) atomicAdd(&sm.dest[(in[i] >> shift) & 255u], 1u);
        __syncthreads();
        if (tid < 256) sum = sm.dest[tid];
        __syncthreads();
    }
    if (tid < 256) {
        if (tile > 0) *word = (sum + own) | kSortSum;
        sm.start[tid] = first;
        sm.dest[tid] = base + (uint32_t)sum - first;
    }
    __syncthreads();
    // the tile in digit order
#pragma unroll
    for (int c = 0; c < kSortItems; ++c) {
        if (w0 + c * 32 + lane >= n) continue;
        const uint32_t d = (uint32_t)((key[c] >> shift) & 255u);
        const uint32_t slot = sm.start[d] + sm.cnt[warp][d] + rank[c];
        sm.key[slot] = key[c];
        if (kVals) sm.val[slot] = val[c];
    }
    __syncthreads();
    for (int slot = tid; slot < count; slot += kSortThreads) {
        const uint64_t k = sm.key[slot];
        const uint32_t at = sm.dest[(k >> shift) & 255u] + (uint32_t)slot;
        out[at] = k;
        if (kVals) vout[at] = sm.val[slot];
    }
}

template <bool kVals>
struct SmallSmem {
    uint64_t key[kSmallKeys];
    uint32_t val[kVals ? kSmallKeys : 1];
    uint32_t cnt[kSmallThreads / 32][256];
    uint32_t start[256], wsum[8];
};

// All digits of at most kSmallKeys keys, in place.
template <bool kVals>
__global__ void __launch_bounds__(kSmallThreads) k_sort_small(uint64_t *keys, uint32_t *vals, int n, int bits) {
    extern __shared__ __align__(16) unsigned char smem[];
    SmallSmem<kVals> &sm = *reinterpret_cast<SmallSmem<kVals> *>(smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = ((n + kSmallThreads - 1) / kSmallThreads) * 32;  // keys of a warp's run
    const int w0 = warp * per;
    const int left = min(per, n - w0);
    uint64_t key[kSmallItems];
    uint32_t val[kSmallItems], rank[kSmallItems];
#pragma unroll
    for (int c = 0; c < kSmallItems; ++c) {
        const bool in = c * 32 + lane < left;
        key[c] = in ? keys[w0 + c * 32 + lane] : 0ull;
        val[c] = kVals && in ? vals[w0 + c * 32 + lane] : 0u;
    }
    for (int shift = 0; shift < bits; shift += 8) {
        for (int q = tid; q < kSmallThreads / 32 * 256; q += kSmallThreads) (&sm.cnt[0][0])[q] = 0u;
        __syncthreads();
        warp_ranks<kSmallItems>(key, left, shift, sm.cnt[warp], rank);
        __syncthreads();
        const uint32_t first = scan256(digit_total<kSmallThreads / 32>(sm.cnt), sm.wsum);
        if (tid < 256) sm.start[tid] = first;
        __syncthreads();
#pragma unroll
        for (int c = 0; c < kSmallItems; ++c) {
            if (c * 32 + lane >= left) continue;
            const uint32_t d = (uint32_t)((key[c] >> shift) & 255u);
            const uint32_t slot = sm.start[d] + sm.cnt[warp][d] + rank[c];
            sm.key[slot] = key[c];
            if (kVals) sm.val[slot] = val[c];
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < kSmallItems; ++c) {
            if (c * 32 + lane >= left) continue;
            key[c] = sm.key[w0 + c * 32 + lane];
            if (kVals) val[c] = sm.val[w0 + c * 32 + lane];
        }
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < kSmallItems; ++c) {
        if (c * 32 + lane >= left) continue;
        keys[w0 + c * 32 + lane] = key[c];
        if (kVals) vals[w0 + c * 32 + lane] = val[c];
    }
}

template <bool kVals>
int sort_impl(uint64_t *keys, uint64_t *tmp, uint32_t *vals, uint32_t *vtmp, int64_t n, int bits,
              cudaStream_t s, uint64_t **result, uint32_t **vresult, int looks) {
    *result = keys;
    if (vresult) *vresult = vals;
    if (n <= 1 || bits <= 0) return TG_OK;
    if (n >= (int64_t)UINT32_MAX) return TG_EOVERFLOW;
    if (n <= kSmallKeys) {
        TG_TRY(tg_allow_max_smem((const void *)k_sort_small<kVals>));
        k_sort_small<kVals><<<1, kSmallThreads, sizeof(SmallSmem<kVals>), s>>>(keys, vals, (int)n, bits);
        tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
        return TG_OK;
    }
    const int passes = (bits + 7) / 8;
    const int64_t tiles = (n + kSortTile - 1) / kSortTile;
    // one zeroed block: tickets, digit counts, tile words
    const size_t words = (size_t)tiles * 256 * passes;
    DevBuf<unsigned long long> buf;
    if (!buf.alloc(words + (size_t)passes * 129, s)) return TG_ENOMEM;
    TG_TRY_CUDA(cudaMemsetAsync(buf.p, 0, (words + (size_t)passes * 129) * 8, s));
    uint32_t *counts = reinterpret_cast<uint32_t *>(buf.p + words), *tickets = counts + passes * 256;
    const int64_t hgrid = std::min<int64_t>((n + 4 * kSortThreads - 1) / (4 * kSortThreads), (int64_t)tg_num_sms() * 4);
    k_sort_digits<<<(unsigned)hgrid, kSortThreads, (size_t)passes * 1024, s>>>(keys, n, passes, counts);
    tg_note_launch();
    TG_TRY_CUDA(cudaGetLastError());
    TG_TRY(tg_allow_max_smem((const void *)k_sort_digit<kVals>));
    uint64_t *a = keys, *b = tmp;
    uint32_t *va = vals, *vb = vtmp;
    for (int p = 0; p < passes; ++p) {
        k_sort_digit<kVals><<<(unsigned)tiles, kSortThreads, sizeof(SortSmem<kVals>), s>>>(
            a, b, va, vb, n, 8 * p, counts + p * 256, buf.p + (size_t)p * tiles * 256, tickets + p, looks);
        tg_note_launch();
        TG_TRY_CUDA(cudaGetLastError());
        std::swap(a, b);
        std::swap(va, vb);
    }
    *result = a;
    if (vresult) *vresult = va;
    return TG_OK;
}

}  // namespace

int tg_radix_sort_kv(uint64_t *keys, uint64_t *tmp, uint32_t *vals, uint32_t *vtmp, int64_t n,
                     int bits, cudaStream_t s, uint64_t **result, uint32_t **vresult, int looks) {
    return sort_impl<true>(keys, tmp, vals, vtmp, n, bits, s, result, vresult, looks);
}

int tg_radix_sort_u64(uint64_t *keys, uint64_t *tmp, int64_t n, int bits, cudaStream_t s,
                      uint64_t **result, int looks) {
    return sort_impl<false>(keys, tmp, nullptr, nullptr, n, bits, s, result, nullptr, looks);
}
