// cs_order.cu -- the single-set interval count of product orders
// (cs_order.cuh): ranks of the two coordinates, the table D, the pair count.
//
// Ranks.  Callers' coordinates may be distributed anyhow.  Up to 8192 elements
// one CTA ranks them by buckets in shared memory, or, where a bucket holds many of
// them, sorts them there.  Beyond, the ranks come from sorted tiles: every tile of 4096 elements is sorted in shared
// memory, and an element's rank is the sum over the tiles of its lower (or
// upper) bound -- n / 4096 binary searches of twelve steps, under 1% of the
// n^2 / 2 pairs counted after it and the same for every distribution.
#include <atomic>

#include "cs_kernels.cuh"
#include "cs_launch.cuh"
#include "cs_order.cuh"

namespace cs {

namespace {

constexpr int kTile = 4096;          // elements per sorted tile
constexpr int kSortThreads = 1024;   // two compare-exchanges per thread and stage
constexpr int64_t kSmallSet = 8192;  // largest set ranked by one CTA

// The two orders' keys: u ascending, v descending, and the other way round.
// Coordinates lie in [0, 2^31).  Elements equal in both coordinates are
// ordered by label in u and against it in v (their ranks then never agree, as
// unrelated elements' must not).
__device__ __forceinline__ uint64_t order_key(const int32_t* __restrict__ coords, int64_t n, int64_t e, int stream) {
    const uint32_t u = uint32_t(coords[e]), v = uint32_t(coords[n + e]);
    return stream == 0 ? (uint64_t(u) << 31) | (0x7FFFFFFFu - v) : (uint64_t(v) << 31) | (0x7FFFFFFFu - u);
}

// Sort tile blockIdx.x of stream blockIdx.y: its keys ascending to sorted,
// each element's place in its tile to place.  A bitonic network of
// (key, label) pairs.
__global__ void __launch_bounds__(kSortThreads) k_order_sort(const int32_t* __restrict__ coords, int64_t n, int stream0,
                                                          uint64_t* __restrict__ sorted,
                                                          uint16_t* __restrict__ place) {
    __shared__ uint64_t sk[kTile];
    __shared__ uint16_t si[kTile];
    const int stream = stream0 + blockIdx.y;
    const int64_t e0 = int64_t(blockIdx.x) * kTile;
    const int64_t npad = int64_t(gridDim.x) * kTile;
    for (int i = threadIdx.x; i < kTile; i += kSortThreads) {
        sk[i] = e0 + i < n ? order_key(coords, n, e0 + i, stream) : ~0ull;  // past n: behind every key
        // v: equal keys in descending label, so the label's complement is compared
        si[i] = uint16_t(stream == 0 ? i : kTile - 1 - i);
    }
    for (int size = 2; size <= kTile; size <<= 1) {
        for (int j = size >> 1; j > 0; j >>= 1) {
            __syncthreads();
#pragma unroll
            for (int t = threadIdx.x; t < kTile / 2; t += kSortThreads) {
                const int lo = 2 * t - (t & (j - 1)), hi = lo + j;
                const uint64_t a = sk[lo], b = sk[hi];
                const uint16_t ia = si[lo], ib = si[hi];
                const bool greater = a > b || (a == b && ia > ib);
                if (greater == ((lo & size) == 0)) {
                    sk[lo] = b;
                    sk[hi] = a;
                    si[lo] = ib;
                    si[hi] = ia;
                }
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kTile; i += kSortThreads) {
        const int64_t at = int64_t(blockIdx.y) * npad + e0;
        sorted[at + i] = sk[i];
        place[at + (stream == 0 ? si[i] : kTile - 1 - si[i])] = uint16_t(i);
    }
}

// Rank contributions of sorted tile blockIdx.y to every element of tiles
// blockIdx.x.., added into rank[stream] (zeroed before).  An equal key in an
// earlier tile comes first in u and last in v.
constexpr int kRankElems = 4;  // elements per thread
__global__ void __launch_bounds__(256) k_order_rank(const int32_t* __restrict__ coords, int64_t n, int stream0,
                                                    const uint64_t* __restrict__ sorted,
                                                    const uint16_t* __restrict__ place, int64_t npad,
                                                    uint32_t* __restrict__ rank) {
    __shared__ uint64_t sk[kTile];
    const int stream = stream0 + blockIdx.z;
    const int64_t tile = blockIdx.y;
    const uint64_t* src = sorted + int64_t(blockIdx.z) * npad + tile * kTile;
    for (int i = threadIdx.x; i < kTile; i += 256) sk[i] = src[i];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRankElems; ++k) {
        const int64_t e = int64_t(blockIdx.x) * (256 * kRankElems) + k * 256 + threadIdx.x;
        if (e >= n) return;
        uint32_t r;
        if (e / kTile == tile) {
            r = place[int64_t(blockIdx.z) * npad + e];
        } else {
            const uint64_t key = order_key(coords, n, e, stream);
            const bool upper = (tile < e / kTile) == (stream == 0);  // count the tile's equal keys too
            const uint64_t bound = upper ? key + 1 : key;            // keys below 2^62: #{< key + 1} = #{<= key}
            r = 0;
#pragma unroll
            for (int step = kTile / 2; step > 0; step >>= 1) r += sk[r + step - 1] < bound ? step : 0;
            r += sk[r] < bound ? 1u : 0u;
        }
        atomicAdd(rank + int64_t(blockIdx.z) * n + e, r);
    }
}

// p and its inverse.  rank_u NULL: the labels are in u order already.
__global__ void __launch_bounds__(256) k_order_scatter(int64_t n, const uint32_t* __restrict__ rank_u,
                                                       const uint32_t* __restrict__ rank_v, int32_t* __restrict__ p,
                                                       int32_t* __restrict__ q) {
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n; e += int64_t(gridDim.x) * blockDim.x) {
        const int32_t a = rank_u ? int32_t(rank_u[e]) : int32_t(e), v = int32_t(rank_v[e]);
        p[a] = v;
        q[v] = a;
    }
}

// A small set: the ranks of v by one CTA, and those of u by the other CTA of
// a cluster of two when the labels are not in u order; then p and q, and the
// histogram cleared.  (One CTA after the other took 9 us more at n = 4096.)
template <bool kByU>
__device__ __forceinline__ void order_ranks_small(const int32_t* __restrict__ coords, int n, int lgP,
                                                  uint32_t* rank_u, uint32_t* rank_v, int32_t* __restrict__ p,
                                                  int32_t* __restrict__ q, unsigned long long* __restrict__ hist,
                                                  int len) {
    extern __shared__ __align__(16) uint8_t smem_ord[];
    const int P = 1 << lgP, ctas = kByU ? 1 : 2;
    uint64_t* sk = reinterpret_cast<uint64_t*>(smem_ord);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(sk + P);
    uint32_t* slot = cnt + P;
    uint32_t* rank = slot + P;
    launch_dependents();
    for (int k = blockIdx.x * kRankThreads + threadIdx.x; k < len; k += ctas * kRankThreads) hist[k] = 0ull;
    const bool v = kByU || blockIdx.x == 1;
    order_keys_smem(v ? coords + n : coords, v ? coords : coords + n, n, sk);
    if (v)
        rank_keys_smem<true, true>(n, lgP, sk, cnt, slot, rank);
    else
        rank_keys_smem<false, true>(n, lgP, sk, cnt, slot, rank);
    if (kByU) {
        for (int e = threadIdx.x; e < n; e += kRankThreads) {
            const int r = int(rank[e]);
            p[e] = r;
            q[r] = e;
        }
        return;
    }
    for (int e = threadIdx.x; e < n; e += kRankThreads) (v ? rank_v : rank_u)[e] = rank[e];
    cluster_sync();
    for (int e = blockIdx.x * kRankThreads + threadIdx.x; e < n; e += 2 * kRankThreads) {
        const int a = int(__ldcg(rank_u + e)), r = int(__ldcg(rank_v + e));
        p[a] = r;
        q[r] = a;
    }
}
__global__ void __launch_bounds__(kRankThreads) k_order_ranks_v(const int32_t* __restrict__ coords, int n, int lgP,
                                                                int32_t* __restrict__ p, int32_t* __restrict__ q,
                                                                unsigned long long* __restrict__ hist, int len) {
    order_ranks_small<true>(coords, n, lgP, nullptr, nullptr, p, q, hist, len);
}
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kRankThreads)
    k_order_ranks_uv(const int32_t* __restrict__ coords, int n, int lgP, uint32_t* rank_u, uint32_t* rank_v,
                     int32_t* __restrict__ p, int32_t* __restrict__ q, unsigned long long* __restrict__ hist, int len) {
    order_ranks_small<false>(coords, n, lgP, rank_u, rank_v, p, q, hist, len);
}

__global__ void __launch_bounds__(kOrdBuildThreads) k_order_table(OrderSet s) {
    launch_dependents();
    wait_for_primary();
    order_build_rows(s, blockIdx.x);
}

constexpr int kCountWarps = 32;
constexpr int kCountThreads = 32 * kCountWarps;
constexpr int kCountStage = kCountWarps * 32 * int(sizeof(int2));
// Bins of the shared histogram: all that one CTA's shared memory holds
// beside the warps' stages.  A 2D order's counts fall off with k (3% of the
// pairs of a 2^17 order lie past 55296 bins), so wide sets spill little.
constexpr int kCountBins = 55296;

// Bands per column chunk, at most, and the tasks a warp takes between two
// flushes of the bins: a CTA's adds in between stay below 2^32 however few CTAs
// share the pairs, and so does every bin.  (One flush at the end holds up to n = 2^20 on 152 SMs, not on
// 128.)  Up to n = 2^18 a warp's whole share is less than this on 152 SMs.
constexpr int kCountMaxM = 16;
constexpr int64_t kFlushTasks = 256;
static_assert(kFlushTasks * kCountWarps * kOrdBand * (kOrdBand * kCountMaxM) < (int64_t(1) << 32),
              "a bin holds every pair between two flushes");

// One CTA per SM, its warps striding over the tasks.
__global__ void __launch_bounds__(kCountThreads, 1) k_count_order(OrderSet s, int64_t tasks, int m, int bins,
                                                                  unsigned long long* hist) {
    extern __shared__ __align__(16) uint8_t smem_ord[];
    int2* stage = reinterpret_cast<int2*>(smem_ord) + 32 * (threadIdx.x >> 5);
    uint32_t* shist = reinterpret_cast<uint32_t*>(smem_ord + kCountStage);
    for (int k = threadIdx.x; k < bins; k += kCountThreads) shist[k] = 0u;
    wait_for_primary();
    __syncthreads();
    const uint32_t hist_s = smem_u32(shist);
    const int64_t warps = int64_t(gridDim.x) * kCountWarps;
    int64_t t = int64_t(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    for (int64_t end = kFlushTasks * warps;; end += kFlushTasks * warps) {
        for (const int64_t stop = end < tasks ? end : tasks; t < stop; t += warps) {
            int A, C;
            order_decode(t, m, A, C);
            order_task(s, A, C, kOrdBand * m, hist_s, bins, hist, stage);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < bins; k += kCountThreads) {
            const uint32_t c = shist[k];
            if (c) {
                atomicAdd(hist + k, (unsigned long long)c);
                shist[k] = 0u;
            }
        }
        if (end >= tasks) return;
        __syncthreads();
    }
}

struct OrderLayout {
    size_t p, q, R, rank, place, sorted, D, total;
    int64_t npad;
};

OrderLayout order_layout(int64_t n) {
    OrderLayout L;
    L.npad = (n + kTile - 1) / kTile * kTile;
    size_t off = sizeof(WsHeader);
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    L.p = take(size_t(n) * 4);
    L.q = take(size_t(n) * 4);
    L.R = take(size_t(n) * 4);
    L.D = take(order_table_bytes(n));
    // the ranks' scratch ends before the table begins to be written
    size_t at = L.D;
    auto alias = [&](size_t bytes) {
        const size_t x = at;
        at = align_up(at + bytes, 256);
        return x;
    };
    L.sorted = L.place = at;
    L.rank = alias(size_t(n) * 8);
    if (n > kSmallSet) {
        L.sorted = alias(size_t(L.npad) * 16);
        L.place = alias(size_t(L.npad) * 4);
    }
    L.total = off > at ? off : at;
    return L;
}

std::atomic<bool> g_order_attr[64];  // per device: the large-shared-memory attributes are set

}  // namespace

bool order_kind(int kind) { return kind == CS_2D_ORDER || kind == CS_2D_DIAMOND || kind == CS_2D_SQUARE; }

// Up to the largest set that the count is checked at (its table takes 4.3 GB there).
bool order_count_fits(int kind, int64_t n) { return order_kind(kind) && n >= 2 && n <= (int64_t(1) << 20); }

size_t order_workspace_bytes(int64_t n) { return order_layout(n).total; }

cudaError_t launch_count_order(int kind, int64_t n, const int32_t* coords, int64_t* hist, void* workspace,
                               cudaStream_t st) {
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    const OrderLayout L = order_layout(n);
    const bool by_u = kind == CS_2D_ORDER;  // labels are in u order: only v is ranked
    const int streams = by_u ? 1 : 2, stream0 = by_u ? 1 : 0;
    uint64_t* sorted = reinterpret_cast<uint64_t*>(ws + L.sorted);
    uint16_t* place = reinterpret_cast<uint16_t*>(ws + L.place);
    uint32_t* rank = reinterpret_cast<uint32_t*>(ws + L.rank);
    OrderSet s;
    int32_t* p = reinterpret_cast<int32_t*>(ws + L.p);
    int32_t* q = reinterpret_cast<int32_t*>(ws + L.q);
    s.p = p;
    s.q = q;
    s.R = reinterpret_cast<int32_t*>(ws + L.R);
    s.D = reinterpret_cast<uint2*>(ws + L.D);
    s.n = int32_t(n);
    s.W = order_words(n);
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const int64_t len = n > 1 ? n - 1 : 1;
    const int most = kCountStage + (kCountBins + 1) * 4;
    if (!g_order_attr[dev]) {
        if ((err = cudaFuncSetAttribute(k_count_order, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) !=
                cudaSuccess ||
            (err = cudaFuncSetAttribute(k_order_ranks_v, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        int(kSmallSet) * 20)) != cudaSuccess ||
            (err = cudaFuncSetAttribute(k_order_ranks_uv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        int(kSmallSet) * 20)) != cudaSuccess)
            return err;
        g_order_attr[dev] = true;
    }
    if (n <= kSmallSet) {
        int lgP = 10;
        while ((int64_t(1) << lgP) < n) ++lgP;
        unsigned long long* h = reinterpret_cast<unsigned long long*>(hist);
        if (by_u)
            k_order_ranks_v<<<1, kRankThreads, size_t(20) << lgP, st>>>(coords, int(n), lgP, p, q, h, int(len));
        else
            k_order_ranks_uv<<<2, kRankThreads, size_t(20) << lgP, st>>>(coords, int(n), lgP, rank, rank + n, p, q, h,
                                                                        int(len));
    } else {
        if ((err = cudaMemsetAsync(hist, 0, size_t(len) * 8, st)) != cudaSuccess ||
            (err = cudaMemsetAsync(rank, 0, size_t(streams) * size_t(n) * 4, st)) != cudaSuccess)
            return err;
        const unsigned tiles = unsigned(L.npad / kTile);
        k_order_sort<<<dim3(tiles, unsigned(streams)), kSortThreads, 0, st>>>(coords, n, stream0, sorted, place);
        k_order_rank<<<dim3(unsigned((n + 256 * kRankElems - 1) / (256 * kRankElems)), tiles, unsigned(streams)), 256,
                       0, st>>>(coords, n, stream0, sorted, place, L.npad, rank);
        const int64_t blocks = (n + 255) / 256;
        k_order_scatter<<<unsigned(blocks < 2432 ? blocks : 2432), 256, 0, st>>>(n, by_u ? nullptr : rank,
                                                                              by_u ? rank : rank + n, p, q);
    }
    if ((err = cudaGetLastError()) != cudaSuccess ||
        (err = launch_after(k_order_table, dim3(unsigned(order_build_blocks(n))), kOrdBuildThreads, 0, st, s)) !=
            cudaSuccess)
        return err;

    // Column chunks of 64 m: long enough to amortise a task's start (two
    // dependent gathers), short enough that the warps get several tasks each.
    const int sms = device_sm_count();
    int m = kCountMaxM;
    while (m > 1 && order_tasks(n, m) < int64_t(sms) * kCountWarps * 12) m >>= 1;
    const int64_t tasks = order_tasks(n, m);
    const int bins = int(len < kCountBins ? len : kCountBins);
    const int smem = kCountStage + (bins + 1) * 4;
    // small sets: at least a warp task for each of a few warps of a CTA, so
    // that few CTAs flush their histograms
    int64_t grid = (tasks + 7) / 8;
    if (grid > sms) grid = sms;
    unsigned long long* h = reinterpret_cast<unsigned long long*>(hist);
    return launch_after(k_count_order, dim3(unsigned(grid)), kCountThreads, size_t(smem), st, s, tasks, m, bins, h);
}

}  // namespace cs
