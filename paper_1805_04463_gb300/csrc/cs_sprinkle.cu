// cs_sprinkle.cu -- sprinkling on the device (Section "Coordinate Generation",
// Appendix "Causal Set Sprinklings": 1+1, 2+1 and 3+1 Minkowski diamonds and
// the 1+1 de Sitter slab of Section "Spacetime Region Considered").
//
// Coordinates are drawn independently per element from the counter-based
// generator, then elements are sorted by time (Section "Pairwise
// Relations").  The sort is an exact ranking: every element gets
// rank = #{f : (key_f, f) < (key_e, e)}.  Keys are bucketed on their top 10
// to 16 bits, about one bucket per element (counted while the keys are drawn,
// a scan, a fill), and each element compares itself only with its bucket --
// O(n) work for the hashed / uniform keys used here, and the same ranks for
// any bucket fill order.  Four launches; the first form, with one launch per
// step and key stream and a one-block scan, spent 125 us on a set of 16384
// elements and 240 us on a 2D order of 1024.
#include <atomic>
#include <cmath>
#include <mutex>
#include <vector>

#include "cs_kernels.cuh"
#include "cs_launch.cuh"
#include "cs_sprinkle.cuh"

namespace cs {

namespace {

constexpr int kMaxDevices = 64;

// Cumulative sec^2 mass of the slab up to the end of each eta cell, scaled to
// 2^53.  With unit = 2 pi / 2^20 and t0 = tan((G + 1/2) unit), cell g ends
// at x_g = (tan((g + 1/2) unit) + t0) / (2 t0) (the density sec^2(eta) /
// (2 tan eta_0) integrated from -eta_0); this exact expression, in double
// with the C library's tan, is part of the generator's definition, so the
// table is built on the host.
static __device__ uint64_t g_ds_thresholds[kDsTable];
std::atomic<const uint64_t*> g_ds_ptr[kMaxDevices];
std::mutex g_ds_mu;

std::vector<uint64_t> ds_thresholds_host() {
    std::vector<uint64_t> t(kDsTable);
    const double unit = 2.0 * 3.14159265358979323846 / 1048576.0;
    const double t0 = std::tan((double(kDsCells) + 0.5) * unit);
    for (int i = 0; i < kDsTable; ++i) {
        const double g = double(i - kDsCells);
        const double x = (std::tan((g + 0.5) * unit) + t0) / (2.0 * t0);
        t[i] = static_cast<uint64_t>(x * 9007199254740992.0);  // x * 2^53
    }
    return t;
}

constexpr int kMinBucketBits = 10, kMaxBucketBits = 16;
constexpr int kThreads = 256;
constexpr int kScanBuckets = 1024;  // buckets per block of the scan
constexpr int64_t kSmallSet = 2048;  // largest set one CTA sprinkles alone

// About one bucket per element: the ranks stay O(n) and a small set does not
// scan 65536 buckets.
int bucket_bits(int64_t n) {
    int b = kMinBucketBits;
    while (b < kMaxBucketBits && (int64_t(1) << b) < n) ++b;
    return b;
}

// Scratch of a sprinkle.  A 2D order ranks two key streams (u and v), side by
// side in the same launches; the other kinds rank one and keep the drawn
// coordinates in raw.
struct SprinkleScratch {
    uint64_t* key[2];
    int32_t* raw;        // [dim][n], not for a 2D order
    uint32_t* arrival[2];  // position of an element within its bucket
    uint32_t* slot[2];     // bucket by bucket, the elements
    uint32_t* count[2];    // elements per bucket (zeroed before the keys)
    uint32_t* start[2];    // first slot of a bucket; start[buckets] = n
};

// Draw element e < n of a set: its sort key (two for a 2D order) and, for the
// other kinds, its coordinates.  All lanes of a warp (e = n or more: nothing
// is drawn).  false: no rejection attempt was accepted.
template <int KIND>
__device__ __forceinline__ bool draw_element(uint64_t seed, int64_t n, int64_t e, const uint64_t* __restrict__ thr,
                                             int32_t (&c)[4], uint64_t (&key)[2]) {
    if constexpr (KIND == CS_3D_DIAMOND || KIND == CS_4D_DIAMOND) {
        constexpr int D = KIND == CS_3D_DIAMOND ? 3 : 4;
        const uint32_t todo = __ballot_sync(0xffffffffu, e < n);
        return draw_diamond<D>(todo, stream_key(seed, D == 3 ? kStreamDiamond3 : kStreamDiamond4), e, c, key[0]) || e >= n;
    }
    if (e >= n) return true;
    if constexpr (KIND == CS_2D_ORDER)
        draw_2d_order(stream_key(seed, kStreamOrderU), stream_key(seed, kStreamOrderV), e, key[0], key[1]);
    else if constexpr (KIND == CS_2D_DIAMOND)
        key[0] = draw_2d_diamond(stream_key(seed, kStreamDiamond2), e, c[0], c[1]);
    else if constexpr (KIND == CS_2D_SQUARE)
        key[0] = draw_2d_square(stream_key(seed, kStreamSquare), e, c[0], c[1]);
    else if constexpr (KIND == CS_2D_CYLINDER)
        key[0] = draw_2d_cylinder(stream_key(seed, kStreamCylinder), e, c[0], c[1]);
    else if constexpr (KIND == CS_2D_DS_SLAB)
        key[0] = draw_ds_slab(stream_key(seed, kStreamDeSitter), e, thr, c[0], c[1]);
    return true;
}

constexpr int kind_dim(int kind) { return kind == CS_4D_DIAMOND ? 4 : kind == CS_3D_DIAMOND ? 3 : 2; }

// Keys, raw coordinates and bucket counts in one pass; the count's old value
// is the element's place in its bucket, so the fill needs no second atomic.
template <int KIND>
__global__ void __launch_bounds__(kThreads) k_keys(int64_t n, uint64_t seed, const uint64_t* __restrict__ thr,
                                                   SprinkleScratch s, int bits, WsHeader* hdr) {
    launch_dependents();
    const int64_t first = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    for (int64_t e = first; e - (threadIdx.x & 31) < n; e += int64_t(gridDim.x) * blockDim.x) {  // whole warps
        int32_t c[4];
        uint64_t key[2];
        if (!draw_element<KIND>(seed, n, e, thr, c, key)) set_status(hdr, CS_ERANGE);
        if (e >= n) continue;
#pragma unroll
        for (int q = 0; q < (KIND == CS_2D_ORDER ? 2 : 1); ++q) {
            s.key[q][e] = key[q];
            s.arrival[q][e] = atomicAdd(&s.count[q][key[q] >> (64 - bits)], 1u);
        }
        if constexpr (KIND != CS_2D_ORDER) {
#pragma unroll
            for (int k = 0; k < kind_dim(KIND); ++k) s.raw[k * n + e] = c[k];
        }
    }
}

// Exclusive scan of the bucket counts, grid (buckets / 1024, key streams).
// Each block sums every count before its own 1024 (at most 256 KB, read from
// L2 in 16-byte words) and scans its own, so the blocks need not wait on one
// another.  One block that walked all 65536 buckets, each thread its own run
// of 64, took 103-110 us whatever n was (16-byte sectors of 64 separate
// lines per thread and store); this takes about 5.
constexpr int kScanThreads = 1024;  // the last blocks' sums in two rounds of loads
__global__ void __launch_bounds__(kScanThreads) k_bucket_scan(SprinkleScratch s, int64_t n) {
    launch_dependents();
    wait_for_primary();
    const uint32_t* count = s.count[blockIdx.y];
    uint32_t* start = s.start[blockIdx.y];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint4* c4 = reinterpret_cast<const uint4*>(count);
    uint32_t before = 0;
#pragma unroll 8
    for (int g = t; g < int(blockIdx.x) * (kScanBuckets / 4); g += kScanThreads) {
        const uint4 v = c4[g];
        before += v.x + v.y + v.z + v.w;
    }
    const bool mine = t < kScanBuckets / 4;  // threads with own buckets, four each
    const uint4 own = mine ? c4[blockIdx.x * (kScanBuckets / 4) + t] : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t sum = own.x + own.y + own.z + own.w;
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
        before += __shfl_xor_sync(0xffffffffu, before, o);
    }
    __shared__ uint32_t wsum[kScanThreads / 32], wbefore[kScanThreads / 32];
    if (lane == 31) wsum[warp] = incl;
    if (lane == 0) wbefore[warp] = before;
    __syncthreads();
    if (!mine) return;
    uint32_t at = incl - sum + __reduce_add_sync(0xffffffffu, wbefore[lane] + (lane < warp ? wsum[lane] : 0u));
    reinterpret_cast<uint4*>(start)[blockIdx.x * (kScanBuckets / 4) + t] =
        make_uint4(at, at + own.x, at + own.x + own.y, at + own.x + own.y + own.z);
    if (t == kScanBuckets / 4 - 1 && blockIdx.x == gridDim.x - 1) start[gridDim.x * kScanBuckets] = uint32_t(n);
}

__global__ void __launch_bounds__(kThreads) k_bucket_fill(int64_t n, SprinkleScratch s, int bits) {
    launch_dependents();
    wait_for_primary();
    const int q = blockIdx.y;
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n; e += int64_t(gridDim.x) * blockDim.x)
        s.slot[q][s.start[q][s.key[q][e] >> (64 - bits)] + s.arrival[q][e]] = uint32_t(e);
}

// Rank of element e's key, ties by index.
__device__ __forceinline__ uint32_t rank_of(const uint64_t* key, const uint32_t* start, const uint32_t* slot, int bits,
                                            int64_t e) {
    const uint64_t ke = key[e];
    const uint32_t b = uint32_t(ke >> (64 - bits));
    const uint32_t begin = start[b], end = start[b + 1];
    uint32_t r = begin;
    for (uint32_t p = begin; p < end; ++p) {
        const uint32_t f = slot[p];
        const uint64_t kf = key[f];
        r += (kf < ke) || (kf == ke && f < uint32_t(e));
    }
    return r;
}

// Ranks and, with them, the time-sorted coordinates.
__global__ void __launch_bounds__(kThreads) k_rank_scatter(int64_t n, int dim, bool order2d, SprinkleScratch s, int bits,
                                                           int32_t* coords) {
    wait_for_primary();
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n; e += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t r = rank_of(s.key[0], s.start[0], s.slot[0], bits, e);
        if (order2d) {
            coords[r] = int32_t(r);
            coords[n + r] = int32_t(rank_of(s.key[1], s.start[1], s.slot[1], bits, e));
        } else {
            for (int c = 0; c < dim; ++c) coords[c * n + r] = s.raw[c * n + e];
        }
    }
}

// A whole small set in one CTA: draws, ranks in shared memory, coordinates
// out; no scratch in the workspace.  Four launches of a handful of blocks
// are all latency there.
template <int KIND>
__global__ void __launch_bounds__(kRankThreads) k_sprinkle_small(int n, int lgP, uint64_t seed,
                                                                 const uint64_t* __restrict__ thr,
                                                                 int32_t* __restrict__ coords, WsHeader* hdr) {
    extern __shared__ uint8_t smem_raw[];
    constexpr int kPer = int(kSmallSet) / kRankThreads;
    const int P = 1 << lgP;
    uint64_t* sk = reinterpret_cast<uint64_t*>(smem_raw);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(sk + P);
    uint32_t* slot = cnt + P;
    uint32_t* rank = slot + P;
    if (threadIdx.x == 0) hdr->status = 0;
    __syncthreads();
    int32_t c[kPer][4];
    uint64_t key[kPer][2];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int e = int(threadIdx.x) + q * kRankThreads;
        if (!draw_element<KIND>(seed, n, e, thr, c[q], key[q])) set_status(hdr, CS_ERANGE);
        if (e < n) sk[e] = key[q][0];
    }
    rank_keys_smem(n, lgP, sk, cnt, slot, rank);
    if constexpr (KIND == CS_2D_ORDER) {
        uint32_t ru[kPer];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int e = int(threadIdx.x) + q * kRankThreads;
            if (e >= n) continue;
            ru[q] = rank[e];
            sk[e] = key[q][1];
        }
        __syncthreads();
        rank_keys_smem(n, lgP, sk, cnt, slot, rank);
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int e = int(threadIdx.x) + q * kRankThreads;
            if (e >= n) continue;
            coords[ru[q]] = int32_t(ru[q]);
            coords[n + ru[q]] = int32_t(rank[e]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int e = int(threadIdx.x) + q * kRankThreads;
            if (e >= n) continue;
#pragma unroll
            for (int k = 0; k < kind_dim(KIND); ++k) coords[k * n + rank[e]] = c[q][k];
        }
    }
}

struct SprinkleLayout {
    size_t key0, key1, raw, arrival, slot0, slot1, count, start, total;
    int bits;
};

// The bucket counts follow the header, so one memset clears both.  A 2D
// order's arrivals take raw's place and its second slots the arrivals'.
SprinkleLayout sprinkle_layout(int64_t n) {
    SprinkleLayout L;
    L.bits = bucket_bits(n);
    const size_t buckets = size_t(1) << L.bits;
    size_t off = sizeof(WsHeader);
    auto take = [&](size_t bytes) {
        size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    const size_t un = size_t(n);
    L.count = take(2 * buckets * 4);
    L.start = take(2 * (buckets + 64) * 4);
    L.key0 = take(un * 8);
    L.key1 = take(un * 8);
    L.raw = take(un * 16);
    L.slot0 = take(un * 4);
    L.slot1 = take(un * 4);
    L.arrival = L.slot1;
    L.total = off;
    return L;
}

int grid_for(int64_t n) {
    int64_t b = (n + kThreads - 1) / kThreads;
    if (b < 1) b = 1;
    if (b > int64_t(device_sm_count()) * 16) b = int64_t(device_sm_count()) * 16;
    return int(b);
}

template <int KIND>
cudaError_t sprinkle_kind(int64_t n, uint64_t seed, const uint64_t* thr, int32_t* coords, uint8_t* ws,
                          cudaStream_t st) {
    WsHeader* hdr = reinterpret_cast<WsHeader*>(ws);
    const SprinkleLayout L = sprinkle_layout(n);
    if (n <= kSmallSet) {
        // 20 bytes per bucket: at most 40 KB, below the 48 KB any launch may take
        k_sprinkle_small<KIND><<<1, kRankThreads, (size_t(1) << L.bits) * 20, st>>>(int(n), L.bits, seed, thr, coords,
                                                                                   hdr);
        return cudaGetLastError();
    }
    constexpr bool kOrder = KIND == CS_2D_ORDER;
    constexpr int kStreams = kOrder ? 2 : 1;
    const size_t buckets = size_t(1) << L.bits;
    auto u32 = [&](size_t at) { return reinterpret_cast<uint32_t*>(ws + at); };
    SprinkleScratch s;
    s.key[0] = reinterpret_cast<uint64_t*>(ws + L.key0);
    s.key[1] = reinterpret_cast<uint64_t*>(ws + L.key1);
    s.raw = kOrder ? nullptr : reinterpret_cast<int32_t*>(ws + L.raw);
    s.arrival[0] = kOrder ? u32(L.raw) : u32(L.arrival);
    s.arrival[1] = u32(L.raw) + n;
    s.slot[0] = u32(L.slot0);
    s.slot[1] = u32(L.slot1);
    for (int q = 0; q < 2; ++q) {
        s.count[q] = u32(L.count) + q * buckets;
        s.start[q] = u32(L.start) + q * (buckets + 64);
    }
    // the status word and the counts of the streams in use
    cudaError_t err = cudaMemsetAsync(ws, 0, L.count + kStreams * buckets * 4, st);
    if (err != cudaSuccess) return err;
    const unsigned g = unsigned(grid_for(n));
    k_keys<KIND><<<g, kThreads, 0, st>>>(n, seed, thr, s, L.bits, hdr);
    if ((err = cudaGetLastError()) != cudaSuccess ||
        (err = launch_after(k_bucket_scan, dim3(unsigned(buckets / kScanBuckets), kStreams), kScanThreads, 0, st, s,
                            n)) != cudaSuccess ||
        (err = launch_after(k_bucket_fill, dim3(g, kStreams), kThreads, 0, st, n, s, L.bits)) != cudaSuccess)
        return err;
    return launch_after(k_rank_scatter, dim3(g), kThreads, 0, st, n, kind_dim(KIND), kOrder, s, L.bits, coords);
}

}  // namespace

const uint64_t* ds_table_device() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    if (const uint64_t* p = g_ds_ptr[dev].load(std::memory_order_acquire)) return p;
    // Upload under the lock; the pointer is published only after a
    // successful upload, so a failed first attempt (e.g. made during stream
    // capture, where the synchronous copy is not allowed) is retried by the
    // next call instead of disabling the kind for the process.
    std::lock_guard<std::mutex> lk(g_ds_mu);
    if (const uint64_t* p = g_ds_ptr[dev].load(std::memory_order_acquire)) return p;
    static const std::vector<uint64_t> host = ds_thresholds_host();
    void* p = nullptr;
    if (cudaMemcpyToSymbol(g_ds_thresholds, host.data(), host.size() * sizeof(uint64_t)) != cudaSuccess ||
        cudaGetSymbolAddress(&p, g_ds_thresholds) != cudaSuccess) {
        cudaGetLastError();  // not sticky: clear it for the caller's next call
        return nullptr;
    }
    g_ds_ptr[dev].store(static_cast<const uint64_t*>(p), std::memory_order_release);
    return static_cast<const uint64_t*>(p);
}

size_t sprinkle_workspace_bytes(int64_t n) { return sprinkle_layout(n).total; }

cudaError_t launch_sprinkle(int kind, int64_t n, uint64_t seed, int32_t* coords, void* workspace,
                            cudaStream_t st) {
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    switch (kind) {
        case CS_2D_ORDER: return sprinkle_kind<CS_2D_ORDER>(n, seed, nullptr, coords, ws, st);
        case CS_2D_DIAMOND: return sprinkle_kind<CS_2D_DIAMOND>(n, seed, nullptr, coords, ws, st);
        case CS_2D_SQUARE: return sprinkle_kind<CS_2D_SQUARE>(n, seed, nullptr, coords, ws, st);
        case CS_2D_CYLINDER: return sprinkle_kind<CS_2D_CYLINDER>(n, seed, nullptr, coords, ws, st);
        case CS_3D_DIAMOND: return sprinkle_kind<CS_3D_DIAMOND>(n, seed, nullptr, coords, ws, st);
        case CS_4D_DIAMOND: return sprinkle_kind<CS_4D_DIAMOND>(n, seed, nullptr, coords, ws, st);
        default: {
            const uint64_t* thr = ds_table_device();
            return thr ? sprinkle_kind<CS_2D_DS_SLAB>(n, seed, thr, coords, ws, st) : cudaErrorInvalidValue;
        }
    }
}

}  // namespace cs
