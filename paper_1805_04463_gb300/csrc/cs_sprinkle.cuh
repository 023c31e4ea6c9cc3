// cs_sprinkle.cuh -- per-element draws of the sprinklers (Appendix "Causal Set
// Sprinklings"), shared by the single-set and batched sprinkle kernels.
#pragma once

#include "cs_internal.cuh"

namespace cs {

// Stream numbers of the generator specification.
constexpr uint32_t kStreamOrderU = 0, kStreamOrderV = 1, kStreamDiamond2 = 2, kStreamDiamond4 = 3,
                   kStreamDiamond3 = 4, kStreamDeSitter = 5, kStreamSquare = 6, kStreamCylinder = 7;

// de Sitter slab: eta is drawn in coarse cells -kDsCells .. kDsCells of
// 2 pi / 2^20 rad (eta_0 = 0.5 rad), then uniformly among the kDsSub fine
// units (2 pi / 2^32 rad) of the cell; theta is a uint32, a full turn 2^32.
constexpr int kDsCells = 83443;
constexpr int kDsTable = 2 * kDsCells + 1;
constexpr int kDsSub = 4096;

// Random 2D order: the two 64-bit keys whose ranks are u and v.
__device__ __forceinline__ void draw_2d_order(uint64_t su, uint64_t sv, int64_t e, uint64_t& ku, uint64_t& kv) {
    ku = draw_from(su, uint64_t(e), 0);
    kv = draw_from(sv, uint64_t(e), 0);
}

// 2D diamond: u, v on the 2^31 grid (grid-null pairs, du = 0 or dv = 0, are
// then negligible); sort key (u + v) in the top 32 bits.
__device__ __forceinline__ uint64_t draw_2d_diamond(uint64_t s, int64_t e, int32_t& u, int32_t& v) {
    const uint32_t uu = uint32_t(draw_from(s, uint64_t(e), 0) >> 33);
    const uint32_t vv = uint32_t(draw_from(s, uint64_t(e), 1) >> 33);
    u = int32_t(uu);
    v = int32_t(vv);
    return uint64_t(uu + vv) << 32;
}

// Lane of the k-th (from 0) set bit of m, k < popc(m).
__device__ __forceinline__ int nth_lane(uint32_t m, int k) {
    int at = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int c = __popc((m >> at) & ((1u << w) - 1u));
        if (k >= c) {
            k -= c;
            at += w;
        }
    }
    return at;
}

// D-dimensional diamond of height 1 (D = 3: 2+1, D = 4: 3+1): rejection
// sampling in the box t in [0, 2^20), spatial coordinates in [-2^19, 2^19),
// accepting |x|^2 < min(t, 2^20-t)^2; attempt a uses slots D*a .. D*a+D-1.
// Sort key t in the top 20 bits.  Returns false if no attempt was accepted.
//
// All 32 lanes of the warp call it; those of `todo` draw an element (seed s,
// number e) each.  An attempt is accepted with probability pi/24 (3+1) or
// pi/12, so lane by lane a warp went on until its unluckiest one, about 29
// (13) rounds; here the lanes of accepted elements take later attempts of
// the others, 2^lg side by side, and the first accepted one of an element is
// its draw: about 11 (7) rounds, the same coordinates.
template <int D>
__device__ __forceinline__ bool draw_diamond(uint32_t todo, uint64_t s, int64_t e, int32_t (&c)[4], uint64_t& key) {
    constexpr uint32_t kAll = 0xffffffffu;
    const int64_t half = kGrid / 2;
    const int lane = threadIdx.x & 31;
    uint32_t left = todo;  // uniform
    bool ok = false;
    if ((todo >> lane) & 1u) {
        c[0] = c[1] = c[2] = c[3] = 0;
        key = 0;
    }
    for (int a = 0; left && a < kMaxAttempts;) {
        const int u = __popc(left), lg = __clz(u - 1) - 27;  // the largest 2^lg <= 32 / u
        const bool live = (lane >> lg) < u;
        const int owner = live ? nth_lane(left, lane >> lg) : lane;
        const uint64_t se = __shfl_sync(kAll, s, owner);
        const int64_t ee = __shfl_sync(kAll, e, owner);
        const int at = a + (lane & ((1 << lg) - 1));
        int32_t q[D];
        int64_t r2 = 0;
#pragma unroll
        for (int k = 0; k < D; ++k)
            q[k] = int32_t(int64_t(draw_from(se, uint64_t(ee), uint32_t(D * at + k)) >> (64 - kGridBits)));
#pragma unroll
        for (int k = 1; k < D; ++k) {
            q[k] -= int32_t(half);
            r2 += int64_t(q[k]) * q[k];
        }
        const int64_t h = q[0] < kGrid - q[0] ? q[0] : kGrid - q[0];
        const uint32_t accepted = __ballot_sync(kAll, live && at < kMaxAttempts && r2 < h * h);
        // an element's attempts: lanes [r 2^lg, (r + 1) 2^lg) for its place r in left
        const bool mine = (left >> lane) & 1u;
        const int r = __popc(left & ((1u << lane) - 1u));
        const uint32_t group = mine ? (kAll >> (32 - (1 << lg))) << (r << lg) : 0u;
        const uint32_t hit = accepted & group;
        const int src = hit ? __ffs(int(hit)) - 1 : lane;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const int32_t v = __shfl_sync(kAll, q[k], src);
            if (hit) c[k] = v;
        }
        if (hit) ok = true;
        left = __ballot_sync(kAll, mine && !hit);
        a += 1 << lg;
    }
    if (ok) key = uint64_t(uint32_t(c[0])) << (64 - kGridBits);
    return ok;
}

// 1+1 de Sitter slab (spherical foliation, Eq. ds_metric): theta uniform on
// 2^32 fine units; the coarse eta cell is the inverse CDF of the sec^2 mass,
// found by a binary search of the 53-bit uniform U against the cumulative
// thresholds `thr` (thr[g + kDsCells] for cell g, the last one 2^53), and eta
// is uniform among the cell's fine units.  Sort key: eta + 2^31 in the top
// 32 bits.
__device__ __forceinline__ uint64_t draw_ds_slab(uint64_t s, int64_t e, const uint64_t* __restrict__ thr,
                                                 int32_t& eta, int32_t& theta) {
    theta = int32_t(uint32_t(draw_from(s, uint64_t(e), 0) >> 32));
    const uint64_t u = draw_from(s, uint64_t(e), 1) >> 11;
    int lo = 0, hi = kDsTable - 1;  // smallest index with u < thr[index]
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (u < thr[mid]) hi = mid; else lo = mid + 1;
    }
    const int32_t off = int32_t(draw_from(s, uint64_t(e), 2) >> 52);
    eta = (lo - kDsCells) * kDsSub - kDsSub / 2 + off;
    return uint64_t(uint32_t(eta) ^ 0x80000000u) << 32;
}

// 1+1 square t in [-1/2, 1/2), x in [-1/2, 1/2) on a grid of 2^30 per unit,
// stored in light-cone coordinates u = t + x + 2^30, v = t - x + 2^30 (both
// in [0, 2^31), so the diamond's light-cone test applies); sort key
// u + v = 2 t + 2^31 in the top 32 bits.
__device__ __forceinline__ uint64_t draw_2d_square(uint64_t s, int64_t e, int32_t& u, int32_t& v) {
    const int32_t t = int32_t(draw_from(s, uint64_t(e), 0) >> 34) - (1 << 29);
    const int32_t x = int32_t(draw_from(s, uint64_t(e), 1) >> 34) - (1 << 29);
    u = t + x + (1 << 30);
    v = t - x + (1 << 30);
    return uint64_t(uint32_t(u) + uint32_t(v)) << 32;
}

// 1+1 cylinder: theta uniform on 2^32 fine units (a full turn), t uniform on
// [-T, T) fine units with T = floor(2^31 / pi), one radian (t0 = 1), by a
// 32 x 32-bit multiply of a uniform word by 2T.  Sort key: t + 2^31 in the
// top 32 bits.
constexpr uint32_t kCylinderT = 683565275u;
__device__ __forceinline__ uint64_t draw_2d_cylinder(uint64_t s, int64_t e, int32_t& t, int32_t& theta) {
    theta = int32_t(uint32_t(draw_from(s, uint64_t(e), 0) >> 32));
    const uint64_t r = draw_from(s, uint64_t(e), 1) >> 32;
    t = int32_t(int64_t((r * uint64_t(2u * kCylinderT)) >> 32) - int64_t(kCylinderT));
    return uint64_t(uint32_t(t) ^ 0x80000000u) << 32;
}

// Exact ranks of a set's n keys (ties by index: the order "sorted by time,
// ties by generation index") in shared memory, O(n): count the keys into P
// buckets by their top log2(P) bits (P the power of two >= n; the keys are
// a time coordinate in the top bits, or random, so a bucket holds about
// one key and at most a few), an exclusive scan of the counts, fill the
// buckets, then rank each key within its bucket by comparison.  After the
// fill, cnt[b] is the end of bucket b and cnt[b - 1] its start.  (A bitonic
// sort of the (key, index) pairs, O(n log^2 n), took 0.38 ms for the
// 768-set ensemble.)  sk holds the keys on entry, written before a barrier or
// by their own threads (key i by thread i % kRankThreads).  All kRankThreads
// threads; rank[e] receives the rank.  kLastFirst: equal keys rank the later
// element first.  kAny: the keys may lie anyhow (a caller's coordinates); when a bucket
// holds more than kMostInBucket of them they are sorted instead, since every element
// compares itself with its whole bucket (a diamond of 8192 equal elements, whole
// evaluation: 3360 us by buckets, 208 sorted, spread-out coordinates 130).  sk then holds P keys' room.
constexpr int kRankThreads = 1024;
constexpr uint32_t kMostInBucket = 32;

// The same ranks by a bitonic network over the P >= n places, whatever the keys (all
// below ~0).  sk is sorted.
template <bool kLastFirst>
__device__ __forceinline__ void rank_keys_sorted(int n, int lgP, uint64_t* sk, uint32_t* slot, uint32_t* rank) {
    const int P = 1 << lgP;
    // equal keys by label, or against it
    for (int i = threadIdx.x; i < P; i += kRankThreads) {
        if (i >= n) sk[i] = ~0ull;
        slot[i] = uint32_t(kLastFirst ? P - 1 - i : i);
    }
    for (int size = 2; size <= P; size <<= 1) {
        for (int j = size >> 1; j > 0; j >>= 1) {
            __syncthreads();
            for (int t = threadIdx.x; t < P / 2; t += kRankThreads) {
                const int lo = 2 * t - (t & (j - 1)), hi = lo + j;
                const uint64_t a = sk[lo], b = sk[hi];
                const uint32_t ia = slot[lo], ib = slot[hi];
                const bool greater = a > b || (a == b && ia > ib);
                if (greater == ((lo & size) == 0)) {
                    sk[lo] = b;
                    sk[hi] = a;
                    slot[lo] = ib;
                    slot[hi] = ia;
                }
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kRankThreads) rank[kLastFirst ? P - 1 - int(slot[i]) : int(slot[i])] = uint32_t(i);
    __syncthreads();
}

template <bool kLastFirst = false, bool kAny = false>
__device__ __forceinline__ void rank_keys_smem(int n, int lgP, uint64_t* sk, uint32_t* cnt, uint32_t* slot,
                                               uint32_t* rank) {
    const int P = 1 << lgP, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int shift = 64 - lgP;
    for (int i = tid; i < P; i += kRankThreads) cnt[i] = 0u;
    __syncthreads();
    for (int i = tid; i < n; i += kRankThreads) atomicAdd(&cnt[sk[i] >> shift], 1u);
    __syncthreads();
    // exclusive scan: each thread a run of P / kRankThreads buckets (P >= 1024
    // is ensured by the caller), warp and block offsets through shuffles
    const int per = P / kRankThreads;
    uint32_t run = 0, most = 0;
    for (int k = 0; k < per; ++k) {
        run += cnt[tid * per + k];
        most = max(most, cnt[tid * per + k]);
    }
    if (kAny && __syncthreads_or(most > kMostInBucket)) {
        rank_keys_sorted<kLastFirst>(n, lgP, sk, slot, rank);
        return;
    }
    uint32_t incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    __shared__ uint32_t wsum[kRankThreads / 32];
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < kRankThreads / 32 ? wsum[lane] : 0u, wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < kRankThreads / 32) wsum[lane] = wi - w;  // exclusive warp offsets
    }
    __syncthreads();
    uint32_t at = wsum[warp] + incl - run;
    for (int k = 0; k < per; ++k) {
        const uint32_t c = cnt[tid * per + k];
        cnt[tid * per + k] = at;  // start of the bucket, then its fill cursor
        at += c;
    }
    __syncthreads();
    for (int i = tid; i < n; i += kRankThreads) slot[atomicAdd(&cnt[sk[i] >> shift], 1u)] = uint32_t(i);
    __syncthreads();
    for (int i = tid; i < n; i += kRankThreads) {
        const uint64_t ke = sk[i];
        const uint32_t bk = uint32_t(ke >> shift);
        const uint32_t s0 = bk ? cnt[bk - 1] : 0u, s1 = cnt[bk];
        uint32_t r = s0;
        for (uint32_t q = s0; q < s1; ++q) {
            const uint32_t f = slot[q];
            const uint64_t kf = sk[f];
            r += (kf < ke) || (kf == ke && (kLastFirst ? f > uint32_t(i) : f < uint32_t(i)));
        }
        rank[i] = r;
    }
    __syncthreads();
}

}  // namespace cs
