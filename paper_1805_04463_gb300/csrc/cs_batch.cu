// cs_batch.cu -- batched ensembles: many causal sets of different kinds and
// sizes evaluated by one fixed sequence of launches (memsets and kernels
// only, so the sequence can be captured into a CUDA graph and replayed).
//
// Pipeline per launch, every kernel covering all sets at once:
//   k_batch_keys    per element: random keys / raw coordinates (same draws as
//                   cs_sprinkle, so every set equals its single-set result);
//   k_batch_rank    one CTA per set: exact ranks of the keys by a bucket
//                   count in shared memory give the time order; scatter
//                   coordinates;
//   k_batch_ctab    the column tables of the light-cone sets' bitsets;
//   k_batch_relate  every relate chunk (32 words of a 64-row tile, from its
//                   diagonal word) of every bitset, one launch per geometry
//                   (light cone: k_batch_relate_cone, from the tables);
//   k_batch_mirror  the lower triangle of every bitset, the transpose of the
//                   upper one (the past rows);
//   order table, order count   on CS_PATH_AUTO, for the product orders (2D
//                   orders, the 1+1 diamond and square): the table of prefix
//                   ranks and the pair count from it (cs_order.cuh), in
//                   place of relate, mirror and the count below;
//   count           the multi-set POPC kernel, or expand + multi-set tcgen05
//                   kernel: one persistent grid over the tiles of all sets,
//                   largest sets first (longest-processing-time order);
//   k_batch_coef    the smearing coefficients and cutoffs;
//   k_batch_action  one CTA per (set, eps): bracket and smeared sums.
// Ensembles of Poisson-sized sprinklings are the thesis's experimental unit
// (Section "Simulations and Scaling Evaluations": ten graphs per size; the
// appendix's sprinklings draw N from a Poisson distribution).
#include <algorithm>
#include <cstring>
#include <new>
#include <numeric>
#include <vector>

#include "cs_action.cuh"
#include <atomic>

#include "cs_kernels.cuh"
#include "cs_launch.cuh"
#include "cs_order.cuh"
#include "cs_relate.cuh"
#include "cs_sprinkle.cuh"

namespace cs {

namespace {

// Per set, device-resident.
struct BatchSet {
    int32_t kind, dim;
    int64_t n;
    uint64_t seed;
    int32_t* coords;
    uint64_t* bits;
    int64_t row_words;
    uint64_t* key0;
    uint64_t* key1;
    int32_t* raw;
    int64_t elem_begin;    // first element of this set in the concatenated element range
    int64_t rblock_begin;  // first relate block
    int64_t vwords;        // valid words per row = row tiles = ceil(n / 64)
    int64_t mblock_begin;  // first mirror block (lower part by symmetry)
    int64_t mir_side;      // mirror super-tiles per side
    int64_t hist_off;      // offset of this set's histogram in the batch histogram
    ConeTable* ctab;       // light-cone kinds: one column table per column tile (else null)
    int64_t tile_begin;    // first column tile of this set in the concatenated tile range
    OrderSet order;        // counted as a product order (p not null): its arrays, and no bits
    int64_t ord_block;     // first block of this set in the order table build
    int64_t ord_task;      // first of its tasks in the order count
};

// A set counted from its prefix-rank table.
__host__ __device__ __forceinline__ bool by_order(const BatchSet& b) { return b.order.p != nullptr; }

// Bands per column chunk of the order count's tasks, and its threads: two
// CTAs per SM, so that one counts while the other flushes.
constexpr int kBatchOrderM = 2;
constexpr int kBatchOrderThreads = 512;

// The set of element idx, by the whole warp (idx uniform): 32 probes at a
// time, where a search by halves is ten dependent loads for a thousand sets.
__device__ __forceinline__ int find_set_warp(const BatchSet* sets, int nsets, int64_t idx) {
    const int lane = threadIdx.x & 31;
    int lo = 0, count = nsets;  // sets[lo].elem_begin <= idx, the next one's after lo + count is not
    while (count > 1) {
        const int step = (count + 31) / 32, i = lane * step;
        const uint32_t m = __ballot_sync(0xffffffffu, i < count && sets[lo + (i < count ? i : 0)].elem_begin <= idx);
        const int j = (31 - __clz(m)) * step;
        lo += j;
        count = count - j < step ? count - j : step;
    }
    return lo;
}

__global__ void __launch_bounds__(256) k_batch_keys(const BatchSet* __restrict__ sets, int nsets, int64_t total,
                                                    const uint64_t* __restrict__ ds_thr, WsHeader* hdr) {
    const int lane = threadIdx.x & 31;
    for (int64_t at = blockIdx.x * int64_t(blockDim.x) + (threadIdx.x & ~31); at < total;
         at += int64_t(gridDim.x) * blockDim.x) {  // whole warps
        const int64_t idx = at + lane;
        int set = find_set_warp(sets, nsets, at);
        while (set + 1 < nsets && sets[set + 1].elem_begin <= idx) ++set;
        const BatchSet& b = sets[set];
        const int64_t e = idx - b.elem_begin;
        int32_t c[4];
        uint64_t key;
        const bool in = idx < total;
        const uint32_t in3 = __ballot_sync(0xffffffffu, in && b.kind == CS_3D_DIAMOND);
        const uint32_t in4 = __ballot_sync(0xffffffffu, in && b.kind == CS_4D_DIAMOND);
        bool ok = false;
        if (in3) ok |= draw_diamond<3>(in3, stream_key(b.seed, kStreamDiamond3), e, c, key);
        if (in4) ok |= draw_diamond<4>(in4, stream_key(b.seed, kStreamDiamond4), e, c, key);
        if (!in) continue;
        if (b.kind == CS_2D_ORDER) {
            draw_2d_order(stream_key(b.seed, kStreamOrderU), stream_key(b.seed, kStreamOrderV), e, b.key0[e],
                          b.key1[e]);
        } else if (b.kind == CS_2D_DIAMOND) {
            b.key0[e] = draw_2d_diamond(stream_key(b.seed, kStreamDiamond2), e, b.raw[e], b.raw[b.n + e]);
        } else if (b.kind == CS_2D_SQUARE) {
            b.key0[e] = draw_2d_square(stream_key(b.seed, kStreamSquare), e, b.raw[e], b.raw[b.n + e]);
        } else if (b.kind == CS_2D_CYLINDER) {
            b.key0[e] = draw_2d_cylinder(stream_key(b.seed, kStreamCylinder), e, b.raw[e], b.raw[b.n + e]);
        } else if (b.kind == CS_2D_DS_SLAB) {
            b.key0[e] = draw_ds_slab(stream_key(b.seed, kStreamDeSitter), e, ds_thr, b.raw[e], b.raw[b.n + e]);
        } else {
            b.key0[e] = key;
            if (!ok) set_status(hdr, CS_ERANGE);
            for (int k = 0; k < b.dim; ++k) b.raw[k * b.n + e] = c[k];
        }
    }
}

// One CTA per set: exact rank of each element (ties by index), then the
// time-sorted coordinates.  Shared memory: keys 8n, bucket cursors 4P,
// bucket slots 4n, ranks 4n (and the u ranks 4n of a 2D order), P <= max(n, 1024).
__global__ void __launch_bounds__(kRankThreads) k_batch_rank(const BatchSet* __restrict__ sets) {
    wait_for_primary();
    extern __shared__ uint8_t smem_raw[];
    const BatchSet& b = sets[blockIdx.x];
    const int n = int(b.n);
    int lgP = 10;  // at least kRankThreads buckets (the scan's runs), one to two elements each
    while ((2 << lgP) <= n) ++lgP;
    const int P = 1 << lgP;
    uint64_t* sk = reinterpret_cast<uint64_t*>(smem_raw);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(sk + n);
    uint32_t* slot = cnt + P;
    uint32_t* rank = slot + n;
    uint32_t* ru = rank + n;
    int32_t* op = const_cast<int32_t*>(b.order.p);
    int32_t* oq = const_cast<int32_t*>(b.order.q);
    if (by_order(b) && b.kind != CS_2D_ORDER) {  // the count needs the ranks of u and v, not the time order
        order_ranks_smem(b.raw, b.raw + n, false, n, lgP, smem_raw, op, oq);
        return;
    }
    auto load = [&](const uint64_t* key) {
        for (int i = threadIdx.x; i < n; i += kRankThreads) sk[i] = key[i];
    };
    load(b.key0);
    rank_keys_smem(n, lgP, sk, cnt, slot, rank);
    if (b.kind == CS_2D_ORDER) {
        for (int e = threadIdx.x; e < n; e += kRankThreads) ru[e] = rank[e];  // u rank of element e
        __syncthreads();
        load(b.key1);
        rank_keys_smem(n, lgP, sk, cnt, slot, rank);
        for (int e = threadIdx.x; e < n; e += kRankThreads) {
            if (by_order(b)) {
                op[ru[e]] = int32_t(rank[e]);
                oq[rank[e]] = int32_t(ru[e]);
            } else {
                b.coords[ru[e]] = int32_t(ru[e]);
                b.coords[n + ru[e]] = int32_t(rank[e]);
            }
        }
    } else {
        for (int e = threadIdx.x; e < n; e += kRankThreads) {
            const uint32_t p = rank[e];  // the time-sorted position of element e
            for (int c = 0; c < b.dim; ++c) b.coords[c * n + p] = b.raw[c * n + e];
        }
    }
}

// Column tables of the light-cone sets (after k_batch_rank has written the
// time-sorted coordinates), one warp per column tile of the concatenated
// tile range, the set read from a table built at create time.
__global__ void __launch_bounds__(256) k_batch_ctab(const BatchSet* __restrict__ sets,
                                                    const int32_t* __restrict__ tile_set, int64_t tiles) {
    wait_for_primary();
    const int64_t g = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5;  // warp-uniform
    if (g >= tiles) return;
    const BatchSet& b = sets[tile_set[g]];
    if (b.ctab) build_cone_table(b.coords, b.n, g - b.tile_begin, b.kind == CS_2D_ORDER, b.ctab + (g - b.tile_begin));
}

// The prefix-rank tables of the sets counted as product orders, eight rows
// per block, the set read from a table.
__global__ void __launch_bounds__(kOrdBuildThreads) k_batch_order_table(const BatchSet* __restrict__ sets,
                                                                        const int32_t* __restrict__ block_set) {
    wait_for_primary();
    const BatchSet& b = sets[block_set[blockIdx.x]];
    order_build_rows(b.order, int(int64_t(blockIdx.x) - b.ord_block));
}

// Their pair counts.  Each CTA takes an equal, contiguous share of the
// concatenated task list (tasks cost alike), so it meets few sets: its warps
// stride over the share's tasks of a set, then the CTA adds its shared
// histogram to the set's and clears it.  order_sets: the sets in task order.
__global__ void __launch_bounds__(kBatchOrderThreads, 2) k_batch_order_count(const BatchSet* __restrict__ sets,
                                                                          const int32_t* __restrict__ order_sets,
                                                                          int n_order, int64_t tasks, int64_t* hist_base) {
    wait_for_primary();
    constexpr int kWarps = kBatchOrderThreads / 32;
    extern __shared__ __align__(16) uint8_t smem_ord[];
    const int warp = threadIdx.x >> 5;
    int2* stage = reinterpret_cast<int2*>(smem_ord) + 32 * warp;
    uint32_t* shist = reinterpret_cast<uint32_t*>(smem_ord + kWarps * 32 * sizeof(int2));
    const uint32_t hist_s = smem_u32(shist);
    int64_t t = tasks * blockIdx.x / gridDim.x;
    const int64_t end = tasks * (blockIdx.x + 1) / gridDim.x;
    int r = 0;  // the last set whose tasks begin at or before t
    for (int hi = n_order - 1; r < hi;) {
        const int mid = (r + hi + 1) >> 1;
        if (sets[order_sets[mid]].ord_task <= t) r = mid; else hi = mid - 1;
    }
    for (; t < end; ++r) {
        const BatchSet& b = sets[order_sets[r]];
        const OrderSet s = b.order;
        const int bins = s.n > 1 ? s.n - 1 : 1;  // every count of the set
        unsigned long long* hist = reinterpret_cast<unsigned long long*>(hist_base + b.hist_off);
        for (int k = threadIdx.x; k < bins; k += kBatchOrderThreads) shist[k] = 0u;
        __syncthreads();
        const int64_t own = b.ord_task + order_tasks(s.n, kBatchOrderM);  // end of the set's tasks
        const int64_t stop = own < end ? own : end;
        for (int64_t q = t + warp; q < stop; q += kWarps) {
            int A, C;
            order_decode(q - b.ord_task, kBatchOrderM, A, C);
            order_task(s, A, C, kOrdBand * kBatchOrderM, hist_s, bins, hist, stage);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < bins; k += kBatchOrderThreads) {
            const uint32_t c = shist[k];
            if (c) atomicAdd(hist + k, (unsigned long long)c);
        }
        t = stop;
        __syncthreads();
    }
}

// Relate chunks.  Row tile rb of a set with V valid words needs words
// [rb, V) (the words before it are mirrored); they are covered by chunks of
// 32 words from word 4 floor(rb / 4) on (a warp's words are one 32-byte
// sector of a row), so no block holds whole groups of padding.  In units of four words,
// V4 = ceil(V / 4), row tile rb has ceil((V4 - rb / 4) / 8) chunks.
// chunk_sum8(x) = sum_{m=1..x} ceil(m / 8).
__host__ __device__ __forceinline__ int64_t chunk_sum8(int64_t x) {
    const int64_t a = x / 8, b = x % 8;
    return 8 * a * (a + 1) / 2 + b * (a + 1);
}
// Chunks of the row tiles before rb; of all of them for rb = V.
__host__ __device__ __forceinline__ int64_t chunks_before(int64_t V, int64_t rb) {
    const int64_t V4 = (V + 3) / 4, g = rb / 4, left = V4 - g;
    return 4 * (chunk_sum8(V4) - chunk_sum8(left)) + (rb & 3) * ((left + 7) / 8);
}

// Relation geometry of a kind.
__host__ __device__ __forceinline__ int batch_geom(int kind) {
    return kind == CS_4D_DIAMOND                               ? kGeom4
           : kind == CS_3D_DIAMOND                             ? kGeom3
           : (kind == CS_2D_DS_SLAB || kind == CS_2D_CYLINDER) ? kGeomDeSitter
                                                               : kGeomLightCone;
}

// Relate block `local` of a set: its row tile rb, first word w0 and, for a
// row tile's last chunk, the first padding word to zero (else -1).
__device__ __forceinline__ void decode_rblock(const BatchSet& b, int64_t local, int64_t& rb, int64_t& w0,
                                              int64_t& zero_from) {
    const int64_t V = b.vwords;
    int64_t lo = 0, hi = V - 1;  // last row tile whose first chunk is at or before `local`
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (chunks_before(V, mid) <= local) lo = mid; else hi = mid - 1;
    }
    rb = lo;
    w0 = (rb & ~int64_t(3)) + (local - chunks_before(V, rb)) * kRelWordsPerBlock;
    zero_from = w0 + kRelWordsPerBlock >= V ? w0 + kRelWordsPerBlock : -1;
}

// One block per relate chunk of one set, the set read from a table built at
// create time, the (row tile, chunk) by a binary search over row tiles.  The
// last chunk of a row tile also zeroes the row's padding words.  One
// instance per geometry, each launched over that geometry's chunks only (a
// table groups the chunks by geometry), so that every geometry's code gets
// the registers it needs for itself.  Block x of a geometry's launch: relate block order[x] (the launch's slice
// of the blocks grouped by geometry), of set rblock_set[order[x]].
template <int G>
__global__ void __launch_bounds__(kRelThreads) k_batch_relate(const BatchSet* __restrict__ sets,
                                                              const int32_t* __restrict__ rblock_set,
                                                              const int32_t* __restrict__ order) {
    wait_for_primary();
    __shared__ __align__(16) uint8_t sm[relate_stage_bytes(G)];
    const int64_t blk = order[blockIdx.x];
    const BatchSet& b = sets[rblock_set[blk]];
    if (batch_geom(b.kind) != G) return;  // never, by the order's construction
    int64_t rb, w0, zero_from;
    decode_rblock(b, blk - b.rblock_begin, rb, w0, zero_from);
    relate_block<G>(b.coords, b.n, b.bits, b.row_words, rb, w0, sm, zero_from);
}

// The light-cone kinds, from the column tables of k_batch_ctab (one
// look-up per word instead of 64 cone tests).
__global__ void __launch_bounds__(kRelThreads, 4) k_batch_relate_cone(const BatchSet* __restrict__ sets,
                                                                   const int32_t* __restrict__ rblock_set,
                                                                   const int32_t* __restrict__ order,
                                                                   WsHeader* hdr) {
    wait_for_primary();
    extern __shared__ __align__(16) uint8_t smem_rel[];
    const int64_t blk = order[blockIdx.x];
    const BatchSet& b = sets[rblock_set[blk]];
    if (batch_geom(b.kind) != kGeomLightCone) return;  // never, by the order's construction
    int64_t rb, w0, zero_from;
    decode_rblock(b, blk - b.rblock_begin, rb, w0, zero_from);
    relate_block_tables(b.coords, b.n, b.bits, b.row_words, rb, w0, b.ctab, smem_rel, b.kind == CS_2D_ORDER,
                        zero_from, hdr);
}

// One block per mirror super-tile of one set (the lower part of its bitset
// as the transpose of the upper part), the set read from a table.
__global__ void __launch_bounds__(kRelThreads) k_batch_mirror(const BatchSet* __restrict__ sets,
                                                              const int32_t* __restrict__ mblock_set) {
    wait_for_primary();
    __shared__ uint64_t sm[kMirRows][kMirTiles + 1];
    const BatchSet& b = sets[mblock_set[blockIdx.x]];
    const int64_t local = int64_t(blockIdx.x) - b.mblock_begin;
    mirror_block(b.bits, b.n, b.row_words, local / b.mir_side, local % b.mir_side, sm);
}

// Smeared-sum coefficients f_d(k, eps) (Eqs. f2, f3, f4), one table per
// dimension present and eps, shared by every set of that dimension: a set's
// cutoff never exceeds that of the dimension's largest set (smear_cutoff
// grows with n), which sizes the table.  Dimension slot: d - 2.
constexpr int kDimSlots = 3;
struct CoefArgs {
    int64_t base[kDimSlots];              // first table entry of the slot
    int64_t stride[kDimSlots];            // entries per eps (the slot's largest n)
    int64_t kcap[kDimSlots][kMaxEps];     // entries computed per (slot, eps)
    int64_t seg[kDimSlots * kMaxEps + 1];  // prefix sums of kcap in (slot, eps) order
    dd factor[kDimSlots][kMaxEps];         // action_factor per (slot, eps)
};

// The same launch finds each (set, eps) cutoff once (kends), after the
// table entries: a fixed-point iteration of about 1500 FP64 operations, too
// costly to repeat in every thread of the action kernel.
struct BatchPowers {
    EpsPowers e[kMaxEps];
    SmearCoef c[kDimSlots][kMaxEps];
};
__global__ void __launch_bounds__(32) k_batch_coef(dd* coef, CoefArgs c, EpsArgs eps,
                                                    const __grid_constant__ BatchPowers powers,
                                                    const BatchSet* __restrict__ sets, int nsets,
                                                    int64_t* kends) {
    launch_dependents();
    wait_for_primary();
    const int64_t total = c.seg[kDimSlots * kMaxEps];
    const int64_t all = total + int64_t(nsets) * eps.n;
    for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < all; t += int64_t(gridDim.x) * blockDim.x) {
        if (t >= total) {
            const int set = int((t - total) / eps.n), e = int((t - total) % eps.n);
            const double ep = eps.v[e];
            const BatchSet& b = sets[set];
            const int64_t len = b.n > 1 ? b.n - 1 : 1;
            const int64_t kc = is_local(ep) ? 0 : smear_cutoff(b.dim, ep, 0.5 * double(b.n) * double(b.n), len);
            const int64_t cap = c.kcap[b.dim - 2][e];
            kends[int64_t(set) * kMaxEps + e] = kc < cap ? kc : cap;  // never beyond the table
            continue;
        }
        int g = 0;
        while (c.seg[g + 1] <= t) ++g;  // at most 48 segments
        const int slot = g / kMaxEps, e = g % kMaxEps, dim = slot + 2;
        const int64_t k = t - c.seg[g];
        coef[c.base[slot] + e * c.stride[slot] + k] =
            smear_term(dim, powers.c[slot][e], powers.e[e], k);
    }
}

// One CTA per (set, eps): the set's bracket (written by its eps-0 CTA) and
// one local or smeared action; the smeared sums take their coefficients from
// the shared table.  A CTA per set walking its eps values one after another
// left the FP64 pipe waiting on the sums' dependency chains (0.29 ms for 768
// sets and three smeared eps).
__global__ void __launch_bounds__(kActThreads) k_batch_action(const BatchSet* __restrict__ sets,
                                                              const int64_t* hist_base, EpsArgs eps,
                                                              const dd* coef, CoefArgs c, const int64_t* kends,
                                                              double* actions, int64_t* brackets) {
    wait_for_primary();
    __shared__ dd red[kActThreads];
    const int per = eps.n > 0 ? eps.n : 1;  // no eps: one CTA per set for the bracket
    const int set = blockIdx.x / per, e = blockIdx.x % per;
    const BatchSet& b = sets[set];
    const int dim = b.dim, slot = dim - 2;
    const int64_t n = b.n, len = n > 1 ? n - 1 : 1;
    const int64_t* hist = hist_base + b.hist_off;
    const int tid = threadIdx.x;
    int64_t h4[4] = {0, 0, 0, 0};
    for (int k = 0; k < 4 && k < len; ++k) h4[k] = hist[k];
    const int64_t br = bracket_of(dim, n, h4);
    if (tid == 0 && e == 0 && brackets) brackets[set] = br;
    if (e >= eps.n) return;
    const double ep = eps.v[e];
    if (is_local(ep)) {  // uniform across the CTA
        if (tid == 0 && actions) {
            const dd s = local_action(c.factor[slot][e], br);
            actions[int64_t(set) * eps.n + e] = s.hi + s.lo;
        }
        return;
    }
    const int64_t kend = kends[int64_t(set) * kMaxEps + e];  // k_batch_coef's cutoff
    const dd* f = coef + c.base[slot] + e * c.stride[slot];
    dd sum = dd_from(0.0);
    for (int64_t k = tid; k < kend; k += kActThreads) {
        const int64_t hk = hist[k];
        if (hk != 0) sum = dd_add(sum, dd_times_i64(f[k], hk));
    }
    red[tid] = sum;
    __syncthreads();
    for (int s = kActThreads / 2; s > 0; s >>= 1) {
        if (tid < s) red[tid] = dd_add(red[tid], red[tid + s]);
        __syncthreads();
    }
    if (tid == 0 && actions) {
        const dd s = smeared_action(dim, n, ep, c.factor[slot][e], red[0]);
        actions[int64_t(set) * eps.n + e] = s.hi + s.lo;
    }
}

std::atomic<bool> g_rank_attr[64];  // per device: the rank kernel's shared-memory attribute is set
std::atomic<bool> g_cone_attr[64];  // per device: the light-cone relate's shared-memory attribute is set

}  // namespace

}  // namespace cs

using namespace cs;

// Host-side plan of a batch (the device tables live in the workspace).
struct cs_batch {
    int nsets = 0;
    int path = CS_PATH_POPC;
    uint8_t* ws = nullptr;
    WsHeader* hdr = nullptr;
    BatchSet* sets_dev = nullptr;
    PopcSetEntry* popc_dev = nullptr;
    MmaSetEntry* mma_dev = nullptr;
    int64_t total_elems = 0, total_rblocks = 0, total_items = 0, total_chunks = 0, total_hist = 0;
    int32_t* rtab = nullptr;  // relate block -> set
    int32_t* rorder = nullptr;  // relate blocks grouped by geometry (each launch covers its own)
    int64_t geo_begin[8] = {0, 0, 0, 0, 0, 0, 0, 0}, geo_count[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int32_t* etab = nullptr;  // expansion chunk -> count-table entry
    int32_t* mtab = nullptr;  // mirror block -> set
    int64_t total_mblocks = 0;
    int64_t total_tiles = 0;  // column tiles of all sets (k_batch_ctab's warps)
    int32_t* ttab = nullptr;  // column tile -> set
    int n_general = 0;  // sets counted from their causal matrix
    int n_order = 0;    // sets counted as product orders
    int32_t* otab = nullptr;   // order table block -> set
    int32_t* osets = nullptr;  // the product orders, in task order
    int64_t ord_blocks = 0, ord_tasks = 0;
    int64_t ord_nmax = 0;      // the largest of them
    unsigned geoms = 0;  // bit G: some set relates with geometry G
    int64_t n_largest = 1;
    const uint64_t* ds_thr = nullptr;  // de Sitter thresholds, when a set needs them
    dd* coef = nullptr;                 // smeared-sum coefficient tables
    int64_t* kends = nullptr;           // per (set, eps): smeared-sum cutoff [set * kMaxEps + e]
    int64_t nmax[kDimSlots] = {0, 0, 0};  // largest n per dimension slot (0: absent)
    int64_t coef_base[kDimSlots] = {0, 0, 0};
    // cs_batch_poll: each launch copies the status word here (pinned) and
    // records `done` after it.
    int32_t* status_host = nullptr;
    cudaEvent_t done = nullptr;
    ~cs_batch() {
        if (done) cudaEventDestroy(done);
        if (status_host) cudaFreeHost(status_host);
    }
};

namespace {

struct Layout {
    size_t sets, entries, rtab, rorder, etab, mtab, ttab, otab, osets, coef, kends, total;
    std::vector<size_t> coords, bits, key0, key1, raw, ctab, op0, op1;
    std::vector<size_t> ord_p, ord_q, ord_r, ord_d;  // product orders
};

bool batch_valid(const cs_set_desc* sets, int n_sets) {
    if (!sets || n_sets < 1 || n_sets > CS_BATCH_MAX_SETS) return false;
    for (int s = 0; s < n_sets; ++s)
        if (cs_dim(sets[s].kind) == 0 || sets[s].n < 1 || sets[s].n > CS_BATCH_MAX_N || sets[s].reserved != 0)
            return false;
    return true;
}

int batch_path(const cs_set_desc* sets, int n_sets, int path) {
    if (path != CS_PATH_AUTO) return path;
    return batch_auto_path();
}

bool tensor_path(int path) { return path == CS_PATH_MMA || path == CS_PATH_MMA4; }

// On CS_PATH_AUTO a product order is counted from its coordinates.  (Every
// size: in a batch the route's launches are shared by all sets.)
bool set_by_order(const cs_set_desc& d, bool auto_path) { return auto_path && order_kind(d.kind) && d.n >= 2; }

Layout batch_layout(const cs_set_desc* sets, int n_sets, int path, bool auto_path) {
    Layout L;
    size_t off = sizeof(WsHeader);
    auto take = [&](size_t bytes) {
        size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    L.sets = take(sizeof(BatchSet) * size_t(n_sets));
    off = align_up(off, 128);
    L.entries = take((tensor_path(path) ? sizeof(MmaSetEntry) : sizeof(PopcSetEntry)) * size_t(n_sets));
    int64_t rblocks = 0, chunks = 0, mblocks = 0, tiles = 0, oblocks = 0;
    for (int s = 0; s < n_sets; ++s) {
        const int64_t n = sets[s].n;
        if (set_by_order(sets[s], auto_path)) {
            oblocks += order_build_blocks(n);
            continue;
        }
        rblocks += chunks_before((n + 63) / 64, (n + 63) / 64);
        tiles += (n + 63) / 64;
        const int64_t side = ((n + 63) / 64 + kMirTiles - 1) / kMirTiles;
        mblocks += side * side;
        if (tensor_path(path)) chunks += mma_expand_chunks(n);
    }
    L.rtab = take(size_t(rblocks) * 4);  // relate block -> set
    L.rorder = take(size_t(rblocks) * 4);  // relate blocks by geometry
    L.etab = take(size_t(chunks) * 4);   // expansion chunk -> set
    L.mtab = take(size_t(mblocks) * 4);  // mirror block -> set
    L.ttab = take(size_t(tiles) * 4);    // column tile -> set
    L.otab = take(size_t(oblocks) * 4);  // order table block -> set
    L.osets = take(size_t(n_sets) * 4);  // the product orders
    int64_t nmax[kDimSlots] = {0, 0, 0};
    for (int s = 0; s < n_sets; ++s) {
        int64_t& m = nmax[cs_dim(sets[s].kind) - 2];
        m = sets[s].n > m ? sets[s].n : m;
    }
    L.coef = take(size_t(nmax[0] + nmax[1] + nmax[2]) * kMaxEps * sizeof(dd));  // coefficient tables
    L.kends = take(size_t(n_sets) * kMaxEps * 8);                                 // smeared-sum cutoffs
    for (auto* v : {&L.coords, &L.bits, &L.key0, &L.key1, &L.raw, &L.ctab, &L.op0, &L.op1, &L.ord_p, &L.ord_q, &L.ord_r,
                    &L.ord_d})
        v->reserve(size_t(n_sets));
    for (int s = 0; s < n_sets; ++s) {
        const int64_t n = sets[s].n;
        const int dim = cs_dim(sets[s].kind);
        const bool order = set_by_order(sets[s], auto_path);
        L.ord_p.push_back(order ? take(size_t(n) * 4) : 0);
        L.ord_q.push_back(order ? take(size_t(n) * 4) : 0);
        L.ord_r.push_back(order ? take(size_t(n) * 4) : 0);
        L.ord_d.push_back(order ? take(order_table_bytes(n)) : 0);
        L.coords.push_back(order ? 0 : take(size_t(n) * dim * 4));
        L.bits.push_back(order ? 0 : take(size_t(n) * size_t(cs_row_words(n)) * 8));
        L.key0.push_back(take(size_t(n) * 8));
        L.key1.push_back(take(size_t(n) * 8));
        L.raw.push_back(take(size_t(n) * 16));
        L.ctab.push_back(!order && batch_geom(sets[s].kind) == kGeomLightCone
                             ? take(size_t((n + 63) / 64) * sizeof(ConeTable))
                             : 0);
        if (order) {
            L.op0.push_back(0);
            L.op1.push_back(0);
        } else if (tensor_path(path)) {
            off = align_up(off, 1024);
            L.op0.push_back(take(mma_operand_bytes(n, path == CS_PATH_MMA4, 0)));
            off = align_up(off, 1024);
            L.op1.push_back(take(mma_operand_bytes(n, path == CS_PATH_MMA4, 1)));
        }
    }
    L.total = off;
    return L;
}

}  // namespace

extern "C" {

size_t cs_batch_workspace_bytes(const cs_set_desc* sets, int n_sets, int path) {
    if (!batch_valid(sets, n_sets) || path < CS_PATH_AUTO || path > CS_PATH_MMA4) return 0;
    return batch_layout(sets, n_sets, batch_path(sets, n_sets, path), path == CS_PATH_AUTO).total;
}

int64_t cs_batch_hist_len(const cs_set_desc* sets, int n_sets) {
    if (!batch_valid(sets, n_sets)) return -1;
    int64_t t = 0;
    for (int s = 0; s < n_sets; ++s) t += cs_hist_len(sets[s].n);
    return t;
}

int cs_batch_create(const cs_set_desc* sets, int n_sets, int path, void* workspace_dev, size_t workspace_bytes,
                    cs_batch** out, void* stream) {
    CS_TRACE("cs_batch_create");
    if (!out) return CS_EINVAL;
    *out = nullptr;
    if (!batch_valid(sets, n_sets) || path < CS_PATH_AUTO || path > CS_PATH_MMA4 || !workspace_dev ||
        (reinterpret_cast<uintptr_t>(workspace_dev) % 1024) != 0)
        return CS_EINVAL;
    const int p = batch_path(sets, n_sets, path);
    if (tensor_path(p) && !device_has_tcgen05()) return CS_EUNSUPPORTED;
    const bool auto_path = path == CS_PATH_AUTO;
    const Layout L = batch_layout(sets, n_sets, p, auto_path);
    if (workspace_bytes < L.total) return CS_ENOMEM;
    const uint64_t* ds_thr = nullptr;
    for (int s = 0; s < n_sets && !ds_thr; ++s)
        if (sets[s].kind == CS_2D_DS_SLAB && !(ds_thr = ds_table_device())) return CS_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace_dev);

    std::vector<BatchSet> bs(static_cast<size_t>(n_sets));
    int64_t elem = 0, rblk = 0, mblk = 0, hoff = 0, tiles = 0;
    int64_t ord_blocks = 0, ord_tasks = 0, ord_nmax = 0;
    std::vector<int32_t> otab, osets;
    int64_t n_largest = 1;
    for (int s = 0; s < n_sets; ++s) {
        BatchSet& b = bs[s];
        b.kind = sets[s].kind;
        b.dim = cs_dim(b.kind);
        b.n = sets[s].n;
        b.seed = sets[s].seed;
        const bool order = set_by_order(sets[s], auto_path);
        b.coords = order ? nullptr : reinterpret_cast<int32_t*>(ws + L.coords[s]);
        b.bits = order ? nullptr : reinterpret_cast<uint64_t*>(ws + L.bits[s]);
        b.order = OrderSet{};
        if (order) {
            b.order.p = reinterpret_cast<int32_t*>(ws + L.ord_p[s]);
            b.order.q = reinterpret_cast<int32_t*>(ws + L.ord_q[s]);
            b.order.R = reinterpret_cast<int32_t*>(ws + L.ord_r[s]);
            b.order.D = reinterpret_cast<uint2*>(ws + L.ord_d[s]);
            b.order.n = int32_t(b.n);
            b.order.W = order_words(b.n);
            b.ord_block = ord_blocks;
            b.ord_task = ord_tasks;
            ord_blocks += order_build_blocks(b.n);
            ord_tasks += order_tasks(b.n, kBatchOrderM);
            ord_nmax = b.n > ord_nmax ? b.n : ord_nmax;
            otab.insert(otab.end(), size_t(order_build_blocks(b.n)), int32_t(s));
            osets.push_back(int32_t(s));
        }
        b.row_words = cs_row_words(b.n);
        b.key0 = reinterpret_cast<uint64_t*>(ws + L.key0[s]);
        b.key1 = reinterpret_cast<uint64_t*>(ws + L.key1[s]);
        b.raw = reinterpret_cast<int32_t*>(ws + L.raw[s]);
        b.ctab = L.ctab[s] ? reinterpret_cast<ConeTable*>(ws + L.ctab[s]) : nullptr;
        b.elem_begin = elem;
        elem += b.n;
        b.vwords = order ? 0 : (b.n + 63) / 64;  // a product order has no bitset: no tiles, no blocks
        b.rblock_begin = rblk;
        rblk += chunks_before(b.vwords, b.vwords);
        b.mir_side = (b.vwords + kMirTiles - 1) / kMirTiles;
        b.mblock_begin = mblk;
        b.tile_begin = tiles;
        tiles += b.vwords;
        mblk += b.mir_side * b.mir_side;
        b.hist_off = hoff;
        hoff += cs_hist_len(b.n);
        n_largest = b.n > n_largest ? b.n : n_largest;
    }
    auto rblocks_end = [&](int s) { return s + 1 < n_sets ? bs[s + 1].rblock_begin : rblk; };
    // Count tables in decreasing set size (the largest sets' tiles go first).
    std::vector<int> order(static_cast<size_t>(n_sets));
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return bs[a].n > bs[b].n; });
    int64_t items = 0, chunks = 0;
    std::vector<int32_t> rtab(static_cast<size_t>(rblk)), etab, mtab(static_cast<size_t>(mblk)),
        ttab(static_cast<size_t>(tiles));
    for (int s = 0; s < n_sets; ++s)
        std::fill(ttab.begin() + bs[s].tile_begin, ttab.begin() + bs[s].tile_begin + bs[s].vwords, int32_t(s));
    for (int s = 0; s < n_sets; ++s)
        std::fill(mtab.begin() + bs[s].mblock_begin, mtab.begin() + bs[s].mblock_begin + bs[s].mir_side * bs[s].mir_side,
                  int32_t(s));
    for (int s = 0; s < n_sets; ++s)
        std::fill(rtab.begin() + bs[s].rblock_begin, rtab.begin() + rblocks_end(s), int32_t(s));
    // the relate blocks grouped by geometry, so that each geometry's launch
    // covers only its own blocks (blocks of the other geometries returning at
    // once had cost their dispatch)
    std::vector<int32_t> rorder;
    rorder.reserve(rtab.size());
    int64_t geo_begin[8], geo_count[8];
    for (int g = 0; g < 8; ++g) {
        geo_begin[g] = int64_t(rorder.size());
        for (int s = 0; s < n_sets; ++s)
            if (batch_geom(bs[s].kind) == g)
                for (int64_t k = bs[s].rblock_begin, end = rblocks_end(s); k < end; ++k) rorder.push_back(int32_t(k));
        geo_count[g] = int64_t(rorder.size()) - geo_begin[g];
    }
    std::vector<PopcSetEntry> pe;
    std::vector<MmaSetEntry> me;
    for (int r = 0; r < n_sets; ++r) {
        const BatchSet& b = bs[order[r]];
        if (by_order(b)) continue;
        if (tensor_path(p)) {
            // FP4 pairs count in supertiles, FP8 in 128-row tiles
            const bool fp4 = p == CS_PATH_MMA4;
            MmaSetEntry e;
            std::memset(static_cast<void*>(&e), 0, sizeof(e));
            if (mma_fill_entry(&e, b.bits, b.n, b.row_words, ws + L.op0[order[r]], ws + L.op1[order[r]], fp4) !=
                CUDA_SUCCESS)
                return CS_ECUDA;
            e.item_begin = items;
            e.item_offset = 0;
            items += fp4 ? mma4_units(b.n) : mma_items(b.n);
            e.hist_off = b.hist_off * 8;
            e.chunk_begin = chunks;
            chunks += mma_expand_chunks(b.n);
            etab.insert(etab.end(), size_t(mma_expand_chunks(b.n)), int32_t(me.size()));  // its entry of the table
            me.push_back(e);
        } else {
            PopcSetEntry e;
            std::memset(static_cast<void*>(&e), 0, sizeof(e));
            popc_fill_entry(&e, b.bits, b.n, b.row_words);
            if (popc_encode_map(&e.map, b.bits, b.n, b.row_words) != CUDA_SUCCESS) return CS_ECUDA;
            e.item_begin = items;
            e.item_offset = 0;
            items += popc_tiles(b.n);
            e.hist_off = b.hist_off * 8;
            pe.push_back(e);
        }
    }
    cs_batch* h = new (std::nothrow) cs_batch;
    if (!h) return CS_ENOMEM;
    if (cudaHostAlloc(reinterpret_cast<void**>(&h->status_host), sizeof(int32_t), cudaHostAllocDefault) !=
            cudaSuccess ||
        cudaEventCreateWithFlags(&h->done, cudaEventDisableTiming) != cudaSuccess) {
        delete h;
        return CS_ECUDA;
    }
    *h->status_host = CS_OK;
    h->nsets = n_sets;
    h->path = p;
    h->ws = ws;
    h->hdr = reinterpret_cast<WsHeader*>(ws);
    h->sets_dev = reinterpret_cast<BatchSet*>(ws + L.sets);
    h->total_elems = elem;
    h->total_rblocks = rblk;
    for (int s = 0; s < n_sets; ++s)
        if (!by_order(bs[s])) h->geoms |= 1u << batch_geom(sets[s].kind);
    h->n_order = int(osets.size());
    h->n_general = n_sets - h->n_order;
    h->otab = reinterpret_cast<int32_t*>(ws + L.otab);
    h->osets = reinterpret_cast<int32_t*>(ws + L.osets);
    h->ord_blocks = ord_blocks;
    h->ord_tasks = ord_tasks;
    h->ord_nmax = ord_nmax;
    h->total_items = items;
    h->total_chunks = chunks;
    h->rtab = reinterpret_cast<int32_t*>(ws + L.rtab);
    h->rorder = reinterpret_cast<int32_t*>(ws + L.rorder);
    for (int g = 0; g < 8; ++g) {
        h->geo_begin[g] = geo_begin[g];
        h->geo_count[g] = geo_count[g];
    }
    h->mtab = reinterpret_cast<int32_t*>(ws + L.mtab);
    h->total_mblocks = mblk;
    h->total_tiles = tiles;
    h->ttab = reinterpret_cast<int32_t*>(ws + L.ttab);
    h->etab = reinterpret_cast<int32_t*>(ws + L.etab);
    h->total_hist = hoff;
    h->n_largest = n_largest;
    h->ds_thr = ds_thr;
    h->coef = reinterpret_cast<dd*>(ws + L.coef);
    h->kends = reinterpret_cast<int64_t*>(ws + L.kends);
    for (int s = 0; s < n_sets; ++s) {
        int64_t& m = h->nmax[bs[s].dim - 2];
        m = bs[s].n > m ? bs[s].n : m;
    }
    int64_t at = 0;
    for (int d = 0; d < kDimSlots; ++d) {
        h->coef_base[d] = at;
        at += h->nmax[d] * kMaxEps;
    }
    cudaError_t e = cudaMemcpyAsync(h->sets_dev, bs.data(), sizeof(BatchSet) * bs.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !rtab.empty())
        e = cudaMemcpyAsync(h->rtab, rtab.data(), rtab.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !rorder.empty())
        e = cudaMemcpyAsync(h->rorder, rorder.data(), rorder.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !mtab.empty())
        e = cudaMemcpyAsync(h->mtab, mtab.data(), mtab.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !ttab.empty())
        e = cudaMemcpyAsync(h->ttab, ttab.data(), ttab.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !otab.empty())
        e = cudaMemcpyAsync(h->otab, otab.data(), otab.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !osets.empty())
        e = cudaMemcpyAsync(h->osets, osets.data(), osets.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !etab.empty())
        e = cudaMemcpyAsync(h->etab, etab.data(), etab.size() * 4, cudaMemcpyHostToDevice, st);
    if (tensor_path(p)) {
        h->mma_dev = reinterpret_cast<MmaSetEntry*>(ws + L.entries);
        if (e == cudaSuccess && !me.empty())
            e = cudaMemcpyAsync(h->mma_dev, me.data(), sizeof(MmaSetEntry) * me.size(), cudaMemcpyHostToDevice, st);
    } else {
        h->popc_dev = reinterpret_cast<PopcSetEntry*>(ws + L.entries);
        if (e == cudaSuccess && !pe.empty())
            e = cudaMemcpyAsync(h->popc_dev, pe.data(), sizeof(PopcSetEntry) * pe.size(), cudaMemcpyHostToDevice, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // the host tables go out of scope
    if (e != cudaSuccess) {
        delete h;
        return CS_ECUDA;
    }
    *out = h;
    return CS_OK;
}

int cs_batch_launch(const cs_batch* b, const double* eps_host, int n_eps, int64_t* hist_dev, double* actions_dev,
                    int64_t* brackets_dev, void* stream) {
    CS_TRACE("cs_batch_launch");
    if (!b || !hist_dev || n_eps < 0 || n_eps > kMaxEps || (n_eps > 0 && (!eps_host || !actions_dev)) ||
        (reinterpret_cast<uintptr_t>(hist_dev) % 8) != 0)
        return CS_EINVAL;
    EpsArgs a;
    a.n = n_eps;
    for (int e = 0; e < kMaxEps; ++e) {
        a.v[e] = e < n_eps ? eps_host[e] : 0.0;
        a.kend[e] = 0;  // per set, in the kernel
        a.factor[e] = dd_from(0.0);  // per dimension, in CoefArgs
        if (e < n_eps && !(a.v[e] <= 1.0)) return CS_EINVAL;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t err = cudaMemsetAsync(&b->hdr->status, 0, sizeof(int32_t), st);
    if (err == cudaSuccess) err = cudaMemsetAsync(hist_dev, 0, size_t(b->total_hist) * 8, st);
    if (err != cudaSuccess) return CS_ECUDA;
    const int sms = device_sm_count();

    int64_t g = (b->total_elems + 255) / 256;
    if (g > int64_t(sms) * 16) g = int64_t(sms) * 16;
    k_batch_keys<<<unsigned(g), 256, 0, st>>>(b->sets_dev, b->nsets, b->total_elems, b->ds_thr, b->hdr);

    // sized by the largest set itself: rounded up to a power of two, a batch
    // whose sets scatter around 4096 left room for one CTA per SM instead of two
    const size_t rank_smem = size_t(b->n_largest) * 20 + size_t(b->n_largest > kRankThreads ? b->n_largest : kRankThreads) * 4;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CS_ECUDA;
    if (dev >= 0 && dev < 64 && !g_rank_attr[dev]) {
        if (cudaFuncSetAttribute(k_batch_rank, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(size_t(CS_BATCH_MAX_N) * 24)) != cudaSuccess)
            return CS_ECUDA;
        g_rank_attr[dev] = true;
    }
    if ((b->geoms & (1u << kGeomLightCone)) && dev >= 0 && dev < 64 && !g_cone_attr[dev]) {
        if (cudaFuncSetAttribute(k_batch_relate_cone, cudaFuncAttributeMaxDynamicSharedMemorySize, kConeTableSmem) !=
            cudaSuccess)
            return CS_ECUDA;
        g_cone_attr[dev] = true;
    }
    // One after another by launch_after: each kernel down to the mirror, and
    // the actions' two, waits for the one before it.  Small batch (160 slabs of
    // 600, 96 2+1 diamonds) 240 -> 227 us, the ensemble's 768 sets 2.636 -> 2.620
    // ms; with early triggers in the kernels before the order count, too,
    // whose blocks then share SMs with its own, 2.668.
    auto unsig = [](int64_t v) { return dim3(unsigned(v)); };
    if ((err = cudaGetLastError()) != cudaSuccess ||
        (err = launch_after(k_batch_rank, unsig(b->nsets), kRankThreads, rank_smem, st, b->sets_dev)) != cudaSuccess)
        return CS_ECUDA;
    if (b->n_order > 0) {
        // at most 16 x 256 bytes of stages and 8192 bins: below the 48 KB any launch may take
        const int64_t grid = (b->ord_tasks + 15) / 16 < int64_t(sms) * 2 ? (b->ord_tasks + 15) / 16 : int64_t(sms) * 2;
        if ((err = launch_after(k_batch_order_table, unsig(b->ord_blocks), kOrdBuildThreads, 0, st, b->sets_dev,
                                b->otab)) != cudaSuccess ||
            (err = launch_after(k_batch_order_count, unsig(grid), kBatchOrderThreads,
                                kBatchOrderThreads * sizeof(int2) + size_t(b->ord_nmax) * 4, st, b->sets_dev, b->osets,
                                b->n_order, b->ord_tasks, hist_dev)) != cudaSuccess)
            return CS_ECUDA;
    }
    if ((b->geoms & (1u << kGeomLightCone)) &&
        launch_after(k_batch_ctab, unsig((b->total_tiles * 32 + 255) / 256), 256, 0, st, b->sets_dev, b->ttab,
                     b->total_tiles) != cudaSuccess)
        return CS_ECUDA;

    if (b->total_rblocks > int64_t(0x7fffffff)) return CS_EINVAL;
    // one launch per geometry present, over that geometry's blocks only
    auto range = [&](int g) { return b->rorder + b->geo_begin[g]; };
    if (b->geo_count[kGeomLightCone] &&
        launch_after(k_batch_relate_cone, unsig(b->geo_count[kGeomLightCone]), kRelThreads, kConeTableSmem, st,
                     b->sets_dev, b->rtab, range(kGeomLightCone), b->hdr) != cudaSuccess)
        return CS_ECUDA;
    auto relate = [&](auto kernel, int g) {
        return b->geo_count[g] ? launch_after(kernel, unsig(b->geo_count[g]), kRelThreads, 0, st, b->sets_dev, b->rtab,
                                              range(g))
                               : cudaSuccess;
    };
    if (relate(k_batch_relate<kGeom3>, kGeom3) != cudaSuccess || relate(k_batch_relate<kGeom4>, kGeom4) != cudaSuccess ||
        relate(k_batch_relate<kGeomDeSitter>, kGeomDeSitter) != cudaSuccess)
        return CS_ECUDA;
    if (b->total_mblocks > int64_t(0x7fffffff)) return CS_EINVAL;
    if (b->total_mblocks > 0 && launch_after(k_batch_mirror, unsig(b->total_mblocks), kRelThreads, 0, st, b->sets_dev,
                                             b->mtab) != cudaSuccess)
        return CS_ECUDA;

    if (b->n_general == 0) {
        err = cudaSuccess;
    } else if (b->path == CS_PATH_MMA) {
        if ((err = launch_expand_multi(b->mma_dev, b->etab, b->total_chunks, st)) != cudaSuccess) return CS_ECUDA;
        err = launch_count_mma_multi(b->mma_dev, b->n_general, b->total_items, reinterpret_cast<uintptr_t>(hist_dev),
                                     b->hdr, 0, st);
    } else if (b->path == CS_PATH_MMA4) {
        if ((err = launch_expand_multi(b->mma_dev, b->etab, b->total_chunks, st, true)) != cudaSuccess)
            return CS_ECUDA;
        err = launch_count_mma4_multi(b->mma_dev, b->n_general, b->total_items, reinterpret_cast<uintptr_t>(hist_dev),
                                      b->hdr, st);
    } else {
        err = launch_count_popc_multi(b->popc_dev, b->n_general, b->total_items, reinterpret_cast<uintptr_t>(hist_dev),
                                      b->hdr, 0, st);
    }
    if (err != cudaSuccess) return CS_ECUDA;
    if (n_eps > 0 || brackets_dev) {
        CoefArgs c;
        std::memset(static_cast<void*>(&c), 0, sizeof(c));
        int64_t at = 0;
        for (int d = 0; d < kDimSlots; ++d) {
            c.base[d] = b->coef_base[d];
            c.stride[d] = b->nmax[d];
            const int64_t nm = b->nmax[d], len = nm > 1 ? nm - 1 : 1;
            for (int e = 0; e < kMaxEps; ++e) {
                c.kcap[d][e] = (nm > 0 && e < n_eps && !is_local(a.v[e]))
                                   ? smear_cutoff(d + 2, a.v[e], 0.5 * double(nm) * double(nm), len)
                                   : 0;
                c.seg[d * kMaxEps + e] = at;
                at += c.kcap[d][e];
                c.factor[d][e] = nm > 0 && e < n_eps ? action_factor(d + 2, a.v[e]) : dd_from(0.0);
            }
        }
        c.seg[kDimSlots * kMaxEps] = at;
        if (at > 0) {
            // one warp per block: the FP64 work (table entries, then the
            // cutoffs) spreads over every SM's FP64 pipe
            int64_t g = (at + int64_t(b->nsets) * a.n + 31) / 32;
            if (g > int64_t(sms) * 16) g = int64_t(sms) * 16;
            BatchPowers powers;
            for (int e = 0; e < kMaxEps; ++e)
                if (e < n_eps && !is_local(a.v[e])) {
                    powers.e[e] = eps_powers(a.v[e]);
                    for (int d = 0; d < kDimSlots; ++d) powers.c[d][e] = smear_coef(d + 2, a.v[e]);
                }
            if (launch_after(k_batch_coef, unsig(g), 32, 0, st, b->coef, c, a, powers, b->sets_dev, b->nsets,
                             b->kends) != cudaSuccess)
                return CS_ECUDA;
        }
        if (launch_after(k_batch_action, unsig(b->nsets * (a.n > 0 ? a.n : 1)), kActThreads, 0, st, b->sets_dev,
                         hist_dev, a, b->coef, c, b->kends, actions_dev, brackets_dev) != cudaSuccess)
            return CS_ECUDA;
    }
    // For cs_batch_poll: the status word to the plan's pinned copy, then the
    // event (recorded as an external event node when the stream is captured).
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if ((err = cudaStreamIsCapturing(st, &cap)) != cudaSuccess) return cuda_status(err);
    if ((err = cudaMemcpyAsync(b->status_host, &b->hdr->status, sizeof(int32_t), cudaMemcpyDeviceToHost, st)) !=
        cudaSuccess)
        return cuda_status(err);
    err = cap == cudaStreamCaptureStatusActive ? cudaEventRecordWithFlags(b->done, st, cudaEventRecordExternal)
                                               : cudaEventRecord(b->done, st);
    return cuda_status(err);
}

int cs_batch_poll(const cs_batch* b) {
    if (!b) return CS_EINVAL;
    const cudaError_t q = cudaEventQuery(b->done);
    if (q == cudaErrorNotReady) {
        cudaGetLastError();  // not sticky; keep it from the caller's next check
        return CS_PENDING;
    }
    if (q != cudaSuccess) return CS_ECUDA;
    return *static_cast<volatile int32_t*>(b->status_host);
}

int cs_batch_path(const cs_batch* b) { return b ? b->path : -1; }

void cs_batch_destroy(cs_batch* b) { delete b; }

}  // extern "C"
