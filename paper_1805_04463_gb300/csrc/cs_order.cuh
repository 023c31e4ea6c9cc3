// cs_order.cuh -- interval abundances of sets whose relation is the product
// order of two coordinates (random 2D orders, the 1+1 diamond and square in
// light-cone coordinates), shared by the single-set and batched counts.
//
// Relabel the elements by u and let p[a] be the rank of v of element a (u
// ascending, v descending on equal u; v ascending, u descending on equal v,
// so that two elements equal in a coordinate are never in order): a precedes
// b iff a < b and p[a] < p[b], and an abundance does not depend on labels.
// With D(x, y) = #{c < x : p[c] < y},
//   |A_ab| = #{a < c < b : p[a] < p[c] < p[b]}
//          = (R_b - D(a + 1, p[b])) - (D(b, p[a]) - R_a),   R_c = D(c, p[c]):
// the elements after a below p[b], less those below p[a].  A count is four
// lookups instead of a sum over the interval, O(n^2) for the whole set where
// the contraction takes n^3 / 3 multiply-adds.
#pragma once

#include "cs_internal.cuh"
#include "cs_sprinkle.cuh"

namespace cs {

// One set.  Rows of D at every 64th element: word w of row X holds, as a
// bitmask, which y in [32 w, 32 w + 32) are the p of an element before 64 X,
// and how many such y lie before 32 w, so D(64 X, y) is one 8-byte load and
// a population count.  n^2 / 256 bytes.
struct OrderSet {
    const int32_t* p;  // rank of v by u rank
    const int32_t* q;  // its inverse
    int32_t* R;        // R_a = D(a, p[a])
    uint2* D;          // [bands][W]: {mask, elements before the word}
    int32_t n, W;      // W = ceil(n / 32)
};

constexpr int kOrdBand = 64;         // rows of a warp task: two per lane
constexpr int kOrdRowsPerBlock = 8;  // rows of D a block builds (one per warp)
constexpr int kOrdBuildThreads = 32 * kOrdRowsPerBlock;
constexpr int kOrdBuildWords = 512;  // words of those rows per step

__host__ __device__ inline int order_words(int64_t n) { return int((n + 31) / 32); }
__host__ __device__ inline int order_bands(int64_t n) { return int((n + kOrdBand - 1) / kOrdBand); }
__host__ __device__ inline size_t order_table_bytes(int64_t n) {
    return size_t(order_bands(n)) * size_t(order_words(n)) * sizeof(uint2);
}
__host__ __device__ inline int order_build_blocks(int64_t n) {
    return (order_bands(n) + kOrdRowsPerBlock - 1) / kOrdRowsPerBlock;
}

// D(64 X, y), 0 <= y < n.
__device__ __forceinline__ int order_lookup(const uint2* D, int W, int X, int y) {
    const uint2 e = D[size_t(X) * W + (y >> 5)];
    return int(e.y) + __popc(e.x & ((1u << (y & 31)) - 1u));
}

// Sort keys of one coordinate of a set of at most 8192 elements for
// rank_keys_smem: val ascending, sec descending on equal val, shifted so that
// the set's largest val - smallest val fills the top bits (the buckets then
// hold about one key each for any spread-out coordinates, whatever their
// range: ranks 0..n-1 and 31-bit light-cone coordinates alike).  Values in
// [0, 2^31).  All kRankThreads threads; sk[i] is written by thread
// i % kRankThreads.
__device__ __forceinline__ void order_keys_smem(const int32_t* val, const int32_t* sec, int n,
                                                uint64_t* sk) {
    __shared__ int lo_w[kRankThreads / 32], hi_w[kRankThreads / 32];
    int lo = INT32_MAX, hi = INT32_MIN;
    for (int i = threadIdx.x; i < n; i += kRankThreads) {
        const int v = val[i];
        lo = min(lo, v);
        hi = max(hi, v);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        lo_w[threadIdx.x >> 5] = lo;
        hi_w[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lo_w[threadIdx.x & 31]);
    hi = __reduce_max_sync(0xffffffffu, hi_w[threadIdx.x & 31]);
    const int nb = 32 - __clz(max(uint32_t(hi) - uint32_t(lo), 1u));
    for (int i = threadIdx.x; i < n; i += kRankThreads)
        sk[i] = (uint64_t(uint32_t(val[i]) - uint32_t(lo)) << (64 - nb)) |
                (uint64_t((0x7FFFFFFFu - uint32_t(sec[i])) & 0x7FFFFFFFu) << (33 - nb));
}

// p and q of a set of at most 8192 elements by one CTA of kRankThreads
// threads; by_u: the labels are in u order.  smem: 20 n bytes (keys, slots,
// ranks, u ranks) and 4 << lgP (bucket counts), 2^lgP >= kRankThreads.
__device__ __forceinline__ void order_ranks_smem(const int32_t* __restrict__ u, const int32_t* __restrict__ v, bool by_u,
                                                 int n, int lgP, uint8_t* smem, int32_t* __restrict__ p,
                                                 int32_t* __restrict__ q) {
    const int P = 1 << lgP;
    uint64_t* sk = reinterpret_cast<uint64_t*>(smem);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(sk + n);
    uint32_t* slot = cnt + P;
    uint32_t* rank = slot + n;
    uint32_t* ru = rank + n;
    if (!by_u) {
        order_keys_smem(u, v, n, sk);
        rank_keys_smem(n, lgP, sk, cnt, slot, ru);
    }
    order_keys_smem(v, u, n, sk);
    rank_keys_smem<true>(n, lgP, sk, cnt, slot, rank);
    for (int e = threadIdx.x; e < n; e += kRankThreads) {
        const int a = by_u ? e : int(ru[e]), r = int(rank[e]);
        p[a] = r;
        q[r] = a;
    }
}

// Rows [8 g, 8 g + 8) of D and R of their elements.  The masks of the first
// row are ballots of q[y] < 512 g, sixteen words' loads in flight (load and
// ballot one after another left the build latency-bound, 242 against 92 us
// at n = 131072 with 32-row bands); each next row adds its band's 64
// elements, which their p scatter into a shared array.  Then warp x scans row
// 8 g + x.  All kOrdBuildThreads threads.
__device__ __forceinline__ void order_build_rows(const OrderSet& s, int g) {
    __shared__ uint32_t m[kOrdRowsPerBlock][kOrdBuildWords];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int X0 = g * kOrdRowsPerBlock, X = X0 + warp;
    const int a0 = kOrdBand * X + lane;  // this thread's elements: a0 and a0 + 32
    const int p0 = a0 < s.n ? s.p[a0] : INT32_MAX, p1 = a0 + 32 < s.n ? s.p[a0 + 32] : INT32_MAX;
    const bool row = X < order_bands(s.n);  // warp-uniform
    uint32_t carry = 0;  // elements before the step's words, in row X
    for (int w0 = 0; w0 < s.W; w0 += kOrdBuildWords) {
        const int nw = min(kOrdBuildWords, s.W - w0);
        for (int w = threadIdx.x; w < (kOrdRowsPerBlock - 1) * kOrdBuildWords; w += kOrdBuildThreads)
            m[1 + w / kOrdBuildWords][w % kOrdBuildWords] = 0u;
        for (int wb = warp; wb < nw; wb += 16 * kOrdRowsPerBlock) {
            int qy[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int y = 32 * (w0 + wb + k * kOrdRowsPerBlock) + lane;
                qy[k] = s.q[min(y, s.n - 1)];
                if (y >= s.n) qy[k] = INT32_MAX;
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const uint32_t b = __ballot_sync(0xffffffffu, qy[k] < kOrdBand * X0);
                const int w = wb + k * kOrdRowsPerBlock;
                if (lane == 0 && w < nw) m[0][w] = b;
            }
        }
        __syncthreads();
        // row x > 0 holds row x - 1 and band x - 1
        if (warp < kOrdRowsPerBlock - 1) {
            if (unsigned((p0 >> 5) - w0) < unsigned(nw)) atomicOr(&m[warp + 1][(p0 >> 5) - w0], 1u << (p0 & 31));
            if (unsigned((p1 >> 5) - w0) < unsigned(nw)) atomicOr(&m[warp + 1][(p1 >> 5) - w0], 1u << (p1 & 31));
        }
        __syncthreads();
        if (row) {
            for (int wb = 0; wb < nw; wb += 32) {
                const int w = wb + lane;
                uint32_t mask = 0u;
                if (w < nw) {
                    mask = m[0][w];
#pragma unroll
                    for (int x = 1; x < kOrdRowsPerBlock; ++x)
                        if (x <= warp) mask |= m[x][w];
                }
                const uint32_t c = __popc(mask);
                uint32_t incl = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                if (w < nw) s.D[size_t(X) * s.W + w0 + w] = make_uint2(mask, carry + incl - c);
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
        }
        __syncthreads();  // the masks are read; and the row's words are visible to the block
    }
    if (row) {
        // R: the row's count plus the elements of the band before a and below p[a]
        auto base = [&](int pa) {
            if (pa == INT32_MAX) return 0;
            const uint2 e = s.D[size_t(X) * s.W + (pa >> 5)];
            return int(e.y) + __popc(e.x & ((1u << (pa & 31)) - 1u));
        };
        int r0 = base(p0), r1 = base(p1);
#pragma unroll 8
        for (int c = 0; c < 32; ++c) {
            const int c0 = __shfl_sync(0xffffffffu, p0, c), c1 = __shfl_sync(0xffffffffu, p1, c);
            r0 += c < lane && c0 < p0;
            r1 += (c0 < p1) + (c < lane && c1 < p1);
        }
        if (a0 < s.n) s.R[a0] = r0;
        if (a0 + 32 < s.n) s.R[a0 + 32] = r1;
    }
}

// Warp tasks: band A (rows [64 A, 64 A + 64)) against column chunk C
// (columns [chunk C, chunk C + chunk), chunk = 64 m), of the chunks that reach
// past the band's first row.  Chunk C has m (C + 1) candidate bands;
// m C (C + 1) / 2 tasks come before it.
__host__ __device__ inline int64_t order_tasks(int64_t n, int m) {
    const int64_t chunks = (order_bands(n) + m - 1) / m;
    return m * chunks * (chunks + 1) / 2;
}

__device__ __forceinline__ void order_decode(int64_t t, int m, int& A, int& C) {
    const int64_t k = t / m;  // triangle index of the chunk pair
    int64_t c = int64_t((sqrtf(1.0f + 8.0f * float(k)) - 1.0f) * 0.5f);  // corrected below
    while (c * (c + 1) / 2 > k) --c;
    while ((c + 1) * (c + 2) / 2 <= k) ++c;
    C = int(c);
    A = int(t - m * (c * (c + 1) / 2));
}

// One column of 64 pairs: lane l's rows 2 l and 2 l + 1 of the band against
// column (pb, xb).  With c = #{rows a <= 2 l of the band : p_a < pb} (row
// 2 l + 1 counts itself too; that one is in its y from the start),
//   at = y + xb - 4 c;  a related row adds 1 at [at], the other ones
//   (p > pb) lower their y by 4 and add to the spare bin (red_shared_one:
//   every lane adds, and the constant 1).
// le / lt: the lanes at or before / before this one.
struct OrderRows {
    int p0, p1;
    uint32_t y0, y1, le, lt;
};
__device__ __forceinline__ void order_column(OrderRows& r, int pb, int xb, uint32_t spare) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b32 m, c, t, u;\n\t"
        "setp.lt.s32 p, %2, %6;\n\t"
        "setp.lt.s32 q, %3, %6;\n\t"
        "vote.sync.ballot.b32 m, p, 0xffffffff;\n\t"
        "vote.sync.ballot.b32 c, q, 0xffffffff;\n\t"
        "and.b32 m, m, %4;\n\t"
        "and.b32 c, c, %5;\n\t"
        "popc.b32 m, m;\n\t"
        "popc.b32 c, c;\n\t"
        "add.s32 c, c, m;\n\t"
        "mad.lo.s32 t, c, -4, %7;\n\t"
        "add.s32 u, %1, t;\n\t"
        "add.s32 t, %0, t;\n\t"
        "selp.b32 t, t, %8, p;\n\t"
        "selp.b32 u, u, %8, q;\n\t"
        "red.shared.add.u32 [t], 1;\n\t"
        "red.shared.add.u32 [u], 1;\n\t"
        "@!p add.s32 %0, %0, -4;\n\t"
        "@!q add.s32 %1, %1, -4;\n\t}"
        : "+r"(r.y0), "+r"(r.y1)
        : "r"(r.p0), "r"(r.p1), "r"(r.le), "r"(r.lt), "r"(pb), "r"(xb), "r"(spare)
        : "memory");
}

// A column of the band itself: only its rows before band column own count.
__device__ __forceinline__ void order_column_own(OrderRows& r, int pb, int xb, uint32_t spare, int row, int own) {
    asm volatile(
        "{\n\t.reg .pred p, q, f, g;\n\t.reg .b32 m, c, t, u;\n\t"
        "setp.lt.s32 p, %2, %6;\n\t"
        "setp.lt.s32 q, %3, %6;\n\t"
        "vote.sync.ballot.b32 m, p, 0xffffffff;\n\t"
        "vote.sync.ballot.b32 c, q, 0xffffffff;\n\t"
        "and.b32 m, m, %4;\n\t"
        "and.b32 c, c, %5;\n\t"
        "popc.b32 m, m;\n\t"
        "popc.b32 c, c;\n\t"
        "add.s32 c, c, m;\n\t"
        "mad.lo.s32 t, c, -4, %7;\n\t"
        "add.s32 u, %1, t;\n\t"
        "add.s32 t, %0, t;\n\t"
        "setp.lt.and.s32 f, %9, %10, p;\n\t"
        "add.s32 c, %9, 1;\n\t"
        "setp.lt.and.s32 g, c, %10, q;\n\t"
        "selp.b32 t, t, %8, f;\n\t"
        "selp.b32 u, u, %8, g;\n\t"
        "red.shared.add.u32 [t], 1;\n\t"
        "red.shared.add.u32 [u], 1;\n\t"
        "setp.gt.s32 p, %2, %6;\n\t"
        "setp.gt.s32 q, %3, %6;\n\t"
        "@p add.s32 %0, %0, -4;\n\t"
        "@q add.s32 %1, %1, -4;\n\t}"
        : "+r"(r.y0), "+r"(r.y1)
        : "r"(r.p0), "r"(r.p1), "r"(r.le), "r"(r.lt), "r"(pb), "r"(xb), "r"(spare), "r"(row), "r"(own)
        : "memory");
}

// A column whose counts may lie at or past the bins: those add to hist_g.
__device__ __forceinline__ void order_column_wide(OrderRows& r, int pb, int xb, int row, int own, uint32_t hist_s,
                                                  uint32_t spare, unsigned long long* hist_g) {
    const bool p = r.p0 < pb, q = r.p1 < pb;
    const uint32_t c = __popc(__ballot_sync(0xffffffffu, p) & r.le) + __popc(__ballot_sync(0xffffffffu, q) & r.lt);
    const uint32_t t = r.y0 + uint32_t(xb) - 4u * c, u = r.y1 + uint32_t(xb) - 4u * c;
    const bool cp = p && row < own, cq = q && row + 1 < own;
    red_shared_one(cp && t < spare ? t : spare);
    red_shared_one(cq && u < spare ? u : spare);
    if (cp && t >= spare) atomicAdd(hist_g + ((t - hist_s) >> 2), 1ull);
    if (cq && u >= spare) atomicAdd(hist_g + ((u - hist_s) >> 2), 1ull);
    if (pb < r.p0) r.y0 -= 4u;
    if (pb < r.p1) r.y1 -= 4u;
}

// Histogram the pairs of one task.  Lane l holds rows a = 64 A + 2 l and the
// next and, for the columns b one after another, y = R_a - D(b, p_a), which
// falls by one at every b with p_b < p_a.  x_b = R_b - D(64 A, p_b) is found
// once per band by lane b of each 32-column step (loaded a step ahead) and
// read back by all lanes; the rows of the band at or before a that lie below
// p_b are two ballots and population counts.  Per 32 pairs nine instructions,
// one of them the shared add; what bounds the count is the shared-memory
// pipe (adds 2.4 passes each, the broadcast of the column half of one).
// hist_s: shared address of the bins [0, bins) and a spare one; counts at or
// past bins go to hist_g.  stage: 32 int2 of the warp.
__device__ __forceinline__ void order_task(const OrderSet& s, int A, int C, int chunk, uint32_t hist_s, int bins,
                                           unsigned long long* hist_g, int2* stage) {
    const int lane = threadIdx.x & 31, n = s.n, W = s.W;
    const int a0 = kOrdBand * A;
    const int c0 = C * chunk, cend = min(c0 + chunk, n);
    if (a0 >= cend) return;
    const int b0 = c0 > a0 ? c0 : a0;
    const uint32_t spare = hist_s + 4u * uint32_t(bins);
    OrderRows r;
    r.le = 0xffffffffu >> (31 - lane);
    r.lt = r.le >> 1;
    // y in bytes of the histogram, with its address; x likewise.  A row past n
    // precedes nothing.
    const int a = a0 + 2 * lane;
    r.p0 = r.p1 = INT32_MAX;
    r.y0 = r.y1 = hist_s;
    if (a < n) {
        r.p0 = s.p[a];
        r.y0 += 4u * uint32_t(s.R[a] - order_lookup(s.D, W, b0 / kOrdBand, r.p0));
    }
    if (a + 1 < n) {
        r.p1 = s.p[a + 1];
        r.y1 += 4u * uint32_t(s.R[a + 1] - order_lookup(s.D, W, b0 / kOrdBand, r.p1)) - 4u;
    }
    // A count is below b - a, and at most y + x: in a task where it can pass the
    // bins only the columns where y + x does, for the largest y, take the
    // general form.  (All columns of such tasks took it: 4.11 against 3.79 ms
    // for a 2D order of 131072, a third of whose tasks lie there.)
    const bool wide = cend - 1 - a0 > bins;
    // column c of a step and its x
    auto column_of = [&](int b) {
        int2 v = make_int2(-1, 0);
        if (b < cend) {
            v.x = s.p[b];
            v.y = 4 * (s.R[b] - order_lookup(s.D, W, A, v.x));
        }
        return v;
    };
    int2 next = column_of(b0 + lane);
    for (int bc = b0; bc < cend; bc += 32) {
        const int nb = min(32, cend - bc);
        const int2 st = next;
        next = column_of(bc + 32 + lane);
        __syncwarp();  // the previous step's reads are done
        stage[lane] = st;
        __syncwarp();
        uint32_t over = 0u;
        if (wide) {
            const int top = __reduce_max_sync(0xffffffffu, max(int(r.y0), int(r.y1)));
            over = __ballot_sync(0xffffffffu, top + st.y >= int(spare));
        }
        if (over) {
            if (bc < a0 + kOrdBand) over = 0xffffffffu;
#pragma unroll 2
            for (int c = 0; c < nb; ++c) {
                const int2 v = stage[c];
                if ((over >> c) & 1u)
                    order_column_wide(r, v.x, v.y, 2 * lane, bc + c - a0, hist_s, spare, hist_g);
                else
                    order_column(r, v.x, v.y, spare);
            }
        } else if (bc < a0 + kOrdBand) {
#pragma unroll 4
            for (int c = 0; c < nb; ++c)
                order_column_own(r, stage[c].x, stage[c].y, spare, 2 * lane, bc + c - a0);
        } else if (nb < 32) {
#pragma unroll 4
            for (int c = 0; c < nb; ++c) order_column(r, stage[c].x, stage[c].y, spare);
        } else {
            const int4* s4 = reinterpret_cast<const int4*>(stage);
#pragma unroll 4
            for (int c = 0; c < 16; ++c) {
                const int4 v = s4[c];
                order_column(r, v.x, v.y, spare);
                order_column(r, v.z, v.w, spare);
            }
        }
    }
}

}  // namespace cs
