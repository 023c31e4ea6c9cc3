// cs_relate.cuh -- one block of the causal-matrix build (2048 columns x 64
// rows), shared by the single-set and batched relate kernels.
#pragma once

#include "cs_internal.cuh"

namespace cs {

constexpr int kRelColsPerBlock = 2048;
constexpr int kRelWordsPerBlock = kRelColsPerBlock / 64;
constexpr int kRelRowsPerBlock = 64;
constexpr int kRelThreads = 256;
constexpr int kRelWarpWords = kRelWordsPerBlock / (kRelThreads / 32);  // words of one warp: a 32-byte sector
static_assert(kRelWarpWords == 4, "a warp's words of a row are one sector");

// Geometries of the relation test; the number of coordinates is geom_dim(G).
constexpr int kGeomLightCone = 2, kGeom3 = 3, kGeom4 = 4, kGeomDeSitter = 5;
constexpr int geom_dim(int g) { return g == kGeom3 || g == kGeom4 ? g : 2; }

// Symmetric timelike test between two elements (coordinates a, b): du * dv > 0 (1+1,
// light-cone coordinates), dt^2 - |dx|^2 > 0 (2+1, 3+1) exact in int64, or,
// on a circle (the de Sitter slab's conformal grid, Eq. ds_metric, and the
// 1+1 cylinder), the angular separation below the (conformal-)time
// separation.
template <int G>
__device__ __forceinline__ bool rel_related(const int32_t (&a)[geom_dim(G)], const int32_t (&b)[geom_dim(G)]) {
    if constexpr (G == kGeomDeSitter) {
        // |eta| < 2^30 (slab: < 2^29, cylinder: < 2^31 / pi), so de fits
        // int32; theta differences wrap modulo 2^32, one full turn.
        const int32_t de = b[0] - a[0];
        const uint32_t d = uint32_t(b[1]) - uint32_t(a[1]);
        const uint32_t circ = min(d, 0u - d);
        return circ < uint32_t(abs(de));
    } else if constexpr (G == kGeomLightCone) {
        // du * dv > 0 as a sign test (|du|, |dv| < 2^31 fit int32)
        const int32_t du = b[0] - a[0];
        const int32_t dv = b[1] - a[1];
        return (du ^ dv) >= 0 && du != 0 && dv != 0;
    } else {
        // |coordinates| < 2^29: differences fit int32 and each square is one
        // widening multiply-add into the int64 sum (< 2^62, exact)
        const int32_t dt = b[0] - a[0];
        int64_t s2 = int64_t(dt) * dt;
#pragma unroll
        for (int d = 1; d < G; ++d) {
            const int32_t dx = b[d] - a[d];
            s2 -= int64_t(dx) * dx;
        }
        return s2 > 0;
    }
}

// A word of the matrix, exactly, by a whole warp: lane l holds columns
// 64 W + l and 64 W + l + 32, two ballots fold the tests of a row.  Columns
// at or beyond n are 0.
template <int G>
struct ExactWord {
    static constexpr int D = geom_dim(G);
    int32_t b[2][D];
    int64_t j0;
    bool in[2];
    __device__ __forceinline__ ExactWord(const int32_t* __restrict__ coords, int64_t n, int64_t W) {
        j0 = 64 * W + (threadIdx.x & 31);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            in[k] = j0 + 32 * k < n;
#pragma unroll
            for (int d = 0; d < D; ++d) b[k][d] = in[k] ? coords[d * n + j0 + 32 * k] : 0;
        }
    }
    __device__ __forceinline__ uint64_t row(const int32_t* __restrict__ coords, int64_t n, int64_t i) const {
        int32_t a[D];
#pragma unroll
        for (int d = 0; d < D; ++d) a[d] = coords[d * n + i];
        const uint32_t lo = __ballot_sync(0xffffffffu, in[0] && rel_related<G>(a, b[0]));
        const uint32_t hi = __ballot_sync(0xffffffffu, in[1] && rel_related<G>(a, b[1]));
        return (uint64_t(hi) << 32) | lo;
    }
};

// FP32 filter for the 2+1 and 3+1 tests.  With every coordinate in
// [-kFilterRange, kFilterRange] = [-2^20, 2^20],
//   s = 2^23 - (dt^2 - |dx|^2) = A_j + B_i + 2 t_i t_j - 2 x_i . x_j,
//   B = |x|^2 - t^2, A = B + 2^23,
// one add and D fused multiply-adds per pair.  A and B are off by less than
// 2^18.6 each (every square is below 2^40, the sum below 2^42); A + B and the
// partial sums stay below 2^43.8, so the add rounds by at most 2^18, the first
// multiply-add by 2^18 and the others by 2^19: the value lies within 2^22 of
// the exact one.  Negative means s2 > 2^23 - 2^22 > 0 (related), above 2^24
// means s2 < 0, and only a value in [0, 2^24] needs the exact test (about one
// word in a thousand holds one).
constexpr int32_t kFilterRange = 1 << 20;
constexpr float kFilterSlack = 8388608.0f;  // 2^23
// Bits of the float 2^24: a value in [+0, 2^24] has bits at most this as an
// unsigned integer, and every negative value (sign bit set) has more.
constexpr uint32_t kBandBits = 0x4B800000u;

// |x|^2 - t^2 in FP32.
template <int D>
__device__ __forceinline__ float filter_norm(const int32_t (&c)[D]) {
    const float t = float(c[0]);
    float s = -t * t;
#pragma unroll
    for (int d = 1; d < D; ++d) s = fmaf(float(c[d]), float(c[d]), s);
    return s;
}

// Two FP32 values side by side, each operation rounded like the scalar one.
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// x * one + y as a multiply-add (one is 1 at run time).
__device__ __forceinline__ int32_t cone_mad(int32_t x, int32_t one, int32_t y) {
    int32_t d;
    asm("mad.lo.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(x), "r"(one), "r"(y));
    return d;
}

// |d| - (ej - ei) modulo 2^32.
__device__ __forceinline__ int32_t circle_gap(int32_t d, int32_t ei, int32_t ej) {
    uint32_t a;
    asm("abs.s32 %0, %1;" : "=r"(a) : "r"(d));  // 2^31 for d = -2^31
    return int32_t(a + uint32_t(ei) - uint32_t(ej));
}

// Staged bytes per column: u and v (light cone, circle), the coordinates and
// A (filtered 2+1, 3+1).
__host__ __device__ constexpr int relate_stage_bytes(int g) {
    return kRelColsPerBlock * (g == kGeomLightCone || g == kGeomDeSitter ? 8 : g == kGeom3 ? 16 : 20) +
           16;  // and a runtime 1 (the multiplier)
}

// A row as the tests see it: light cone ~u and ~v; circle eta and -theta;
// filtered 2+1 and 3+1 the multipliers (2 t, -2 x, ..) and B, each twice.
template <int G>
struct RelRow {
    int32_t nu, nv;
};
template <>
struct RelRow<kGeom3> {
    uint64_t k[3], b;
};
template <>
struct RelRow<kGeom4> {
    uint64_t k[4], b;
};

// acc shifted left by one, x's sign bit shifted in.
__device__ __forceinline__ uint32_t push_sign(uint32_t x, uint32_t acc) {
    uint32_t r;
    asm("shf.l.wrap.b32 %0, %1, %2, 1;" : "=r"(r) : "r"(x), "r"(acc));
    return r;
}

// The sign bits of a lane's two rows against the 64 staged columns from pair
// pbase on: acc[row][half], and (2+1, 3+1) the unsigned minimum of the
// filter's bits.  kOwn: the row tile's own word, where column lane (+ 32 for
// the second row) is the row itself, whose value lies in the band and is left
// out of the minimum.
template <int G, bool kOwn>
__device__ __forceinline__ void relate_word(const uint8_t* __restrict__ smem, int pbase, const RelRow<G> (&row)[2],
                                            int32_t one, uint32_t (&acc)[2][2], uint32_t (&band)[2]) {
    constexpr bool kFilter = G == kGeom3 || G == kGeom4;
    band[0] = band[1] = ~0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t s0 = 0u, s1 = 0u;
        // highest column first: after 32 shifts column 32 h is bit 0
        if constexpr (kFilter) {
            const ulonglong2* q0 = reinterpret_cast<const ulonglong2*>(smem) + pbase;
            const ulonglong2* q1 = q0 + kRelColsPerBlock / 2;
            const uint64_t* q2 = reinterpret_cast<const uint64_t*>(smem) + 2 * kRelColsPerBlock + pbase;
#pragma unroll 4
            for (int p = 16 * h + 15; p >= 16 * h; --p) {
                const ulonglong2 tx = q0[p], yz = q1[p];
                const uint64_t A = G == kGeom4 ? q2[p] : yz.y;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    uint64_t s = f2_add(A, row[r].b);
                    s = f2_fma(row[r].k[0], tx.x, s);
                    s = f2_fma(row[r].k[1], tx.y, s);
                    s = f2_fma(row[r].k[2], yz.x, s);
                    if constexpr (G == kGeom4) s = f2_fma(row[r].k[geom_dim(G) - 1], yz.y, s);
                    const uint32_t lo = uint32_t(s), hi = uint32_t(s >> 32);
                    uint32_t& a = r == 0 ? s0 : s1;
                    a = push_sign(hi, a);
                    a = push_sign(lo, a);
                    if constexpr (kOwn) {
                        const int d = int(threadIdx.x & 31) + 32 * r - 2 * p;  // 0 or 1: this pair holds the row itself
                        band[r] = min(band[r], min(d == 0 ? ~0u : lo, d == 1 ? ~0u : hi));
                    } else {
                        band[r] = min(band[r], min(lo, hi));
                    }
                }
            }
        } else {
            const int4* q = reinterpret_cast<const int4*>(smem) + pbase;  // two columns
#pragma unroll
            for (int p = 16 * h + 15; p >= 16 * h; --p) {
                const int4 x = q[p];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    int32_t d1 = cone_mad(x.w, one, row[r].nv), d0 = cone_mad(x.y, one, row[r].nv);
                    if constexpr (G == kGeomDeSitter) {
                        d1 = circle_gap(d1, row[r].nu, x.z);
                        d0 = circle_gap(d0, row[r].nu, x.x);
                    } else {
                        d1 |= cone_mad(x.z, one, row[r].nu);
                        d0 |= cone_mad(x.x, one, row[r].nu);
                    }
                    uint32_t& a = r == 0 ? s0 : s1;
                    a = push_sign(uint32_t(d1), a);
                    a = push_sign(uint32_t(d0), a);
                }
            }
        }
        acc[0][h] = s0;
        acc[1][h] = s1;
    }
}

// Rows [64 rb, 64 rb + 64) x words [w0, w0 + 32) of the bitset, less the words
// before the row tile (word < rb): the relation is symmetric, so mirror_block
// fills those as transposes.  w0 is a multiple of 4.  zero_from >= 0: the
// block also zeroes each row's words [zero_from, row_words) (padding past a
// row's last chunk).  smem: relate_stage_bytes(G), 16-byte aligned.  All 256
// threads.
//
// A lane owns two rows (l and l + 32 of the tile) and a warp four words, so
// that a row's words leave as one whole 32-byte sector, and every column's
// values are read once by broadcast for 64 rows: with a lane per word instead
// (32 lanes reading 32 different columns for two rows) the shared-memory
// reads cost as much as the tests.  Labels are in time order, so a word after
// the row tile needs only the future cone.  The words are built from sign
// bits, funnel-shifted in one column at a time:
//   light cone: x_j - x_i - 1 < 0 for u or v (coordinates in [0, 2^31): no
//     overflow), one integer multiply-add each (x_j * 1 + ~x_i, the multiplier a runtime 1
//     that keeps it on the FMA pipe; compares and ORs held the integer pipe);
//   circle: |dtheta| - deta < 0, dtheta modulo 2^32 in [-2^31, 2^31) and
//     0 <= deta < 2^31: exact in 32 bits but where deta = 0 and |dtheta| = 2^31,
//     so a word whose first column has the row's eta is found exactly;
//   2+1, 3+1: the FP32 filter, two columns per packed operation, four
//     instructions per test where differences and squares took ten; a word
//     with a value near the cone is found exactly.
// The integer tests' own word of the row tile (it holds the diagonal and both
// cones) is found exactly; the filter is symmetric and takes it too.
// kWords: words per warp (4), or 1 for a set whose chunks leave SMs idle; the
// block then covers 8 words (w0 a multiple of 8).
template <int G, int kWords = kRelWarpWords>
__device__ __forceinline__ void relate_block(const int32_t* __restrict__ coords, int64_t n,
                                             uint64_t* __restrict__ bits, int64_t row_words, int64_t rb, int64_t w0,
                                             uint8_t* smem, int64_t zero_from = -1) {
    constexpr int D = geom_dim(G);
    constexpr bool kFilter = G == kGeom3 || G == kGeom4;
    constexpr int kBlockWords = kWords * (kRelThreads / 32);
    if (w0 + kBlockWords <= rb) return;  // wholly below the diagonal
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t V = (n + 63) >> 6;  // valid words
    const int64_t c0 = w0 * 64, r0 = rb * kRelRowsPerBlock;
    const int64_t wfirst = rb > w0 ? rb : w0;  // first word tested here
    int32_t* one_s = reinterpret_cast<int32_t*>(smem + relate_stage_bytes(G) - 16);

    // ---- stage the columns, two per thread and step
    const int first = int(wfirst - w0) * 32;  // in column pairs
    bool fast = true;
    if constexpr (kFilter) {
        int out = 0;
        ulonglong2* q0 = reinterpret_cast<ulonglong2*>(smem);      // (t, t), (x, x)
        ulonglong2* q1 = q0 + kRelColsPerBlock / 2;                // (y, y), (z, z); 2+1: (y, y), (A, A)
        uint64_t* q2 = reinterpret_cast<uint64_t*>(q1 + kRelColsPerBlock / 2);  // 3+1: (A, A)
        for (int p = first + threadIdx.x; p < 32 * kBlockWords; p += kRelThreads) {
            int32_t c[2][D];
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    const int64_t j = c0 + 2 * p + k;
                    c[k][d] = j < n ? coords[d * n + j] : 0;
                    out |= c[k][d] < -kFilterRange || c[k][d] > kFilterRange;
                }
            auto pair = [&](int d) { return f2_pack(float(c[0][d]), float(c[1][d])); };
            const uint64_t A = f2_pack(filter_norm<D>(c[0]) + kFilterSlack, filter_norm<D>(c[1]) + kFilterSlack);
            q0[p] = make_ulonglong2(pair(0), pair(1));
            if constexpr (G == kGeom4) {
                q1[p] = make_ulonglong2(pair(2), pair(3));
                q2[p] = A;
            } else {
                q1[p] = make_ulonglong2(pair(2), A);
            }
        }
        if (threadIdx.x < 64 && r0 + threadIdx.x < n) {
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const int32_t x = coords[d * n + r0 + threadIdx.x];
                out |= x < -kFilterRange || x > kFilterRange;
            }
        }
        fast = !__syncthreads_or(out);
    } else {
        for (int p = first + threadIdx.x; p < 32 * kBlockWords; p += kRelThreads) {
            int32_t c[2][2];
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    const int64_t j = c0 + 2 * p + k;
                    c[k][d] = j < n ? coords[d * n + j] : 0;
                }
            reinterpret_cast<int4*>(smem)[p] = make_int4(c[0][0], c[0][1], c[1][0], c[1][1]);
        }
        if (threadIdx.x == 0) *one_s = 1;
        __syncthreads();
    }

    int32_t one = 1;
    if constexpr (!kFilter) one = *one_s;
    // ---- this lane's two rows
    RelRow<G> row[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int64_t i = r0 + lane + 32 * r;
        int32_t c[D];
#pragma unroll
        for (int d = 0; d < D; ++d) c[d] = i < n ? coords[d * n + i] : 0;
        if constexpr (kFilter) {
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const float k = (d == 0 ? 2.0f : -2.0f) * float(c[d]);
                row[r].k[d] = f2_pack(k, k);
            }
            const float b = filter_norm<D>(c);
            row[r].b = f2_pack(b, b);
        } else if constexpr (G == kGeomDeSitter) {
            row[r].nu = c[0];
            row[r].nv = int32_t(0u - uint32_t(c[1]));
        } else {
            row[r].nu = ~c[0];
            row[r].nv = ~c[1];
        }
    }
    const int64_t wb = w0 + kWords * warp;  // this warp's first word
    if (wb + kWords > rb && wb < row_words) {  // warp-uniform: some word at or after the row tile
        // [word][row]; the words shift down as they are found, so that the loop
        // is one copy of the tests (unrolled, the instruction cache missed)
        uint64_t word[kWords][2] = {};
#pragma unroll 1
        for (int k = 0; k < kWords; ++k) {
            const int64_t W = wb + k;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
#pragma unroll
                for (int x = 0; x + 1 < kWords; ++x) word[x][r] = word[x + 1][r];
                word[kWords - 1][r] = 0ull;
            }
            uint64_t (&found)[2] = word[kWords - 1];
            if (W < rb || W >= V) continue;  // warp-uniform
            // rows to find exactly: the own word of the integer tests, coordinates beyond the
            // filter's range, and below the rows whose tests could not decide
            bool exact[2] = {W == rb || !fast, W == rb || !fast};
            if (kFilter ? fast : W != rb) {
                const int pbase = int(W - w0) * 32;
                uint32_t acc[2][2], band[2];
                if (kFilter && W == rb)
                    relate_word<G, true>(smem, pbase, row, one, acc, band);
                else
                    relate_word<G, false>(smem, pbase, row, one, acc, band);
                const int64_t left = n - 64 * W;
                const uint64_t valid = left >= 64 ? ~0ull : (1ull << left) - 1ull;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    uint64_t x = (uint64_t(acc[r][1]) << 32) | acc[r][0];
                    if constexpr (G == kGeomLightCone) x = ~x;  // sign set: not in the future cone
                    found[r] = x & valid;
                    if constexpr (kFilter) exact[r] = band[r] <= kBandBits;
                    if constexpr (G == kGeomDeSitter) exact[r] = row[r].nu == coords[64 * W];
                }
            }
            const uint32_t todo0 = __ballot_sync(0xffffffffu, exact[0] && r0 + lane < n);
            const uint32_t todo1 = __ballot_sync(0xffffffffu, exact[1] && r0 + lane + 32 < n);
            if (todo0 | todo1) {  // warp-uniform
                const ExactWord<G> ex(coords, n, W);
                if ((!kFilter && W == rb) || !fast) {  // every row: their loads overlap
#pragma unroll 4
                    for (int q = 0; q < 32; ++q) {
                        const uint64_t y0 = ex.row(coords, n, r0 + q < n ? r0 + q : n - 1);
                        const uint64_t y1 = ex.row(coords, n, r0 + 32 + q < n ? r0 + 32 + q : n - 1);
                        if (lane == q) {
                            found[0] = y0;
                            found[1] = y1;
                        }
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < 2; ++r)
                        for (uint32_t todo = r == 0 ? todo0 : todo1; todo; todo &= todo - 1u) {
                            const int q = __ffs(int(todo)) - 1;
                            const uint64_t y = ex.row(coords, n, r0 + 32 * r + q);
                            if (lane == q) found[r] = y;
                        }
                }
            }
        }
        // a row's four words as one 32-byte store; words before the row tile are mirror_block's
        const bool whole = kWords == kRelWarpWords && wb >= rb && (reinterpret_cast<uintptr_t>(bits) & 31) == 0;  // warp-uniform
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int64_t i = r0 + lane + 32 * r;
            if (i >= n) continue;
            uint64_t* dst = bits + i * row_words + wb;
            if (whole) {
                asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(dst), "l"(word[0][r]),
                             "l"(word[1 % kWords][r]), "l"(word[2 % kWords][r]), "l"(word[3 % kWords][r])
                             : "memory");
            } else {
#pragma unroll
                for (int k = 0; k < kWords; ++k)
                    if (wb + k >= rb) dst[k] = word[k][r];
            }
        }
    }
    if (zero_from >= 0 && zero_from < row_words)
        for (int64_t i = r0 + warp; i < r0 + 64 && i < n; i += kRelThreads / 32)
            for (int64_t w = zero_from + lane; w < row_words; w += 32) bits[i * row_words + w] = 0ull;
}

// ------------------------------------------- light-cone kinds, a lane per word
//
// Labels are in time order, so in a word wholly after the row tile only the
// future cone can hold (u_j > u_i and v_j > v_i); for a random 2D order labelled
// by u the u test is implied by j > i and only v is compared (kUseU = false).
// Each lane owns one word (64 columns) of the block's 32 and tests its columns one by one, for
// four rows at a time, with no ballots: one or two multiply-adds per test as above, an OR with u,
// and a funnel shift that appends the sign bit to the half-word's
// accumulator (the complement of the relation bits).
// The column coordinates are staged transposed, st[c][w] = column 64 w + c
// (row pitch kConePitch: the lanes' reads of one offset c hit consecutive
// banks); columns at or beyond n are staged as 0, which no cone test
// passes.  The row tile's own word (lane rb - w0) takes the full symmetric test
// by ballots in all eight warps; words before the row tile are left to mirror_block.
constexpr int kConePitch = kRelWordsPerBlock + 1;  // staged words per column offset
constexpr int kConeRows = 4;                       // rows a lane tests together
constexpr int kConeOne = 2 * 64 * kConePitch;      // after the (u, v) staging: a runtime 1 (the multiplier)
constexpr int kConeInts = kConeOne + 1;

// The 64 rows from r0 of one block whose columns are staged in st; ws: the own word, < 0: none.
template <bool kUseU>
__device__ __forceinline__ void relate_rows_cone(const int32_t* __restrict__ coords, int64_t n,
                                                 uint64_t* __restrict__ bits, int64_t row_words, int64_t w0,
                                                 int64_t r0, int64_t r1, int ws, const int32_t* __restrict__ st) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kWarps = kRelThreads / 32;
    const int2* st2 = reinterpret_cast<const int2*>(st);  // kUseU: (u, v) pairs
    const int wbeg = ws > 0 ? ws : 0;
    const int32_t one = st[kConeOne];
    for (int64_t ib = r0 + int64_t(warp) * kConeRows; ib < r1; ib += int64_t(kWarps) * kConeRows) {
        int32_t ru[kConeRows], rv[kConeRows], nu[kConeRows], nv[kConeRows];
        uint32_t lo[kConeRows], hi[kConeRows];
#pragma unroll
        for (int r = 0; r < kConeRows; ++r) {
            const int64_t i = ib + r;
            ru[r] = i < r1 ? coords[i] : INT32_MAX;  // a missing row passes no test
            rv[r] = i < r1 ? coords[n + i] : INT32_MAX;
            nu[r] = ~ru[r];  // -x_i - 1
            nv[r] = ~rv[r];
            lo[r] = hi[r] = 0u;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // the word's low and high halves
            // highest column first: after 32 shifts column 32 h is bit 0
#pragma unroll 8
            for (int c = 32 * h + 31; c >= 32 * h; --c) {
                int32_t xu = 0, xv;
                if constexpr (kUseU) {
                    const int2 x = st2[c * kConePitch + lane];
                    xu = x.x;
                    xv = x.y;
                } else {
                    xv = st[c * kConePitch + lane];
                }
#pragma unroll
                for (int r = 0; r < kConeRows; ++r) {
                    // sign bit set iff the column is not in the future cone
                    const int32_t d = kUseU ? (cone_mad(xu, one, nu[r]) | cone_mad(xv, one, nv[r]))
                                            : cone_mad(xv, one, nv[r]);
                    if (h == 0)
                        lo[r] = __funnelshift_l(uint32_t(d), lo[r], 1);
                    else
                        hi[r] = __funnelshift_l(uint32_t(d), hi[r], 1);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < kConeRows; ++r) {
            const int64_t i = ib + r;
            if (i >= r1) break;  // warp-uniform
            uint64_t word = ~((uint64_t(hi[r]) << 32) | lo[r]);
            if (ws >= 0) {  // the row tile's own word: full test (warp-uniform)
                bool b[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = lane + 32 * h;  // column offset in the word
                    const int64_t j = (w0 + ws) * 64 + k;
                    if constexpr (kUseU) {
                        const int2 x = st2[k * kConePitch + ws];
                        const int32_t du = x.x - ru[r], dv = x.y - rv[r];
                        b[h] = j < n && (du ^ dv) >= 0 && du != 0 && dv != 0;
                    } else {  // u increases with the label
                        const int32_t xv = st[k * kConePitch + ws];
                        b[h] = j < n && (j > i ? xv > rv[r] : (j < i && xv < rv[r]));
                    }
                }
                const uint64_t d = (uint64_t(__ballot_sync(0xffffffffu, b[1])) << 32) | __ballot_sync(0xffffffffu, b[0]);
                if (lane == ws) word = d;
            }
            if (lane >= wbeg && w0 + lane < row_words) bits[i * row_words + w0 + lane] = word;
        }
    }
}

// Rows [64 rb, 64 rb + 64) x words [w0, w0 + 32), w0 a multiple of 32.  order2d: only v is
// staged and tested.  st: kConeInts ints, 16-byte aligned (no __restrict__: the threads
// read one another's columns).  All 256 threads.
__device__ __forceinline__ void relate_block_cone(const int32_t* __restrict__ coords, int64_t n,
                                                  uint64_t* __restrict__ bits, int64_t row_words, int64_t rb,
                                                  int64_t w0, int32_t* st, bool order2d) {
    if (w0 + kRelWordsPerBlock <= rb) return;  // wholly below the diagonal
    const int ws = rb < w0 ? -1 : int(rb - w0);
    const int wbeg = ws > 0 ? ws : 0;
    const int64_t c0 = w0 * 64, r0 = rb * kRelRowsPerBlock;
    const int64_t r1 = r0 + kRelRowsPerBlock < n ? r0 + kRelRowsPerBlock : n;
    for (int t = threadIdx.x + 64 * wbeg; t < kRelColsPerBlock; t += kRelThreads) {
        const int64_t col = c0 + t;
        const int at = (t & 63) * kConePitch + (t >> 6);
        if (order2d)
            st[at] = col < n ? coords[n + col] : 0;
        else
            reinterpret_cast<int2*>(st)[at] = col < n ? make_int2(coords[col], coords[n + col]) : make_int2(0, 0);
    }
    if (threadIdx.x == 0) st[kConeOne] = 1;
    __syncthreads();
    if (order2d)
        relate_rows_cone<false>(coords, n, bits, row_words, w0, r0, r1, ws, st);
    else
        relate_rows_cone<true>(coords, n, bits, row_words, w0, r0, r1, ws, st);
}

// ------------------------------------------------ light-cone column tables
//
// In the light-cone kinds a row i and a column tile C wholly after i's row
// tile relate exactly where u_j > u_i and v_j > v_i (the future cone; labels
// are in time order).  Sorting the tile's 64 values of one coordinate turns
// "the columns whose value exceeds y" into a suffix of the sorted order, so
// with the suffix masks precomputed the whole 64-bit word is
//   above_u[#{p : us[p] <= u_i}] & above_v[#{p : vs[p] <= v_i}],
// two binary searches of six steps instead of 64 tests (for a random 2D
// order, whose u increases with the label, the v term alone).  Columns at or
// beyond n hold -1, which exceeds no coordinate (all lie in [0, 2^31)).
struct alignas(16) ConeTable {
    int32_t xs[2][64];      // u and v of the tile's columns, each sorted ascending
    uint64_t above[2][66];  // above[x][m], m <= 64: the columns at sorted positions >= m of coordinate x
    uint32_t pad[4];        // 1584 bytes: consecutive tables start at different 16-byte offsets of
};                          // a 128-byte line, so the lanes' bucket loads spread over the banks
static_assert(sizeof(ConeTable) == 1584, "cone table layout");

// Table of column tile C, one full warp.  The 64 keys (value + 1) << 6 |
// column, two per lane (element lane + 32 h), go through a bitonic network
// (partners at distance 32 inside the lane, the others by shuffles); after
// it element e is the e-th smallest, and a suffix OR over the elements gives
// the masks.  order2d: only the v table (its u is the label order).
__device__ __forceinline__ void build_cone_table(const int32_t* __restrict__ coords, int64_t n, int64_t C,
                                                 bool order2d, ConeTable* __restrict__ t) {
    const int lane = threadIdx.x & 31;
    for (int x = order2d ? 1 : 0; x < 2; ++x) {
        uint64_t k[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t col = 64 * C + lane + 32 * h;
            const int32_t v = col < n ? coords[x * n + col] : -1;
            k[h] = (uint64_t(uint32_t(v + 1)) << 6) | uint64_t(lane + 32 * h);
        }
#pragma unroll
        for (int size = 2; size <= 64; size <<= 1) {
#pragma unroll
            for (int j = size >> 1; j > 0; j >>= 1) {
                if (j == 32) {  // size 64: ascending, partner e + 32 in the same lane
                    const uint64_t lo = k[0] < k[1] ? k[0] : k[1], hi = k[0] < k[1] ? k[1] : k[0];
                    k[0] = lo;
                    k[1] = hi;
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int e = lane + 32 * h;
                        const uint64_t p = __shfl_xor_sync(0xffffffffu, k[h], j);
                        const bool keep_min = ((e & j) == 0) == ((e & size) == 0);
                        k[h] = keep_min ? (k[h] < p ? k[h] : p) : (k[h] < p ? p : k[h]);
                    }
                }
            }
        }
        t->xs[x][lane] = int32_t(uint32_t(k[0] >> 6)) - 1;
        t->xs[x][lane + 32] = int32_t(uint32_t(k[1] >> 6)) - 1;
        uint64_t s0 = 1ull << (k[0] & 63), s1 = 1ull << (k[1] & 63);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t a = __shfl_down_sync(0xffffffffu, s0, o), b = __shfl_down_sync(0xffffffffu, s1, o);
            if (lane + o < 32) {
                s0 |= a;
                s1 |= b;
            }
        }
        s0 |= __shfl_sync(0xffffffffu, s1, 0);  // every element of the upper half follows the lower half
        t->above[x][lane] = s0;
        t->above[x][lane + 32] = s1;
        if (lane == 0) t->above[x][64] = 0ull;
    }
}

// #{m < 7 : s[m] <= y} for ascending s, by binary lifting with selects
// (steps of 4, 2, 1): three compares instead of seven.
__device__ __forceinline__ int cone_lift7(int32_t s0, int32_t s1, int32_t s2, int32_t s3, int32_t s4, int32_t s5,
                                          int32_t s6, int32_t y) {
    const bool a = s3 <= y;
    const bool b = (a ? s5 : s1) <= y;
    const bool d = (a ? (b ? s6 : s4) : (b ? s2 : s0)) <= y;
    return (a ? 4 : 0) + (b ? 2 : 0) + (d ? 1 : 0);
}

// #{p : xs[p] <= y} over 64 ascending values, and the mask of the columns
// above y.  s[m] = xs[8 m + 7] (m < 7) are the bucket splitters, kept in
// registers: they give the buckets wholly at or below y, then the one
// 32-byte bucket that may straddle y is loaded and counted the same way.
__device__ __forceinline__ uint64_t cone_above(const int32_t* __restrict__ xs, const uint64_t* __restrict__ above,
                                               const int32_t (&s)[7], int32_t y) {
    const int c1 = cone_lift7(s[0], s[1], s[2], s[3], s[4], s[5], s[6], y);
    const int4 a = reinterpret_cast<const int4*>(xs)[2 * c1], b = reinterpret_cast<const int4*>(xs)[2 * c1 + 1];
    const int c = 8 * c1 + cone_lift7(a.x, a.y, a.z, a.w, b.x, b.y, b.z, y) + (b.w <= y ? 1 : 0);
    return above[c];
}

// Bytes of dynamic shared memory of relate_block_tables: 32 tables, the own
// tile's columns, the copy's mbarrier.
constexpr int kConeTableSmem = kRelWordsPerBlock * int(sizeof(ConeTable)) + 128 * 4 + 16;

// Rows [64 rb, 64 rb + 64) x words [w0, w0 + 32) (less the words before rb) of
// a light-cone set from its column tables (tables[C] for column tile C): the row tile's
// own word rb by the exact symmetric test folded with ballots, every word
// after it by the table look-ups, words at or past the last valid one zeroed
// (and, with zero_from >= 0, the row's words [zero_from, row_words)).  The
// block's tables arrive by one bulk copy.  smem: kConeTableSmem bytes,
// 16-byte aligned.  All 256 threads.  Returns false (status recorded) if the
// copy did not complete in time.
__device__ __forceinline__ bool relate_block_tables(const int32_t* __restrict__ coords, int64_t n,
                                                    uint64_t* __restrict__ bits, int64_t row_words, int64_t rb,
                                                    int64_t w0, const ConeTable* __restrict__ tables, uint8_t* smem,
                                                    bool order2d, int64_t zero_from, WsHeader* hdr) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kWarps = kRelThreads / 32;
    ConeTable* st = reinterpret_cast<ConeTable*>(smem);
    // u, v of the row tile's elements: the rows here, and the columns of the own word
    int32_t* own = reinterpret_cast<int32_t*>(smem + kRelWordsPerBlock * sizeof(ConeTable));
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + kRelWordsPerBlock * sizeof(ConeTable) + 128 * 4);
    const int64_t V = (n + 63) >> 6;
    const int64_t r0 = rb * 64, r1 = r0 + 64 < n ? r0 + 64 : n;
    const int64_t wt = w0 > rb ? w0 : rb + 1;                                      // first table word
    const int64_t we = w0 + kRelWordsPerBlock < V ? w0 + kRelWordsPerBlock : V;  // end of the valid words
    const int nt = wt < we ? int(we - wt) : 0;
    const bool has_own = rb >= w0;
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t bytes = uint32_t(nt) * uint32_t(sizeof(ConeTable));
        mbar_arrive_expect_tx(bar, bytes);
        if (bytes) bulk_load(st, tables + wt, bytes, bar);
    }
    if (threadIdx.x < 128) {
        const int64_t e = r0 + (threadIdx.x & 63);
        own[threadIdx.x] = e < n ? coords[(threadIdx.x >> 6) * n + e] : 0;
    }
    __syncthreads();
    if (has_own) {
        for (int64_t i = r0 + warp; i < r1; i += kWarps) {
            const int32_t ui = own[i - r0], vi = own[64 + (i - r0)];
            bool b[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = lane + 32 * h;
                const int64_t j = r0 + k;
                const int32_t du = own[k] - ui, dv = own[64 + k] - vi;
                b[h] = j < n && (order2d ? (j > i ? dv > 0 : (j < i && dv < 0))
                                         : ((du ^ dv) >= 0 && du != 0 && dv != 0));
            }
            const uint64_t d = (uint64_t(__ballot_sync(0xffffffffu, b[1])) << 32) | __ballot_sync(0xffffffffu, b[0]);
            if (lane == 0) bits[i * row_words + rb] = d;
        }
    }
    if (!mbar_wait_bounded(bar, 0, hdr)) {
        mbar_wait_bounded(bar, 0, hdr);  // the copy may still be writing: wait once more before leaving
        return false;
    }
    // lane l: word w0 + l of each of the warp's rows, 32 consecutive words per row and warp
    const int64_t w = w0 + lane;
    const bool tab = w >= wt && w < we;
    if (tab || (w >= V && w < row_words)) {
        const ConeTable& T = st[tab ? int(w - wt) : 0];
        int32_t su[7], sv[7];
#pragma unroll
        for (int m = 0; m < 7; ++m) {
            sv[m] = tab ? T.xs[1][8 * m + 7] : 0;
            su[m] = tab && !order2d ? T.xs[0][8 * m + 7] : 0;
        }
#pragma unroll 2
        for (int64_t i = r0 + warp; i < r1; i += kWarps) {
            uint64_t word = 0ull;
            if (tab) {
                word = cone_above(T.xs[1], T.above[1], sv, own[64 + (i - r0)]);
                if (!order2d) word &= cone_above(T.xs[0], T.above[0], su, own[i - r0]);
            }
            bits[i * row_words + w] = word;
        }
    }
    if (zero_from >= 0)
        for (int64_t i = r0 + warp; i < r1; i += kWarps)
            for (int64_t z = zero_from + lane; z < row_words; z += 32) bits[i * row_words + z] = 0ull;
    return true;
}

// ------------------------------------------------ the lower part by symmetry
//
// A 64 x 64 tile wholly below the diagonal (row tile A, word B < A) is the
// transpose of tile (B, A) above it.  mirror_block fills one super-tile of
// 512 output rows x 8 output words (8 x 8 tiles): the 512 source rows x 8
// source words land in shared memory with 64-byte reads, each warp
// transposes its output row tile's 8 tiles in registers (six butterfly
// stages, five of them across lanes) and writes its row tile's words
// below the diagonal back through shared memory, 64 contiguous bytes per
// output row off the diagonal super-tiles, four lanes to a row.
constexpr int kMirTiles = 8;                    // tiles per super-tile side
constexpr int kMirRows = 64 * kMirTiles;        // 512 source / output rows

// Transposes of bit tiles held one row per lane (bit c = column c).  Stage
// j of the recursive block swap exchanges, between lanes l and l ^ j, the
// j-bit groups that lie off the diagonal: the lane with (l & j) == 0 keeps
// its low groups and takes its partner's low groups into its high ones, the
// other keeps its high groups and takes its partner's high groups into its
// low ones.  Per lane constants make every stage lane-uniform: for j = 16
// and 8 a byte permute of the lane's word and its partner's; for j = 4, 2, 1
// each lane sends its word rotated toward its partner's positions (right by
// j, or by 32 - j, i.e. left by j) and masked to the groups the partner
// takes, and keeps (own & mask) | received.
struct Tr32 {
    uint32_t s16, s8;       // byte-permute selectors
    uint32_t r[3], m[3];    // rotations and kept masks for j = 4, 2, 1
};
__device__ __forceinline__ Tr32 tr32_consts(int lane) {
    Tr32 c;
    c.s16 = (lane & 16) ? 0x3276u : 0x5410u;  // high: partner's bytes 2,3 then own 2,3; low: own 0,1 then partner's 0,1
    c.s8 = (lane & 8) ? 0x3715u : 0x6240u;    // high: p1 v1 p3 v3; low: v0 p0 v2 p2
    const uint32_t mk[3] = {0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int j = 4 >> s;
        const bool high = (lane & j) != 0;
        c.r[s] = high ? uint32_t(32 - j) : uint32_t(j);
        c.m[s] = high ? ~mk[s] : mk[s];
    }
    return c;
}
__device__ __forceinline__ uint32_t transpose32(uint32_t v, const Tr32& c) {
    v = __byte_perm(v, __shfl_xor_sync(0xffffffffu, v, 16), c.s16);
    v = __byte_perm(v, __shfl_xor_sync(0xffffffffu, v, 8), c.s8);
#pragma unroll
    for (int s = 0; s < 3; ++s)
        v = (v & c.m[s]) | __shfl_xor_sync(0xffffffffu, __funnelshift_r(v, v, c.r[s]) & c.m[s], 4 >> s);
    return v;
}

// Transpose the 64 x 64 bit tile whose rows l and l + 32 lane l holds: the
// stage j = 32 inside the lane (x's high half with y's low half), then the
// four 32 x 32 quarters independently.
__device__ __forceinline__ void transpose64(uint64_t& x, uint64_t& y, const Tr32& c) {
    const uint64_t t = ((x >> 32) ^ y) & 0x00000000FFFFFFFFull;
    y ^= t;
    x ^= t << 32;
    x = uint64_t(transpose32(uint32_t(x), c)) | (uint64_t(transpose32(uint32_t(x >> 32), c)) << 32);
    y = uint64_t(transpose32(uint32_t(y), c)) | (uint64_t(transpose32(uint32_t(y >> 32), c)) << 32);
}

// Super-tile (A8, B8): output rows [512 A8, 512 A8 + 512), output words
// [8 B8, 8 B8 + 8).  sm: 512 x 9 words of shared memory.  All 256 threads.
__device__ __forceinline__ void mirror_block(uint64_t* bits, int64_t n, int64_t row_words, int64_t A8,
                                             int64_t B8, uint64_t (*sm)[kMirTiles + 1]) {
    const int64_t tiles = (n + 63) >> 6;  // row tiles = valid words
    const int64_t A0 = A8 * kMirTiles, B0 = B8 * kMirTiles;
    // anything to do here? (uniform: some tile with B < A < tiles)
    if (A0 >= tiles || B0 >= (A0 + kMirTiles - 1 < tiles ? A0 + kMirTiles - 1 : tiles - 1)) return;
    // source rows 64 B0 .. + 512, source words A0 .. A0 + 8, as 16-byte word
    // pairs (A0 is even and rows are 16-word multiples), every load of a
    // thread issued before the first shared-memory store: with one load in
    // flight per thread the kernel waited on memory latency at a quarter of
    // the HBM rate.  The second word of a pair at the last valid word is a
    // padding word of the row (loaded, then replaced by 0).
    constexpr int kPairs = kMirRows * kMirTiles / 2, kPerThread = kPairs / kRelThreads;
    static_assert(kPairs % kRelThreads == 0 && kMirTiles % 2 == 0, "word pairs split evenly over the block");
    ulonglong2 v[kPerThread];
#pragma unroll
    for (int s = 0; s < kPerThread; ++s) {
        const int t = threadIdx.x + s * kRelThreads;
        const int64_t row = 64 * B0 + t / (kMirTiles / 2), word = A0 + 2 * (t % (kMirTiles / 2));
        v[s] = (row < n && word < tiles) ? __ldcg(reinterpret_cast<const ulonglong2*>(bits + row * row_words + word))
                                         : make_ulonglong2(0ull, 0ull);
    }
#pragma unroll
    for (int s = 0; s < kPerThread; ++s) {
        const int t = threadIdx.x + s * kRelThreads;
        const int r = t / (kMirTiles / 2), w = 2 * (t % (kMirTiles / 2));
        sm[r][w] = v[s].x;
        sm[r][w + 1] = A0 + w + 1 < tiles ? v[s].y : 0ull;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t A = A0 + warp;  // this warp's output row tile
    const bool active = A < tiles && B0 < A;  // warp-uniform
    uint64_t ox[kMirTiles], oy[kMirTiles];
    if (active) {
        const Tr32 tc = tr32_consts(lane);
#pragma unroll
        for (int qb = 0; qb < kMirTiles; ++qb) {
            uint64_t x = sm[64 * qb + lane][warp], y = sm[64 * qb + lane + 32][warp];
            transpose64(x, y, tc);
            ox[qb] = x;
            oy[qb] = y;
        }
    }
    __syncthreads();  // every warp has read its column of the source words
    if (active) {
        // The warp's 64 output rows go through its own 64 rows of shared
        // memory, then out with four lanes per row (16 bytes each): every
        // row's 64 bytes leave as two whole 32-byte sectors.  Words B0 + w
        // < A only (all inside the row: B < A < tiles).
        uint64_t (*out)[kMirTiles + 1] = sm + 64 * warp;
#pragma unroll
        for (int qb = 0; qb < kMirTiles; ++qb) {
            out[lane][qb] = ox[qb];
            out[lane + 32][qb] = oy[qb];
        }
        __syncwarp();
        const int w = 2 * (lane & 3);  // this lane's word pair
        static_assert(kMirTiles == 8, "four lanes cover a row's eight words");
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int r = 8 * s + (lane >> 2);
            const int64_t row = 64 * A + r;
            if (row < n && B0 + w < A) {
                uint64_t* dst = bits + row * row_words + B0 + w;
                if (B0 + w + 1 < A)
                    *reinterpret_cast<ulonglong2*>(dst) = make_ulonglong2(out[r][w], out[r][w + 1]);
                else
                    *dst = out[r][w];
            }
        }
    }
}

}  // namespace cs
