// cs_chains.cu -- longest chains and greedy maximal antichains on the bitset
// (Section "Set Partitions": Algorithms "Maximal Chain Length" and "Maximal
// Antichain").
//
// Longest chain.  The thesis recurses through the Alexandroff set, caching
// the distance of each element to the top.  On the GPU the same length comes
// from peeling: the set S (A_ij for a pair, every element for the whole set)
// loses all its minimal elements -- those with no predecessor left in S --
// once per round; the number of rounds is the number of elements of the
// longest chain in S.  Each element remembers the word of its row that last
// held a predecessor in S: S only shrinks, so the words nearer than it stay
// empty, and over all rounds a row is scanned once.
//
// Greedy antichain.  Each round takes the candidate j with the largest c_j =
// |A - J(j)|, the smallest label on ties, as in the algorithm's scan, and
// removes J(k) from A and J(k) + {k} from the candidates.  Maximising c_j is
// minimising the overlap o_j = |A & J(j)|; the candidates removed in a round
// are what every other overlap loses.
//
// Both run all their rounds in one cooperative launch, one CTA per SM, each
// with its own copy of the set (S, or the candidates) in shared memory, so
// that a round takes one bounded grid barrier; where a cooperative launch is
// not available they fall back to batches of kBatch launches between host
// checks of the number of elements left (rounds after the last one find
// nothing to do).
#include "cs_kernels.cuh"
#include "cs_relate.cuh"

namespace cs {

namespace {

constexpr int kBatch = 32;

struct ChainState {
    unsigned long long best;  // antichain: packed (c, ~label) of the best candidate
    int32_t found;            // chain: this round removed something
    int32_t related;          // chain: i precedes j
    int64_t rounds;           // rounds that removed something; -1 until known
    int64_t left;             // elements left in S (chain) or candidates left (antichain)
    // persistent (cooperative) kernels
    unsigned int arrived;         // grid barrier: blocks that arrived, all rounds together
    int32_t status;               // the kernel's cs_status
    unsigned long long best3[3];  // antichain: smallest (overlap, label) of a round, rounds in turn
};

struct ChainLayout {
    size_t state, s, m, total;
};

ChainLayout chain_layout(int64_t row_words) {
    ChainLayout L;
    size_t off = sizeof(WsHeader);
    L.state = off;
    off = align_up(off + sizeof(ChainState), 256);
    L.s = off;
    off = align_up(off + size_t(row_words) * 8, 256);
    L.m = off;  // chain: the elements removed in a round, three rounds in turn
    off = align_up(off + 3 * size_t(row_words) * 8, 256);
    L.total = off;
    return L;
}

// The workspace header stands before the state.
__device__ __forceinline__ WsHeader* header_of(ChainState* st) {
    return reinterpret_cast<WsHeader*>(reinterpret_cast<uint8_t*>(st) - sizeof(WsHeader));
}

__device__ __forceinline__ bool bit_of(const uint64_t* row, int64_t k) { return (row[k >> 6] >> (k & 63)) & 1ull; }

// Bits of word w strictly between columns lo and hi (lo < col < hi).
__device__ __forceinline__ uint64_t between_mask(int64_t w, int64_t lo, int64_t hi) {
    const int64_t c0 = 64 * w;
    uint64_t m = ~0ull;
    if (lo + 1 > c0) m = lo + 1 - c0 >= 64 ? 0ull : m & (~0ull << (lo + 1 - c0));
    if (hi < c0 + 64) m = hi <= c0 ? 0ull : m & (~0ull >> (c0 + 64 - hi));
    return m;
}

__device__ __forceinline__ int warp_or(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// S = A_ij (bits strictly between i and j set in both rows), or all of [0, n).
__global__ void k_chain_init(const uint64_t* __restrict__ bits, int64_t n, int64_t row_words, int64_t i, int64_t j,
                             uint64_t* __restrict__ S, uint64_t* __restrict__ M, ChainState* st) {
    const bool whole = i < 0;
    const int64_t lo = whole ? -1 : i, hi = whole ? n : j;
    for (int64_t w = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; w < row_words;
         w += int64_t(gridDim.x) * blockDim.x) {
        uint64_t x = between_mask(w, lo, hi);
        if (!whole) x &= __ldg(bits + i * row_words + w) & __ldg(bits + j * row_words + w);
        S[w] = x;
        M[w] = 0ull;
        M[row_words + w] = 0ull;
        M[2 * row_words + w] = 0ull;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->found = 0;
        st->arrived = 0u;
        st->status = 0;
        header_of(st)->status = 0;
        st->rounds = 0;
        st->related = whole ? 1 : int(bit_of(bits + i * row_words, j));
        st->left = 1;
    }
}

// One peeling round: the elements of S with no predecessor in S go to M.
__global__ void __launch_bounds__(256) k_chain_peel(const uint64_t* __restrict__ bits, int64_t row_words,
                                                    int64_t lo, int64_t hi, const uint64_t* __restrict__ S,
                                                    uint64_t* __restrict__ M, ChainState* st) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    const int64_t wlo = lo < 0 ? 0 : lo >> 6;
    for (int64_t k = lo + 1 + int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); k < hi; k += warps) {
        if (!bit_of(S, k)) continue;  // warp-uniform
        const int64_t wk = k >> 6;
        int any = 0;
        for (int64_t w = wlo + lane; w <= wk && !any; w += 32) {
            uint64_t x = __ldg(bits + k * row_words + w) & S[w];
            if (w == wk) x &= (k & 63) ? ((1ull << (k & 63)) - 1ull) : 0ull;  // predecessors only
            any = x != 0ull;
        }
        if (!warp_or(any) && lane == 0) {
            atomicOr(reinterpret_cast<unsigned long long*>(M + wk), 1ull << (k & 63));
            st->found = 1;
        }
    }
}

// Close a round: S -= M, count it if it removed anything, count what is left.
__global__ void __launch_bounds__(1024) k_chain_apply(int64_t row_words, uint64_t* __restrict__ S,
                                                      uint64_t* __restrict__ M, ChainState* st) {
    __shared__ unsigned long long left;
    __shared__ int found;
    if (threadIdx.x == 0) {
        left = 0;
        found = st->found;
    }
    __syncthreads();
    unsigned long long mine = 0;
    for (int64_t w = threadIdx.x; w < row_words; w += blockDim.x) {
        const uint64_t x = S[w] & ~M[w];
        S[w] = x;
        M[w] = 0ull;
        mine += __popcll(x);
    }
    atomicAdd(&left, mine);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (found) st->rounds += 1;
        st->found = 0;
        st->left = int64_t(left);
    }
}

// Antichain start: X = elements unrelated to the seed, A = X + {seed}.
__global__ void k_anti_init(const uint64_t* __restrict__ bits, int64_t n, int64_t row_words, int64_t seed,
                            uint64_t* __restrict__ A, uint64_t* __restrict__ X, ChainState* st) {
    for (int64_t w = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; w < row_words;
         w += int64_t(gridDim.x) * blockDim.x) {
        uint64_t x = ~__ldg(bits + seed * row_words + w) & between_mask(w, -1, n);
        if (w == (seed >> 6)) x &= ~(1ull << (seed & 63));
        X[w] = x;
        A[w] = w == (seed >> 6) ? x | (1ull << (seed & 63)) : x;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->best = 0ull;
        st->left = 1;
        st->arrived = 0u;
        st->status = 0;
        header_of(st)->status = 0;
        st->rounds = -1;
        for (int k = 0; k < 3; ++k) st->best3[k] = ~0ull;
    }
}

// Score every candidate j by |A - J(j)|; keep the best (largest, then first).
__global__ void __launch_bounds__(256) k_anti_score(const uint64_t* __restrict__ bits, int64_t n, int64_t row_words,
                                                    const uint64_t* __restrict__ A, const uint64_t* __restrict__ X,
                                                    ChainState* st) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (n + 63) >> 6;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    for (int64_t k = int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); k < n; k += warps) {
        if (!bit_of(X, k)) continue;  // warp-uniform
        int c = 0;
        for (int64_t w = lane; w < nw; w += 32) c += __popcll(A[w] & ~__ldg(bits + k * row_words + w));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (lane == 0)
            atomicMax(&st->best, (static_cast<unsigned long long>(c) << 32) | (0xFFFFFFFFull - uint64_t(k)));
    }
}

// Take the best candidate k: A -= J(k), X -= J(k) + {k}.
__global__ void __launch_bounds__(1024) k_anti_apply(const uint64_t* __restrict__ bits, int64_t row_words,
                                                     uint64_t* __restrict__ A, uint64_t* __restrict__ X,
                                                     ChainState* st) {
    __shared__ unsigned long long left;
    __shared__ unsigned long long best;
    if (threadIdx.x == 0) {
        left = 0;
        best = st->best;
    }
    __syncthreads();
    const bool take = best != 0ull;
    const int64_t k = int64_t(0xFFFFFFFFull - (best & 0xFFFFFFFFull));
    unsigned long long mine = 0;
    for (int64_t w = threadIdx.x; w < row_words; w += blockDim.x) {
        uint64_t x = X[w];
        if (take) {
            const uint64_t r = __ldg(bits + k * row_words + w);
            A[w] &= ~r;
            x &= ~r;
            if (w == (k >> 6)) x &= ~(1ull << (k & 63));
            X[w] = x;
        }
        mine += __popcll(x);
    }
    atomicAdd(&left, mine);
    __syncthreads();
    if (threadIdx.x == 0) {
        st->best = 0ull;
        st->left = int64_t(left);
    }
}

// Number of set bits of a bitset into st->rounds.
__global__ void __launch_bounds__(1024) k_count_bits(const uint64_t* __restrict__ A, int64_t row_words,
                                                     ChainState* st) {
    __shared__ unsigned long long total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    unsigned long long mine = 0;
    for (int64_t w = threadIdx.x; w < row_words; w += blockDim.x) mine += __popcll(A[w]);
    atomicAdd(&total, mine);
    __syncthreads();
    if (threadIdx.x == 0) st->rounds = int64_t(total);
}

// ------------------------------------------- persistent (cooperative) rounds
//
// With a cooperative launch every block is resident, so the rounds can run in
// one kernel separated by grid barriers instead of two launches per round.
// The barrier's wait is bounded: after 4 s it records CS_ETIMEOUT and the
// kernel returns (every later barrier of the other blocks then times out
// too), so a fault cannot hang the GPU.

constexpr int kPersistThreads = 1024;
constexpr int kPersistWarps = kPersistThreads / 32;

// Barrier number r (from 0) of all blocks: the blocks' writes before it are
// visible after it (read them with __ldcg).  One counter that only grows: no
// reset to wait for.
__device__ bool grid_barrier(ChainState* st, unsigned int r) {
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0 && gridDim.x > 1) {
        const unsigned int target = (r + 1) * gridDim.x;
        __threadfence();
        atomicAdd(&st->arrived, 1u);
        const unsigned long long t0 = global_timer_ns();
        for (unsigned int spin = 1;; ++spin) {
            unsigned int seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&st->arrived) : "memory");
            if (int(seen - target) >= 0) break;
            if ((spin & 63u) == 0u && global_timer_ns() - t0 > kWaitLimitNs) {
                atomicCAS(&st->status, 0, int(CS_ETIMEOUT));
                set_status(header_of(st), CS_ETIMEOUT);
                ok = 0;
                break;
            }
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

// All peeling rounds, one barrier each.  Element lo + 1 + e belongs to lane
// (e / warps) % 32 of warp e % warps (neighbours, which lose their
// predecessors together, to different SMs); slot t holds its 32 t-th on.
// Per slot the lane keeps the word w of its row that last met S, and that
// word's predecessor bits x.  A round: S minus the last round's removals in
// every block's shared copy; an element whose x no longer meets S has its
// row searched by the whole warp from w down, 64 words a step; one that finds
// nothing is minimal and enters this round's removals.  rounds = the number
// of rounds run until S is empty.
//
// Two barriers a round of 1216 small blocks, and every element's row scanned
// from its label down each round, took 20 us a round at n = 32768 (7.2 ms
// for the 355 of a 2D order); this takes 5.9 us.
constexpr int kWide = 8;
template <int kSlots>
__global__ void __launch_bounds__(kPersistThreads) k_chain_persist(const uint64_t* __restrict__ bits,
                                                                   int64_t row_words, int64_t lo, int64_t hi,
                                                                   int64_t max_rounds, const uint64_t* __restrict__ S0,
                                                                   uint64_t* M, ChainState* st) {
    extern __shared__ __align__(16) uint64_t S[];  // [row_words]
    if (!st->related) return;  // the same in every block
    const int lane = threadIdx.x & 31;
    const int64_t warps = int64_t(gridDim.x) * kPersistWarps;
    const int64_t gwarp = int64_t(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const int64_t wlo = lo < 0 ? 0 : lo >> 6, whi = hi > 0 ? (hi - 1) >> 6 : 0;  // words S may touch
    int any = 0;
    for (int64_t w = threadIdx.x; w < row_words; w += kPersistThreads) {
        S[w] = __ldg(S0 + w);
        any |= S[w] != 0ull;
    }
    if (!__syncthreads_or(any)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) st->rounds = 0;
        return;
    }
    // Predecessors of element k in word w of its row.
    auto preds = [&](int64_t k, int64_t w, uint64_t x) {
        return w == (k >> 6) ? x & ((1ull << (k & 63)) - 1ull) : x;
    };
    int w[kSlots];        // -1: no element, or removed
    uint64_t x[kSlots];
#pragma unroll
    for (int t = 0; t < kSlots; ++t) {
        const int64_t k = lo + 1 + (int64_t(32 * t + lane)) * warps + gwarp;
        const bool in = k < hi && ((S[k >> 6] >> (k & 63)) & 1ull);
        w[t] = in ? int(k >> 6) : -1;
        x[t] = in ? preds(k, k >> 6, __ldg(bits + k * row_words + (k >> 6))) : 0ull;
    }
    for (int64_t r = 0; r < max_rounds; ++r) {
        uint64_t* Mr = M + (r % 3) * row_words;
#pragma unroll
        for (int t = 0; t < kSlots; ++t) {
            const bool lost = w[t] >= 0 && (x[t] & S[w[t]]) == 0ull;
            for (uint32_t todo = __ballot_sync(0xffffffffu, lost); todo; todo &= todo - 1u) {
                const int f = __ffs(int(todo)) - 1;
                const int64_t k = lo + 1 + (int64_t(32 * t + f)) * warps + gwarp;
                const uint64_t* row = bits + k * row_words;
                int64_t w1 = __shfl_sync(0xffffffffu, w[t], f) - 1;  // the next word to look at
                int64_t at = -1;
                uint64_t found = 0ull;
                // 64 words at first, where the next one usually is, then 256 at a
                // time: a round waits for its longest search
                for (int width = 2; w1 >= wlo; w1 -= 32 * width, width = kWide) {
                    uint64_t y[kWide];  // lane l: words w1 - l - 32 c
#pragma unroll
                    for (int c = 0; c < kWide; ++c) {
                        const int64_t wc = w1 - lane - 32 * c;
                        y[c] = c < width && wc >= wlo ? __ldg(row + wc) : 0ull;
                    }
#pragma unroll
                    for (int c = 0; c < kWide; ++c) {
                        const int64_t wc = w1 - lane - 32 * c;
                        const uint32_t m = __ballot_sync(0xffffffffu, wc >= wlo && (y[c] & S[wc < 0 ? 0 : wc]) != 0ull);
                        if (m && at < 0) {  // the nearest one
                            const int q = __ffs(int(m)) - 1;
                            at = w1 - q - 32 * c;
                            found = __shfl_sync(0xffffffffu, y[c], q);
                        }
                    }
                    if (at >= 0) break;
                }
                if (lane == f) {
                    w[t] = int(at);
                    x[t] = found;
                    if (at < 0) atomicOr(reinterpret_cast<unsigned long long*>(Mr + (k >> 6)), 1ull << (k & 63));
                }
            }
        }
        // clear the next round's removals (last read in the round before this one)
        uint64_t* Mn = M + ((r + 1) % 3) * row_words;
        for (int64_t q = int64_t(blockIdx.x) * kPersistThreads + threadIdx.x; q < row_words;
             q += int64_t(gridDim.x) * kPersistThreads)
            Mn[q] = 0ull;
        if (!grid_barrier(st, unsigned(r))) return;
        int left = 0;
        for (int64_t q = wlo + threadIdx.x; q <= whi; q += kPersistThreads) {
            const uint64_t y = S[q] & ~__ldcg(Mr + q);
            S[q] = y;
            left |= y != 0ull;
        }
        if (!__syncthreads_or(left)) {
            if (blockIdx.x == 0 && threadIdx.x == 0) st->rounds = r + 1;
            return;
        }
    }
}

// All greedy rounds, one barrier each.  Block b owns the candidates of its
// share of the 32-column groups and keeps their overlaps in shared memory;
// every block keeps all candidates X.  A round: the block's smallest (o_j, j),
// one 64-bit atomicMin, barrier; then every block for itself reads row k and
// takes J(k) and k out of X, lists the candidates R that this removed (A loses
// exactly these: the members are unrelated to every candidate), and lowers
// its overlaps by the number of R's elements related to j, 32 rows by 32
// candidates at a time (bit transposes), the warps of a group in turn.  The
// overlaps are counted in full once, at the start.  Three barriers a round
// and one thread per candidate walking R took 37 us a round at n = 32768.
constexpr int kListCap = 4096;  // elements of R listed at a time
__global__ void __launch_bounds__(kPersistThreads) k_anti_persist(const uint64_t* __restrict__ bits, int64_t n,
                                                                  int64_t row_words, int64_t seed, int64_t max_rounds,
                                                                  uint64_t* members,
                                                                  const uint64_t* __restrict__ X0, int64_t groups_per_block,
                                                                  ChainState* st) {
    extern __shared__ __align__(16) uint64_t X[];  // [row_words], then the overlaps, the list
    int32_t* over = reinterpret_cast<int32_t*>(X + row_words);
    int32_t* list = over + 32 * groups_per_block;
    __shared__ int listed, valid;  // elements offered to the list, and listed without a gap
    __shared__ unsigned long long least;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nw = (n + 63) >> 6;
    const int64_t g0 = int64_t(blockIdx.x) * groups_per_block;
    const int64_t groups = (n + 31) / 32;
    const int ng = int(g0 >= groups ? 0 : (groups - g0 < groups_per_block ? groups - g0 : groups_per_block));
    for (int64_t w = threadIdx.x; w < row_words; w += kPersistThreads) {
        X[w] = __ldg(X0 + w);
        if (blockIdx.x == 0) members[w] = w == (seed >> 6) ? 1ull << (seed & 63) : 0ull;
    }
    __syncthreads();
    for (int c = warp; c < 32 * ng; c += kPersistWarps) {
        const int64_t j = 32 * g0 + c;
        int o = 0;
        if (j < n && bit_of(X, j)) {  // warp-uniform
#pragma unroll 4
            for (int64_t w = lane; w < nw; w += 32) o += __popcll(X[w] & __ldg(bits + j * row_words + w));
            o = int(__reduce_add_sync(0xffffffffu, unsigned(o)));
        }
        if (lane == 0) over[c] = o;
    }
    __syncthreads();
    const Tr32 tc = tr32_consts(lane);
    // warps per group (a group per warp, in turn, when there are more groups)
    const int share = ng > 0 && ng < kPersistWarps ? kPersistWarps / ng : 1;
    int64_t taken = 0;
    for (int64_t r = 0; r < max_rounds; ++r) {
        if (threadIdx.x == 0) least = ~0ull;
        __syncthreads();
        unsigned long long mine = ~0ull;
        for (int c = threadIdx.x; c < 32 * ng; c += kPersistThreads) {
            const int64_t j = 32 * g0 + c;
            if (j < n && bit_of(X, j)) {
                const unsigned long long key = (static_cast<unsigned long long>(over[c]) << 32) | uint64_t(j);
                mine = key < mine ? key : mine;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, mine, o);
            mine = y < mine ? y : mine;
        }
        if (lane == 0 && mine != ~0ull) atomicMin(&least, mine);
        __syncthreads();
        if (threadIdx.x == 0) {
            if (least != ~0ull) atomicMin(&st->best3[r % 3], least);
            if (blockIdx.x == 0) st->best3[(r + 1) % 3] = ~0ull;  // last read in the round before last
        }
        if (!grid_barrier(st, unsigned(r))) return;
        const unsigned long long best = __ldcg(&st->best3[r % 3]);
        if (best == ~0ull) break;  // no candidates (every block sees the same value)
        ++taken;
        const int64_t k = int64_t(best & 0xFFFFFFFFull);
        if (threadIdx.x == 0) {
            X[k >> 6] &= ~(1ull << (k & 63));
            if (blockIdx.x == 0) members[k >> 6] |= 1ull << (k & 63);
        }
        for (bool more = true; more;) {
            __syncthreads();
            if (threadIdx.x == 0) {
                listed = 0;
                valid = kListCap;
            }
            __syncthreads();
            int rest = 0;
            for (int64_t w = threadIdx.x; w < nw; w += kPersistThreads) {
                uint64_t y = X[w] & __ldg(bits + k * row_words + w);
                if (!y) continue;
                const int c = __popcll(y), at = atomicAdd(&listed, c);
                if (at + c > kListCap) {  // stays in X; its turn comes in the next pass
                    atomicMin(&valid, at);
                    rest = 1;
                    continue;
                }
                X[w] &= ~y;
                for (int q = at; y; y &= y - 1ull, ++q)
                    list[q] = int32_t(64 * w + __ffsll(static_cast<long long>(y)) - 1);
            }
            more = __syncthreads_or(rest) != 0;
            const int nr = listed < valid ? listed : valid;
            for (int g = warp / share; g < ng; g += kPersistWarps / share) {
                if (warp / share >= kPersistWarps / share) break;  // the warps left over
                // 32 rows at a time: lane l reads its row's word of the group,
                // the transpose gives lane l the 32 rows' bits of column l
                const uint32_t* col = reinterpret_cast<const uint32_t*>(bits) + (g0 + g);
                int d = 0;
#pragma unroll 2
                for (int t = 32 * (warp % share); t < nr; t += 32 * share) {
                    const uint32_t v = t + lane < nr ? __ldg(col + int64_t(list[t + lane]) * row_words * 2) : 0u;
                    d += __popc(transpose32(v, tc));
                }
                if (d) atomicSub(&over[32 * g + lane], d);
            }
        }
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) st->rounds = taken + 1;  // and the seed
}

// Blocks of a cooperative launch of `kernel` with `smem` bytes, one per SM at
// most and `need` of them at most; 0 where it is not possible.
int coop_grid(const void* kernel, int smem, int64_t need) {
    int dev = 0, coop = 0, per_sm = 0, most = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || smem > most - 1024)
        return 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kPersistThreads, smem) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        return 0;
    }
    const int64_t sms = device_sm_count();
    return int(need < 1 ? 1 : need < sms ? need : sms);
}

int warp_grid(int64_t rows) {
    int64_t g = (rows + 7) / 8;
    const int64_t cap = int64_t(device_sm_count()) * 16;
    return int(g < 1 ? 1 : (g > cap ? cap : g));
}

bool chain_args_ok(int64_t n, const uint64_t* bits, int64_t row_words, void* ws) {
    return n >= 1 && n <= kMaxN && bits && (reinterpret_cast<uintptr_t>(bits) % 16) == 0 &&
           row_words >= cs_row_words(n) && row_words % 16 == 0 && ws && (reinterpret_cast<uintptr_t>(ws) % 256) == 0;
}

cudaError_t read_state(const ChainState* dev, ChainState* host, cudaStream_t st) {
    cudaError_t e = cudaMemcpyAsync(host, dev, sizeof(ChainState), cudaMemcpyDeviceToHost, st);
    return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

}  // namespace

}  // namespace cs

using namespace cs;

extern "C" size_t cs_chain_workspace_bytes(int64_t n) {
    if (n < 1 || n > kMaxN) return 0;
    return chain_layout(cs_row_words(n)).total;
}

extern "C" int cs_longest_chain(int64_t n, const uint64_t* bits_dev, int64_t row_words, int64_t i, int64_t j,
                                int64_t* length, void* workspace_dev, size_t workspace_bytes, void* stream) {
    CS_TRACE("cs_longest_chain");
    if (!chain_args_ok(n, bits_dev, row_words, workspace_dev) || !length) return CS_EINVAL;
    const bool whole = i < 0 && j < 0;
    if (!whole && (i < 0 || j < 0 || i >= n || j >= n)) return CS_EINVAL;
    const ChainLayout L = chain_layout(row_words);
    if (workspace_bytes < L.total) return CS_ENOMEM;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace_dev);
    ChainState* sd = reinterpret_cast<ChainState*>(ws + L.state);
    uint64_t* S = reinterpret_cast<uint64_t*>(ws + L.s);
    uint64_t* M = reinterpret_cast<uint64_t*>(ws + L.m);
    if (!whole && j <= i) {
        *length = -1;
        return CS_OK;
    }
    const int64_t lo = whole ? -1 : i, hi = whole ? n : j;
    int64_t g = (row_words + 255) / 256;
    k_chain_init<<<unsigned(g < 1 ? 1 : g), 256, 0, st>>>(bits_dev, n, row_words, whole ? -1 : i, j, S, M, sd);
    ChainState h{};
    // one cooperative launch for all rounds when the device allows it: about
    // four elements per warp where the set does not fill the SMs
    const int64_t count = hi - lo - 1;
    const int smem = int(row_words * 8);
    const int64_t per_slot = int64_t(device_sm_count()) * kPersistThreads;
    const auto kernel = count <= per_slot       ? k_chain_persist<1>
                        : count <= 4 * per_slot ? k_chain_persist<4>
                                                : k_chain_persist<12>;
    const int64_t blocks = (count + 4 * kPersistWarps - 1) / (4 * kPersistWarps);
    const int cg = count <= 12 * per_slot ? coop_grid(reinterpret_cast<const void*>(kernel), smem, blocks) : 0;
    if (cg > 0) {
        int64_t max_rounds = n + 1;
        const uint64_t* S0 = S;
        void* args[] = {const_cast<uint64_t**>(&bits_dev), &row_words, const_cast<int64_t*>(&lo),
                        const_cast<int64_t*>(&hi), &max_rounds, &S0, &M, &sd};
        if (cudaMemsetAsync(&sd->rounds, 0xFF, sizeof(int64_t), st) != cudaSuccess) return CS_ECUDA;  // -1 until the last round
        if (cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kernel), dim3(unsigned(cg)),
                                        dim3(kPersistThreads), args, size_t(smem), st) == cudaSuccess) {
            if (read_state(sd, &h, st) != cudaSuccess) return CS_ECUDA;
            if (h.status != 0) return h.status;
            if (!h.related) {
                *length = -1;
                return CS_OK;
            }
            if (h.rounds < 0) return CS_ERANGE;  // cannot happen for a transitive relation
            *length = whole ? h.rounds : h.rounds + 1;  // no round: a link, or an empty set
            return CS_OK;
        }
        cudaGetLastError();  // not launched: clear and take the multi-launch path
        k_chain_init<<<unsigned(g < 1 ? 1 : g), 256, 0, st>>>(bits_dev, n, row_words, whole ? -1 : i, j, S, M, sd);
    }
    for (int64_t done = 0; done <= n; done += kBatch) {  // at most n + 1 rounds remove anything
        for (int r = 0; r < kBatch; ++r) {
            k_chain_peel<<<warp_grid(hi - lo - 1), 256, 0, st>>>(bits_dev, row_words, lo, hi, S, M, sd);
            k_chain_apply<<<1, 1024, 0, st>>>(row_words, S, M, sd);
        }
        if (cudaGetLastError() != cudaSuccess || read_state(sd, &h, st) != cudaSuccess) return CS_ECUDA;
        if (h.left == 0 || !h.related) break;
    }
    if (h.left != 0 && h.related) return CS_ERANGE;  // cannot happen for a transitive relation
    *length = whole ? h.rounds : (h.related ? h.rounds + 1 : -1);
    return CS_OK;
}

extern "C" int cs_greedy_antichain(int64_t n, const uint64_t* bits_dev, int64_t row_words, int64_t seed,
                                   uint64_t* members_dev, int64_t* size, void* workspace_dev, size_t workspace_bytes,
                                   void* stream) {
    CS_TRACE("cs_greedy_antichain");
    if (!chain_args_ok(n, bits_dev, row_words, workspace_dev) || seed < 0 || seed >= n || !members_dev ||
        (reinterpret_cast<uintptr_t>(members_dev) % 8) != 0 || !size)
        return CS_EINVAL;
    const ChainLayout L = chain_layout(row_words);
    if (workspace_bytes < L.total) return CS_ENOMEM;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(workspace_dev);
    ChainState* sd = reinterpret_cast<ChainState*>(ws + L.state);
    uint64_t* X = reinterpret_cast<uint64_t*>(ws + L.s);
    int64_t g = (row_words + 255) / 256;
    k_anti_init<<<unsigned(g < 1 ? 1 : g), 256, 0, st>>>(bits_dev, n, row_words, seed, members_dev, X, sd);
    ChainState h{};
    const int64_t groups = (n + 31) / 32;
    const int64_t sms = device_sm_count();
    // at least four groups of 32 candidates per block, at most the SMs' share
    int64_t per = (groups + sms - 1) / sms;
    if (per < 4) per = 4;
    const int64_t blocks = (groups + per - 1) / per;
    const int smem = int(row_words * 8 + 32 * per * 4 + kListCap * 4);
    const int cg = coop_grid(reinterpret_cast<const void*>(k_anti_persist), smem, blocks);
    if (cg == blocks) {
        int64_t max_rounds = n + 1;
        const uint64_t* X0 = X;
        void* args[] = {const_cast<uint64_t**>(&bits_dev), &n, &row_words, &seed, &max_rounds, &members_dev, &X0, &per, &sd};
        if (cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_anti_persist), dim3(unsigned(cg)),
                                        dim3(kPersistThreads), args, size_t(smem), st) == cudaSuccess) {
            if (read_state(sd, &h, st) != cudaSuccess) return CS_ECUDA;
            if (h.status != 0) return h.status;
            if (h.rounds < 0) return CS_ERANGE;
            *size = h.rounds;
            return CS_OK;
        }
        cudaGetLastError();
        k_anti_init<<<unsigned(g < 1 ? 1 : g), 256, 0, st>>>(bits_dev, n, row_words, seed, members_dev, X, sd);
    }
    bool done = false;
    for (int64_t rounds = 0; !done && rounds <= n; rounds += kBatch) {  // multi-launch path
        for (int r = 0; r < kBatch; ++r) {
            k_anti_score<<<warp_grid(n), 256, 0, st>>>(bits_dev, n, row_words, members_dev, X, sd);
            k_anti_apply<<<1, 1024, 0, st>>>(bits_dev, row_words, members_dev, X, sd);
        }
        if (cudaGetLastError() != cudaSuccess || read_state(sd, &h, st) != cudaSuccess) return CS_ECUDA;
        if (h.left == 0) done = true;
    }
    if (!done) return CS_ERANGE;
    k_count_bits<<<1, 1024, 0, st>>>(members_dev, row_words, sd);
    if (cudaGetLastError() != cudaSuccess || read_state(sd, &h, st) != cudaSuccess) return CS_ECUDA;
    *size = h.rounds;
    return CS_OK;
}

