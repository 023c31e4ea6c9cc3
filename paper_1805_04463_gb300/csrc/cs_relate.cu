// cs_relate.cu -- the causal matrix as row bitsets (Section "Data Structures
// for Totally Ordered Sets": the symmetrised matrix P + P^T, one bitset per
// row; Section "Lorentzian Geometry": related iff Delta s^2 < 0).
//
// A block owns 2048 columns (32 words) and 64 rows (relate_block): column
// values are staged once in shared memory and read by broadcast, each lane
// builds the words of two rows from the sign bits of integer multiply-adds
// (circle) or of an FP32 filter with an exact int64 recompute near the cone
// (2+1, 3+1); the row tile's own word, which holds the diagonal, takes the full
// symmetric test by two ballots.  The light-cone kinds have a lane per word
// instead (relate_block_cone).  64 x 64 tiles
// wholly below the diagonal are not tested: k_mirror fills them as bit
// transposes of the tiles above (the relation is symmetric), which halves
// the tests.
#include "cs_kernels.cuh"
#include "cs_launch.cuh"
#include "cs_relate.cuh"

namespace cs {

namespace {

// Relate kernel alone, before (a lane per word, or 64 tests per two ballots
// for the circle) / now: 3+1 n = 16384 102 / 45 us, 2+1 n = 20011 150 / 57 us,
// de Sitter slab n = 50021 632 / 253 us.  What bounds it now is the integer pipe (the
// circle 83%), in 3+1 the FMA pipe (53%) with it (44%).
//
// The mirror is launched behind it without an early trigger: its blocks
// come when the last ones here end.  Triggered at the start they crowded onto the few SMs that
// still had room, four to an SM: with the mirror, early / so, 2D order n = 5000 16.8 / 12.2 us,
// slab n = 4099 19.3 / 13.3, 3+1 n = 7000 29.5 / 25.4, n >= 12000 alike (an ordinary
// launch: 14.8, 16.9, 29.2).
template <int G, int kWords>
__global__ void __launch_bounds__(kRelThreads) k_relate(const int32_t* __restrict__ coords, int64_t n,
                                                        uint64_t* __restrict__ bits, int64_t row_words) {
    __shared__ __align__(16) uint8_t sm[relate_stage_bytes(G)];
    relate_block<G, kWords>(coords, n, bits, row_words, blockIdx.x,
                            int64_t(blockIdx.y) * (kWords * (kRelThreads / 32)), sm);
}

// The light-cone kinds, five blocks per SM (48 registers; at four, 57 registers, the diamond of
// 131072 takes 1915 us with the mirror instead of 1720).
__global__ void __launch_bounds__(kRelThreads, 5) k_relate_cone(const int32_t* __restrict__ coords, int64_t n,
                                                                uint64_t* __restrict__ bits, int64_t row_words,
                                                                bool order2d) {
    __shared__ __align__(16) int32_t st[kConeInts];
    relate_block_cone(coords, n, bits, row_words, blockIdx.x, int64_t(blockIdx.y) * kRelWordsPerBlock, st, order2d);
}

// Chunks of 32 words; of 8, one per warp, where those would be fewer than two
// per SM (n up to 6144): a chunk is then
// latency, four words in turn.  With the mirror, 32 / 8 words, back to back: 3+1
// n = 1024 12.4 / 10.4 us, n = 4099 15.2 / 12.9, slab n = 2000 12.5 / 10.1, n = 4099 13.4 / 13.3.
// The light cone by broadcast columns only there (diamond n = 2000 11.1 us, a lane per word 12.2;
// n = 6100 15.3 / 14.5, n = 131072 1767 / 1720), the 2D order never (n = 2000 14.5 / 10.5 us,
// its own words' exact tests the longest chain; n = 131072 1276 / 1273).
template <int G>
void launch_upper(const int32_t* coords, int64_t n, uint64_t* bits, int64_t row_words, bool order2d, cudaStream_t st) {
    const unsigned rows = unsigned((n + kRelRowsPerBlock - 1) / kRelRowsPerBlock);
    const dim3 grid(rows, unsigned((row_words + kRelWordsPerBlock - 1) / kRelWordsPerBlock));
    if (!order2d && int64_t(rows) * grid.y < 2 * int64_t(device_sm_count()))
        k_relate<G, 1><<<dim3(rows, unsigned((row_words + 7) / 8)), kRelThreads, 0, st>>>(coords, n, bits, row_words);
    else if constexpr (G == kGeomLightCone)
        k_relate_cone<<<grid, kRelThreads, 0, st>>>(coords, n, bits, row_words, order2d);
    else
        k_relate<G, kRelWarpWords><<<grid, kRelThreads, 0, st>>>(coords, n, bits, row_words);
}

__global__ void __launch_bounds__(kRelThreads, 4) k_mirror(uint64_t* bits, int64_t n, int64_t row_words) {
    __shared__ uint64_t sm[kMirRows][kMirTiles + 1];
    wait_for_primary();
    mirror_block(bits, n, row_words, blockIdx.x, blockIdx.y, sm);
}

}  // namespace

cudaError_t launch_relate(int kind, int64_t n, const int32_t* coords, uint64_t* bits, int64_t row_words,
                          cudaStream_t st) {
    if (kind == CS_4D_DIAMOND)
        launch_upper<kGeom4>(coords, n, bits, row_words, false, st);
    else if (kind == CS_3D_DIAMOND)
        launch_upper<kGeom3>(coords, n, bits, row_words, false, st);
    else if (kind == CS_2D_DS_SLAB || kind == CS_2D_CYLINDER)
        launch_upper<kGeomDeSitter>(coords, n, bits, row_words, false, st);
    else
        launch_upper<kGeomLightCone>(coords, n, bits, row_words, kind == CS_2D_ORDER, st);
    const int64_t st8 = ((n + 63) / 64 + kMirTiles - 1) / kMirTiles;  // super-tiles per side
    const cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess || st8 <= 0) return err;
    return launch_after(k_mirror, dim3(unsigned(st8), unsigned(st8)), kRelThreads, 0, st, bits, n, row_words);
}

}  // namespace cs
