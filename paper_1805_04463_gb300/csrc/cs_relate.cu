// cs_relate.cu -- the causal matrix as row bitsets (Section "Data Structures
// for Totally Ordered Sets": the symmetrised matrix P + P^T, one bitset per
// row; Section "Lorentzian Geometry": related iff Delta s^2 < 0).
//
// A block owns 2048 columns (32 words) and 64 rows (relate_block): column
// values are staged once in shared memory and read by broadcast, each lane
// builds the words of two rows from the sign bits of integer multiply-adds
// (light cone, circle) or of an FP32 filter with an exact int64 recompute
// near the cone (2+1, 3+1); the row tile's own word, which holds the
// diagonal, takes the full symmetric test by two ballots.  64 x 64 tiles
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
// de Sitter slab n = 50021 632 / 253 us, 1+1 diamond n = 30011 79 / 79 us, 2D
// order n = 131072 789 / 802 us.  What bounds it now is the integer pipe (the
// circle 83%, the light cone 70%), in 3+1 the FMA pipe (53%) with it (44%).
//
// The mirror is launched behind it without an early trigger: its blocks
// come when the last ones here end.  Triggered at the start they crowded onto the few SMs that
// still had room, four to an SM: with the mirror, early / so, slab n = 4099 19.3 / 13.3 us,
// 3+1 n = 7000 29.5 / 25.4, n >= 12000 alike (an ordinary launch: 16.9, 29.2).
template <int G, int kWords>
__global__ void __launch_bounds__(kRelThreads) k_relate(const int32_t* __restrict__ coords, int64_t n,
                                                        uint64_t* __restrict__ bits, int64_t row_words) {
    __shared__ __align__(16) uint8_t sm[relate_stage_bytes(G)];
    relate_block<G, kWords>(coords, n, bits, row_words, blockIdx.x,
                            int64_t(blockIdx.y) * (kWords * (kRelThreads / 32)), sm);
}

// Chunks of 32 words; of 8, one per warp, where those would be fewer than two
// per SM (n up to 6144): a chunk is then
// latency, four words in turn.  With the mirror, 32 / 8 words, back to back: 1+1
// diamond n = 2048 12.1 / 9.0 us, 3+1 n = 1024 10.2 / 7.4, n = 4099 12.9 / 10.7,
// 2D order 2048 13.7 / 11.9, 4099 13.9 / 14.2 (its own words' exact tests are the
// longest chain).
template <int G>
void launch_upper(const int32_t* coords, int64_t n, uint64_t* bits, int64_t row_words, cudaStream_t st) {
    const unsigned rows = unsigned((n + kRelRowsPerBlock - 1) / kRelRowsPerBlock);
    const int64_t chunks = (row_words + kRelWordsPerBlock - 1) / kRelWordsPerBlock;
    if (int64_t(rows) * chunks < 2 * int64_t(device_sm_count()))
        k_relate<G, 1><<<dim3(rows, unsigned((row_words + 7) / 8)), kRelThreads, 0, st>>>(coords, n, bits, row_words);
    else
        k_relate<G, kRelWarpWords><<<dim3(rows, unsigned(chunks)), kRelThreads, 0, st>>>(coords, n, bits, row_words);
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
        launch_upper<kGeom4>(coords, n, bits, row_words, st);
    else if (kind == CS_3D_DIAMOND)
        launch_upper<kGeom3>(coords, n, bits, row_words, st);
    else if (kind == CS_2D_DS_SLAB || kind == CS_2D_CYLINDER)
        launch_upper<kGeomDeSitter>(coords, n, bits, row_words, st);
    else if (kind == CS_2D_ORDER)
        launch_upper<kGeomOrder>(coords, n, bits, row_words, st);
    else
        launch_upper<kGeomLightCone>(coords, n, bits, row_words, st);
    const int64_t st8 = ((n + 63) / 64 + kMirTiles - 1) / kMirTiles;  // super-tiles per side
    const cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess || st8 <= 0) return err;
    return launch_after(k_mirror, dim3(unsigned(st8), unsigned(st8)), kRelThreads, 0, st, bits, n, row_words);
}

}  // namespace cs
