// Chunks of the Frobenius products (reduce.cu) and their split over blocks: an np x np matrix is read
// in chunks of kChunkBytes consecutive bytes of a row, those on or above the diagonal, a block
// taking consecutive ones. Host-compilable, for a host test.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define FO_GS __host__ __device__
#else
#define FO_GS
#endif

namespace fo {

constexpr int kChunkBytes = 512;    // one chunk of one matrix: 128 float32 / 64 float64
constexpr int kGChunks = 64;        // most chunks per block
constexpr int kGramBlocks = 300;    // blocks that float64 plans aim at: two per SM

// Upper chunks of an np x np matrix: row r holds chunks floor(r / kc) .. np / kc - 1.
FO_GS inline int64_t upper_chunks(int64_t np, int kc) {
    const int64_t cpr = np / kc;
    return (int64_t)kc * cpr * (cpr + 1) / 2;
}

// Chunks per block of a plan of `count` instances. float32: kGChunks (the partial sums' grouping is
// part of the result's bits). float64: as few as give the whole batch about kGramBlocks blocks, since
// the float64 FMAs bound the kernel and one small matrix would otherwise use few SMs (N = 256 alone:
// 10 blocks of 64 chunks, 0.37 ms; 320 of two 0.10). A block ends with 125 float64 adds per warp and
// tile, as many as the FMAs of two chunks, so that a batch that fills the SMs by itself keeps long
// blocks: 64 matrices of N = 256 take 1.6 ms in blocks of 64 chunks, 3.8 in blocks of two.
inline int gram_chunks(const int64_t* np, int count, bool is64) {
    if (!is64) return kGChunks;
    int64_t total = 0;
    for (int i = 0; i < count; ++i) total += upper_chunks(np[i], kChunkBytes / 8);
    const int64_t c = total / kGramBlocks;
    return c < 2 ? 2 : (c > kGChunks ? kGChunks : (int)c);
}

}  // namespace fo
