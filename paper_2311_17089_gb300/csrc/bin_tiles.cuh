// The tile lists of one frame from a depth order of its Gaussians, without
// materialising (tile, index) pairs.  Defined in bin_tiles.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace msgs {

constexpr int kMaxColBlocks = 512;  // blocks of the column scan (and tile_sums words)

struct TileListArgs {
    const uint32_t *order;   // Gaussian indices in depth order
    const uint32_t *n32;     // their count (device)
    const uint32_t *n_tiles;
    const uint2 *rect;
    int64_t n;               // length of n_tiles and rect, upper bound of the count
    int tiles_x;
    int64_t tiles;
    int64_t cap;             // entries gauss_idx holds
    uint32_t *gauss_idx, *ranges;
    unsigned long long *err;
    // scratch: a 64-bit word per block of the order (tile_block_count(n)),
    // 2 words per block and 4 more (8-byte aligned), item and idx n
    // entries each (idx may be the order itself), the matrix's bytes
    // (16-byte aligned)
    unsigned long long *block_sums;
    uint32_t *block_words;
    uint2 *item;
    uint32_t *idx;
    uint32_t *matrix;
    size_t matrix_bytes;
    uint32_t *meta;          // [8] words
    uint32_t *tile_sums;     // [kMaxColBlocks] zeroed words
};

// Blocks of an order of n Gaussians (1024 positions each, or a multiple).
int64_t tile_block_count(int64_t n);
int launch_tile_lists(const TileListArgs &a, cudaStream_t st);

}  // namespace msgs
