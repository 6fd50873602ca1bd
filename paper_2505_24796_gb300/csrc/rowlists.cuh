// rowlists.cuh -- the sorting stage by tile-row lists (rowlists.cu), as binsort.cu calls it.
#pragma once

#include "common.cuh"

namespace tcgs {

// Grids of at most this many tile columns and rows are sorted by row lists: a run's row and first and
// last column then take 8 bits each, beside the 8-bit index of its Gaussian in its block.
constexpr int kRowListsMaxGrid = 256;

struct RowLists {
    DevCamera cam;
    uint32_t P;
    const uint32_t* order;   // the P Gaussians by depth
    const float* mean2d;
    const int32_t* radius;
    const float* conic;      // exact coverage only
    const float* opacity;    // exact coverage only
    bool exact;
    bool fill_rows;          // exact: a wide Gaussian's row is one run from its first to its last reached tile
    int64_t capacity;
    char* scratch;           // 256-byte aligned, at least row_lists_scratch_bytes(P, capacity)
    uint32_t* ids_sorted;
    uint32_t* ranges;
    int64_t* n_splats;
    int32_t* status;
};

size_t row_lists_scratch_bytes(int64_t P, int64_t capacity);

// Depth keys (radius <= 0 last) and indices of the P Gaussians; zeroes the tile ranges, the first
// digit pass's totals (256 words) and the counters at the start of `scratch`.
void launch_row_keys(const RowLists& a, const float* depth, uint32_t* keys, uint32_t* vals, uint32_t* digit_total0,
                     cudaStream_t s);

// From the depth order to the sorted lists, ranges, N and status.
void launch_row_lists(const RowLists& a, cudaStream_t s);

}  // namespace tcgs
