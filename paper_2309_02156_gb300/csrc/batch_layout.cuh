// Shared memory of a block of the batched step: the guess, then the resident CG.
#pragma once

#include "common.cuh"
#include "resident.cuh"
#include "sketch_tile.cuh"

namespace sa {

constexpr int kBatchMaxM = 16;
constexpr int kBatchMaxS = 64;
constexpr int kSketchTeams = 4;           // teams of four warps that sketch a sequence

// The sketch takes its teams' regions and an FP64 accumulator per team.  Its sum
// W ends in the first accumulator; the regions then hold the least squares
// (block_lsq), y and, in a cluster, the total of W, so that the largest guess
// (M = 16, s = 64) takes 104 KB and two blocks fit on an SM (131 KB when each
// had a place of its own).
__host__ __device__ inline size_t sketch_regions_doubles(int s, int ncol) {
    return kSketchTeams * (sketch_team_bytes(s, ncol) / 8);
}
__host__ __device__ inline size_t lsq_ws_doubles(int s, int M) {
    return 2 * (size_t)s * M + 3 * (size_t)s + 5 * (size_t)M;
}
__host__ __device__ inline size_t after_sketch_doubles(int s, int M) {
    return lsq_ws_doubles(s, M) + kBatchMaxM + (size_t)s * (M + 1);
}

// Bytes of one block, or one CTA of a cluster, for s sketch rows and M columns.
inline size_t batch_smem_bytes(int s, int M) {
    const int ncol = M + 1;
    const size_t guess = 8 * (sketch_regions_doubles(s, ncol) + kSketchTeams * (size_t)s * ncol);
    const size_t stage = sizeof(double) * 32 * (size_t)kTileChunks * 32;   // up to 32 warps
    return guess > stage ? guess : stage;
}

// Layout of a sequence's resident CG over `ctas` CTAs; false: it takes the form
// whose vectors lie in global memory.  A CTA of a cluster also forms the direction
// on the rows within reach on both sides: with more of those than rows of its own
// it is slower for it (clusters of 8 and of 4, 64 sequences, ms a step, global
// form and resident: 10,000 rows, reach 5,000, 1.12 and 1.41, 0.67 and 0.74, reach
// 2,000 1.19 and 1.26, 0.71 and 0.72, reach 100 1.17 and 1.11, 0.70 and 0.65;
// 64,000 rows, reach 1,600, 3.02 and 2.83, 2.37 and 2.23).
__host__ __device__ inline bool batch_resident(int n, int W, int reach, int ctas, size_t budget,
                                               ResLayout* L) {
    return res_layout(n, W, reach, ctas, sizeof(float), budget, L) &&
           (ctas == 1 || 2LL * reach <= 32LL * L->per);
}

}  // namespace sa
