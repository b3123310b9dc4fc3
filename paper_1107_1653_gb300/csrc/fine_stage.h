// Shared-memory staging of the finest level's wide phases (fine.cuh): sizes
// only, in plain C++, so that they can be checked on the CPU for every grid.
#pragma once

#ifdef __CUDACC__
#define GS_STAGE_FN __host__ __device__ constexpr
#else
#define GS_STAGE_FN constexpr
#endif

namespace gs {

// The restriction stages the residuals of the colour-0 points of 2 k + 1 rows for
// k coarse rows, (side + 1) / 2 values per row; the last relaxation stages
// whole rows of side + 1 values.  64 KB hold that for grids of side up to 8191;
// the largest accepted side, 16383, needs three half rows (96 KB).
constexpr int kFineStage = 16384;

// Floats of one launch's staging.
GS_STAGE_FN int fine_stage_floats(int side) {
    const int least = 3 * ((side + 1) / 2);
    return least > kFineStage ? least : kFineStage;
}

// Coarse rows the restriction takes at a time.
GS_STAGE_FN int fine_restrict_chunk(int side) { return (fine_stage_floats(side) / ((side + 1) / 2) - 1) / 2; }

// Rows the last relaxation takes at a time.
GS_STAGE_FN int fine_update_chunk(int side) { return fine_stage_floats(side) / (side + 1); }

}  // namespace gs
