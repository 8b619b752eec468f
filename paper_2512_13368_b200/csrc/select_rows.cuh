// First stage of the selection with a lane per query row (select_rows.cu).
#pragma once
#include "select_geom.cuh"

namespace blossom {

struct RowsGeom {
  int cols, pitch;  // candidates in the table of means; pitch of a row's table of exponentials (floats)
  int means;        // floats of the table of means
  int lg_heads;     // (per position) log2 of the heads of the group that as many warps take at once
  int list;         // what is not certain goes to the list (else the kernel decides it itself)
};
// Whether the kernel takes the problem (up to 128 scored and selection blocks), its plan and its shared memory.
bool rows_geom(const Shape &sh, const SelGeom &g, int dtype, RowsGeom *rg, size_t *smem);
// Writes the certain index rows and, with rg.list, appends the others to `list` (per block: unit * M + block; per
// position: unit * L + position).
int launch_score_rows(const Shape &sh, const SelGeom &g, const RowsGeom &rg, size_t smem, int dtype, const void *q,
                      const float *mean32, const float *norm, const double *mean, const int32_t *seq_lens, int32_t *idx,
                      int32_t *list, int32_t *count, cudaStream_t st);

}  // namespace blossom
