// Descriptor of one matrix of a batched product (shared by api.cu, which
// fills it on the host, and batched.cu, whose persistent kernel reads it).
#pragma once
#include <cuda_runtime.h>

#include "launch.h"

namespace gbs {

// Tiles of one MERGE work item: one per warp of the batch's CTAs for block vectors (2048 to 4096
// nonzeros at k = 8), four for a vector, whose tiles are 256 nonzeros.
__host__ __device__ inline int batch_item_tiles(int k) { return k == 1 ? 32 : 8; }

template <typename T>
struct BatchDesc {
  int m, n, nnz, k;
  const int* row_ptr;
  const int* col_idx;
  const T* vals;
  const T* X;
  T* Y;
  long long ldx, ldy;
  int variant;     // GBS_VARIANT_ROWS or GBS_VARIANT_MERGE
  int lanes;       // ROWS: lanes per row (k == 1) or column lanes (k > 1)
  int tile;        // ROWS: nonzeros staged per pass
  int share;       // MERGE: nonzeros per merge thread of the nonzero-split walk
  int tiles;       // MERGE: its tiles (warps)
  int item_begin;  // first work item of this matrix in the batch's work list
  int nitems;      // its work items: row blocks (ROWS) or groups of tiles (MERGE)
  const SplitWord* words;  // MERGE: A's split index and the carries (plan-owned)
  const int* ids;
  const int* empty;
  int nempty;
  int wide;
  int* carry_row;
  T* carry_val;
  int fix_begin;   // MERGE: first block of this matrix in the fix-up launch, and its carry blocks
  int fix_carry_blocks;
  int aligned_vals, aligned_cols;
};

}  // namespace gbs
