// Plan-time index of the SPLIT variant (see split_kernel.cuh): per 32 nonzeros, the bitmap of row
// ends and the ordinal of the first nonzero's row; the row numbers of the non-empty rows; the
// empty rows.  One thread per row, the words of a long row written by its whole warp.
#include <algorithm>

#include "launch.h"

namespace gbs {

__global__ void __launch_bounds__(256) nonempty_kernel(const int* __restrict__ rp, int m, int* __restrict__ flag) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) flag[i] = rp[i + 1] > rp[i];
}

__global__ void __launch_bounds__(256) split_words_kernel(const int* __restrict__ rp, int m,
                                                          const int* __restrict__ ord, SplitWord* __restrict__ words,
                                                          int* __restrict__ ids, int* __restrict__ empty) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int w0 = 0, w1 = 0, o = 0;  // words [w0, w1) begin inside this thread's row
  if (i < m) {
    const int s = rp[i], e = rp[i + 1];
    o = ord ? ord[i] : i;
    if (e > s) {
      if (ids) ids[o] = i;
      atomicOr(&words[(e - 1) >> 5].ends, 1u << ((e - 1) & 31));
      w0 = (int)((s + 31u) >> 5);
      w1 = (int)((e + 31u) >> 5);
    } else if (empty) {
      empty[i - o] = i;
    }
  }
  const bool is_long = w1 - w0 > 32;
  if (!is_long)
    for (int w = w0; w < w1; ++w) words[w].first = o;
  unsigned todo = __ballot_sync(0xffffffffu, is_long);
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    const int a = __shfl_sync(0xffffffffu, w0, src), b = __shfl_sync(0xffffffffu, w1, src);
    const int v = __shfl_sync(0xffffffffu, o, src);
    for (int w = a + lane; w < b; w += 32) words[w].first = v;
  }
}

cudaError_t split_build(int m, int nnz, const int* row_ptr, SplitWord* words, int* ids, int* empty, int* ord,
                        int* scan_ws, cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(words, 0, sizeof(SplitWord) * (size_t)(((long long)nnz + 31) / 32), s);
  if (e != cudaSuccess) return e;
  const int grid = (m + 255) / 256;
  if (ord) {
    nonempty_kernel<<<grid, 256, 0, s>>>(row_ptr, m, ord);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = exclusive_scan_i32(ord, ord, m, scan_ws, s)) != cudaSuccess) return e;
  }
  split_words_kernel<<<grid, 256, 0, s>>>(row_ptr, m, ord, words, ids, empty);
  return cudaGetLastError();
}

long long split_tiles(int nnz, int g, int share) {
  const long long per = (long long)(32 / g) * share;
  return std::max(1LL, (nnz + per - 1) / per);
}

}  // namespace gbs
