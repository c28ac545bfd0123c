// The index of the SPLIT variant (see split_kernel.cuh): per 32 nonzeros, the bitmap of row ends and
// the ordinal of the first nonzero's row; the row numbers of the non-empty rows; the empty rows.
// A one-shot call makes it each time and cannot afford a general scan's launches: at most
// kSplitBlocks blocks of consecutive rows, whose non-empty rows the first kernel counts (it also
// clears the words); in the second every block adds up the counts before its own, and the words of
// a long row are written by its whole warp.
#include <algorithm>

#include "dependent.cuh"
#include "gbspmv.h"
#include "launch.h"

namespace gbs {

// Marks the row's end in its word and numbers the words that begin in it (the whole warp calls it).
__device__ __forceinline__ void split_mark(int s, int e, int number, SplitWord* __restrict__ words) {
  const int lane = threadIdx.x & 31;
  int w0 = 0, w1 = 0;  // words [w0, w1) begin inside this thread's row
  if (e > s) {
    atomicOr(&words[(e - 1) >> 5].ends, 1u << ((e - 1) & 31));
    w0 = (int)((s + 31u) >> 5);
    w1 = (int)((e + 31u) >> 5);
  }
  const bool is_long = w1 - w0 > 32;
  if (!is_long)
    for (int w = w0; w < w1; ++w) words[w].first = number;
  unsigned todo = __ballot_sync(0xffffffffu, is_long);
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    const int a = __shfl_sync(0xffffffffu, w0, src), b = __shfl_sync(0xffffffffu, w1, src);
    const int v = __shfl_sync(0xffffffffu, number, src);
    for (int w = a + lane; w < b; w += 32) words[w].first = v;
  }
}

__global__ void __launch_bounds__(256) split_count_kernel(const int* __restrict__ rp, int m, int rows_per_block,
                                                          SplitWord* __restrict__ words, int nwords,
                                                          int* __restrict__ counts) {
  allow_next();
  for (long long w = (long long)blockIdx.x * 256 + threadIdx.x; w < nwords; w += (long long)gridDim.x * 256)
    words[w] = SplitWord{0u, 0};
  const long long r0 = (long long)blockIdx.x * rows_per_block, r1 = min((long long)m, r0 + rows_per_block);
  int c = 0;
  for (long long i = r0 + threadIdx.x; i < r1; i += 256) c += rp[i + 1] > rp[i];
  __shared__ int part[8];
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) c += part[w];
    counts[blockIdx.x] = c;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) split_number_kernel(const int* __restrict__ rp, int m, int rows_per_block,
                                                         SplitWord* __restrict__ words, int* __restrict__ ids,
                                                         int* __restrict__ nonempty, int* __restrict__ empty,
                                                         const int* __restrict__ counts, int k, T* __restrict__ Y,
                                                         long long ldy) {
  __shared__ int part[2][8];
  wait_for_previous();
  allow_next();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int before = 0;
  for (int b = threadIdx.x; b < (int)blockIdx.x; b += 256) before += counts[b];
  before = __reduce_add_sync(0xffffffffu, before);
  if (lane == 0) part[0][w] = before;
  __syncthreads();
  before = 0;
  for (int v = 0; v < 8; ++v) before += part[0][v];
  const long long r0 = (long long)blockIdx.x * rows_per_block, r1 = min((long long)m, r0 + rows_per_block);
  int buf = 1;  // the warps' counts of one round are read while the next round writes the other half
  for (long long base = r0; base < r1; base += 256) {
    const long long i = base + threadIdx.x;
    int s = 0, e = 0;
    if (i < r1) {
      s = rp[i];
      e = rp[i + 1];
    }
    const unsigned full = __ballot_sync(0xffffffffu, e > s);
    if (lane == 0) part[buf][w] = __popc(full);
    __syncthreads();
    int ord = before + __popc(full & ((1u << lane) - 1u));
    for (int v = 0; v < 8; ++v) {
      const int c = part[buf][v];
      if (v < w) ord += c;
      before += c;
    }
    buf ^= 1;
    if (e > s) {
      if (ids) ids[ord] = (int)i;
    } else if (i < r1) {
      if (empty) empty[i - ord] = (int)i;
      for (int c = 0; c < k; ++c) Y[i * ldy + c] = T(0);
    }
    split_mark(s, e, ord, words);
  }
  if (nonempty && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *nonempty = before;
}

cudaError_t split_build(int dtype, int m, int nnz, const int* row_ptr, SplitWord* words, int* ids, int* nonempty,
                        int* empty, int* counts, int k, void* Y, long long ldy, cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  const int per = (int)std::max<long long>(256, (((long long)m + kSplitBlocks - 1) / kSplitBlocks + 255) / 256 * 256);
  const int grid = (int)(((long long)m + per - 1) / per);
  split_count_kernel<<<grid, 256, 0, s>>>(row_ptr, m, per, words, (int)(((long long)nnz + 31) / 32), counts);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (dtype == GBS_F64)
    return launch_dependent(split_number_kernel<double>, grid, 256, 0, s, row_ptr, m, per, words, ids, nonempty, empty,
                            counts, k, static_cast<double*>(Y), ldy);
  return launch_dependent(split_number_kernel<float>, grid, 256, 0, s, row_ptr, m, per, words, ids, nonempty, empty, counts,
                          k, static_cast<float*>(Y), ldy);
}

long long split_tiles(int nnz, int g, int share) {
  const long long per = (long long)(32 / g) * share;
  return std::max(1LL, (nnz + per - 1) / per);
}

}  // namespace gbs
