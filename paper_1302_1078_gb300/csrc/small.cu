// One-shot SpMV of a small matrix in one launch.
//
// Up to some ten thousand nonzeros a call is bound by its launches and allocations, not by the
// GPU: merge-path needs scratch and three kernels.  Here L lanes take a row (L from the mean row
// length, which the host knows), and a row much longer than that is left to the whole CTA, so that
// no row length needs statistics or a second kernel; a CTA that owned every nonzero of the largest
// matrix sent here would take about as long as merge-path's launches.  64 x 64 grid, 20,224
// nonzeros: 23.9 -> 14.8 us a call (the C call alone 4 us).
#include <algorithm>

#include "device_common.cuh"
#include "gbspmv.h"
#include "launch.h"

namespace gbs {

constexpr int kSmallThreads = 512;

// The other lane's sum added to a's.  float: the lanes of a row hold a few products each, so most of
// the sum's roundings are made here: by TwoSum, both parts.
__device__ __forceinline__ void merge(Acc<double>& a, double s, double) { a.s += s; }
__device__ __forceinline__ void merge(Acc<float>& a, float s, float c) {
  a.add_partial(s);
  a.c = __fadd_rn(a.c, c);
}
__device__ __forceinline__ void tree_add(Acc<double>& a, int o) { merge(a, __shfl_xor_sync(0xffffffffu, a.s, o), 0.0); }
__device__ __forceinline__ void tree_add(Acc<float>& a, int o) {
  const float s = __shfl_xor_sync(0xffffffffu, a.s, o), c = __shfl_xor_sync(0xffffffffu, a.c, o);
  merge(a, s, c);
}

// Products of nonzeros p, p + step, ... < e, four gathers in flight.
template <typename T>
__device__ __forceinline__ Acc<T> small_walk(const int* __restrict__ ci, const T* __restrict__ v,
                                             const T* __restrict__ x, int p, int e, int step) {
  Acc<T> acc;
  for (; p < e; p += 4 * step) {
    T a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = p + u * step;
      a[u] = b[u] = T(0);
      if (q < e) {
        a[u] = __ldg(v + q);
        b[u] = __ldg(x + __ldg(ci + q));
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (p + u * step < e) acc.add(a[u], b[u]);
  }
  return acc;
}

template <typename T, int L>
__global__ void __launch_bounds__(kSmallThreads) small_spmv_kernel(int m, const int* __restrict__ rp,
                                                                   const int* __restrict__ ci, const T* __restrict__ v,
                                                                   const T* __restrict__ x, T* __restrict__ y) {
  constexpr int R = kSmallThreads / L, LONG = 64 * L;
  __shared__ int long_rows[R];
  __shared__ int nlong;
  __shared__ T part_s[kSmallThreads / 32], part_c[kSmallThreads / 32];  // part_c: floats only
  if (threadIdx.x == 0) nlong = 0;
  __syncthreads();
  const int lane = threadIdx.x % L, row = blockIdx.x * R + threadIdx.x / L;
  int s = 0, e = 0;
  if (row < m) {
    s = __ldg(rp + row);
    e = __ldg(rp + row + 1);
  }
  const bool is_long = e - s > LONG;
  if (is_long && lane == 0) long_rows[atomicAdd(&nlong, 1)] = row;  // in any order: each row is summed by itself
  Acc<T> acc = small_walk<T>(ci, v, x, is_long ? e : s + lane, e, L);
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) tree_add(acc, o);
  if (row < m && lane == 0 && !is_long) y[row] = acc.value();
  __syncthreads();
  for (int i = 0; i < nlong; ++i) {
    const int r = long_rows[i];
    Acc<T> a = small_walk<T>(ci, v, x, __ldg(rp + r) + threadIdx.x, __ldg(rp + r + 1), kSmallThreads);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tree_add(a, o);
    if ((threadIdx.x & 31) == 0) {
      part_s[threadIdx.x >> 5] = a.s;
      if constexpr (sizeof(T) == 4) part_c[threadIdx.x >> 5] = a.c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kSmallThreads / 32; ++w) merge(a, part_s[w], sizeof(T) == 4 ? part_c[w] : T(0));
      y[r] = a.value();
    }
    __syncthreads();
  }
}

template <typename T>
static cudaError_t small_t(const CsrView& A, const void* x, void* y, cudaStream_t s) {
  const T* v = static_cast<const T*>(A.vals);
  const T* xx = static_cast<const T*>(x);
  T* yy = static_cast<T*>(y);
  int l = 1;  // about two nonzeros per lane of a mean row
  while (l < 32 && 2LL * l * A.m < A.nnz) l <<= 1;
  const int rows = kSmallThreads / l;
  const unsigned grid = (unsigned)(((long long)A.m + rows - 1) / rows);
  auto go = [&](auto kernel) {
    kernel<<<grid, kSmallThreads, 0, s>>>(A.m, A.row_ptr, A.col_idx, v, xx, yy);
    return cudaGetLastError();
  };
  switch (l) {
    case 1: return go(small_spmv_kernel<T, 1>);
    case 2: return go(small_spmv_kernel<T, 2>);
    case 4: return go(small_spmv_kernel<T, 4>);
    case 8: return go(small_spmv_kernel<T, 8>);
    case 16: return go(small_spmv_kernel<T, 16>);
    default: return go(small_spmv_kernel<T, 32>);
  }
}

cudaError_t launch_small_spmv(int dtype, const CsrView& A, const void* x, void* y, cudaStream_t s) {
  return dtype == GBS_F64 ? small_t<double>(A, x, y, s) : small_t<float>(A, x, y, s);
}

}  // namespace gbs
