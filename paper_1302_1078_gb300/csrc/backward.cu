// Backward pass of Y = A X with respect to the stored values (the paper has
// no backward pass): the sampled dense-dense product over A's pattern
//   dvals[p] = sum_c dY[row(p), c] * X[col_idx[p], c].
// Every lane takes 8 consecutive nonzeros and sums each one's k products in column order, so no
// FP64 reduction across lanes is needed (on GB300 every FP64 instruction counts).  The rows come
// from A's SPLIT index (split_kernel.cuh; 8 bytes per 32 nonzeros where a stored row per nonzero
// is 128), so a lane knows where its row changes and reads a slice of dY once per row, not once
// per nonzero; the column ids arrive and the results leave in whole 32-byte sectors, and an X row
// is gathered in slices of 32 bytes.  What bounds it is the L1 lookups of those gathers, one per
// slice and nonzero (128-bit slices take two, and a dY slice per nonzero as many again): R-MAT 20,
// FP32, k = 4 and 8: 95 -> 69 and 123 -> 94 us, FP64, k = 8: 250 -> 228 us (the FP64 pipe needs
// 200); k = 1 is the same 64 us, its row numbers' loads costing what the stored rows' did.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "device_common.cuh"
#include "gbspmv.h"
#include "launch.h"
#include "split_kernel.cuh"

namespace gbs {

// VEC consecutive elements of a gathered row: 32 bytes, 16 bytes or one element.
template <typename T, int VEC>
__device__ __forceinline__ void ld_slice(const T* p, uint64_t pol, T* v) {
  if constexpr (VEC * sizeof(T) == 32 && sizeof(T) == 8) {
    asm volatile("ld.global.nc.L2::cache_hint.v4.f64 {%0,%1,%2,%3}, [%4], %5;"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                 : "l"(p), "l"(pol));
  } else if constexpr (VEC * sizeof(T) == 32) {
    asm volatile("ld.global.nc.L2::cache_hint.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p), "l"(pol));
  } else {
    const Vec<T, VEC> r = ld_keep_vec<T, VEC>(p, pol);
#pragma unroll
    for (int j = 0; j < VEC; ++j) v[j] = r.v[j];
  }
}

// K1: k == 1 with contiguous X and dY.
template <typename T, int VEC, bool K1>
__global__ void __launch_bounds__(128, K1 ? 10 : VEC * sizeof(T) == 32 ? 6 : 8) sddmm_kernel(int nnz, int k, const SplitWord* __restrict__ words,
                                                    const int* __restrict__ ids_in, const int* __restrict__ nonempty,
                                                    int m, const int* __restrict__ col_idx, const T* __restrict__ X,
                                                    long long ldx, const T* __restrict__ dY, long long lddy,
                                                    T* __restrict__ dvals, bool wide_cols, bool wide_out) {
  const uint64_t pol_keep = policy_evict_last(), pol_stream = policy_evict_first();
  const long long p0 = 8 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (p0 >= nnz) return;
  const int p = (int)p0, cnt = min(8, nnz - p);
  const int* __restrict__ ids = nonempty && __ldg(nonempty) == m ? nullptr : ids_in;
  const uint2 w = __ldg(reinterpret_cast<const uint2*>(words) + (p >> 5));
  const uint32_t ends = (w.x >> (p & 31)) & 0xffu;
  const int ord0 = (int)w.y + __popc(w.x & ((1u << (p & 31)) - 1u));
  int c[8];
  if (wide_cols && cnt == 8) {
    uint32_t q[8];
    ld_stream_8w(col_idx + p, pol_stream, q);
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = (int)q[u];
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = u < cnt ? ld_stream(col_idx + p + u, pol_stream) : -1;
  }
  // the row of every nonzero, fetched together: a row's number or its dY slice fetched only when
  // the walk reaches it would put two round trips into every row change
  int row[8];
  row[0] = split_row(ids, ord0);
#pragma unroll
  for (int u = 1; u < 8; ++u) {
    row[u] = row[u - 1];
    if ((ends >> (u - 1) & 1u) && u < cnt) row[u] = split_row(ids, ord0 + __popc(ends & ((1u << u) - 1u)));
  }
  Acc<T> acc[8];
  if constexpr (K1) {
    T x[8], y[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (c[u] >= 0) x[u] = ld_keep(X + c[u], pol_keep);
    y[0] = ld_keep(dY + row[0], pol_keep);
#pragma unroll
    for (int u = 1; u < 8; ++u) {
      y[u] = y[u - 1];
      if (row[u] != row[u - 1]) y[u] = ld_keep(dY + row[u], pol_keep);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (c[u] >= 0) acc[u].add(y[u], x[u]);
  }
  auto columns = [&](int c0, auto width) {
    constexpr int V = decltype(width)::value, H = V * sizeof(T) == 32 ? 2 : 4;  // X slices in flight
    T y[V];
    const T* __restrict__ yc = dY + c0;
#pragma unroll
    for (int h = 0; h < 8; h += H) {
      T x[H][V];
#pragma unroll
      for (int u = 0; u < H; ++u)
        if (c[h + u] >= 0) ld_slice<T, V>(X + c0 + (uint64_t)(uint32_t)c[h + u] * (uint32_t)ldx, pol_keep, x[u]);
#pragma unroll
      for (int u = 0; u < H; ++u) {
        if (h + u == 0 || row[h + u] != row[h + u - 1]) ld_slice<T, V>(yc + (uint64_t)(uint32_t)row[h + u] * (uint32_t)lddy, pol_keep, y);
        if (c[h + u] >= 0) {
#pragma unroll
          for (int j = 0; j < V; ++j) acc[h + u].add(y[j], x[u][j]);
        }
      }
    }
  };
  int c0 = 0;
  if constexpr (VEC > 1)
    for (; c0 + VEC <= k; c0 += VEC) columns(c0, std::integral_constant<int, VEC>{});
  if constexpr (!K1)
    for (; c0 < k; ++c0) columns(c0, std::integral_constant<int, 1>{});
  if (wide_out && cnt == 8) {
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int u = 0; u < 8; u += 4)
        asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(dvals + p + u), "d"(acc[u].value()),
                     "d"(acc[u + 1].value()), "d"(acc[u + 2].value()), "d"(acc[u + 3].value())
                     : "memory");
    } else {
      asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dvals + p), "f"(acc[0].value()),
                   "f"(acc[1].value()), "f"(acc[2].value()), "f"(acc[3].value()), "f"(acc[4].value()),
                   "f"(acc[5].value()), "f"(acc[6].value()), "f"(acc[7].value())
                   : "memory");
    }
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u < cnt) st_stream(dvals + p + u, acc[u].value());
  }
}

template <typename T>
static cudaError_t sddmm_t(int nnz, int k, const SplitIndex& I, int m, const int* col_idx, const void* X,
                           long long ldx, const void* dY, long long lddy, void* dvals, cudaStream_t s) {
  if (nnz == 0) return cudaSuccess;
  // the widest slice that X, dY and their leading dimensions allow: 32, 16 bytes or an element
  const long long es = sizeof(T);
  const unsigned long long all = reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(dY) |
                                 (unsigned long long)(ldx * es) | (unsigned long long)(lddy * es);
  const bool wide_cols = reinterpret_cast<uintptr_t>(col_idx) % 32 == 0;
  const bool wide_out = reinterpret_cast<uintptr_t>(dvals) % 32 == 0;
  const unsigned grid = (unsigned)((((long long)nnz + 7) / 8 + 127) / 128);
  const T* x = static_cast<const T*>(X);
  const T* dy = static_cast<const T*>(dY);
  T* dv = static_cast<T*>(dvals);
  constexpr int W = 32 / (int)sizeof(T), H = W / 2;
  auto go = [&](auto kernel) {
    kernel<<<grid, 128, 0, s>>>(nnz, k, I.words, I.ids, I.nonempty, m, col_idx, x, k == 1 ? 1 : ldx, dy,
                                k == 1 ? 1 : lddy, dv, wide_cols, wide_out);
    return cudaGetLastError();
  };
  if (k == 1) return go(sddmm_kernel<T, 1, true>);
  if (k >= W && all % 32 == 0) return go(sddmm_kernel<T, W, false>);
  if (k >= H && all % 16 == 0) return go(sddmm_kernel<T, H, false>);
  return go(sddmm_kernel<T, 1, false>);
}

cudaError_t launch_sddmm(int dtype, int nnz, int k, const SplitIndex& I, int m, const int* col_idx, const void* X,
                         long long ldx, const void* dY, long long lddy, void* dvals, cudaStream_t s) {
  return dtype == GBS_F64 ? sddmm_t<double>(nnz, k, I, m, col_idx, X, ldx, dY, lddy, dvals, s)
                          : sddmm_t<float>(nnz, k, I, m, col_idx, X, ldx, dY, lddy, dvals, s);
}

}  // namespace gbs
