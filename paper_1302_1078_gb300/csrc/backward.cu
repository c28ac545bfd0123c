// Backward pass of Y = A X with respect to the stored values (the paper has
// no backward pass): the sampled dense-dense product over A's pattern
//   dvals[p] = sum_c dY[row(p), c] * X[col_idx[p], c].
// Each nonzero's k products are summed by one lane in column order, so no FP64 reduction across lanes
// is needed (on GB300 every FP64 instruction counts).  The rows come from A's SPLIT index
// (split_kernel.cuh; 8 bytes per 32 nonzeros where a stored row per nonzero is 128).  What bounds the
// pass is the L1 lookups of the gathered rows of X and dY and the loads in flight, and which of two
// layouts serves that better depends on how many slices a row takes (sddmm_t):
//   - sddmm_kernel: a lane takes 8 consecutive nonzeros, knows where its row changes and reads a slice of
//     dY once per row; the column ids arrive and the results leave in whole 32-byte sectors, and an X row
//     is gathered in slices of 32 bytes.  Best where a row is a slice or a few, or the slices are wide
//     and many: R-MAT 20, FP32, k = 4 and 8: 95 -> 72 and 123 -> 94 us, FP64, k = 16: 497 -> 433 us.  It
//     holds 256 rows of X per warp between two slices, more than L1 keeps if the slices are narrow and many.
//   - sddmm_lane_kernel: a warp takes 32 consecutive nonzeros, two such groups at a time, whose dY rows are
//     the same few lines; the ids and rows of the next two groups are fetched before the sums.  R-MAT 20,
//     k = 13, odd rows: FP64 633 us in the other layout, 473 in this one; FP32 582 and 345.
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
  if constexpr (VEC * sizeof(T) == 32)
    if (c0 + VEC / 2 <= k) {
      columns(c0, std::integral_constant<int, VEC / 2>{});
      c0 += VEC / 2;
    }
  if constexpr (!K1 && !(sizeof(T) == 4 && VEC != 4)) {
    for (; c0 < k; ++c0) columns(c0, std::integral_constant<int, 1>{});
  } else if constexpr (!K1) {
    // single columns: all that are left of two nonzeros before the next two, so that an X row's lines are
    // used up while they are in L1 (k = 13 in rows of 16 floats, R-MAT 20: 323 -> 197 us; the other
    // instances have no registers for it)
    if (c0 < k) {
#pragma unroll
      for (int h = 0; h < 8; h += 2) {
        const bool in[2] = {c[h] >= 0, c[h + 1] >= 0}, same = row[h + 1] == row[h];
        const T *xr[2], *yr[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          xr[u] = X + (uint64_t)(uint32_t)max(c[h + u], 0) * (uint32_t)ldx;
          yr[u] = dY + (uint64_t)(uint32_t)row[h + u] * (uint32_t)lddy;
        }
        auto part = [&](int q, auto width) {
          constexpr int V = decltype(width)::value;
          T x[2][V], y[2][V];
#pragma unroll
          for (int j = 0; j < V; ++j) {
            if (in[0]) x[0][j] = ld_keep(xr[0] + q + j, pol_keep);
            if (in[1]) x[1][j] = ld_keep(xr[1] + q + j, pol_keep);
            y[0][j] = ld_keep(yr[0] + q + j, pol_keep);
          }
#pragma unroll
          for (int j = 0; j < V; ++j) {
            y[1][j] = y[0][j];
            if (!same) y[1][j] = ld_keep(yr[1] + q + j, pol_keep);
          }
#pragma unroll
          for (int j = 0; j < V; ++j) {
            if (in[0]) acc[h].add(y[0][j], x[0][j]);
            if (in[1]) acc[h + 1].add(y[1][j], x[1][j]);
          }
        };
        constexpr int CH = VEC == 1 ? 2 : 1;
        int q = c0;
        for (; q + CH <= k; q += CH) part(q, std::integral_constant<int, CH>{});
        for (; q < k; ++q) part(q, std::integral_constant<int, 1>{});
      }
    }
  }
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

// FEW: a few single columns (few registers, many warps); else as many loads in flight as four CTAs
// leave registers for.
template <typename T, int VEC, bool FEW>
__global__ void __launch_bounds__(256, FEW ? 6 : 4) sddmm_lane_kernel(int nnz, int k, const SplitWord* __restrict__ words,
                                                         const int* __restrict__ ids_in, const int* __restrict__ nonempty,
                                                         int m, const int* __restrict__ col_idx, const T* __restrict__ X,
                                                         long long ldx, const T* __restrict__ dY, long long lddy,
                                                         T* __restrict__ dvals) {
  constexpr int U = 2, VU = 2, SU = FEW ? 1 : 4;
  const uint64_t pol_keep = policy_evict_last(), pol_stream = policy_evict_first();
  const int* __restrict__ ids = nonempty && __ldg(nonempty) == m ? nullptr : ids_in;
  const int lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u, lx = (uint32_t)ldx, ly = (uint32_t)lddy;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long step = ((long long)gridDim.x * blockDim.x >> 5) * 32 * U;
  uint32_t col_next[U], row_next[U];
  auto fetch = [&](long long base) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long p = base + 32 * u + lane;
      col_next[u] = row_next[u] = 0;  // (past the end: the first rows of X and dY, whose sum is not stored)
      if (p < nnz) {
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(words) + (p >> 5));
        col_next[u] = (uint32_t)ld_stream(col_idx + p, pol_stream);
        row_next[u] = (uint32_t)split_row(ids, (int)w.y + __popc(w.x & below));
      }
    }
  };
  long long base = warp * 32 * U;
  fetch(base);
  for (; base < nnz; base += step) {
    uint32_t col[U], row[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      col[u] = col_next[u];
      row[u] = row_next[u];
    }
    fetch(base + step);
    Acc<T> acc[U];
    int c = 0;
    if constexpr (VEC > 1) {
#pragma unroll VU
      for (; c + VEC <= k; c += VEC) {
        Vec<T, VEC> x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          x[u] = ld_keep_vec<T, VEC>(X + (uint64_t)col[u] * lx + c, pol_keep);
          y[u] = ld_keep_vec<T, VEC>(dY + (uint64_t)row[u] * ly + c, pol_keep);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int j = 0; j < VEC; ++j) acc[u].add(y[u].v[j], x[u].v[j]);
      }
    }
#pragma unroll SU
    for (; c < k; ++c) {
      T x[U], y[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        x[u] = ld_keep(X + (uint64_t)col[u] * lx + c, pol_keep);
        y[u] = ld_keep(dY + (uint64_t)row[u] * ly + c, pol_keep);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) acc[u].add(y[u], x[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (base + 32 * u + lane < nnz) st_stream(dvals + base + 32 * u + lane, acc[u].value());
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
  auto go_lanes = [&](auto kernel) {
    const unsigned ctas = (unsigned)std::min<long long>(152LL * 16, ((long long)nnz + 511) / 512);
    kernel<<<ctas, 256, 0, s>>>(nnz, k, I.words, I.ids, I.nonempty, m, col_idx, x, ldx, dy, lddy, dv);
    return cudaGetLastError();
  };
  // Rows of fewer than six nonzeros change inside nearly every lane's eight (5-point 1000^2, sddmm_kernel
  // and sddmm_lane_kernel: FP64 k = 16 181 and 158 us, FP32 74 and 66; with six in a row 155 and 168, 70
  // and 74), up to four slices of 32 bytes: FP32 k = 32 133 and 157.
  const bool short_rows = nnz < 6LL * m;
  if constexpr (sizeof(T) == 8) {
    // one 16-byte slice: banded 200,003 x 41, k = 2 36 and 45 us; k = 4 66 and 66, 12 175 and 170, 16 230 and
    // 256; k = 8 R-MAT 20 (15 in a row) 227 and 235, banded 500,000 x 9 76 and 71
    if (k < 4 && k >= H && all % 16 == 0) return go(sddmm_kernel<T, H, false>);
    if (all % 32 == 0 && (k > 12 ? !short_rows : k == 8 && nnz >= 12LL * m)) return go(sddmm_kernel<T, W, false>);
    if (k >= H && all % 16 == 0) return go_lanes(sddmm_lane_kernel<T, H, false>);
    // single columns; registers for more loads from k = 8 (banded 500,000 x 9: k = 5 51 and 51 us, k = 3
    // 34 and 35, k = 13 135 and 124)
    return k < 8 ? go_lanes(sddmm_lane_kernel<T, 1, true>) : go_lanes(sddmm_lane_kernel<T, 1, false>);
  } else {
    if (k >= W && all % 32 == 0 && !(short_rows && k > W && k < 4 * W)) return go(sddmm_kernel<T, W, false>);
    // one 16-byte slice or a few single columns: R-MAT 20, k = 4 72 and 81 us, k = 3 101 and 108; k = 12 167 and
    // 160; 5-point 1000^2, k = 5, single columns, 33 and 29 us
    if (k == H && all % 16 == 0) return go(sddmm_kernel<T, H, false>);
    if (k >= H && all % 16 == 0) return go_lanes(sddmm_lane_kernel<T, H, false>);
    return k < H && !(short_rows && k > 2) ? go(sddmm_kernel<T, 1, false>) : go_lanes(sddmm_lane_kernel<T, 1, false>);
  }
}

cudaError_t launch_sddmm(int dtype, int nnz, int k, const SplitIndex& I, int m, const int* col_idx, const void* X,
                         long long ldx, const void* dY, long long lddy, void* dvals, cudaStream_t s) {
  return dtype == GBS_F64 ? sddmm_t<double>(nnz, k, I, m, col_idx, X, ldx, dY, lddy, dvals, s)
                          : sddmm_t<float>(nnz, k, I, m, col_idx, X, ldx, dY, lddy, dvals, s);
}

}  // namespace gbs
