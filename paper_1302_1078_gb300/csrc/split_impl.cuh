// Template launchers of the SPLIT variant, instantiated once per dtype (split_f64.cu, split_f32.cu).
#pragma once
#include "launch_impl.cuh"
#include "split_kernel.cuh"

namespace gbs {

template <typename T, bool PERM>
static cudaError_t split_spmv_go(const SplitArgs<T>& a, int grid, int threads, cudaStream_t s) {
  static L1Split split;
  const cudaError_t e = prefer_l1(split_spmv_kernel<T, PERM>, threads, 0, split);
  if (e != cudaSuccess) return e;
  return launch_dependent(split_spmv_kernel<T, PERM>, grid, threads, 0, s, a);
}

template <typename T, int VEC, int G, bool PERM>
static cudaError_t split_spmm_go(const SplitArgs<T>& a, int grid, int threads, cudaStream_t s) {
  static L1Split split;
  const cudaError_t e = prefer_l1(split_spmm_kernel<T, VEC, G, PERM>, threads, 0, split);
  if (e != cudaSuccess) return e;
  return launch_dependent(split_spmm_kernel<T, VEC, G, PERM>, grid, threads, 0, s, a);
}

template <typename T, int VEC, bool PERM>
static cudaError_t split_spmm_g(const SplitArgs<T>& a, int g, int grid, int threads, cudaStream_t s) {
  switch (g) {
    case 1: return split_spmm_go<T, VEC, 1, PERM>(a, grid, threads, s);
    case 2: return split_spmm_go<T, VEC, 2, PERM>(a, grid, threads, s);
    case 4: return split_spmm_go<T, VEC, 4, PERM>(a, grid, threads, s);
    case 8: return split_spmm_go<T, VEC, 8, PERM>(a, grid, threads, s);
    case 16: return split_spmm_go<T, VEC, 16, PERM>(a, grid, threads, s);
    case 32: return split_spmm_go<T, VEC, 32, PERM>(a, grid, threads, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, bool PERM>
static cudaError_t split_dispatch(SplitArgs<T>& a, bool vec16, int threads, int share, cudaStream_t s) {
  constexpr int V = 16 / (int)sizeof(T);
  const bool spmv = a.k == 1 && a.ldx == 1 && a.ldy == 1;
  int g = 1;
  if (spmv) {
    share = kSplitShare;
  } else {
    while (g < 32 && g * (vec16 && a.k > 1 ? V : 1) < a.k) g <<= 1;
    if (share % 32) share = 32;
  }
  a.share = share;
  a.tiles = (int)split_tiles(a.nnz, g, share);
  const int grid = (int)((a.tiles * 32LL + threads - 1) / threads);
  if (spmv) return split_spmv_go<T, PERM>(a, grid, threads, s);
  if (vec16 && a.k > 1) return split_spmm_g<T, V, PERM>(a, g, grid, threads, s);
  return split_spmm_g<T, 1, PERM>(a, g, grid, threads, s);
}

template <typename T>
cudaError_t launch_split_t(const CsrView& A, const SplitIndex& I, const DenseView& D, bool vec16, int threads,
                           int share, const SplitScratch& S, cudaStream_t s) {
  if (A.m == 0) return cudaSuccess;
  SplitArgs<T> a;
  a.m = A.m;
  a.k = D.k;
  a.nnz = A.nnz;
  a.col_idx = A.col_idx;
  a.vals = static_cast<const T*>(A.vals);
  a.perm = A.perm;
  a.X = static_cast<const T*>(D.X);
  a.Y = static_cast<T*>(D.Y);
  a.ldx = D.ldx;
  a.ldy = D.ldy;
  a.words = I.words;
  a.nwords = (int)(((long long)A.nnz + 31) / 32);
  a.ids = I.ids;
  a.nonempty = I.nonempty;
  a.carry_row = S.carry_row;
  a.carry_val = static_cast<T*>(S.carry_val);
  const void* v = A.perm ? static_cast<const void*>(A.perm) : A.vals;
  a.wide = ((reinterpret_cast<uintptr_t>(v) | reinterpret_cast<uintptr_t>(A.col_idx)) & 31) == 0;
  a.tiles = 0;
  if (A.nnz > 0) {
    const cudaError_t e = A.perm ? split_dispatch<T, true>(a, vec16, threads, share, s)
                                 : split_dispatch<T, false>(a, vec16, threads, share, s);
    if (e != cudaSuccess) return e;
  }
  if (a.tiles <= 1 && I.nempty == 0) return cudaSuccess;
  const int lg = split_fixup_lg(a.k);
  const long long carry_blocks = (((long long)a.tiles << lg) + 255) >> 8, empty_blocks = (((long long)I.nempty << lg) + 255) >> 8;
  return launch_dependent(split_fixup_kernel<T>, (unsigned)(carry_blocks + empty_blocks), 256, 0, s, a.tiles, a.k, lg,
                          a.carry_row, a.carry_val, a.Y, a.ldy, I.empty, I.nempty, (int)carry_blocks);
}

}  // namespace gbs
