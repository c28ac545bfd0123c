// Batched mode: many CSR products in one persistent launch.
//
// The paper multiplies one matrix at a time (Sec. 4, Sec. 5).  Serving many
// small and uneven matrices one launch each leaves most of GB300's 152 SMs idle
// for the small ones and pays a launch per matrix.  Here one persistent kernel
// walks a work list of (matrix, row block | merge tile) items.  A CTA takes the
// next unclaimed item from a device counter (reset by the graph before every
// launch), so the SMs stay busy until the list is exhausted whatever the items'
// costs; the matrix comes from a binary search of the descriptors' first items
// (a CTA's items only increase, so the search starts at its previous matrix),
// and each item runs exactly the device function the standalone kernels run
// (rows_block / split_spmv_tile / split_spmm_tile) with the matrix's own
// configuration, so the batched result equals the per-matrix loop bitwise:
// which CTA runs an item does not change what the item computes.
//
// A MERGE matrix runs as the nonzero-split walk (split_kernel.cuh): every warp
// takes a tile, without shared memory or barriers, and a second, small node of
// the graph adds every matrix's carries and writes the empty rows' zeros.  (With
// the fix-up in the kernel, by the CTA that retired a matrix's last item, the
// largest matrices' carries were a serial tail: 2.2 ms for 128 matrices of
// k = 8.)  On that batch the staged merge-path tiles this replaced, with three
// barriers and 54 KB of staging each, kept the FP64 pipe 81% busy:
// 1776 -> 1564 us.
#include <cstdint>

#include "batched.cuh"
#include "gbspmv.h"
#include "launch.h"
#include "rows_kernel.cuh"
#include "split_kernel.cuh"

namespace gbs {

// Resident CTAs of the batched kernel: the nonzero-split walk wants 80 registers (three CTAs), and
// 64 cost it 60 bytes of spill, but a fourth CTA is worth more (128 matrices, k = 8: 1.69 and 1.61 ms).
constexpr int kBatchCtas = 4;

template <typename T>
__device__ __forceinline__ RowsArgs<T> rows_args(const BatchDesc<T>& d) {
  RowsArgs<T> a;
  a.m = d.m;
  a.k = d.k;
  a.row_ptr = d.row_ptr;
  a.col_idx = d.col_idx;
  a.vals = d.vals;
  a.X = d.X;
  a.Y = d.Y;
  a.ldx = d.ldx;
  a.ldy = d.ldy;
  a.tile = d.tile;
  a.row_base = 0;
  a.aligned_vals = d.aligned_vals;
  a.aligned_cols = d.aligned_cols;
  return a;
}

template <typename T>
__device__ __forceinline__ SplitArgs<T> split_args(const BatchDesc<T>& d) {
  SplitArgs<T> a;
  a.m = d.m;
  a.k = d.k;
  a.nnz = d.nnz;
  a.col_idx = d.col_idx;
  a.vals = d.vals;
  a.perm = nullptr;
  a.X = d.X;
  a.Y = d.Y;
  a.ldx = d.ldx;
  a.ldy = d.ldy;
  a.words = d.words;
  a.nwords = (int)(((long long)d.nnz + 31) / 32);
  a.ids = d.ids;
  a.nonempty = nullptr;
  a.share = d.share;
  a.tiles = d.tiles;
  a.carry_row = d.carry_row;
  a.carry_val = d.carry_val;
  a.wide = d.wide != 0;
  return a;
}

// SPLIT (k == 1): ROWS lanes vary per matrix.  !SPLIT (k > 1): every matrix uses G column lanes.
// (ROWS_DIRECT items are not offered: they lost every whole-batch policy, and their code cost this
// register-bound kernel spills.)
template <typename T, int VEC, bool SPLIT, int G>
__global__ void __launch_bounds__(256, kBatchCtas) batched_kernel(const BatchDesc<T>* __restrict__ descs, int nmat,
                                                      int total_items, int* __restrict__ next_item) {
  __shared__ int s_item;
  int lo = 0;  // matrix of this CTA's previous item
  // items are claimed one ahead: the claim of the next item is issued when the current one
  // starts, so the atomic's round trip overlaps the current item's work
  if (threadIdx.x == 0) s_item = atomicAdd(next_item, 1);
  __syncthreads();
  for (;;) {
    const int item = s_item;
    if (item >= total_items) break;
    int claimed = 0;
    if (threadIdx.x == 0) claimed = atomicAdd(next_item, 1);
    int hi = nmat - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(&descs[mid].item_begin) <= item)
        lo = mid;
      else
        hi = mid - 1;
    }
    const BatchDesc<T> d = descs[lo];
    const int local = item - d.item_begin;
    if (d.variant == GBS_VARIANT_ROWS) {
      const RowsArgs<T> a = rows_args(d);
      if constexpr (SPLIT) {
        switch (d.lanes) {
          case 1: rows_block<T, 1, 1, true>(a, local); break;
          case 2: rows_block<T, 1, 2, true>(a, local); break;
          case 4: rows_block<T, 1, 4, true>(a, local); break;
          case 8: rows_block<T, 1, 8, true>(a, local); break;
          case 16: rows_block<T, 1, 16, true>(a, local); break;
          default: rows_block<T, 1, 32, true>(a, local); break;
        }
      } else {
        rows_block<T, VEC, G, false>(a, local);
      }
    } else {
      const SplitArgs<T> a = split_args(d);
      const int per = batch_item_tiles(d.k);
      const int t1 = min(a.tiles, (local + 1) * per);
      for (int t = local * per + ((int)threadIdx.x >> 5); t < t1; t += 8) {
        if constexpr (SPLIT)
          split_spmv_tile<T, false>(a, t);
        else
          split_spmm_tile<T, VEC, G, false>(a, t);
      }
    }
    // the next item's index is published, and a ROWS item's shared memory handed over, with one
    // barrier after the item and one before the next (a MERGE item has none of its own)
    __syncthreads();
    if (threadIdx.x == 0) s_item = claimed;
    __syncthreads();
  }
}

// The carries and the empty rows of every MERGE matrix, as split_fixup_kernel for each: block b
// belongs to the last matrix whose fix_begin is at most b (ROWS matrices have no blocks).
template <typename T>
__global__ void __launch_bounds__(256) batched_fixup_kernel(const BatchDesc<T>* __restrict__ descs, int nmat) {
  int lo = 0, hi = nmat - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(&descs[mid].fix_begin) <= (int)blockIdx.x)
      lo = mid;
    else
      hi = mid - 1;
  }
  const BatchDesc<T>& d = descs[lo];
  const int lg = split_fixup_lg(d.k), sub = threadIdx.x & ((1 << lg) - 1), local = (int)blockIdx.x - d.fix_begin;
  if (local >= d.fix_carry_blocks) {
    split_zero_row<T>((((long long)local - d.fix_carry_blocks) * 256 + threadIdx.x) >> lg, d.k, lg, sub, d.empty, d.nempty,
                      d.Y, d.ldy);
    return;
  }
  const long long b = ((long long)local * 256 + threadIdx.x) >> lg;
  split_fixup_tile<T>(b < d.tiles ? (int)b : d.tiles, d.tiles, d.k, lg, sub, d.carry_row, d.carry_val, d.Y, d.ldy);
}

cudaError_t batched_fixup(int dtype, const void* descs, int nmat, int blocks, cudaStream_t s) {
  if (blocks <= 0) return cudaSuccess;
  if (dtype == GBS_F64)
    batched_fixup_kernel<double><<<blocks, 256, 0, s>>>(static_cast<const BatchDesc<double>*>(descs), nmat);
  else
    batched_fixup_kernel<float><<<blocks, 256, 0, s>>>(static_cast<const BatchDesc<float>*>(descs), nmat);
  return cudaGetLastError();
}

template <typename T, int VEC, bool SPLIT, int G>
static cudaError_t batched_go(bool launch, const void* descs, int nmat, int total_items, int* next_item, int grid,
                              size_t smem, int* blocks_per_sm, cudaStream_t s) {
  auto kern = batched_kernel<T, VEC, SPLIT, G>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (!launch) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kern, 256, smem);
  kern<<<grid, 256, smem, s>>>(static_cast<const BatchDesc<T>*>(descs), nmat, total_items, next_item);
  return cudaGetLastError();
}

template <typename T, int VEC>
static cudaError_t batched_g(bool launch, bool split, int G, const void* descs, int nmat, int total_items,
                             int* next_item, int grid, size_t smem, int* bps, cudaStream_t s) {
  if (split) return batched_go<T, 1, true, 1>(launch, descs, nmat, total_items, next_item, grid, smem, bps, s);
  switch (G) {
    case 1: return batched_go<T, VEC, false, 1>(launch, descs, nmat, total_items, next_item, grid, smem, bps, s);
    case 2: return batched_go<T, VEC, false, 2>(launch, descs, nmat, total_items, next_item, grid, smem, bps, s);
    case 4: return batched_go<T, VEC, false, 4>(launch, descs, nmat, total_items, next_item, grid, smem, bps, s);
    case 8: return batched_go<T, VEC, false, 8>(launch, descs, nmat, total_items, next_item, grid, smem, bps, s);
    case 16: return batched_go<T, VEC, false, 16>(launch, descs, nmat, total_items, next_item, grid, smem, bps, s);
    case 32: return batched_go<T, VEC, false, 32>(launch, descs, nmat, total_items, next_item, grid, smem, bps, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t batched_kernel_call(bool launch, int dtype, bool split, int G, bool vec16, const void* descs, int nmat,
                                int total_items, int* next_item, int grid, size_t smem, int* blocks_per_sm,
                                cudaStream_t s) {
  if (dtype == GBS_F64)
    return vec16 ? batched_g<double, 2>(launch, split, G, descs, nmat, total_items, next_item, grid, smem,
                                        blocks_per_sm, s)
                 : batched_g<double, 1>(launch, split, G, descs, nmat, total_items, next_item, grid, smem,
                                        blocks_per_sm, s);
  return vec16 ? batched_g<float, 4>(launch, split, G, descs, nmat, total_items, next_item, grid, smem, blocks_per_sm,
                                     s)
               : batched_g<float, 1>(launch, split, G, descs, nmat, total_items, next_item, grid, smem, blocks_per_sm,
                                     s);
}

}  // namespace gbs
