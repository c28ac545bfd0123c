// Deterministic CSR transpose (the CRS of A^T, i.e. the CCS of A: Sec. 3
// notes that the two formats are dual) and the transpose plan used by the
// backward pass.
//
// The nonzeros are stably sorted by column id with an LSD radix sort whose
// values are the original positions; the stable order inside each column of A
// is therefore the order of storage, exactly as a counting sort gives it.
// Digits are at most 9 bits wide, the ids' bits shared evenly between the
// passes (131,072 columns: two passes where 8-bit digits need three).  Every
// pass is:
//   1. per tile of 4096 keys, a digit histogram (shared memory);
//   2. an exclusive scan of the histograms in digit-major order;
//   3. a scatter in which each key's rank among equal digits of its tile is
//      computed in position order (warp match + popcount, then a per-digit
//      prefix over warps), so no atomic decides any output position.  The
//      tile is put in order in shared memory first, so that a warp's stores
//      go to a few runs of consecutive positions and not to 32 (the scattered
//      stores were most of the pass: the transpose of 1.9 M nonzeros 219 -> 155 us).
// The first pass takes the positions from the index, the last writes perm.
// row_ptr of A^T comes from the boundaries of the sorted keys, col_idx of
// A^T by gathering the row of each sorted nonzero.  All of it is integer
// work and bit-exact.
#include <algorithm>
#include <cstdint>
#include <string>

#include "gbspmv.h"
#include "launch.h"

namespace gbs {

constexpr int kSortThreads = 512;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;  // 4096 keys per tile
constexpr int kSortBits = 9;                          // widest digit (at most one digit per thread)

// Row of every nonzero: one warp per row writes the row id over its range.
__global__ void expand_rows_kernel(const int* __restrict__ row_ptr, int m, int* __restrict__ rows) {
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = warp; i < m; i += nwarps) {
    const int s = row_ptr[i], e = row_ptr[i + 1];
    for (int p = s + lane; p < e; p += 32) rows[p] = (int)i;
  }
}

__global__ void __launch_bounds__(kSortThreads) radix_upsweep(const int* __restrict__ keys, int n, int shift, int bits,
                                                              int ntiles, int* __restrict__ hist) {
  __shared__ int h[1 << kSortBits];
  const int tile = blockIdx.x, nb = 1 << bits;
  if (threadIdx.x < nb) h[threadIdx.x] = 0;
  __syncthreads();
  const long long base = (long long)tile * kSortTile;
  for (int q = threadIdx.x; q < kSortTile; q += kSortThreads)
    if (base + q < n) atomicAdd(&h[(keys[base + q] >> shift) & (nb - 1)], 1);  // counts only: order-free
  __syncthreads();
  if (threadIdx.x < nb) hist[(size_t)threadIdx.x * ntiles + tile] = h[threadIdx.x];
}

// vals_in NULL: the values are the positions.
__global__ void __launch_bounds__(kSortThreads) radix_downsweep(const int* __restrict__ keys_in,
                                                                const int* __restrict__ vals_in,
                                                                int* __restrict__ keys_out, int* __restrict__ vals_out,
                                                                int n, int shift, int bits, int ntiles,
                                                                const int* __restrict__ offs) {
  constexpr int W = kSortThreads / 32, NB = 1 << kSortBits;
  __shared__ __align__(16) unsigned short wcnt[W][NB];  // a warp holds 256 keys
  __shared__ int start[NB], dest[NB];     // a digit's first place in the tile; that place's position in the output, less it
  __shared__ int wsum[W];
  __shared__ int s_key[kSortTile];
  static_assert(sizeof(wcnt) >= kSortTile * sizeof(int), "the values take the counts' place");
  int* s_val = reinterpret_cast<int*>(&wcnt[0][0]);
  const int tile = blockIdx.x, nb = 1 << bits;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = threadIdx.x; q < W * NB / 2; q += kSortThreads) reinterpret_cast<unsigned int*>(&wcnt[0][0])[q] = 0u;
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
  const long long base = (long long)tile * kSortTile;
  int key[kSortItems], dig[kSortItems], wr[kSortItems];
  // warp w owns the contiguous run [w*256, w*256 + 256) of the tile, 32 keys per round
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const long long idx = base + w * 256 + r * 32 + lane;
    const bool valid = idx < n;
    const int k = valid ? keys_in[idx] : 0;
    const int d = valid ? ((k >> shift) & (nb - 1)) : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, valid ? d : NB + lane);
    const int leader = __ffs(peers) - 1;
    const int before = valid ? wcnt[w][d] : 0;
    __syncwarp();
    if (valid && lane == leader) wcnt[w][d] = (unsigned short)(before + __popc(peers));
    __syncwarp();
    key[r] = k;
    dig[r] = d;
    wr[r] = before + __popc(peers & lt);
  }
  __syncthreads();
  // thread d: digit d's exclusive prefix over the warps (warp order = position order), then its
  // first place in the tile by a scan of the digits' totals
  int total = 0;
  const int d = threadIdx.x;
#pragma unroll
  for (int ww = 0; ww < W; ++ww) {
    const int t = wcnt[ww][d];
    wcnt[ww][d] = (unsigned short)total;
    total += t;
  }
  int inc = total;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  int first = inc - total;
  for (int ww = 0; ww < w; ++ww) first += wsum[ww];
  start[d] = first;
  dest[d] = (d < nb ? offs[(size_t)d * ntiles + tile] : 0) - first;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r)
    if (dig[r] >= 0) wr[r] += start[dig[r]] + wcnt[w][dig[r]];
  __syncthreads();  // the counts have been read
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    if (dig[r] >= 0) {
      const long long idx = base + w * 256 + r * 32 + lane;
      s_key[wr[r]] = key[r];
      s_val[wr[r]] = vals_in ? vals_in[idx] : (int)idx;
    }
  }
  __syncthreads();
  const int cnt = (int)min((long long)kSortTile, n - base);
  for (int i = threadIdx.x; i < cnt; i += kSortThreads) {
    const int k = s_key[i], dst = dest[(k >> shift) & (nb - 1)] + i;
    keys_out[dst] = k;
    vals_out[dst] = s_val[i];
  }
}

// row_ptr of A^T from the sorted column ids: rptrT[j] = first position whose key >= j.
__global__ void boundaries_kernel(const int* __restrict__ skeys, int nnz, int n, int* __restrict__ rptrT) {
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q <= nnz; q += (long long)gridDim.x * blockDim.x) {
    const int lo = q == 0 ? 0 : skeys[q - 1] + 1;  // first column starting at q
    const int hi = q == nnz ? n : skeys[q];         // last column starting at q
    for (int j = lo; j <= hi; ++j) rptrT[j] = q;
  }
}

__global__ void gather_int_kernel(const int* __restrict__ src, const int* __restrict__ idx, int n, int* __restrict__ out) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) out[i] = src[idx[i]];
}

// out[i] = row of nonzero idx[i], from the SPLIT index of A: a 16th of the bytes of a stored row per
// nonzero, which is neither written nor kept (index and gather take the 25-28 us of the stored rows
// on R-MAT 17).
__global__ void gather_rows_kernel(const SplitWord* __restrict__ words, const int* __restrict__ ids_in,
                                   const int* __restrict__ nonempty, int m, const int* __restrict__ idx, int n,
                                   int* __restrict__ out) {
  const int* __restrict__ ids = nonempty && *nonempty == m ? nullptr : ids_in;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int p = idx[i];
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(words) + (p >> 5));
    const int ord = (int)w.y + __popc(w.x & ((1u << (p & 31)) - 1u));
    out[i] = ids ? __ldg(ids + ord) : ord;
  }
}

template <typename T>
__global__ void gather_vals_kernel(const T* __restrict__ src, const int* __restrict__ idx, int n, T* __restrict__ out) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) out[i] = src[idx[i]];
}

static int grid_for(long long work, int threads = 256) {
  return (int)std::min<long long>(152LL * 32, std::max<long long>(1, (work + threads - 1) / threads));
}

// Stable LSD radix sort of n (key, value) pairs by the low `bits` bits of the keys (at least one
// pass); keys must be non-negative.  The passes write the a and b buffers in turn, beginning with b
// (keys / vals may be the a buffers; vals may be NULL, for the positions), except that the last one
// writes its values to `last_vals` if that is not NULL; *keys_out / *vals_out point at the result.
static cudaError_t radix_sort(int n, int bits, const int* keys, const int* vals, int* keys_a, int* keys_b, int* vals_a,
                              int* vals_b, int* last_vals, int* hist, int* scan_ws, int** keys_out, int** vals_out,
                              cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  const int ntiles = (int)(((long long)n + kSortTile - 1) / kSortTile);
  const int passes = std::max(1, (bits + kSortBits - 1) / kSortBits);
  const int width = std::max(1, (bits + passes - 1) / passes);
  const int* ki = keys;
  const int* vi = vals;
  int *ko = keys_b, *vo = vals_b;
  for (int p = 0; p < passes; ++p) {
    const int shift = p * width, b = std::max(1, std::min(width, bits - shift));
    int* out = p == passes - 1 && last_vals ? last_vals : vo;
    radix_upsweep<<<ntiles, kSortThreads, 0, s>>>(ki, n, shift, b, ntiles, hist);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = exclusive_scan_i32(hist, hist, (long long)ntiles << b, scan_ws, s)) != cudaSuccess) return e;
    radix_downsweep<<<ntiles, kSortThreads, 0, s>>>(ki, vi, ko, out, n, shift, b, ntiles, hist);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ki = ko;
    vi = out;
    *keys_out = ko;
    *vals_out = out;
    ko = ko == keys_b ? keys_a : keys_b;
    vo = vo == vals_b ? vals_a : vals_b;
  }
  return e;
}

// The same on keys_a / vals_a in place of given arrays.  hist and scan_ws as for the transpose
// (transpose_hist_ints(n), transpose_scan_ws_ints(n) ints).
cudaError_t radix_sort_pairs(int n, int bits, int* keys_a, int* keys_b, int* vals_a, int* vals_b, int* hist,
                             int* scan_ws, int** keys_out, int** vals_out, cudaStream_t s) {
  *keys_out = keys_a;
  *vals_out = vals_a;
  if (n <= 0 || bits <= 0) return cudaSuccess;
  return radix_sort(n, bits, keys_a, vals_a, keys_a, keys_b, vals_a, vals_b, nullptr, hist, scan_ws, keys_out, vals_out, s);
}

// Transpose with caller-provided device buffers (sizes: launch.h).
// Returns a CUDA error.  tmp must hold 2 * nnz + 2 * nnz ints + hist + scan workspace.
cudaError_t transpose_run(int m, int n, int nnz, const int* row_ptr, const int* col_idx, int* rptrT, int* colT,
                          int* perm, int* rows, int* keys_a, int* keys_b, int* vals_a, int* vals_b, int* hist,
                          int* scan_ws, cudaStream_t s, const SplitIndex* index) {
  cudaError_t e;
  if (m > 0 && nnz > 0 && !index) {
    expand_rows_kernel<<<grid_for((long long)m * 32), 256, 0, s>>>(row_ptr, m, rows);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (nnz == 0) {
    // every column of A^T is empty
    return cudaMemsetAsync(rptrT, 0, sizeof(int) * ((size_t)n + 1), s);
  }
  int bits = 0;
  while (bits < 31 && (1LL << bits) < (long long)n) ++bits;
  int *ki = nullptr, *vi = nullptr;
  if ((e = radix_sort(nnz, bits, col_idx, nullptr, keys_a, keys_b, vals_a, vals_b, perm, hist, scan_ws, &ki, &vi, s)) !=
      cudaSuccess)
    return e;
  // ki: sorted column ids, vi (perm): original positions
  boundaries_kernel<<<grid_for((long long)nnz + 1), 256, 0, s>>>(ki, nnz, n, rptrT);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (index)
    gather_rows_kernel<<<grid_for(nnz), 256, 0, s>>>(index->words, index->ids, index->nonempty, m, vi, nnz, colT);
  else
    gather_int_kernel<<<grid_for(nnz), 256, 0, s>>>(rows, vi, nnz, colT);
  return cudaGetLastError();
}

cudaError_t gather_values(int dtype, const void* src, const int* perm, int nnz, void* out, cudaStream_t s) {
  if (nnz == 0) return cudaSuccess;
  if (dtype == GBS_F64)
    gather_vals_kernel<double><<<grid_for(nnz), 256, 0, s>>>(static_cast<const double*>(src), perm, nnz,
                                                                 static_cast<double*>(out));
  else
    gather_vals_kernel<float><<<grid_for(nnz), 256, 0, s>>>(static_cast<const float*>(src), perm, nnz,
                                                                static_cast<float*>(out));
  return cudaGetLastError();
}

size_t transpose_scan_ws_ints(int nnz) {
  const long long ntiles = ((long long)nnz + kSortTile - 1) / kSortTile;
  return scan_workspace_ints(std::max(ntiles, 1LL) << kSortBits);
}

size_t transpose_hist_ints(int nnz) {
  const long long ntiles = ((long long)nnz + kSortTile - 1) / kSortTile;
  return (size_t)std::max(ntiles, 1LL) << kSortBits;
}

}  // namespace gbs
