// Internal launcher interface between the C-ABI layer (api.cu) and the
// per-dtype kernel translation units.  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>

#include "gbspmv.h"

namespace gbs {

// Stream-ordered device memory from the library's own pool (scratch.cu).
cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s);
cudaError_t scratch_free(void* p, cudaStream_t s);

struct CsrView {
  int m, n, nnz;
  const int* row_ptr;
  const int* col_idx;
  const void* vals;
  const int* perm = nullptr;  // if set, the value of entry p is vals[perm[p]] (ROWS, MERGE, MERGE_DIRECT)
  int hot_cols = 0;           // > 0: columns relabelled hottest first; MERGE_DIRECT SpMV gathers
                              // columns >= hot_cols without L1 allocation
  bool alternate = false;     // ROWS_TMA SpMV: half-warps take alternate rows
};

struct DenseView {
  int k;
  const void* X;
  long long ldx;
  void* Y;
  long long ldy;
};

struct MergeScratch {
  int ctas;
  int2* coords;     // [ctas + 1]
  int* carry_row;   // [ctas]
  void* carry_val;  // [ctas * k] elements of the dtype
};

// Plan-time index of the SPLIT variant (split_kernel.cuh, split_build.cu): one word per 32 nonzeros.
struct SplitWord {
  unsigned int ends;  // bit j: nonzero 32 w + j is the last of its row
  int first;          // ordinal, among the non-empty rows, of the row of nonzero 32 w
};

struct SplitIndex {
  const SplitWord* words;  // [ceil(nnz / 32)]
  const int* ids;          // [non-empty rows] their row numbers; NULL when no row is empty
  const int* empty;        // [nempty] the empty rows still to be written as zero
  int nempty;
  const int* nonempty = nullptr;  // if set, the number of non-empty rows, on the device (ids unused when it is m)
};

struct SplitScratch {
  int* carry_row;   // [split_tiles]
  void* carry_val;  // [split_tiles * k] elements of the dtype
};

// Nonzeros per merge thread of the SPLIT SpMV (x and y contiguous): one 32-byte sector of column ids.
constexpr int kSplitShare = 8;
// Threads per CTA of a SPLIT launch.  A float vector's CTAs of two warps end faster than new ones
// begin: three warps there (2M x 50 banded: 64 threads 204 us, 96 181, 128 187); the others keep two,
// which leave the smallest last wave (doubles: 281, 282, 282; R-MAT 22 257, 258, 261).
inline int split_threads(int dtype, int k) { return k == 1 && dtype == GBS_F32 ? 96 : 64; }

// SPLIT variant.  share: nonzeros per merge thread of SpMM (a multiple of 32).  vec16 as for ROWS; values through A.perm if set.
cudaError_t launch_split_f64(const CsrView& A, const SplitIndex& I, const DenseView& D, bool vec16, int threads,
                             int share, const SplitScratch& S, cudaStream_t s);
cudaError_t launch_split_f32(const CsrView& A, const SplitIndex& I, const DenseView& D, bool vec16, int threads,
                             int share, const SplitScratch& S, cudaStream_t s);
// Warps (tiles) of one launch; SpMM: g lanes per merge thread.
long long split_tiles(int nnz, int g, int share);
// The index in two launches: words, ids [m] (the non-empty rows; may be NULL when there is no empty
// row), nonempty [1] and empty (either may be NULL); counts is a workspace of kSplitBlocks ints.
// Also writes the zeros of Y's empty rows (k columns; k may be 0).
constexpr int kSplitBlocks = 2048;
cudaError_t split_build(int dtype, int m, int nnz, const int* row_ptr, SplitWord* words, int* ids, int* nonempty,
                        int* empty, int* counts, int k, void* Y, long long ldy, cudaStream_t s);

// y = A x of a small matrix of any row lengths in one launch, without scratch (small.cu; contiguous x and y).
constexpr int kSmallNnz = 98304;
cudaError_t launch_small_spmv(int dtype, const CsrView& A, const void* x, void* y, cudaStream_t s);

// ROWS variant.  lanes: 1..32 (power of two); k == 1 -> lanes split nonzeros,
// k > 1 -> lanes split columns (k <= lanes * VEC is required per launch;
// wider k is done in column panels by the caller).  vec16: use 128-bit
// gathers/stores of X/Y (caller checked the alignment).
cudaError_t launch_rows_f64(const CsrView& A, const DenseView& D, int lanes, bool vec16, int threads, int tile,
                            int row_base, int rows, cudaStream_t s);
cudaError_t launch_rows_f32(const CsrView& A, const DenseView& D, int lanes, bool vec16, int threads, int tile,
                            int row_base, int rows, cudaStream_t s);

// ROWS_DIRECT variant (no shared memory, no barriers): lanes split the columns (k > 1; same
// rules as ROWS), one lane per row for k == 1; values are not read through a permutation.
cudaError_t launch_rows_direct_f64(const CsrView& A, const DenseView& D, int lanes, bool vec16, int threads,
                                   cudaStream_t s);
cudaError_t launch_rows_direct_f32(const CsrView& A, const DenseView& D, int lanes, bool vec16, int threads,
                                   cudaStream_t s);

// ROWS_TMA variant (persistent, bulk-copy pipeline).  tile must hold the largest block's
// nonzeros + 8; vals and col_idx 16-byte aligned; status: device int (bit 0 = wait timeout).
// emul (FP64 only, 0..3): products per group of 4 nonzeros computed on the FP32 pipe (df64.cuh).
cudaError_t launch_rows_tma_f64(const CsrView& A, const DenseView& D, int lanes, bool vec16, int threads, int tile,
                                int emul, int* status, cudaStream_t s);
cudaError_t launch_rows_tma_f32(const CsrView& A, const DenseView& D, int lanes, bool vec16, int threads, int tile,
                                int emul, int* status, cudaStream_t s);
size_t rows_tma_smem(int dtype, int rows_per_cta, int tile);

// MERGE variant: partition (coords) must have been computed for (threads / g) * items
// items per CTA.  g lanes per merge thread (columns), g * VEC >= k.  direct: each merge
// thread loads its nonzeros from global memory (MERGE_DIRECT) instead of shared memory.
cudaError_t launch_merge_f64(const CsrView& A, const DenseView& D, int g, bool vec16, bool direct, int threads,
                             int items, const MergeScratch& S, cudaStream_t s);
cudaError_t launch_merge_f32(const CsrView& A, const DenseView& D, int g, bool vec16, bool direct, int threads,
                             int items, const MergeScratch& S, cudaStream_t s);
// The same launchers for a CsrView whose values are read through A.perm (the backward pass's
// A^T on A's values).
cudaError_t launch_rows_perm_f64(const CsrView& A, const DenseView& D, int lanes, bool vec16, int threads, int tile,
                                 int row_base, int rows, cudaStream_t s);
cudaError_t launch_rows_perm_f32(const CsrView& A, const DenseView& D, int lanes, bool vec16, int threads, int tile,
                                 int row_base, int rows, cudaStream_t s);
cudaError_t launch_merge_perm_f64(const CsrView& A, const DenseView& D, int g, bool vec16, bool direct, int threads,
                                  int items, const MergeScratch& S, cudaStream_t s);
cudaError_t launch_merge_perm_f32(const CsrView& A, const DenseView& D, int g, bool vec16, bool direct, int threads,
                                  int items, const MergeScratch& S, cudaStream_t s);
cudaError_t launch_merge_partition(const CsrView& A, long long items_per_cta, const MergeScratch& S, cudaStream_t s);

// Exclusive prefix sum of int32 (in == out allowed); ws holds scan_workspace_ints(count) ints.
cudaError_t exclusive_scan_i32(const int* in, int* out, long long count, int* ws, cudaStream_t s);
size_t scan_workspace_ints(long long count);

// Transpose (transpose.cu).  Buffer sizes: rptrT n+1, colT/perm/rows/keys_a/keys_b/vals_a/vals_b nnz,
// hist transpose_hist_ints(nnz), scan_ws transpose_scan_ws_ints(nnz).
// `index`: if not NULL, the SPLIT index of A, from which the rows are then taken (`rows` unused).
cudaError_t transpose_run(int m, int n, int nnz, const int* row_ptr, const int* col_idx, int* rptrT, int* colT,
                          int* perm, int* rows, int* keys_a, int* keys_b, int* vals_a, int* vals_b, int* hist,
                          int* scan_ws, cudaStream_t s, const SplitIndex* index = nullptr);
size_t transpose_hist_ints(int nnz);
size_t transpose_scan_ws_ints(int nnz);
// Stable LSD radix sort of n (key >= 0, value) pairs by the keys' low `bits` bits (transpose.cu);
// hist / scan_ws sized as for a transpose of n nonzeros.
cudaError_t radix_sort_pairs(int n, int bits, int* keys_a, int* keys_b, int* vals_a, int* vals_b, int* hist,
                             int* scan_ws, int** keys_out, int** vals_out, cudaStream_t s);

// Column relabelling by in-degree, hottest first (relabel.cu).  col_degree_stats: the largest
// column degree and the coefficient of variation of the degrees (synchronises s).  relabel_build:
// newid[n] (rank of each column) and col_rl[nnz] = newid[col_idx] (synchronises s).
// relabel_dense: X'[newid[j], :] = X[j, :] for the n rows of X (k columns; vec16: X, X' and both
// leading dimensions 16-byte aligned).
cudaError_t col_degree_stats(int n, int nnz, const int* col_idx, int* max_deg, double* cv_deg, cudaStream_t s);
cudaError_t relabel_build(int n, int nnz, const int* col_idx, int* newid, int* col_rl, cudaStream_t s);
cudaError_t relabel_dense(int dtype, int n, int k, const void* X, long long ldx, const int* newid, void* Xp,
                          long long ldxp, bool vec16, cudaStream_t s);

// out[q] = src[perm[q]] for values of `dtype`.
cudaError_t gather_values(int dtype, const void* src, const int* perm, int nnz, void* out, cudaStream_t s);

// dvals[p] = sum_c dY[row(p), c] * X[col_idx[p], c], row(p) from A's index  (backward.cu)
cudaError_t launch_sddmm(int dtype, int nnz, int k, const SplitIndex& I, int m, const int* col_idx, const void* X,
                         long long ldx, const void* dY, long long lddy, void* dvals, cudaStream_t s);

// Batched persistent kernel (batched.cu).  launch == false: set the shared-memory
// attribute and report the resident CTAs per SM in *blocks_per_sm; launch == true: launch
// `grid` CTAs of 256 threads over `descs` (device BatchDesc<T>[nmat]); CTAs claim items
// from the device counter *next_item, which must be 0 at launch.
cudaError_t batched_kernel_call(bool launch, int dtype, bool split, int G, bool vec16, const void* descs, int nmat,
                                int total_items, int* next_item, int grid, size_t smem, int* blocks_per_sm,
                                cudaStream_t s);

// The fix-up launch of a batch's MERGE matrices (`blocks` of 256 threads over the same descriptors).
cudaError_t batched_fixup(int dtype, const void* descs, int nmat, int blocks, cudaStream_t s);

// UCLD sums (ucld.cu): acc[0] += sum of nnz_i / (line * lines_i) over non-empty rows in 2^-31
// fixed point, acc[1] += sum of lines_i, acc[2] += non-empty rows.
cudaError_t launch_ucld(const int* row_ptr, const int* col_idx, int m, int line, unsigned long long* acc,
                        cudaStream_t s);

// Reverse Cuthill-McKee permutation of the symmetric pattern of a square A (rcm.cu;
// allocates its scratch stream-ordered and synchronises s), and B = P A P^T (vals and
// bvals may be NULL for the pattern only).
cudaError_t rcm_run(int n, int nnz, const int* row_ptr, const int* col_idx, int* perm, cudaStream_t s);
cudaError_t permute_run(int n, int nnz, const int* row_ptr, const int* col_idx, const void* vals, int dtype,
                        const int* perm, int* brp, int* bcol, void* bvals, cudaStream_t s);

// Register-blocked CRS (bcsr.cu).  bcsr_count fills bptr[mb+1] and *nblocks (synchronises s)
// and leaves the sorted block columns in *scratch (stream-ordered allocation) for bcsr_fill,
// which writes bcol / bval; the caller frees scratch with scratch_free.
cudaError_t bcsr_count(int m, int n, int nnz, const int* row_ptr, const int* col_idx, int a, int b, int* bptr,
                       int** bcol_sorted, int* nblocks, void** scratch, cudaStream_t s);
cudaError_t bcsr_fill(int m, int n, int nnz, const int* row_ptr, const int* col_idx, const void* vals, int dtype,
                      int a, int b, const int* bptr, int* bcol, void* bval, long long nblocks, void* scratch,
                      cudaStream_t s);
cudaError_t bcsr_spmv(int dtype, int a, int b, int m, int n, const int* bptr, const int* bcol, const void* bval,
                      const void* x, void* y, cudaStream_t s);

// Message returned by gbs_last_error() on the calling thread (api.cu).
void set_last_error(const char* msg);

}  // namespace gbs
