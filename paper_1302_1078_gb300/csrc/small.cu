// One-shot SpMV of a small matrix in one launch.
//
// Up to some ten thousand nonzeros a call is bound by its launches and allocations, not by the
// GPU: merge-path needs scratch and three kernels.  Here L lanes take a row (L from the mean row
// length, which the host knows).  The row lengths are not known, and a CTA would be busy for long
// with long rows that happen to lie together (one after another by the whole CTA, 512 rows of 192
// nonzeros took 870 us, merge-path 23).  So the CTAs of a cluster look at all the cluster's rows, and
// if one has more than 16 nonzeros per lane, all take the cluster's rows another way: the nonzeros are
// consecutive, every warp gets an equal part of them, walks 256 at a time, 8 per lane, and finds their
// rows by a search of the row ends in shared memory; a row that crosses lanes is finished by the
// segmented scan of the SPLIT walk (split_kernel.cuh), a row that crosses warps over one carry per
// warp and one per CTA.  One SM gathers about one nonzero per clock, so that eight
// finish the most nonzeros that are sent here, 98,304, in 6 us, and the rest is a chain of loads.
// Back to back, FP64 and FP32: 64 x 64 grid, 20,224 nonzeros, 7 us, of which 6 are the Python call
// (merge-path 23 before the library had a pool of its own, 18 with it); 512 rows of 192 together 17 and
// 13; one row of 98,304 19 and 15 (23 and 21); six rows of 16,000 15 and 11 (20 and 18).
// The kernel alone under ncu, long rows by the CTA that owns them and by the cluster: R-MAT 13 x 9 37 and 10
// us, FP32 22 and 10; 390,000 rows, most of them empty, whose ends eight CTAs look at, 7 and 10.
#include <algorithm>

#include "device_common.cuh"
#include "gbspmv.h"
#include "launch.h"
#include "split_kernel.cuh"

namespace gbs {

constexpr int kSmallThreads = 512, kSmallWarps = kSmallThreads / 32;
constexpr int kSmallCluster = 8;  // CTAs; the largest size that every GPU of the architecture allows

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// The address of a shared variable in the cluster's first CTA.
__device__ __forceinline__ uint32_t in_first_cta(const void* p) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t a, int v) { asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void st_cluster(uint32_t a, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void st_cluster(uint32_t a, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }

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

// Nonzeros [s0, s1) of the rows whose ends are rp[0 .. rows], by one warp; s0 is a multiple of 8, s1 of
// 256 more than s0 unless it is rp[rows], and positions below rp[0] are passed over.  Returns the row
// that goes on behind s1 (-1: none) and in `open` its sum so far; the row that was open at s0 is
// written without what came before.
template <typename T>
__device__ __forceinline__ int small_split(const SplitArgs<T>& a, const int* rp, int rows, int s0, int s1, T* y,
                                           Open<T>& open) {
  constexpr int N = 8;
  const uint64_t pol = policy_evict_first();
  const int lane = threadIdx.x & 31, b0 = rp[0], e = rp[rows];
  int open_row = -1;
  for (int t0 = s0; t0 < s1; t0 += 32 * N) {
    const int p = t0 + lane * N;
    int c[N];
    T v[N], x[N];
    split_load8<T, false>(a, p, a.wide && p + N <= a.nnz, pol, c, v);
#pragma unroll
    for (int u = 0; u < N; ++u) {
      if (p + u < b0 || p + u >= s1) c[u] = -1;
      x[u] = c[u] >= 0 ? __ldg(a.X + c[u]) : T(0);
    }
    int row = 0;  // the last row that begins at or before the first nonzero: it is not empty
    for (int hi = rows; hi - row > 1;) {
      const int mid = (row + hi) >> 1;
      if (rp[mid] <= max(p, b0))
        row = mid;
      else
        hi = mid;
    }
    int next = rp[row + 1], head_row = -1;
    Acc<T> acc, head;
    if (lane == 0) acc = open.acc();
#pragma unroll
    for (int u = 0; u < N; ++u) {
      if (c[u] < 0) continue;
      acc.add(v[u], x[u]);
      if (p + u + 1 == next) {
        if (head_row < 0) {
          head = acc;
          head_row = row;
        } else {
          y[row] = acc.value();
        }
        acc.reset();
        if (next < e) {
          do next = rp[++row + 1];
          while (next == p + u + 1);
        }
      }
    }
    const unsigned closed = __ballot_sync(0xffffffffu, head_row >= 0);
    const unsigned upto = closed & (0xffffffffu >> (31 - lane));
    const int hs = upto ? 31 - __clz(upto) : 0;
    Open<T> S(acc);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const bool take = lane - d >= hs;
      if (__any_sync(0xffffffffu, take)) {
        const Open<T> o = S.up(d);
        if (take) S.add(o);
      }
    }
    const Open<T> before = S.up(1);
    if (head_row >= 0) {
      Open<T> out(head);
      if (lane > 0) out.add(before);
      y[head_row] = out.value();
    }
    open = S.of(31);
    open_row = __shfl_sync(0xffffffffu, rp[row] < p + N ? row : -1, 31);
  }
  return s0 < s1 && s1 < e ? open_row : -1;
}

// Carries of consecutive warps (or CTAs): row still open behind each, or -1, and its sum's two parts
// (c for floats only).
template <typename T, int N>
struct SmallCarries {
  int row[N];
  T s[N], c[N];
  // Thread t < N: if t is the first of a run of equal rows, the run's sum in `sum`, its row returned (else
  // -1), and in `last` whether the run reaches the last entry.
  __device__ __forceinline__ int run(int t, Open<T>& sum, bool& last) const {
    const int r = row[t];
    if (r < 0 || (t > 0 && row[t - 1] == r)) return -1;
    int q = t;
    for (; q < N && row[q] == r; ++q) {
      Acc<T> a;
      a.s = s[q];
      if constexpr (sizeof(T) == 4) a.c = c[q];
      sum.add(Open<T>(a));
    }
    last = q == N;
    return r;
  }
};

// Adds what came before to a row's last part, which another thread has written.
template <typename T>
__device__ __forceinline__ void small_add(T* y, const Open<T>& sum) {
  Acc<T> a = sum.acc();
  a.add_partial(__ldcg(y));
  *y = a.value();
}

template <typename T, int L>
__global__ void __cluster_dims__(kSmallCluster, 1, 1) __launch_bounds__(kSmallThreads)
    small_spmv_kernel(const int* __restrict__ rp, SplitArgs<T> a) {
  constexpr int R = kSmallThreads / L, LONG = 16 * L;
  constexpr int CR = R * kSmallCluster, CW = kSmallWarps * kSmallCluster;  // rows and warps of the cluster
  const int lane = threadIdx.x % L, row = blockIdx.x * R + threadIdx.x / L;
  const int rank = blockIdx.x % kSmallCluster, first = (int)(blockIdx.x - rank) * R, rows = max(0, min(CR, a.m - first));
  int s = 0, e = 0;
  if (row < a.m) {
    s = __ldg(rp + row);
    e = __ldg(rp + row + 1);
  }
  bool is_long = false;
#pragma unroll
  for (int i = 0; i < CR; i += kSmallThreads) {
    const int r = i + (int)threadIdx.x;
    if (r < rows && __ldg(rp + first + r + 1) - __ldg(rp + first + r) > LONG) is_long = true;
  }
  if (!__syncthreads_or(is_long)) {  // every CTA of the cluster comes to the same answer
    Open<T> sum(small_walk<T>(a.col_idx, a.vals, a.X, s + lane, e, L));
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) sum.add(sum.across(o));
    if (row < a.m && lane == 0) a.Y[row] = sum.value();
    return;
  }
  __shared__ int s_rp[CR + 1];
  __shared__ SmallCarries<T, kSmallWarps> of_warps;
  __shared__ SmallCarries<T, kSmallCluster> of_ctas;  // the first CTA's is used
  cluster_arrive();  // (none writes to the first CTA's memory before that has begun)
  for (int r = threadIdx.x; r <= rows; r += kSmallThreads) s_rp[r] = __ldg(rp + first + r);
  __syncthreads();
  T* y = a.Y + first;
  for (int r = rank * kSmallThreads + threadIdx.x; r < rows; r += kSmallThreads * kSmallCluster)
    if (s_rp[r] == s_rp[r + 1]) y[r] = T(0);
  const int base = s_rp[0] & ~7, end = s_rp[rows], w = (int)(threadIdx.x >> 5);
  const int per = (end - base + 256 * CW - 1) / (256 * CW) * 256;
  const int s0 = base + (rank * kSmallWarps + w) * per, s1 = min(end, s0 + per);
  Open<T> open{Acc<T>()};
  const int open_row = small_split<T>(a, s_rp, rows, s0, s1, y, open);
  if ((threadIdx.x & 31) == 0) {
    of_warps.row[w] = open_row;
    of_warps.s[w] = open.s;
    if constexpr (sizeof(T) == 4) of_warps.c[w] = open.c;
  }
  __syncthreads();
  cluster_wait();
  // rows that end in this CTA get the sums of its warps before that; a row that goes on, or none, is the CTA's carry
  const int t = threadIdx.x;
  if (t < kSmallWarps) {
    Open<T> sum{Acc<T>()};
    bool last = false;
    const int r = of_warps.run(t, sum, last);
    if (r >= 0 && !last) small_add(y + r, sum);
    if (last || (t == kSmallWarps - 1 && of_warps.row[t] < 0)) {
      st_cluster(in_first_cta(&of_ctas.row[rank]), r);
      st_cluster(in_first_cta(&of_ctas.s[rank]), sum.s);
      if constexpr (sizeof(T) == 4) st_cluster(in_first_cta(&of_ctas.c[rank]), sum.c);
    }
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  if (rank == 0 && t < kSmallCluster) {
    Open<T> sum{Acc<T>()};
    bool last = false;
    const int r = of_ctas.run(t, sum, last);
    if (r >= 0) small_add(y + r, sum);
  }
}

template <typename T>
static cudaError_t small_t(const CsrView& A, const void* x, void* y, cudaStream_t s) {
  SplitArgs<T> a{};
  a.m = A.m;
  a.nnz = A.nnz;
  a.col_idx = A.col_idx;
  a.vals = static_cast<const T*>(A.vals);
  a.X = static_cast<const T*>(x);
  a.Y = static_cast<T*>(y);
  a.wide = ((reinterpret_cast<uintptr_t>(A.vals) | reinterpret_cast<uintptr_t>(A.col_idx)) & 31) == 0;
  int l = 1;  // about two nonzeros per lane of a mean row
  while (l < 32 && 2LL * l * A.m < A.nnz) l <<= 1;
  const long long per = (long long)kSmallThreads / l * kSmallCluster;
  const unsigned grid = (unsigned)((A.m + per - 1) / per * kSmallCluster);
  auto go = [&](auto kernel) {
    kernel<<<grid, kSmallThreads, 0, s>>>(A.row_ptr, a);
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
