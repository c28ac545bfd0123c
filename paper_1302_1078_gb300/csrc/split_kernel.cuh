// Nonzero-split CSR kernel ("SPLIT" variant) for SpMV and SpMM.
//
// Power-law rows again (see merge_kernel.cuh), split by nonzeros alone: every
// merge thread takes the same number of consecutive nonzeros, a multiple of 8
// that starts on a multiple of 8.  GB300's FP64 pipe is the scarce resource,
// and a warp FP64 instruction costs its full slot whatever its mask, so equal
// shares of nonzeros (merge-path equalises rows + nonzeros) leave no slot
// without a product, and the aligned shares are read in whole 32-byte sectors
// with 256-bit loads, nothing masked.
//
// What a merge thread has to know about the rows comes from an index (split_build.cu)
// of 8 bytes per 32 nonzeros, which replaces row_ptr and the two binary
// searches per thread of the merge-path walk: SplitWord w holds a bitmap of
// the nonzeros 32w .. 32w+31 that are the last of their row, and the ordinal,
// among the non-empty rows, of the row of nonzero 32w.  The row of any nonzero
// is then an ordinal plus a population count, and a row end is a bit test on a
// register where the merge walk re-reads row_ptr.  `ids` maps ordinals to row
// numbers (NULL when no row is empty); empty rows are written as zero by the
// fix-up kernel from their own list (a one-shot call: by the pass that makes
// the index), so a run of a million empty rows costs its stores and nothing else.
//
// A warp is on its own: no shared memory and no barrier.  The rows that are
// split across merge threads are finished as in the merge kernel, by a
// segmented scan over the warp's merge threads (its segments are known from
// one ballot), and rows split across warps by split_fixup_kernel over one
// carry per warp.  No atomics, every order of summation fixed by the
// structure and the configuration: bitwise reproducible.
//
// PERM: the value of stored entry p is vals[perm[p]] (the backward pass's A^T).
//
// Bounds and measurements (GB300, plans tuned, back to back): SpMV is bound by
// the L1 lookups of its random x gathers; 8 nonzeros per lane keep 40 warps of
// 48 registers on an SM, 16 per lane (80 registers) are 15-20% slower.  R-MAT
// 22 FP64 338 us (direct merge walk) -> 257 us, 0.50 of the measured HBM rate;
// R-MAT 20 forward 95 -> 75 us.  SpMM: FP64 is bound by its pipe (R-MAT 22,
// k = 8: 1346 -> 1008 us, 0.81 of the pipe), FP32 by instruction issue (R-MAT
// 20, k = 8, forward: 233 us staged merge walk, 122 us; the staged walk issued about 150
// warp instructions per 16 nonzeros, most of them in divergent row ends).
#pragma once
#include "dependent.cuh"
#include "device_common.cuh"
#include "launch.h"

namespace gbs {

template <typename T>
struct SplitArgs {
  int m, k, nnz;
  const int* __restrict__ col_idx;
  const T* __restrict__ vals;
  const int* __restrict__ perm;
  const T* __restrict__ X;
  T* __restrict__ Y;
  long long ldx, ldy;
  const SplitWord* __restrict__ words;
  int nwords;
  const int* __restrict__ ids;  // row number of each non-empty row; NULL: its ordinal
  const int* __restrict__ nonempty;  // if set, the device's count of non-empty rows: ids unused when it is m
  int share;                    // SpMM: nonzeros per merge thread (multiple of 32)
  int tiles;                    // warps
  int* __restrict__ carry_row;  // [tiles] row still open at the tile's end, or -1
  T* __restrict__ carry_val;    // [tiles * k]
  bool wide;                    // col_idx and vals (or perm) 32-byte aligned
};

// Eight consecutive 32-bit words (one whole 32-byte sector), skipping L1; ptr 32-byte aligned.
__device__ __forceinline__ void ld_stream_8w(const void* ptr, uint64_t pol, uint32_t* r) {
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(ptr), "l"(pol));
}

// Column ids and values of nonzeros p .. p + 7 (p a multiple of 8).  `whole`: all eight exist and
// the arrays are 32-byte aligned; otherwise element by element, with 0 in the place of those at or
// past nnz (their products are 0 * X[0] = 0 or are skipped by the caller).
template <typename T, bool PERM>
__device__ __forceinline__ void split_load8(const SplitArgs<T>& a, int p, bool whole, uint64_t pol, int* c, T* v) {
  if (whole) {
    uint32_t w[8];
    ld_stream_8w(a.col_idx + p, pol, w);
#pragma unroll
    for (int u = 0; u < 8; ++u) c[u] = (int)w[u];
    if constexpr (PERM) {
      uint32_t q[8];
      ld_stream_8w(a.perm + p, pol, q);
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldg(a.vals + (int)q[u]);
    } else if constexpr (sizeof(T) == 8) {
      ld_stream_4d(reinterpret_cast<const double*>(a.vals + p), pol, reinterpret_cast<double*>(v));
      ld_stream_4d(reinterpret_cast<const double*>(a.vals + p + 4), pol, reinterpret_cast<double*>(v) + 4);
    } else {
      uint32_t q[8];
      ld_stream_8w(a.vals + p, pol, q);
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __uint_as_float(q[u]);
    }
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      c[u] = -1;
      v[u] = T(0);
      if (p + u < a.nnz) {
        c[u] = ld_stream(a.col_idx + p + u, pol);
        if constexpr (PERM)
          v[u] = __ldg(a.vals + ld_stream(a.perm + p + u, pol));
        else
          v[u] = ld_stream(a.vals + p + u, pol);
      }
    }
  }
}

template <typename T>
__device__ __forceinline__ const int* split_ids(const SplitArgs<T>& a) {
  return a.nonempty && __ldg(a.nonempty) == a.m ? nullptr : a.ids;
}
__device__ __forceinline__ int split_row(const int* __restrict__ ids, int ord) { return ids ? __ldg(ids + ord) : ord; }

// The open sum of a merge thread as the carry scan combines it.  float: both parts of the
// accumulator, the sums added with Knuth's TwoSum, so that the scan does not round (error against 64
// bits, with the accumulator of the time: 200,003 x 41 banded SpMV 6.0e-8 by two plain additions, 3.6e-8 by
// TwoSum, merge-path 5.8e-8, for 2% of the time; now 2.7e-8, and R-MAT 20, k = 8, forward and backward
// 3.4e-8, merge-path 6.8e-8).
template <typename T>
struct Open;
template <>
struct Open<double> {
  double s;
  __device__ __forceinline__ explicit Open(const Acc<double>& a) : s(a.s) {}
  __device__ __forceinline__ Open up(int d) const {
    Open o = *this;
    o.s = __shfl_up_sync(0xffffffffu, s, d);
    return o;
  }
  __device__ __forceinline__ Open across(int d) const {
    Open o = *this;
    o.s = __shfl_xor_sync(0xffffffffu, s, d);
    return o;
  }
  __device__ __forceinline__ Open of(int lane) const {
    Open o = *this;
    o.s = __shfl_sync(0xffffffffu, s, lane);
    return o;
  }
  __device__ __forceinline__ Acc<double> acc() const {
    Acc<double> a;
    a.s = s;
    return a;
  }
  __device__ __forceinline__ void add(const Open& o) { s += o.s; }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct Open<float> {
  float s, c;
  __device__ __forceinline__ explicit Open(const Acc<float>& a) : s(a.s), c(a.c) {}
  __device__ __forceinline__ Open up(int d) const {
    Open o = *this;
    o.s = __shfl_up_sync(0xffffffffu, s, d);
    o.c = __shfl_up_sync(0xffffffffu, c, d);
    return o;
  }
  __device__ __forceinline__ Open across(int d) const {
    Open o = *this;
    o.s = __shfl_xor_sync(0xffffffffu, s, d);
    o.c = __shfl_xor_sync(0xffffffffu, c, d);
    return o;
  }
  __device__ __forceinline__ Open of(int lane) const {
    Open o = *this;
    o.s = __shfl_sync(0xffffffffu, s, lane);
    o.c = __shfl_sync(0xffffffffu, c, lane);
    return o;
  }
  __device__ __forceinline__ Acc<float> acc() const {
    Acc<float> a;
    a.s = s;
    a.c = c;
    return a;
  }
  __device__ __forceinline__ void add(const Open& o) {
    const float t = __fadd_rn(s, o.s), b = __fsub_rn(t, s);
    c = __fadd_rn(__fadd_rn(c, o.c), __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(o.s, b)));
    s = t;
  }
  __device__ __forceinline__ float value() const { return __fadd_rn(s, c); }
};

// SpMV: x and y contiguous, one lane per merge thread, N = 8 nonzeros each.
template <typename T, bool PERM>
__device__ __forceinline__ void split_spmv_tile(const SplitArgs<T>& a, int tile) {
  constexpr int N = kSplitShare;
  const int* __restrict__ ids = split_ids(a);
  const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
  const int lane = threadIdx.x & 31;
  // 64-bit: the last tiles' lanes may lie past 2^31
  const long long p0 = (long long)tile * (32 * N) + (long long)lane * N;
  uint32_t ends = 0;
  int ord = 0;
  Acc<T> acc, head;
  if (p0 < a.nnz) {
    const int p = (int)p0;
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(a.words) + (p >> 5));
    const int sh = p & 31;
    ends = (w.x >> sh) & ((1u << N) - 1u);
    ord = (int)w.y + __popc(w.x & ((1u << sh) - 1u));
    bool first = true;
    int c[N];
    T v[N], x[N];
    split_load8<T, PERM>(a, p, a.wide && p + N <= a.nnz, pol_stream, c, v);
#pragma unroll
    for (int u = 0; u < N; ++u) x[u] = c[u] >= 0 ? ld_keep(a.X + c[u], pol_keep) : T(0);
#pragma unroll
    for (int u = 0; u < N; ++u) {
      acc.add(v[u], x[u]);
      if (ends >> u & 1u) {
        if (first) {
          head = acc;
          first = false;
        } else {
          st_stream(a.Y + split_row(ids, ord), acc.value());
        }
        ++ord;
        acc.reset();
      }
    }
  }
  // the row a lane's first end closes began in an earlier lane (or exactly at its first nonzero,
  // when the sum before it is 0): segmented scan of the open sums, a lane with an end starting a
  // new segment.  hs: the segment's first lane.
  const uint32_t closed = __ballot_sync(0xffffffffu, ends != 0);
  const uint32_t upto = closed & (0xffffffffu >> (31 - lane));
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
  if (ends != 0) {
    Open<T> out(head);
    if (lane > 0) out.add(before);
    st_stream(a.Y + split_row(ids, ord - __popc(ends)), out.value());
  }
  if (lane == 31) {
    // the tile's last nonzero lies in a row that goes on unless it ends there or the matrix does
    const bool open = p0 + N < a.nnz && !(ends >> (N - 1) & 1u);
    a.carry_row[tile] = open ? split_row(ids, ord) : -1;
    a.carry_val[tile] = S.value();
  }
}

template <typename T, bool PERM>
__global__ void __launch_bounds__(256, 5) split_spmv_kernel(SplitArgs<T> a) {
  wait_for_previous();
  allow_next();
  const int tile = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  if (tile < a.tiles) split_spmv_tile<T, PERM>(a, tile);
}

// SpMM: G lanes per merge thread, each owning VEC of the k columns (k <= G * VEC); a.share
// nonzeros per merge thread, a multiple of 32.
template <typename T, int VEC, int G, bool PERM>
__device__ __forceinline__ void split_spmm_tile(const SplitArgs<T>& a, int tile) {
  constexpr int MT = 32 / G;  // merge threads per warp
  const int* __restrict__ ids = split_ids(a);
  const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
  const int wl = threadIdx.x & 31, mt = wl / G, c_lo = (wl % G) * VEC;
  const bool col_active = c_lo < a.k, col_full = c_lo + VEC <= a.k;
  const int nwp = a.share >> 5;  // words per merge thread
  const int w0 = (tile * MT + mt) * nwp, w1 = min(w0 + nwp, a.nwords);
  const T* __restrict__ Xc = a.X + c_lo;
  T* __restrict__ Yc = a.Y + c_lo;
  const uint32_t ldx = (uint32_t)a.ldx;  // one 32 x 32 -> 64-bit product per gathered row
  auto store_row = [&](int ord, const T* out) {
    T* y = Yc + (long long)split_row(ids, ord) * a.ldy;
    if (col_full)
      st_stream_vec<T, VEC>(y, out);
    else
      for (int j = 0; j < a.k - c_lo; ++j) st_stream(y + j, out[j]);
  };
  Acc<T> acc[VEC], head[VEC];
  int ord = 0, head_ord = -1;
  bool last_end = true;
  for (int w = w0; w < w1; ++w) {
    const uint2 word = __ldg(reinterpret_cast<const uint2*>(a.words) + w);
    if (w == w0) ord = (int)word.y;
    uint32_t ends = word.x;
    last_end = ends >> 31;
    const int pw = w << 5;
#pragma unroll 1
    for (int b = 0; b < 32 && pw + b < a.nnz; b += 8) {
      const int p = pw + b;
      const bool whole = a.wide && p + 8 <= a.nnz;
      int c[8];
      T v[8];
      split_load8<T, PERM>(a, p, whole, pol_stream, c, v);
#pragma unroll
      for (int h = 0; h < 8; h += 4) {  // four gathers in flight: eight take 110 registers, half the warps
        Vec<T, VEC> x[4];
        if (whole && col_full) {
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = ld_keep_vec<T, VEC>(Xc + (uint64_t)(uint32_t)c[h + u] * ldx, pol_keep);
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int j = 0; j < VEC; ++j)
              x[u].v[j] = c[h + u] >= 0 && c_lo + j < a.k ? ld_keep(Xc + (uint64_t)(uint32_t)c[h + u] * ldx + j, pol_keep) : T(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
          for (int j = 0; j < VEC; ++j) acc[j].add(v[h + u], x[u].v[j]);
          if (ends >> (h + u) & 1u) {
            if (head_ord < 0) {
              head_ord = ord;
#pragma unroll
              for (int j = 0; j < VEC; ++j) head[j] = acc[j];
            } else if (col_active) {
              T out[VEC];
#pragma unroll
              for (int j = 0; j < VEC; ++j) out[j] = acc[j].value();
              store_row(ord, out);
            }
#pragma unroll
            for (int j = 0; j < VEC; ++j) acc[j].reset();
            ++ord;
          }
        }
      }
      ends >>= 8;
    }
  }
  const uint32_t closed = __ballot_sync(0xffffffffu, head_ord >= 0);
  const uint32_t upto = closed & (0xffffffffu >> (31 - wl));
  const int hs = upto ? (31 - __clz(upto)) / G : 0;
  T tail[VEC], out[VEC];
#pragma unroll
  for (int j = 0; j < VEC; ++j) {
    Open<T> S(acc[j]);
#pragma unroll
    for (int d = 1; d < MT; d <<= 1) {
      const bool take = mt - d >= hs;
      if (__any_sync(0xffffffffu, take)) {
        const Open<T> o = S.up(d * G);
        if (take) S.add(o);
      }
    }
    const Open<T> before = S.up(G);
    Open<T> h(head[j]);
    if (mt > 0) h.add(before);
    out[j] = h.value();
    tail[j] = S.value();
  }
  if (head_ord >= 0 && col_active) store_row(head_ord, out);
  if (mt == MT - 1) {
    if (wl == 32 - G) a.carry_row[tile] = w1 - w0 == nwp && (long long)w1 * 32 < a.nnz && !last_end ? split_row(ids, ord) : -1;
    if (col_active)
      for (int j = 0; j < VEC && c_lo + j < a.k; ++j) a.carry_val[(size_t)tile * a.k + c_lo + j] = tail[j];
  }
}

template <typename T, int VEC, int G, bool PERM>
__global__ void __launch_bounds__(256, PERM && sizeof(T) == 8 ? 4 : 3) split_spmm_kernel(SplitArgs<T> a) {
  wait_for_previous();
  allow_next();
  const int tile = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  if (tile < a.tiles) split_spmm_tile<T, VEC, G, PERM>(a, tile);
}

// Adds the tiles' carries to the rows they belong to: lanes sub, sub + 2^lg, ... of the columns of
// tile b (2^lg lanes share a tile; b >= tiles for none), so the reads and writes of a warp are
// coalesced and no index is divided (with a 64-bit division per element the fix-up took 22 us of a
// 271 us R-MAT 20 product of k = 8).  The first tile of a run of equal carry rows sums the run;
// runs of more than eight tiles (hub rows) are summed by the whole warp, each lane every 32nd
// carry and then a fixed shuffle tree, so that a hub of hundreds of tiles costs a few round trips
// (floats keep both parts of their sums up to the end: rounded before a tree of plain additions, the
// sums of rows of 8,192 equal signs k = 64, were off by 0.56 of their last place in the root mean square, 0.28 with both).
// The row's last tile has written its own part of the row already.  Whole warps call it.
template <typename T>
__device__ __forceinline__ void split_fixup_tile(int b, int tiles, int k, int lg, int sub,
                                                 const int* __restrict__ carry_row, const T* __restrict__ carry_val,
                                                 T* __restrict__ Y, long long ldy) {
  constexpr int W = 8;
  const int lane = threadIdx.x & 31;
  int r = -1;
  if (b < tiles) {
    r = __ldcg(carry_row + b);
    if (r >= 0 && b > 0 && __ldcg(carry_row + b - 1) == r) r = -1;
  }
  int len = 0;  // tiles of the run, W + 1 when longer
  if (r >= 0) {
    len = 1;
    while (len <= W && b + len < tiles && __ldcg(carry_row + b + len) == r) ++len;
    if (len <= W) {
      for (int c = sub; c < k; c += 1 << lg) {
        Acc<T> s;
        for (int q = 0; q < len; ++q) s.add_partial(__ldcg(carry_val + (size_t)(b + q) * k + c));
        T* y = Y + (long long)r * ldy + c;
        s.add_partial(__ldcg(y));
        *y = s.value();
      }
    }
  }
  uint32_t todo = __ballot_sync(0xffffffffu, len > W && sub == 0);
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    const int rb = __shfl_sync(0xffffffffu, b, src), rr = __shfl_sync(0xffffffffu, r, src);
    for (int c = 0; c < k; ++c) {
      Acc<T> s;
      T* y = Y + (long long)rr * ldy + c;
      if (lane == 0) s.add_partial(__ldcg(y));
      for (int base = rb; base < tiles; base += 32) {
        const int t = base + lane;
        const bool in = t < tiles && __ldcg(carry_row + t) == rr;
        if (in) s.add_partial(__ldcg(carry_val + (size_t)t * k + c));
        if (!__all_sync(0xffffffffu, in)) break;
      }
      Open<T> sum(s);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum.add(sum.across(o));
      if (lane == 0) *y = sum.value();
    }
  }
}

// The zeros of empty row e (e >= nempty: none), its columns shared like a tile's.
template <typename T>
__device__ __forceinline__ void split_zero_row(long long e, int k, int lg, int sub, const int* __restrict__ empty,
                                               int nempty, T* __restrict__ Y, long long ldy) {
  if (e >= nempty) return;
  T* y = Y + (long long)__ldg(empty + e) * ldy;
  for (int c = sub; c < k; c += 1 << lg) st_stream(y + c, T(0));
}

// Lanes that share a tile in the fix-up, as a power of two.
__host__ __device__ inline int split_fixup_lg(int k) {
  int lg = 0;
  while (lg < 5 && (1 << lg) < k) ++lg;
  return lg;
}

template <typename T>
__global__ void __launch_bounds__(256) split_fixup_kernel(int tiles, int k, int lg, const int* __restrict__ carry_row,
                                                          const T* __restrict__ carry_val, T* __restrict__ Y,
                                                          long long ldy, const int* __restrict__ empty, int nempty,
                                                          int carry_blocks) {
  wait_for_previous();
  const int sub = threadIdx.x & ((1 << lg) - 1);
  if ((int)blockIdx.x >= carry_blocks) {
    split_zero_row<T>((((long long)blockIdx.x - carry_blocks) * 256 + threadIdx.x) >> lg, k, lg, sub, empty, nempty, Y, ldy);
    return;
  }
  const long long b = ((long long)blockIdx.x * 256 + threadIdx.x) >> lg;
  split_fixup_tile<T>(b < tiles ? (int)b : tiles, tiles, k, lg, sub, carry_row, carry_val, Y, ldy);
}

}  // namespace gbs
