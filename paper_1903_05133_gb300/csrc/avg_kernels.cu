// Local and global averages of Algorithm 1 (Sec. 3.1) over a learner-indexed
// fp32 matrix w[P, ld]: in-memory segmented / full means over the learner axis.
//
// Each thread owns one 16-byte column slice (4 consecutive parameters) and walks
// the n rows of its cluster (or of all P learners): loads are 128-bit and a warp
// reads 512 contiguous bytes per row, so every row access is fully coalesced.
// The sum over rows follows the canonical adjacent-pair tree (v[i] += v[i+h] for
// h = 1, 2, 4, ..., unpaired elements carried up), evaluated as a streaming binary
// counter: pushing value i combines it with the pending partials of the same
// size, exactly like incrementing a binary number, so only log2(n)+1 partials
// live in registers.  Then one IEEE division by n and a broadcast write-back.
// The arithmetic is __fadd_rn / __fdiv_rn only (no FMA, no flush to zero), so the
// result is bit-identical to the CPU definition of the same tree.
#include <cstdint>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace ha {
namespace {

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float4 vadd(float4 a, float4 b) {
  return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z),
                     __fadd_rn(a.w, b.w));
}
__device__ __forceinline__ float vdiv(float a, float n) { return __fdiv_rn(a, n); }
__device__ __forceinline__ float4 vdiv(float4 a, float n) {
  return make_float4(__fdiv_rn(a.x, n), __fdiv_rn(a.y, n), __fdiv_rn(a.z, n),
                     __fdiv_rn(a.w, n));
}

// Sum of the 2^LOG consecutive rows starting at p (row stride ld_v in vectors).
template <int LOG, class V>
__device__ __forceinline__ V tree_pow2(const V* __restrict__ p, int64_t ld_v) {
  constexpr int N = 1 << LOG;
  V stack[LOG + 1];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    V x = p[static_cast<int64_t>(i) * ld_v];
    int l = 0;
#pragma unroll
    for (; l < LOG; ++l) {
      if (((i >> l) & 1) == 0) break;
      x = vadd(stack[l], x);
    }
    stack[l] = x;
  }
  return stack[LOG];
}

template <class V>
__device__ __forceinline__ void store_rows(V* p, int64_t ld_v, int n, V m) {
#pragma unroll 8
  for (int i = 0; i < n; ++i) p[static_cast<int64_t>(i) * ld_v] = m;
}

// Rows whose length is no multiple of four: `tail` = 1 to 3 columns follow the cols_v quads, and
// the row's last CTA takes them, a thread per column, with the same tree over floats.  (A second
// launch for them cost 3 to 5 us; the generic kernels, which need none, keep fewer rows in
// flight.  Rows padded to 64, this | the generic kernels | two launches: P = 16, S = 2, D =
// 8000001 local + global 150 | 231 | 163 us; P = 64, S = 8, D = 1000003 local 74.8 | 76.8 | 80.0,
// local + global 87.6 | 121 | 125; P = 128, S = 32, D = 4000001 local + global 618 | 777 | 689.)
// (kTail: kernels of their own, so that the others keep their code: D = 1000000 of 128 rows global
// 160.4 us, 161.3 with the branch in.)
template <bool kTail>
__device__ __forceinline__ bool tail_cta() {
  if constexpr (kTail) return blockIdx.x == gridDim.x - 1;
  return false;
}
__device__ __forceinline__ bool tail_thread(int tail) {
  return threadIdx.y == 0 && static_cast<int>(threadIdx.x) < tail;
}
__device__ __forceinline__ const float* tail_column(const float4* row, int64_t cols_v) {
  return reinterpret_cast<const float*>(row + cols_v) + threadIdx.x;
}
__device__ __forceinline__ float* tail_column(float4* row, int64_t cols_v) {
  return reinterpret_cast<float*>(row + cols_v) + threadIdx.x;
}

// One column (V: of four parameters, or of one) of a group of n = 2^LOG rows: its mean.
template <int LOG, class V>
__device__ __forceinline__ void mean_pow2_column(V* p, int64_t ld_v) {
  const V m = vdiv(tree_pow2<LOG>(p, ld_v), static_cast<float>(1 << LOG));
  store_rows(p, ld_v, 1 << LOG, m);
}

// Group means, n = 2^LOG rows per group; grid.y = group index.
template <int LOG, bool kTail>
__global__ void __launch_bounds__(256) k_mean_pow2(float4* __restrict__ w, int64_t ld_v,
                                                   int64_t cols_v, int tail) {
  grid_dep_wait();
  float4* row = w + static_cast<int64_t>(blockIdx.y) * (int64_t(1) << LOG) * ld_v;
  if (tail_cta<kTail>()) {
    if (tail_thread(tail)) mean_pow2_column<LOG>(tail_column(row, cols_v), 4 * ld_v);
    return;
  }
  const int64_t c = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (c < cols_v) mean_pow2_column<LOG>(row + c, ld_v);
}

// The same group sums divided by div, written once per group, to row blockIdx.y of
// out (row stride out_ld_v): compact cluster means, the rows of w only read.  div is
// the group size, or, when the rows of w are themselves sums of the first tree levels
// (group sums of Q learners), the cluster size.
template <int LOG>
__global__ void __launch_bounds__(256) k_mean_pow2_to(const float4* __restrict__ w, int64_t ld_v,
                                                      int64_t cols_v, float div,
                                                      float4* __restrict__ out, int64_t out_ld_v) {
  grid_dep_wait();
  const int64_t c = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (c >= cols_v) return;
  const float4* p = w + static_cast<int64_t>(blockIdx.y) * (int64_t(1) << LOG) * ld_v + c;
  out[static_cast<int64_t>(blockIdx.y) * out_ld_v + c] = vdiv(tree_pow2<LOG>(p, ld_v), div);
}

// Fused last local average + global average: G = 2^LOGG clusters of S = 2^LOGS.
// The global tree runs over the P values the local average would have written
// (S copies of each cluster mean, in learner order), so the result is the literal
// two-pass result: the S equal copies of a cluster form one complete sub-tree of
// the global tree, whose value is the cluster mean added to itself LOGS times.
// Each cluster's sum is the tree over its 2^(LOGS - LOGQ) rows of src (row stride
// src_ld_v): the learner rows themselves (LOGQ = 0, src = w), or sums of Q = 2^LOGQ
// learners each that hold the first LOGQ levels of the cluster's tree.  The result
// is written to all P rows of w (src may be rows of w: a thread reads its column of
// every source row before it writes).
template <int LOGQ, int LOGS, int LOGG, class V>
__device__ __forceinline__ void local_global_pow2_column(const V* q, int64_t src_ld_v, V* p, int64_t ld_v) {
  constexpr int S = 1 << LOGS, G = 1 << LOGG, N = 1 << (LOGS - LOGQ);
  V stack[LOGG + 1];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    V x = vdiv(tree_pow2<LOGS - LOGQ>(q + static_cast<int64_t>(g) * N * src_ld_v, src_ld_v),
                    static_cast<float>(S));
#pragma unroll
    for (int l = 0; l < LOGS; ++l) x = vadd(x, x);
    int l = 0;
#pragma unroll
    for (; l < LOGG; ++l) {
      if (((g >> l) & 1) == 0) break;
      x = vadd(stack[l], x);
    }
    stack[l] = x;
  }
  const V m = vdiv(stack[LOGG], static_cast<float>(S * G));
  store_rows(p, ld_v, S * G, m);
}
template <int LOGQ, int LOGS, int LOGG, bool kTail>
__global__ void __launch_bounds__(256) k_local_global_pow2(const float4* src, int64_t src_ld_v, float4* w,
                                                           int64_t ld_v, int64_t cols_v, int tail) {
  grid_dep_wait();
  if (tail_cta<kTail>()) {
    if (tail_thread(tail))
      local_global_pow2_column<LOGQ, LOGS, LOGG>(tail_column(src, cols_v), 4 * src_ld_v, tail_column(w, cols_v),
                                                 4 * ld_v);
    return;
  }
  const int64_t c = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (c < cols_v) local_global_pow2_column<LOGQ, LOGS, LOGG>(src + c, src_ld_v, w + c, ld_v);
}

// The same two kernels with each column's rows split between two threads (threadIdx.y),
// for short rows (D small against the GPU): twice the threads, each walking half the
// rows.  The tree over 2^LOG rows is the tree over each half joined by one addition
// (first half + second half), so the result has the same bits.  blockDim = (128, 2).
template <int LOG, bool kTail>
__global__ void __launch_bounds__(256) k_mean_pow2_split(float4* w, int64_t ld_v, int64_t cols_v,
                                                         int tail) {
  __shared__ float4 part[128];
  grid_dep_wait();
  if (tail_cta<kTail>()) {
    float4* row = w + static_cast<int64_t>(blockIdx.y) * (int64_t(1) << LOG) * ld_v;
    if (tail_thread(tail)) mean_pow2_column<LOG>(tail_column(row, cols_v), 4 * ld_v);
    return;
  }
  const int64_t c = static_cast<int64_t>(blockIdx.x) * 128 + threadIdx.x;
  const bool valid = c < cols_v;
  constexpr int H = 1 << (LOG - 1);
  float4* p = w + static_cast<int64_t>(blockIdx.y) * (int64_t(1) << LOG) * ld_v + c +
              static_cast<int64_t>(threadIdx.y) * H * ld_v;
  float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
  if (valid) x = tree_pow2<LOG - 1>(p, ld_v);
  if (threadIdx.y == 1) part[threadIdx.x] = x;
  __syncthreads();
  if (threadIdx.y == 0) part[threadIdx.x] = vdiv(vadd(x, part[threadIdx.x]), static_cast<float>(1 << LOG));
  __syncthreads();
  if (valid) store_rows(p, ld_v, H, part[threadIdx.x]);
}

// (threadIdx.y = which half of the G clusters; the first G / 2 clusters' S copies form a
// complete sub-tree of the global tree.)
template <int LOGQ, int LOGS, int LOGG, bool kTail>
__global__ void __launch_bounds__(256) k_local_global_pow2_split(const float4* src, int64_t src_ld_v,
                                                                 float4* w, int64_t ld_v,
                                                                 int64_t cols_v, int tail) {
  __shared__ float4 part[128];
  grid_dep_wait();
  if (tail_cta<kTail>()) {
    if (tail_thread(tail))
      local_global_pow2_column<LOGQ, LOGS, LOGG>(tail_column(src, cols_v), 4 * src_ld_v, tail_column(w, cols_v),
                                                 4 * ld_v);
    return;
  }
  const int64_t c = static_cast<int64_t>(blockIdx.x) * 128 + threadIdx.x;
  const bool valid = c < cols_v;
  constexpr int S = 1 << LOGS, G2 = 1 << (LOGG - 1), N = 1 << (LOGS - LOGQ);
  const int g0 = static_cast<int>(threadIdx.y) * G2;
  float4 half = make_float4(0.f, 0.f, 0.f, 0.f);
  if (valid) {
    const float4* q = src + c;
    float4 stack[LOGG];
#pragma unroll
    for (int g = 0; g < G2; ++g) {
      float4 x = vdiv(tree_pow2<LOGS - LOGQ>(q + static_cast<int64_t>(g0 + g) * N * src_ld_v, src_ld_v),
                      static_cast<float>(S));
#pragma unroll
      for (int l = 0; l < LOGS; ++l) x = vadd(x, x);
      int l = 0;
#pragma unroll
      for (; l < LOGG - 1; ++l) {
        if (((g >> l) & 1) == 0) break;
        x = vadd(stack[l], x);
      }
      stack[l] = x;
    }
    half = stack[LOGG - 1];
  }
  if (threadIdx.y == 1) part[threadIdx.x] = half;
  __syncthreads();
  if (threadIdx.y == 0)
    part[threadIdx.x] = vdiv(vadd(half, part[threadIdx.x]), static_cast<float>(S * (2 * G2)));
  __syncthreads();
  if (valid) store_rows(w + c + static_cast<int64_t>(g0) * S * ld_v, ld_v, G2 * S, part[threadIdx.x]);
}

// Generic path: any number of rows, any alignment, any row length.  A thread owns four
// columns, which an access policy maps to memory: Quad for rows that start on 16 bytes (four
// neighbours, one 128-bit access; the row's last quad may be partial), Spread for all others
// (columns 256 apart, so that each of the four 32-bit accesses of a warp is contiguous).
// The tree over n rows is the tree over the complete block of each set bit of n, highest bit
// first, folded from the smallest block upward (the binary counter's pending partials), and each
// block is unrolled in registers with its loads in flight.  (One column per thread with the
// counter in a local array had been bound by the latency of its serial loads and stack.
// Unaligned rows, L2 holding the matrix: P = 12, S = 6, D = 1000003 local 23.4 -> 12.5 us, local +
// global 34.0 -> 17.0 us (5.6 TB/s); P = 48, S = 8, D = 8000001 from HBM: local 905 -> 459 us
// (6.7 TB/s), global 880 -> 622, local + global 1067 -> 699.)
struct Quad {
  using V = float4;
  static constexpr int kCols = 4;
  int64_t c;
  int live;
  __device__ __forceinline__ explicit Quad(int64_t cols) {
    c = (static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x) * 4;
    live = cols - c >= 4 ? 4 : cols > c ? static_cast<int>(cols - c) : 0;
  }
  __device__ __forceinline__ float4 load(const float* row) const {
    if (live == 4) return *reinterpret_cast<const float4*>(row + c);
    return make_float4(row[c], live > 1 ? row[c + 1] : 0.f, live > 2 ? row[c + 2] : 0.f, 0.f);
  }
  __device__ __forceinline__ void store(float* row, float4 v) const {
    if (live == 4) {
      *reinterpret_cast<float4*>(row + c) = v;
      return;
    }
    row[c] = v.x;
    if (live > 1) row[c + 1] = v.y;
    if (live > 2) row[c + 2] = v.z;
  }
};
struct Spread {
  using V = float4;
  static constexpr int kCols = 4;
  int64_t c;
  int live;
  __device__ __forceinline__ explicit Spread(int64_t cols) {
    c = static_cast<int64_t>(blockIdx.x) * 1024 + threadIdx.x;
    const int64_t left = cols - c;
    live = left <= 0 ? 0 : left > 768 ? 4 : left > 512 ? 3 : left > 256 ? 2 : 1;
  }
  __device__ __forceinline__ float4 load(const float* row) const {
    const float* p = row + c;
    return make_float4(p[0], live > 1 ? p[256] : 0.f, live > 2 ? p[512] : 0.f, live > 3 ? p[768] : 0.f);
  }
  __device__ __forceinline__ void store(float* row, float4 v) const {
    float* p = row + c;
    p[0] = v.x;
    if (live > 1) p[256] = v.y;
    if (live > 2) p[512] = v.z;
    if (live > 3) p[768] = v.w;
  }
};

// One column per thread, for rows so short that four would leave SMs without a CTA.
struct Single {
  using V = float;
  static constexpr int kCols = 1;
  int64_t c;
  int live;
  __device__ __forceinline__ explicit Single(int64_t cols) {
    c = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
    live = c < cols;
  }
  __device__ __forceinline__ float load(const float* row) const { return row[c]; }
  __device__ __forceinline__ void store(float* row, float v) const { row[c] = v; }
};

// Tree over the 2^LOG rows from p on.
template <int LOG, class A>
__device__ __forceinline__ typename A::V tree_block(const A& a, const float* p, int64_t ld) {
  typename A::V stack[LOG + 1];
#pragma unroll
  for (int i = 0; i < (1 << LOG); ++i) {
    typename A::V x = a.load(p + i * ld);
    int l = 0;
#pragma unroll
    for (; l < LOG; ++l) {
      if (((i >> l) & 1) == 0) break;
      x = vadd(stack[l], x);
    }
    stack[l] = x;
  }
  return stack[LOG];
}

// The binary counter over values pushed in order, with blocks of 2^level values that are
// equal or already summed pushed at once (idx: the block's first value, a multiple of
// 2^level).  The levels are uniform over the CTA.  Unrolled, the partials stay in registers and a
// push costs every level's test; kLoop, a push ends at the level where its block comes to rest
// (every other one at its first) and the partials stand in local memory, where a thread's few
// live ones stay in L1: better for many pushes of small blocks.
template <class V, int LEVELS, bool kLoop = false>
struct Counter {
  V st[LEVELS];
  __device__ __forceinline__ void push(int idx, int level, V x) {
    if constexpr (kLoop) {
      int l = level;
      for (; (idx >> l) & 1; ++l) x = vadd(st[l], x);
      st[l] = x;
    } else {
      bool open = true;
#pragma unroll
      for (int l = 0; l < LEVELS; ++l) {
        if (l < level || !open) continue;
        if ((idx >> l) & 1) {
          x = vadd(st[l], x);
        } else {
          st[l] = x;
          open = false;
        }
      }
    }
  }
  // The pending partials of n values folded from the smallest upward, after `acc` (the sum of
  // smaller blocks that follow them) if have.
  __device__ __forceinline__ V total(int n, V acc, bool have) const {
#pragma unroll
    for (int l = 0; l < LEVELS; ++l)
      if ((n >> l) & 1) {
        acc = have ? vadd(st[l], acc) : st[l];
        have = true;
      }
    return acc;
  }
};

// Tree over n < 2^BITS rows from p on.  The block of bit l is rows [n with bits 0 .. l
// cleared, + 2^l).  Above the last n mod 16 rows, kUnroll has one unrolled block per bit (45
// registers, as many loads in flight as the power-of-two kernels, long code), otherwise
// blocks of 16 go through a counter.
template <int BITS, bool kUnroll, class A>
__device__ __forceinline__ typename A::V tree_rows(const A& a, const float* p, int64_t ld, int n) {
  typename A::V acc{};
  bool have = false;
  auto fold = [&](typename A::V x) {
    acc = have ? vadd(x, acc) : x;
    have = true;
  };
  auto block = [&](int l) { return p + static_cast<int64_t>((n >> l >> 1) << l << 1) * ld; };
  if (n & 1) fold(tree_block<0>(a, block(0), ld));
  if (n & 2) fold(tree_block<1>(a, block(1), ld));
  if (n & 4) fold(tree_block<2>(a, block(2), ld));
  if (n & 8) fold(tree_block<3>(a, block(3), ld));
  if constexpr (BITS > 4 && kUnroll) {
    static_assert(BITS == 8, "one block per bit");
    if (n & 16) fold(tree_block<4>(a, block(4), ld));
    if (n & 32) fold(tree_block<5>(a, block(5), ld));
    if (n & 64) fold(tree_block<6>(a, block(6), ld));
    if (n & 128) fold(tree_block<7>(a, block(7), ld));
  } else if constexpr (BITS > 4) {
    Counter<typename A::V, BITS - 4> cnt;
#pragma unroll 1
    for (int i = 0; i < (n >> 4); ++i) {
      const float* q = p + static_cast<int64_t>(16 * i) * ld;
      const typename A::V x = tree_block<3>(a, q, ld);
      cnt.push(i, 0, vadd(x, tree_block<3>(a, q + 8 * ld, ld)));
    }
    acc = cnt.total(n >> 4, acc, have);
  }
  return acc;
}

// Sums of groups of n rows of src divided by div: written to all n rows of the group (dst =
// src's matrix, row stride ld), or, kTo, once, to row g of dst (row stride dst_ld).
template <class A, int BITS, bool kTo>
__global__ void __launch_bounds__(256) k_mean_any(const float* src, int64_t ld, int64_t cols, int n,
                                                  float div, float* dst, int64_t dst_ld) {
  grid_dep_wait();
  const A a(cols);
  if (a.live == 0) return;
  const int64_t row0 = static_cast<int64_t>(blockIdx.y) * n;
  const typename A::V m = vdiv(tree_rows<BITS, A::kCols == 4 && !kTo>(a, src + row0 * ld, ld, n), div);
  if constexpr (kTo) {
    a.store(dst + static_cast<int64_t>(blockIdx.y) * dst_ld, m);
  } else {
#pragma unroll 8
    for (int i = 0; i < n; ++i) a.store(dst + (row0 + i) * ld, m);
  }
}

// (src, src_ld, n: as in k_local_global_pow2, n = S / Q source rows per cluster.)  The global
// tree runs over S copies of each cluster mean; a complete block of 2^l copies is the mean
// added to itself l times, so a cluster's run is pushed as its maximal aligned blocks.
// (BITS: of n; LEVELS: of P.  Up to 255 rows, three CTAs per SM: without the limit the compiler
// keeps so many rows in flight per thread that one fits, and P = 24, S = 4, D = 5025045 took 407
// instead of 190 us; the kernels for clusters of 16 rows and more spill under it.  Clusters of
// less than 16 rows are many pushes, a looped counter's: P = 48, S = 3, D = 1000003 with padded
// rows 120 -> 67 us.  From 16 rows on there are few, and unrolled levels are as fast or faster up
// to 8 of them (P = 96, S = 96, D = 262145 42.0 us against 47.5 looped), looped ones beyond.)
template <class A, int BITS, int LEVELS>
__global__ void __launch_bounds__(256, LEVELS == 4 ? 4 : LEVELS == 8 ? 3 : 1)
    k_local_global_any(const float* src, int64_t src_ld, int n, float* w, int64_t ld, int64_t cols, int S,
                       int G) {
  grid_dep_wait();
  const A a(cols);
  if (a.live == 0) return;
  Counter<typename A::V, LEVELS, (LEVELS > (BITS == 4 ? 4 : 8))> cnt;
  for (int g = 0; g < G; ++g) {
    const typename A::V m =
        vdiv(tree_rows<BITS, false>(a, src + static_cast<int64_t>(g) * n * src_ld, src_ld, n),
             static_cast<float>(S));
    for (int i = g * S, end = i + S; i < end;) {
      int l = 31 - __clz(end - i);
      if (i != 0) l = min(l, __ffs(i) - 1);
      typename A::V x = m;
      for (int k = 0; k < l; ++k) x = vadd(x, x);
      cnt.push(i, l, x);
      i += 1 << l;
    }
  }
  const int total = S * G;
  const typename A::V m = vdiv(cnt.total(total, typename A::V{}, false), static_cast<float>(total));
#pragma unroll 8
  for (int i = 0; i < total; ++i) a.store(w + static_cast<int64_t>(i) * ld, m);
}

constexpr int kThreads = 256;

int ilog2_exact(int64_t n) {
  if (n < 1 || (n & (n - 1)) != 0) return -1;
  int l = 0;
  while ((int64_t(1) << l) < n) ++l;
  return l;
}

// Fewer columns than about two waves of one-thread-per-column CTAs: split each column's
// rows between two threads.
constexpr int64_t kSplitCols = 2 * kSms * 8 * 256;
bool split_rows(int64_t cols_v, int64_t groups) { return cols_v * groups <= kSplitCols; }

// Grid of the power-of-two kernels: `per` quads per CTA, and a CTA for the columns after them.
dim3 pow2_grid(int64_t cols_v, int per, int tail, int64_t groups) {
  return dim3(static_cast<unsigned>((cols_v + per - 1) / per + (tail != 0)), static_cast<unsigned>(groups));
}

template <int LOG>
void launch_mean_pow2(float4* w, int64_t ld_v, int64_t cols_v, int tail, int64_t groups,
                      cudaStream_t s) {
  if (split_rows(cols_v, groups)) {
    launch_pdl(tail != 0 ? k_mean_pow2_split<LOG, true> : k_mean_pow2_split<LOG, false>,
               pow2_grid(cols_v, 128, tail, groups), dim3(128, 2), 0, s, false, 1, w, ld_v, cols_v, tail);
    return;
  }
  launch_pdl(tail != 0 ? k_mean_pow2<LOG, true> : k_mean_pow2<LOG, false>,
             pow2_grid(cols_v, kThreads, tail, groups), dim3(kThreads), 0, s, false, 1, w, ld_v, cols_v, tail);
}

// (The _to launches: rows of w with stride ld_v, rows of out with stride out_ld_v.)
template <int LOG>
void launch_mean_pow2_to(const float4* w, int64_t ld_v, int64_t cols_v, int64_t groups, float div,
                         float4* out, int64_t out_ld_v, cudaStream_t s) {
  dim3 grid(static_cast<unsigned>((cols_v + kThreads - 1) / kThreads),
            static_cast<unsigned>(groups));
  launch_pdl(k_mean_pow2_to<LOG>, grid, dim3(kThreads), 0, s, false, 1, w, ld_v, cols_v, div, out,
             out_ld_v);
}

bool mean_pow2_to_dispatch(int log, const float4* w, int64_t ld_v, int64_t cols_v, int64_t groups,
                           float div, float4* out, int64_t out_ld_v, cudaStream_t s) {
  switch (log) {
    case 0: launch_mean_pow2_to<0>(w, ld_v, cols_v, groups, div, out, out_ld_v, s); return true;
    case 1: launch_mean_pow2_to<1>(w, ld_v, cols_v, groups, div, out, out_ld_v, s); return true;
    case 2: launch_mean_pow2_to<2>(w, ld_v, cols_v, groups, div, out, out_ld_v, s); return true;
    case 3: launch_mean_pow2_to<3>(w, ld_v, cols_v, groups, div, out, out_ld_v, s); return true;
    case 4: launch_mean_pow2_to<4>(w, ld_v, cols_v, groups, div, out, out_ld_v, s); return true;
    case 5: launch_mean_pow2_to<5>(w, ld_v, cols_v, groups, div, out, out_ld_v, s); return true;
    case 6: launch_mean_pow2_to<6>(w, ld_v, cols_v, groups, div, out, out_ld_v, s); return true;
    case 7: launch_mean_pow2_to<7>(w, ld_v, cols_v, groups, div, out, out_ld_v, s); return true;
    default: return false;
  }
}

bool mean_pow2_dispatch(int log, float4* w, int64_t ld_v, int64_t cols_v, int tail, int64_t groups,
                        cudaStream_t s) {
  switch (log) {
    case 1: launch_mean_pow2<1>(w, ld_v, cols_v, tail, groups, s); return true;
    case 2: launch_mean_pow2<2>(w, ld_v, cols_v, tail, groups, s); return true;
    case 3: launch_mean_pow2<3>(w, ld_v, cols_v, tail, groups, s); return true;
    case 4: launch_mean_pow2<4>(w, ld_v, cols_v, tail, groups, s); return true;
    case 5: launch_mean_pow2<5>(w, ld_v, cols_v, tail, groups, s); return true;
    case 6: launch_mean_pow2<6>(w, ld_v, cols_v, tail, groups, s); return true;
    case 7: launch_mean_pow2<7>(w, ld_v, cols_v, tail, groups, s); return true;
    default: return false;
  }
}

template <int LOGQ, int LOGS, int LOGG>
void launch_lg(const float4* src, int64_t src_ld_v, float4* w, int64_t ld_v, int64_t cols_v,
               int tail, cudaStream_t s) {
  constexpr bool kTail = LOGQ == 0;      // (group sums come in whole quads)
  if constexpr (LOGG >= 1) {
    if (split_rows(cols_v, 1)) {
      launch_pdl(tail != 0 ? k_local_global_pow2_split<LOGQ, LOGS, LOGG, kTail>
                           : k_local_global_pow2_split<LOGQ, LOGS, LOGG, false>,
                 pow2_grid(cols_v, 128, tail, 1), dim3(128, 2), 0, s, false, 1, src, src_ld_v, w, ld_v, cols_v, tail);
      return;
    }
  }
  launch_pdl(tail != 0 ? k_local_global_pow2<LOGQ, LOGS, LOGG, kTail> : k_local_global_pow2<LOGQ, LOGS, LOGG, false>,
             pow2_grid(cols_v, kThreads, tail, 1), dim3(kThreads), 0, s, false, 1, src, src_ld_v, w, ld_v, cols_v,
             tail);
}

template <int LOGQ, int LOGS>
bool lg_dispatch_g(int logg, const float4* src, int64_t src_ld_v, float4* w, int64_t ld_v,
                   int64_t cols_v, int tail, cudaStream_t s) {
  if constexpr (LOGQ <= LOGS) {
#define HA_LG(G_) \
    if constexpr (LOGS + G_ <= 7) \
      if (logg == G_) { launch_lg<LOGQ, LOGS, G_>(src, src_ld_v, w, ld_v, cols_v, tail, s); return true; }
    HA_LG(0) HA_LG(1) HA_LG(2) HA_LG(3) HA_LG(4) HA_LG(5) HA_LG(6)
#undef HA_LG
  }
  return false;
}

template <int LOGQ>
bool lg_dispatch_s(int logs, int logg, const float4* src, int64_t src_ld_v, float4* w,
                   int64_t ld_v, int64_t cols_v, int tail, cudaStream_t s) {
  switch (logs) {
    case 1: return lg_dispatch_g<LOGQ, 1>(logg, src, src_ld_v, w, ld_v, cols_v, tail, s);
    case 2: return lg_dispatch_g<LOGQ, 2>(logg, src, src_ld_v, w, ld_v, cols_v, tail, s);
    case 3: return lg_dispatch_g<LOGQ, 3>(logg, src, src_ld_v, w, ld_v, cols_v, tail, s);
    case 4: return lg_dispatch_g<LOGQ, 4>(logg, src, src_ld_v, w, ld_v, cols_v, tail, s);
    case 5: return lg_dispatch_g<LOGQ, 5>(logg, src, src_ld_v, w, ld_v, cols_v, tail, s);
    default: return false;
  }
}

bool lg_dispatch(int logq, int logs, int logg, const float4* src, int64_t src_ld_v, float4* w,
                 int64_t ld_v, int64_t cols_v, int tail, cudaStream_t s) {
  switch (logq) {
    case 0: return lg_dispatch_s<0>(logs, logg, src, src_ld_v, w, ld_v, cols_v, tail, s);
    case 1: return lg_dispatch_s<1>(logs, logg, src, src_ld_v, w, ld_v, cols_v, tail, s);
    case 2: return lg_dispatch_s<2>(logs, logg, src, src_ld_v, w, ld_v, cols_v, tail, s);
    default: return false;
  }
}

// Grid of the generic kernels: 256 threads of A::kCols columns each.
template <class A>
dim3 any_grid(int64_t cols, int64_t groups) {
  return dim3(static_cast<unsigned>((cols + 256 * A::kCols - 1) / (256 * A::kCols)),
              static_cast<unsigned>(groups));
}

template <class A, bool kTo>
void launch_mean_any(const float* src, int64_t ld, int64_t cols, int n, int64_t groups, float div,
                     float* dst, int64_t dst_ld, cudaStream_t s) {
  launch_pdl(n < 16 ? k_mean_any<A, 4, kTo> : k_mean_any<A, 8, kTo>, any_grid<A>(cols, groups),
             dim3(256), 0, s, false, 1, src, ld, cols, n, div, dst, dst_ld);
}

// Four columns per thread while that gives every SM two CTAs.
bool spread_wide(int64_t cols, int64_t groups) { return cols * groups >= 2 * kSms * 1024; }

template <bool kTo>
void mean_any_dispatch(bool vec, const float* src, int64_t ld, int64_t cols, int n, int64_t groups,
                       float div, float* dst, int64_t dst_ld, cudaStream_t s) {
  if (n >= 256)     // (one column per thread: 27 float partials fit in registers)
    launch_pdl(k_mean_any<Single, 31, kTo>, any_grid<Single>(cols, groups), dim3(256), 0, s, false, 1,
               src, ld, cols, n, div, dst, dst_ld);
  else if (vec)
    launch_mean_any<Quad, kTo>(src, ld, cols, n, groups, div, dst, dst_ld, s);
  else if (spread_wide(cols, groups))
    launch_mean_any<Spread, kTo>(src, ld, cols, n, groups, div, dst, dst_ld, s);
  else
    launch_mean_any<Single, kTo>(src, ld, cols, n, groups, div, dst, dst_ld, s);
}

template <class A>
void launch_lg_any(const float* src, int64_t src_ld, int n, float* w, int64_t ld, int64_t cols, int S,
                   int G, cudaStream_t s) {
  launch_pdl(S * G < 16 ? k_local_global_any<A, 4, 4> : n < 16 ? k_local_global_any<A, 4, 8>
                                                          : k_local_global_any<A, 8, 8>,
             any_grid<A>(cols, 1), dim3(256), 0, s, false, 1, src, src_ld, n, w, ld, cols, S, G);
}

// From 256 rows on, four columns per thread only where clusters of less than 16 rows leave the
// registers for it and the row gives every SM two CTAs: local + global, D = 1000000, quads | one
// column per thread: P = 256, S = 16 749 | 370 us; P = 512, S = 64 1361 | 696.  (Before, | one
// kernel with 31 unrolled levels for all of them, | a counter in a local array for all sizes:
// P = 512, S = 2, D = 1000001 735 | 5310 | 1508 us, P = 300, S = 3, D = 1000000 436 | 3554 | 699,
// P = 300, S = 75 440 | 746 | 614, P = 5000, S = 2, D = 65600 1988 | 4169 | 4456.)
void lg_any_dispatch(bool vec, const float* src, int64_t src_ld, int n, float* w, int64_t ld,
                     int64_t cols, int S, int G, cudaStream_t s) {
  const int64_t P = static_cast<int64_t>(S) * G;
  const bool wide = spread_wide(cols, 1);
  if (P < 256) {
    if (vec)
      launch_lg_any<Quad>(src, src_ld, n, w, ld, cols, S, G, s);
    else if (wide)
      launch_lg_any<Spread>(src, src_ld, n, w, ld, cols, S, G, s);
    else
      launch_lg_any<Single>(src, src_ld, n, w, ld, cols, S, G, s);
  } else if (P < 4096 && n < 16 && wide) {
    launch_pdl(vec ? k_local_global_any<Quad, 4, 12> : k_local_global_any<Spread, 4, 12>, any_grid<Quad>(cols, 1),
               dim3(256), 0, s, false, 1, src, src_ld, n, w, ld, cols, S, G);
  } else {
    launch_pdl(P < 4096 ? n < 16 ? k_local_global_any<Single, 4, 12> : k_local_global_any<Single, 12, 12>
                        : n < 16 ? k_local_global_any<Single, 4, 31> : k_local_global_any<Single, 31, 31>,
               any_grid<Single>(cols, 1), dim3(256), 0, s, false, 1, src, src_ld, n, w, ld, cols, S, G);
  }
}

}  // namespace

// Whether every row starts on 16 bytes.
static bool vec_ok(const float* w, int64_t ld) {
  return (reinterpret_cast<uintptr_t>(w) % 16 == 0) && (ld % 4 == 0);
}

// The power-of-two kernels take aligned rows; other group sizes and alignments, and rows of
// less than a quad, go to the generic kernels.
cudaError_t launch_group_mean(float* w, int64_t P, int64_t n, int64_t D, int64_t ld,
                              cudaStream_t s) {
  if (D == 0 || n == 1) return cudaSuccess;   // a mean of one row is that row
  const int64_t groups = P / n;
  const bool vec = vec_ok(w, ld);
  const int log = ilog2_exact(n);
  if (!(vec && D >= 4 && log >= 1 &&
        mean_pow2_dispatch(log, reinterpret_cast<float4*>(w), ld / 4, D / 4, static_cast<int>(D % 4), groups, s)))
    mean_any_dispatch<false>(vec, w, ld, D, static_cast<int>(n), groups, static_cast<float>(n), w, ld, s);
  return cudaGetLastError();
}

cudaError_t launch_group_mean_to(const float* w, int64_t P, int64_t n, int64_t D, int64_t ld,
                                 float* out, cudaStream_t s) {
  return launch_group_sum_mean_to(w, P, n, D, ld, static_cast<float>(n), out, ld, s);
}

cudaError_t launch_group_sum_mean_to(const float* w, int64_t rows, int64_t n, int64_t D, int64_t ld,
                                     float div, float* out, int64_t out_ld, cudaStream_t s) {
  if (D == 0) return cudaSuccess;
  const int64_t groups = rows / n;
  const bool vec = vec_ok(w, ld) && vec_ok(out, out_ld);
  const int log = ilog2_exact(n);
  if (!(vec && D % 4 == 0 && log >= 0 &&
        mean_pow2_to_dispatch(log, reinterpret_cast<const float4*>(w), ld / 4, D / 4, groups, div,
                              reinterpret_cast<float4*>(out), out_ld / 4, s)))
    mean_any_dispatch<true>(vec, w, ld, D, static_cast<int>(n), groups, div, out, out_ld, s);
  return cudaGetLastError();
}

cudaError_t launch_local_global_mean(float* w, int64_t P, int64_t S, int64_t D, int64_t ld,
                                     cudaStream_t s) {
  if (D == 0) return cudaSuccess;
  // S = 1: the local average is the identity, so the pair is one global mean.
  // (S = P is NOT shortcut: the literal second pass re-averages P equal copies.)
  if (S == 1) return launch_group_mean(w, P, P, D, ld, s);
  return launch_local_global_from_groups(w, ld, 1, w, P, S, D, ld, s);
}

cudaError_t launch_local_global_from_groups(const float* src, int64_t src_ld, int64_t Q, float* w,
                                            int64_t P, int64_t S, int64_t D, int64_t ld,
                                            cudaStream_t s) {
  if (D == 0) return cudaSuccess;
  const int64_t G = P / S, n = S / Q;
  const bool vec = vec_ok(w, ld) && vec_ok(src, src_ld);
  const int logq = ilog2_exact(Q), logs = ilog2_exact(S), logg = ilog2_exact(G);
  if (!(vec && D >= 4 && (D % 4 == 0 || Q == 1) && logq >= 0 && logs >= 1 && logg >= 0 &&
        lg_dispatch(logq, logs, logg, reinterpret_cast<const float4*>(src), src_ld / 4,
                    reinterpret_cast<float4*>(w), ld / 4, D / 4, static_cast<int>(D % 4), s)))
    lg_any_dispatch(vec, src, src_ld, static_cast<int>(n), w, ld, D, static_cast<int>(S), static_cast<int>(G), s);
  return cudaGetLastError();
}

}  // namespace ha
