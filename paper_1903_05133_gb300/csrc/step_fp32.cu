// fp32 learner step on CUDA cores: the precision mode in which every product and
// sum of the local SGD step (Algorithm 1 inner loop, Sec. 3.1) stays in fp32 (FFMA;
// bf16 or tf32 operands are outside this mode's tolerance).
//
//   k_tile_f32<BM, false>  Z = H W^T + b (ReLU)   one tile of 8-64 samples x 64 outputs per CTA
//   k_tile_f32<BM, true>   dZ' = (dZ W) [H > 0]   the same tile shape over samples x inputs
//   k_dw_f32    W -= lr dZ^T H, b -= lr sum dZ   64 outputs x 128 inputs per CTA
//   k_xent_f32, k_xent_f32_cluster               softmax cross-entropy gradient
//   k_head_f32  the whole last layer (forward, cross-entropy, dX, update) when it has at
//               most 16 classes; for a one-layer model several local steps per launch
// (Small nets run whole steps in one launch instead, whichever the precision: step_small.cu.)
// The first layer reads its batch rows straight from X (no gather).  Rows whose length is a
// multiple of four floats move as 16-byte cp.async copies, others as 4-byte ones.
// Rounds against 16 x 16-tile kernels with one output per thread and a serial reduction
// (seven launches per step of a two-layer net): 3072-10 (P = 4, B = 16, 4 steps) 350 -> 29 us,
// 100-37-10 (P = 4, B = 7, 4 steps) 127 -> 49 us, 3072-512-10 (P = 16, B = 32, 8 steps)
// 4965 -> 930 us; error against 64 bits the same or smaller (5e-8 at 3072-10, was 1.2e-7;
// ReLU flips at 3072-512-10 in 6 of 40 seeds' rounds, were in 8).
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace ha {
namespace {

// ------------------------------------------------------------------ cp.async
// Copies that fill with zeros where `ok` is false (src must be a readable address).
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ------------------------------------------------------------------ packed FMA
// Two fp32 FMAs in one instruction, each rounded as fmaf rounds it.  A scalar FFMA of an outer
// product is held up by the register file (three reads per product): 8 x 8 products per thread
// in registers ran at 55 TFLOP/s with FFMA, at 65 with pairs.
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// A warp's lanes as 4 (y) x 8 (x) threads of a tile.  A 128-bit shared-memory read takes two
// cycles when each half-warp's lanes, taken in neighbouring pairs, touch at most 128 bytes,
// and four otherwise: with y in the lane's lowest bit and highest bit both operands of an
// outer product do (measured: x = lane & 7 takes four cycles, x = lane >> 1 & 7 two).
__device__ __forceinline__ int lane_y(int lane) { return (lane >> 4 << 1) | (lane & 1); }
__device__ __forceinline__ int lane_x(int lane) { return lane >> 1 & 7; }

// Columns [k0, k0 + W) of rows [0, R) into dst (row pitch `pitch` floats) by 256 threads;
// row(r) is the address of row r's column 0 (nullptr: zeros), columns from kmax on are
// zeros.  vec: every row starts on 16 bytes and kmax is a multiple of 4.
template <int W, int R, class Row>
__device__ __forceinline__ void load_rows(float* dst, int pitch, int k0, int kmax, bool vec,
                                          const float* any, int t, Row row) {
  if (vec) {
    constexpr int Q = W / 4;
    const int q = t % Q, k = k0 + 4 * q;
    const bool kin = k < kmax;
#pragma unroll
    for (int i = 0; i < (R * Q + 255) / 256; ++i) {
      const int r = t / Q + i * (256 / Q);
      if (R * Q % 256 != 0 && r >= R) break;
      const float* p = row(r);
      const bool ok = p != nullptr && kin;
      cp_async16(dst + r * pitch + 4 * q, ok ? p + k : any, ok);
    }
  } else {
    const int q = t % W, k = k0 + q;
    const bool kin = k < kmax;
#pragma unroll 4
    for (int r = t / W; r < R; r += 256 / W) {
      const float* p = row(r);
      const bool ok = p != nullptr && kin;
      cp_async4(dst + r * pitch + q, ok ? p + k : any, ok);
    }
  }
}
// Weight rows r0 + r < rmax of a row-major matrix W [rmax][in].
struct WRows {
  const float* p;     // row r0
  int64_t in;
  int rows;           // rmax - r0
  __device__ __forceinline__ const float* operator()(int r) const {
    return r < rows ? p + r * in : nullptr;
  }
};

// ------------------------------------------------------------------ forward and dX tiles
// Both contract a [samples x K] operand (H, or dZ) with the weights into a tile of BM
// samples x 64 columns.  The eight warps of a CTA split the reduction, not the tile: each
// warp holds the whole tile (BM = 64: half of its samples) in registers (8 columns by up
// to 8 samples per thread; from 32 samples on a few words of them spill at the 128 registers
// that two CTAs per SM leave), and takes an eighth of every 64-wide chunk of K, so that a
// chunk's 16-byte shared-memory reads feed 16 FFMAs each (half of the shared-memory
// bandwidth at the FFMA rate).  With few tiles a cluster of up to 8 CTAs shares a tile's
// chunks.  The partials meet in shared memory and then through distributed shared memory,
// added in a fixed order (warp, then CTA rank).  Operands arrive by cp.async, three chunks
// deep.  The forward of 3072 -> 512 (P = 16, B = 32) takes 56 us, 29 TFLOP/s: 45 us of products
// and reductions on the SMs with two CTAs (48 chunks, the average is 40), 26 us of loads, not
// wholly overlapped.  (A fourth stage took 63 us: what shared memory takes, L1 lacks for the
// copies in flight.)
constexpr int kThreads = 256;
constexpr int kBN = 64;                 // columns of a tile
constexpr int kKC = 64;                 // reduction chunk
constexpr int kKP = kKC + 4;            // row pitch: consecutive rows on distinct bank groups
constexpr int kRP = kBN + 8;            // row pitch of the partials
constexpr int kStages = 3;

__host__ __device__ constexpr int tile_stage_floats(int BM) { return (BM + kBN) * kKP; }
__host__ __device__ constexpr int tile_smem(int BM) { return kStages * tile_stage_floats(BM) * 4; }
static_assert(8 * 32 * kRP <= kStages * tile_stage_floats(32) && 4 * 64 * kRP <= kStages * tile_stage_floats(64) &&
                  8 * 8 * kRP <= kStages * tile_stage_floats(8) && 8 * 16 * kRP <= kStages * tile_stage_floats(16),
              "the partials reuse the stages");

struct TileArgs {
  // operand rows: learner j's row b at act + j * act_stride + ((row0 + b) mod N) * K
  const float* act;
  int64_t act_stride, N, row0;
  const float* W;              // learner 0's W_l [out][in], learner j at + j * ld
  int64_t ld;
  int in, out, B;
  int vec_act, vec_w;          // 16-byte copies of the activation rows / weight rows
  const float* bias;           // forward: b_l
  int relu;
  const float* mask;           // dX: H_{l-1} [P][B][in]
  float* y;                    // forward: [P][B][out]; dX: dZ_{l-1} [P][B][in]
};

// kDx false: y[b][o] = sum_k act[b][k] W[o][k]; true: y[b][i] = sum_o act[b][o] W[o][i].
template <int BM, bool kDx>
__global__ void __launch_bounds__(kThreads, 2) k_tile_f32(const TileArgs a, int split) {
  constexpr int MW = BM < 32 ? BM : 32;   // samples of a warp
  constexpr int WM = BM / MW;           // warps along the samples
  constexpr int TM = MW / 4;            // samples of a thread
  constexpr int KS = 8 / WM;            // warps along the reduction
  constexpr int KW = kKC / KS;          // reduction indices of a warp in a chunk
  extern __shared__ __align__(16) float sm[];
  __shared__ const float* arow[BM];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int rank = split > 1 ? static_cast<int>(blockIdx.x) % split : 0;
  const int n0 = (split > 1 ? static_cast<int>(blockIdx.x) / split : static_cast<int>(blockIdx.x)) * kBN;
  const int b0 = blockIdx.y * BM;
  const int64_t j = blockIdx.z;
  const int K = kDx ? a.out : a.in, cols = kDx ? a.in : a.out;
  const int nk = (K + kKC - 1) / kKC;
  const int c_lo = rank * nk / split, c_hi = (rank + 1) * nk / split;
  if (t < BM)
    arow[t] = b0 + t < a.B ? a.act + j * a.act_stride + wrap_row(a.row0 + b0 + t, a.N) * K : nullptr;
  const float* W = a.W + j * a.ld;
  __syncthreads();
  grid_dep_wait();

  auto load = [&](int c, int s) {
    float* as = sm + s * tile_stage_floats(BM);
    float* ws = as + BM * kKP;
    load_rows<kKC, BM>(as, kKP, c * kKC, K, a.vec_act, a.W, t, [&](int r) { return arow[r]; });
    if constexpr (kDx)        // rows o of the chunk, columns i of the tile
      load_rows<kBN, kKC>(ws, kBN, n0, a.in, a.vec_w, a.W, t,
                          WRows{W + static_cast<int64_t>(c) * kKC * a.in, a.in, a.out - c * kKC});
    else                      // rows o of the tile, columns k of the chunk
      load_rows<kKC, kBN>(ws, kKP, c * kKC, a.in, a.vec_w, a.W, t,
                          WRows{W + static_cast<int64_t>(n0) * a.in, a.in, a.out - n0});
  };
  const int ks = warp % KS, wm = warp / KS, ly = lane_y(lane), lx = lane_x(lane);
  // dX: pairs of columns, which lie side by side in its weight chunk.  The forward's pairs
  // would be even and odd indices of the reduction, with half the samples per thread and 1.5
  // times the shared-memory reads per product: no faster (56.5 against 56 us), so scalars.
  constexpr int NA = kDx ? 4 : 8;
  using Acc = std::conditional_t<kDx, uint64_t, float>;
  Acc acc[TM][NA];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int n = 0; n < NA; ++n) acc[i][n] = 0;

#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (c_lo + s < c_hi) load(c_lo + s, s);
    cp_async_commit();
  }
  for (int c = c_lo, it = 0; c < c_hi; ++c, ++it) {
    cp_async_wait<kStages - 2>();
    __syncthreads();          // chunk c has arrived, and chunk c - 1's slot is read
    if (c + kStages - 1 < c_hi) load(c + kStages - 1, (it + kStages - 1) % kStages);
    cp_async_commit();
    const float* as = sm + (it % kStages) * tile_stage_floats(BM) + (wm * MW + ly) * kKP + ks * KW;
    const float* ws = sm + (it % kStages) * tile_stage_floats(BM) + BM * kKP;
#pragma unroll
    for (int k = 0; k < KW; k += 4) {
      if constexpr (kDx) {
        float4 av[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4*>(as + 4 * i * kKP + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const float* wr = ws + (ks * KW + k + kk) * kBN + 4 * lx;
          const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(wr);
          const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(wr + 32);
#pragma unroll
          for (int i = 0; i < TM; ++i) {
            const float x = kk == 0 ? av[i].x : kk == 1 ? av[i].y : kk == 2 ? av[i].z : av[i].w;
            const uint64_t xx = pack2(x, x);
            acc[i][0] = fma2(xx, w0.x, acc[i][0]);
            acc[i][1] = fma2(xx, w0.y, acc[i][1]);
            acc[i][2] = fma2(xx, w1.x, acc[i][2]);
            acc[i][3] = fma2(xx, w1.y, acc[i][3]);
          }
        }
      } else {
        float4 av[TM];
#pragma unroll
        for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4*>(as + 4 * i * kKP + k);
#pragma unroll
        for (int n = 0; n < 8; ++n) {
          const float4 wv = *reinterpret_cast<const float4*>(ws + (lx + 8 * n) * kKP + ks * KW + k);
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][n] = fmaf(av[i].x, wv.x, acc[i][n]);
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][n] = fmaf(av[i].y, wv.y, acc[i][n]);
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][n] = fmaf(av[i].z, wv.z, acc[i][n]);
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][n] = fmaf(av[i].w, wv.w, acc[i][n]);
        }
      }
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  // partials [KS][BM][64]: forward columns lx + 8 n, dX columns 4 lx + n and 32 + 4 lx + n
  {
    float* red = sm + (ks * BM + wm * MW + ly) * kRP;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if constexpr (kDx) {
        *reinterpret_cast<ulonglong2*>(red + 4 * i * kRP + 4 * lx) = make_ulonglong2(acc[i][0], acc[i][1]);
        *reinterpret_cast<ulonglong2*>(red + 4 * i * kRP + 32 + 4 * lx) = make_ulonglong2(acc[i][2], acc[i][3]);
      } else {
#pragma unroll
        for (int n = 0; n < 8; ++n) {
          red[4 * i * kRP + lx + 8 * n] = acc[i][n];
        }
      }
    }
  }
  __syncthreads();
  // four columns of one sample per thread and turn: the warps' partials in order ...
  auto warp_sum = [&](int q) {
    const float* p = sm + (q >> 4) * kRP + 4 * (q & 15);
    float4 s = *reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int w = 1; w < KS; ++w) {
      const float4 v = *reinterpret_cast<const float4*>(p + w * BM * kRP);
      s = make_float4(__fadd_rn(s.x, v.x), __fadd_rn(s.y, v.y), __fadd_rn(s.z, v.z), __fadd_rn(s.w, v.w));
    }
    return s;
  };
  auto finish = [&](int q, float4 s) {
    const int b = b0 + (q >> 4), n = n0 + 4 * (q & 15);
    if (b >= a.B) return;
    const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (n + e >= cols) return;
      const int64_t o = (j * a.B + b) * cols + n + e;
      if constexpr (kDx) {
        a.y[o] = a.mask[o] > 0.f ? v[e] : 0.f;
      } else {
        const float z = __fadd_rn(v[e], a.bias[j * a.ld + n + e]);
        a.y[o] = a.relu ? fmaxf(z, 0.f) : z;
      }
    }
  };
  if (split == 1) {
    for (int q = t; q < BM * 16; q += kThreads) finish(q, warp_sum(q));
    return;
  }
  // ... and, with the tile's chunks split over a cluster, the ranks' sums in order, each
  // rank finishing its share of the tile
  for (int q = t; q < BM * 16; q += kThreads) {
    const float4 s = warp_sum(q);
    *reinterpret_cast<float4*>(sm + (q >> 4) * kRP + 4 * (q & 15)) = s;
  }
  cluster_sync_all();
  const int per = BM * 16 / split;       // (split divides 128)
  for (int q = rank * per + t; q < (rank + 1) * per; q += kThreads) {
    const float* p = sm + (q >> 4) * kRP + 4 * (q & 15);
    float4 s = ld_cluster_f4(p, 0);
    for (int r = 1; r < split; ++r) {
      const float4 v = ld_cluster_f4(p, r);
      s = make_float4(__fadd_rn(s.x, v.x), __fadd_rn(s.y, v.y), __fadd_rn(s.z, v.z), __fadd_rn(s.w, v.w));
    }
    finish(q, s);
  }
  cluster_sync_all();                    // the partials have been read: every CTA may exit
}

// ------------------------------------------------------------------ weight update
// W[j][o][i] -= lr * sum_b dZ[j][b][o] H[j][b][i] (samples in ascending order, one FFMA
// chain per weight) and, in the first input tile, b_l -= lr * sum_b dZ.  CTA = 64 outputs x
// 128 inputs, thread = 8 x 8 of them; the weights are loaded into registers before the
// batch arrives, so their latency hides behind the products.  Samples go in chunks of 32
// through two cp.async stages.  3072 -> 512 (P = 16, B = 32): 48 us, 4.2 TB/s, 33 TFLOP/s
// (57 us with scalar FFMAs and lanes 4 x 8 in order, 55 with samples unrolled by two).
constexpr int kDwThreads = 128;
constexpr int kDwO = 64, kDwI = 128, kDwB = 32;
constexpr int kDwStage = kDwB * (kDwO + kDwI);
constexpr int kDwSmem = 2 * kDwStage * 4;

struct DwArgs {
  const float* dZ;             // [P][B][out]
  const float* H;              // learner j's row b at H + j * h_stride + ((row0 + b) mod N) * in
  int64_t h_stride, N, row0;
  float* W;
  float* bias;
  int64_t ld;
  int in, out, B;
  int vec_z;                   // 16-byte copies of dZ rows
  float lr;
};

// kVec (16-byte copies of H and W rows): thread columns 4 lx .. 4 lx + 3 (+ 32), else lx + 8 n.
template <bool kVec>
__global__ void __launch_bounds__(kDwThreads, 3) k_dw_f32(const DwArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, ly = lane_y(lane), lx = lane_x(lane);
  const int i0 = blockIdx.x * kDwI, o0 = blockIdx.y * kDwO;
  const int64_t j = blockIdx.z;
  grid_dep_wait();
  const int ow = 32 * (warp >> 1) + 8 * ly;       // this thread's first output in the tile
  const int iw = 64 * (warp & 1);                 // this warp's first input in the tile
  auto col = [&](int n) { return iw + (kVec ? (n < 4 ? 4 * lx + n : 28 + 4 * lx + n) : lx + 8 * n); };
  const float* Hj = a.H + j * a.h_stride;
  auto load = [&](int c, int s) {
    float* zs = sm + s * kDwStage;
    float* hs = zs + kDwB * kDwO;
    for (int r = warp; r < kDwB; r += kDwThreads / 32) {   // a warp per sample
      const int b = c * kDwB + r;
      const bool live = b < a.B;
      const float* z = a.dZ + (j * a.B + (live ? b : 0)) * a.out;
      const float* h = Hj + wrap_row(a.row0 + (live ? b : 0), a.N) * a.in;
      if (a.vec_z) {
        if (lane < 16) {
          const bool ok = live && o0 + 4 * lane < a.out;
          cp_async16(zs + r * kDwO + 4 * lane, ok ? z + o0 + 4 * lane : a.W, ok);
        }
      } else {
        for (int o = lane; o < kDwO; o += 32) {
          const bool ok = live && o0 + o < a.out;
          cp_async4(zs + r * kDwO + o, ok ? z + o0 + o : a.W, ok);
        }
      }
      if (kVec) {
        const bool ok = live && i0 + 4 * lane < a.in;
        cp_async16(hs + r * kDwI + 4 * lane, ok ? h + i0 + 4 * lane : a.W, ok);
      } else {
        for (int i = lane; i < kDwI; i += 32) {
          const bool ok = live && i0 + i < a.in;
          cp_async4(hs + r * kDwI + i, ok ? h + i0 + i : a.W, ok);
        }
      }
    }
  };
  const int nb = (a.B + kDwB - 1) / kDwB;
  load(0, 0);
  cp_async_commit();
  float* Wj = a.W + j * a.ld + static_cast<int64_t>(o0 + ow) * a.in + i0;
  float w[8][8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const bool orow = o0 + ow + e < a.out;
    if constexpr (kVec) {
#pragma unroll
      for (int n = 0; n < 8; n += 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (orow && i0 + col(n) < a.in)
          v = *reinterpret_cast<const float4*>(Wj + static_cast<int64_t>(e) * a.in + col(n));
        w[e][n] = v.x; w[e][n + 1] = v.y; w[e][n + 2] = v.z; w[e][n + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int n = 0; n < 8; ++n)
        w[e][n] = orow && i0 + col(n) < a.in ? Wj[static_cast<int64_t>(e) * a.in + col(n)] : 0.f;
    }
  }
  uint64_t acc[8][4];                  // columns (0, 1), (2, 3), ... of each output
#pragma unroll
  for (int e = 0; e < 8; ++e)
#pragma unroll
    for (int n = 0; n < 4; ++n) acc[e][n] = 0;
  float db = 0.f;
  for (int c = 0; c < nb; ++c) {
    if (c + 1 < nb) load(c + 1, (c + 1) & 1);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    const float* zs = sm + (c & 1) * kDwStage;
    const float* hs = zs + kDwB * kDwO;
    const int rows = a.B - c * kDwB < kDwB ? a.B - c * kDwB : kDwB;
    for (int r = 0; r < rows; ++r) {
      float z[8];
      uint64_t h[4];
      *reinterpret_cast<float4*>(z) = *reinterpret_cast<const float4*>(zs + r * kDwO + ow);
      *reinterpret_cast<float4*>(z + 4) = *reinterpret_cast<const float4*>(zs + r * kDwO + ow + 4);
      if constexpr (kVec) {
        *reinterpret_cast<ulonglong2*>(h) = *reinterpret_cast<const ulonglong2*>(hs + r * kDwI + col(0));
        *reinterpret_cast<ulonglong2*>(h + 2) = *reinterpret_cast<const ulonglong2*>(hs + r * kDwI + col(4));
      } else {
#pragma unroll
        for (int n = 0; n < 4; ++n) h[n] = pack2(hs[r * kDwI + col(2 * n)], hs[r * kDwI + col(2 * n + 1)]);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint64_t zz = pack2(z[e], z[e]);
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[e][n] = fma2(zz, h[n], acc[e][n]);
      }
    }
    if (blockIdx.x == 0 && t < kDwO)
      for (int r = 0; r < rows; ++r) db = __fadd_rn(db, zs[r * kDwO + t]);
    __syncthreads();           // the stage may be replaced
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (o0 + ow + e >= a.out) break;
#pragma unroll
    for (int n = 0; n < 8; n += 2) {
      const float2 g = unpack2(acc[e][n / 2]);
      w[e][n] = __fsub_rn(w[e][n], __fmul_rn(a.lr, g.x));
      w[e][n + 1] = __fsub_rn(w[e][n + 1], __fmul_rn(a.lr, g.y));
    }
    if constexpr (kVec) {
#pragma unroll
      for (int n = 0; n < 8; n += 4)
        if (i0 + col(n) < a.in)
          *reinterpret_cast<float4*>(Wj + static_cast<int64_t>(e) * a.in + col(n)) =
              make_float4(w[e][n], w[e][n + 1], w[e][n + 2], w[e][n + 3]);
    } else {
#pragma unroll
      for (int n = 0; n < 8; ++n)
        if (i0 + col(n) < a.in) Wj[static_cast<int64_t>(e) * a.in + col(n)] = w[e][n];
    }
  }
  if (blockIdx.x == 0 && t < kDwO && o0 + t < a.out) {
    float* p = a.bias + j * a.ld + o0 + t;
    *p = __fsub_rn(*p, __fmul_rn(a.lr, db));
  }
}

// ------------------------------------------------------------------ cross-entropy
// One CTA per learner, one warp per sample: dZ = (softmax(z_b) - onehot(y_b)) / B, loss =
// mean CE.  Each lane's logits go in blocks of eight loads in flight.
constexpr int kXentThreads = 1024;
__global__ void __launch_bounds__(kXentThreads) k_xent_f32(const float* __restrict__ Z,
                                                          const int32_t* __restrict__ y, int64_t N,
                                                          int64_t row0, int B, int C,
                                                          float* __restrict__ dZ,
                                                          float* __restrict__ loss) {
  extern __shared__ float row_loss[];
  grid_dep_wait();
  const int j = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float fB = static_cast<float>(B);
  for (int b = warp; b < B; b += kXentThreads / 32) {
    const float* z = Z + (static_cast<int64_t>(j) * B + b) * C;
    float* d = dZ + (static_cast<int64_t>(j) * B + b) * C;
    const int yb = y[static_cast<int64_t>(j) * N + (row0 + b) % N];
    float m = -INFINITY;
    for (int c0 = lane; c0 < C; c0 += 256) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = c0 + 32 * k < C ? z[c0 + 32 * k] : -INFINITY;
#pragma unroll
      for (int k = 0; k < 8; ++k) m = fmaxf(m, v[k]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    float s = 0.f;
    for (int c0 = lane; c0 < C; c0 += 256) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = c0 + 32 * k < C ? z[c0 + 32 * k] : 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (c0 + 32 * k < C) s += expf(v[k] - m);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) row_loss[b] = logf(s) + m - z[yb];
    for (int c0 = lane; c0 < C; c0 += 256) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = c0 + 32 * k < C ? z[c0 + 32 * k] : 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int c = c0 + 32 * k;
        if (c < C) d[c] = __fdiv_rn(__fsub_rn(__fdiv_rn(expf(v[k] - m), s), yb == c ? 1.f : 0.f), fB);
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float l = 0.f;
    for (int b = 0; b < B; ++b) l += row_loss[b];
    loss[j] = l / B;
  }
}

// The same over a cluster of up to 8 CTAs per learner, each with `per` samples: one warp per
// sample takes its maximum and sum of exponentials, then all threads form dZ; rank 0 adds the
// samples' losses in order.  Bound by the exponentials and divisions, ~70 instructions per logit
// (8 learners, B = 32, 1496 classes: 18.1 us per launch in one CTA, 11.8 here).  Below about 12 K
// logits per learner the cluster's launch and barriers cost more than it saves (P = 32, 99
// classes, B = 26: a round of 8 steps 680 against 688 us here).
constexpr int kXentcThreads = 256, kXentRanks = 8;
constexpr int kXentSpread = 12288;                 // logits per learner
__global__ void __launch_bounds__(kXentcThreads) k_xent_f32_cluster(const float* __restrict__ Z,
                                                          const int32_t* __restrict__ y, int64_t N,
                                                          int64_t row0, int B, int C, int per,
                                                          float* __restrict__ dZ,
                                                          float* __restrict__ loss) {
  extern __shared__ float sm[];                    // per sample: loss, maximum, sum, label
  __shared__ float gathered[kXentcThreads];
  float *row_loss = sm, *row_max = sm + per, *row_sum = sm + 2 * per;
  int* row_y = reinterpret_cast<int*>(sm + 3 * per);
  grid_dep_wait();
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int64_t j = blockIdx.y;
  const int b0 = blockIdx.x * per, nb = B - b0 < per ? B - b0 : per;
  const float* Zb = Z + (j * B + b0) * C;
  for (int i = warp; i < nb; i += kXentcThreads / 32) {
    const float* z = Zb + static_cast<int64_t>(i) * C;
    float m = -INFINITY;
    for (int c0 = lane; c0 < C; c0 += 256) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = c0 + 32 * k < C ? z[c0 + 32 * k] : -INFINITY;
#pragma unroll
      for (int k = 0; k < 8; ++k) m = fmaxf(m, v[k]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    float s = 0.f;
    for (int c0 = lane; c0 < C; c0 += 256) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = c0 + 32 * k < C ? z[c0 + 32 * k] : 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (c0 + 32 * k < C) s += expf(v[k] - m);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
      const int yb = y[j * N + wrap_row(row0 + b0 + i, N)];
      row_max[i] = m;
      row_sum[i] = s;
      row_y[i] = yb;
      row_loss[i] = logf(s) + m - z[yb];
    }
  }
  __syncthreads();
  cluster_arrive();
  const float fB = static_cast<float>(B);
  float* d = dZ + (j * B + b0) * C;
  for (int c = t; c < C; c += kXentcThreads)
#pragma unroll 4
    for (int i = 0; i < nb; ++i) {
      const int64_t at = static_cast<int64_t>(i) * C + c;
      const float p = __fdiv_rn(expf(Zb[at] - row_max[i]), row_sum[i]);
      d[at] = __fdiv_rn(__fsub_rn(p, row_y[i] == c ? 1.f : 0.f), fB);
    }
  cluster_wait();                                  // every rank's losses are written
  if (blockIdx.x == 0) {
    float l = 0.f;
    for (int base = 0; base < B; base += kXentcThreads) {
      const int b = base + t;
      if (b < B) gathered[t] = ld_cluster_f1(row_loss + b % per, b / per);
      __syncthreads();
      if (t == 0) {
        const int n = B - base < kXentcThreads ? B - base : kXentcThreads;
#pragma unroll 8
        for (int i = 0; i < n; ++i) l += gathered[i];
      }
      __syncthreads();
    }
    if (t == 0) loss[j] = l / B;
  }
  cluster_sync_all();                              // the losses have been read: every CTA may exit
}

// ------------------------------------------------------------------ small last layer
// The last layer with at most 16 classes in one launch: a cluster of S CTAs per learner,
// CTA s owning the input features [s F, s F + F): partial logits, summed over the ranks in
// order through distributed shared memory (every rank alike), softmax cross-entropy, then
// dZ_{L-1} and b_{L-1} (with W_L before its update) and W_L, b_L for its features.  What
// bounds it is latency: one round trip of loads, one cluster barrier, ~1 us of arithmetic
// (6.5 us at 37 -> 10, 10.7 us at 512 -> 10 with 16 learners, B = 32).
// A one-layer model (has_dx = 0, rows from X) may run `steps` local steps in the launch:
// W_L stays in shared memory and the next step's rows load during the current step (two
// steps of 3072 -> 10, P = 4, B = 16: 15 us).
constexpr int kHeadC = 16, kHeadB = 64, kHeadSplit = 8;
constexpr int kHeadSmemMax = 200 * 1024;

// Features per CTA: at least 64, a multiple of 4, at most kHeadSplit slices.
__host__ __device__ inline int head32_slice(int in) {
  const int f = ((in + kHeadSplit - 1) / kHeadSplit + 3) / 4 * 4;
  return f < 64 ? 64 : f;
}
// H slices (bufs) | W slice | zp[2], g | losses, labels[2], b_L
inline int head32_smem(int in, int B, int bufs) {
  return 4 * (head32_slice(in) * (bufs * B + kHeadC) + 3 * kHeadB * kHeadC + 3 * kHeadB + kHeadC);
}

__device__ __forceinline__ float4 fma4(float s, float4 v, float4 a) {
  return make_float4(fmaf(s, v.x, a.x), fmaf(s, v.y, a.y), fmaf(s, v.z, a.z), fmaf(s, v.w, a.w));
}

__global__ void __launch_bounds__(kThreads) k_head_f32(const Head32Args a) {
  extern __shared__ __align__(16) float sm[];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int s = blockIdx.x, S = gridDim.x, C = a.C, B = a.B, in = a.in;
  const int64_t j = blockIdx.y;
  const int F = head32_slice(in), k0 = s * F, kc = in - k0 < F ? in - k0 : F, nq = F / 4;
  float* hs0 = sm;                                   // [bufs][B][F] H rows
  float* ws = hs0 + a.bufs * B * F;                  // [16][F]      W_L
  float* zp0 = ws + kHeadC * F;                      // [2][64][16]  partial logits
  float* g = zp0 + 2 * kHeadB * kHeadC;              // [64][16]     gradient
  float* rl = g + kHeadB * kHeadC;                   // [64]         loss of a sample
  int* ys0 = reinterpret_cast<int*>(rl + kHeadB);    // [2][64]      labels
  float* bls = reinterpret_cast<float*>(ys0 + 2 * kHeadB);   // [16] b_L
  float* W = a.W + j * a.ld;
  const int64_t N = a.N;
  auto load_batch = [&](int step) {
    float* hs = hs0 + (step % a.bufs) * B * F;
    const float* hj = a.H + j * a.h_stride;
    const int64_t r0 = a.x_rows ? a.row0 + static_cast<int64_t>(step) * B : 0;
    if (a.vec) {
      for (int idx = t; idx < B * nq; idx += kThreads) {
        const int b = idx / nq, q = idx - b * nq;
        const bool ok = 4 * q < kc;
        const float* p = hj + (a.x_rows ? wrap_row(r0 + b, N) : b) * in + k0 + 4 * q;
        cp_async16(hs + b * F + 4 * q, ok ? p : W, ok);
      }
    } else {
      for (int idx = t; idx < B * F; idx += kThreads) {
        const int b = idx / F, f = idx - b * F;
        const bool ok = f < kc;
        const float* p = hj + (a.x_rows ? wrap_row(r0 + b, N) : b) * in + k0 + f;
        cp_async4(hs + b * F + f, ok ? p : W, ok);
      }
    }
    if (t < B) ys0[(step & 1) * kHeadB + t] = a.y[j * N + (a.row0 + static_cast<int64_t>(step) * B + t) % N];
  };
  grid_dep_wait();
  load_batch(0);
  if (a.vec) {
    for (int idx = t; idx < kHeadC * nq; idx += kThreads) {
      const int c = idx / nq, q = idx - c * nq;
      const bool ok = c < C && 4 * q < kc;
      cp_async16(ws + c * F + 4 * q, ok ? W + static_cast<int64_t>(c) * in + k0 + 4 * q : W, ok);
    }
  } else {
    for (int idx = t; idx < kHeadC * F; idx += kThreads) {
      const int c = idx / F, f = idx - c * F;
      const bool ok = c < C && f < kc;
      cp_async4(ws + c * F + f, ok ? W + static_cast<int64_t>(c) * in + k0 + f : W, ok);
    }
  }
  cp_async_commit();
  if (t < kHeadC) bls[t] = t < C ? a.bias[j * a.ld + t] : 0.f;

  for (int step = 0; step < a.steps; ++step) {
    const float* hs = hs0 + (step % a.bufs) * B * F;
    const int* ys = ys0 + (step & 1) * kHeadB;
    float* zp = zp0 + (step & 1) * kHeadB * kHeadC;
    cp_async_wait<0>();
    __syncthreads();
    if (a.bufs == 2 && step + 1 < a.steps) {
      load_batch(step + 1);
      cp_async_commit();
    }
    // ---- partial logits: a warp takes 4 samples x 8 classes, its lanes the features
    const int units = (B + 3) / 4 * ((C + 7) / 8);
    for (int u = warp; u < units; u += kThreads / 32) {
      const int bu = (u % ((B + 3) / 4)) * 4, cu = (u / ((B + 3) / 4)) * 8;
      float v[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = 0.f;
      for (int q = lane; q < nq; q += 32) {
        float4 h[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          h[i] = *reinterpret_cast<const float4*>(hs + (bu + i < B ? bu + i : bu) * F + 4 * q);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float4 w = *reinterpret_cast<const float4*>(ws + (cu + c) * F + 4 * q);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float x = v[8 * i + c];
            x = fmaf(h[i].x, w.x, x);
            x = fmaf(h[i].y, w.y, x);
            x = fmaf(h[i].z, w.z, x);
            v[8 * i + c] = fmaf(h[i].w, w.w, x);
          }
        }
      }
      // sum each of the 32 values over the lanes; lane l ends with value l
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < off; ++i) {
          const float send = up ? v[i] : v[i + off], keep = up ? v[i + off] : v[i];
          v[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, off));
        }
      }
      zp[(bu + (lane >> 3)) * kHeadC + cu + (lane & 7)] = v[0];
    }
    // ---- logits (ranks in order) and softmax cross-entropy, 16 lanes per sample.  One
    // cluster barrier per step: zp alternates, and a rank writes it again only after the
    // next step's barrier, which follows every rank's reads here.
    cluster_sync_all();
    float zv[kHeadB * kHeadC / kThreads];          // every turn's remote loads in flight
#pragma unroll
    for (int i = 0; i < kHeadB * kHeadC / kThreads; ++i) {
      const int e = t + i * kThreads, b = e >> 4, c = e & 15;
      zv[i] = 0.f;
      if (b >= B || c >= C) continue;
      float v[kHeadSplit];
#pragma unroll
      for (int r = 0; r < kHeadSplit; ++r) v[r] = r < S ? ld_cluster_f1(zp + e, r) : 0.f;
      float z = v[0];
#pragma unroll
      for (int r = 1; r < kHeadSplit; ++r)
        if (r < S) z = __fadd_rn(z, v[r]);
      zv[i] = __fadd_rn(z, bls[c]);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kHeadB * kHeadC / kThreads; ++i) {
      const int e = t + i * kThreads, b = e >> 4, c = e & 15;
      if (i * kThreads / kHeadC >= B) break;
      const bool live = b < B && c < C;
      const float z = zv[i];
      float m = live ? z : -INFINITY;
#pragma unroll
      for (int off = 1; off < kHeadC; off <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
      const float ex = live ? expf(z - m) : 0.f;
      float sum = ex;
#pragma unroll
      for (int off = 1; off < kHeadC; off <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
      float gv = 0.f;
      if (live) {
        gv = __fdiv_rn(__fsub_rn(__fdiv_rn(ex, sum), c == ys[b] ? 1.f : 0.f), static_cast<float>(B));
        if (c == ys[b]) rl[b] = logf(sum) + m - z;
      }
      g[e] = gv;
    }
    __syncthreads();
    // ---- backward: thread = (feature quad q, group grp of ng)
    const int ng = kThreads / nq, q = t % nq, grp = t / nq;
    if (a.has_dx && grp < ng) {
      // dZ_{L-1} of samples grp, grp + ng, ... (b_{L-1} is updated from it with W_{L-1})
      float4 w[kHeadC];
#pragma unroll
      for (int c = 0; c < kHeadC; ++c) w[c] = *reinterpret_cast<const float4*>(ws + c * F + 4 * q);
      for (int b = grp; b < B; b += ng) {
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < kHeadC; c += 4) {
          const float4 gv = *reinterpret_cast<const float4*>(g + b * kHeadC + c);
          d = fma4(gv.x, w[c], d);
          d = fma4(gv.y, w[c + 1], d);
          d = fma4(gv.z, w[c + 2], d);
          d = fma4(gv.w, w[c + 3], d);
        }
        const float4 h = *reinterpret_cast<const float4*>(hs + b * F + 4 * q);
        d = make_float4(h.x > 0.f ? d.x : 0.f, h.y > 0.f ? d.y : 0.f, h.z > 0.f ? d.z : 0.f,
                        h.w > 0.f ? d.w : 0.f);
        float* o = a.dz_prev + (j * B + b) * in + k0 + 4 * q;
        if (a.vec) {
          if (4 * q < kc) *reinterpret_cast<float4*>(o) = d;
        } else {
          if (4 * q < kc) o[0] = d.x;
          if (4 * q + 1 < kc) o[1] = d.y;
          if (4 * q + 2 < kc) o[2] = d.z;
          if (4 * q + 3 < kc) o[3] = d.w;
        }
      }
    }
    if (a.has_dx) __syncthreads();   // every dX has read W_L before it is updated
    const bool last = step + 1 == a.steps;
    if (grp < ng) {
      // W_L of classes c0 .. c0 + 3: samples in ascending order, one FFMA chain per weight
      for (int c0 = 4 * grp; c0 < C; c0 += 4 * ng) {
        float4 d[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) d[e] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int b = 0; b < B; ++b) {
          const float4 h = *reinterpret_cast<const float4*>(hs + b * F + 4 * q);
          const float4 gv = *reinterpret_cast<const float4*>(g + b * kHeadC + c0);
          d[0] = fma4(gv.x, h, d[0]);
          d[1] = fma4(gv.y, h, d[1]);
          d[2] = fma4(gv.z, h, d[2]);
          d[3] = fma4(gv.w, h, d[3]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (c0 + e >= C) break;
          float4* pw = reinterpret_cast<float4*>(ws + (c0 + e) * F + 4 * q);
          float4 w = *pw;
          w = make_float4(__fsub_rn(w.x, __fmul_rn(a.lr, d[e].x)), __fsub_rn(w.y, __fmul_rn(a.lr, d[e].y)),
                          __fsub_rn(w.z, __fmul_rn(a.lr, d[e].z)), __fsub_rn(w.w, __fmul_rn(a.lr, d[e].w)));
          *pw = w;
          if (!last) continue;
          float* o = W + static_cast<int64_t>(c0 + e) * in + k0 + 4 * q;
          if (a.vec) {
            if (4 * q < kc) *reinterpret_cast<float4*>(o) = w;
          } else {
            if (4 * q < kc) o[0] = w.x;
            if (4 * q + 1 < kc) o[1] = w.y;
            if (4 * q + 2 < kc) o[2] = w.z;
            if (4 * q + 3 < kc) o[3] = w.w;
          }
        }
      }
    }
    // every rank keeps b_L; rank 0 writes it and the loss (the last warp, which has no weights
    // to update where slices are narrow)
    if (t >= kThreads - 32 && lane < C) {
      float db = 0.f;
#pragma unroll 8
      for (int b = 0; b < B; ++b) db = __fadd_rn(db, g[b * kHeadC + lane]);
      bls[lane] = __fsub_rn(bls[lane], __fmul_rn(a.lr, db));
      if (last && s == 0) a.bias[j * a.ld + lane] = bls[lane];
    } else if (last && s == 0 && t == kThreads - 1) {
      float l = 0.f;
#pragma unroll 8
      for (int b = 0; b < B; ++b) l += rl[b];
      a.loss[j] = l / B;
    }
    if (!last && a.bufs == 1) {
      __syncthreads();               // the batch has been read
      load_batch(step + 1);
      cp_async_commit();
    }
  }
  cluster_sync_all();                // the partials have been read: every CTA may exit
}

bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

// CTAs of a cluster that share a tile's reduction (a power of two up to 8, at least two
// chunks each): the least work on the fullest SM, in chunks, with four chunks' worth of
// start and reduction per CTA, and a fifth on top where every SM holds one CTA at most
// (nothing covers its waits).  3072 -> 512 (P = 16, B = 32: 128 tiles of 48 chunks), split
// 1, 2, 4, 8: 63.5, 58.3, 63.2, 68.2 us.
int tile_split(int64_t tiles, int K) {
  const int64_t nk = (K + kKC - 1) / kKC;
  int best = 1;
  int64_t cost = 0;
  for (int s = 1; s <= 8 && (s == 1 || nk >= 2 * s); s *= 2) {
    const int64_t per_sm = (tiles * s + kSms - 1) / kSms;
    const int64_t c = per_sm * ((nk + s - 1) / s + 4) * (per_sm == 1 ? 6 : 5);
    if (s == 1 || c < cost) {
      cost = c;
      best = s;
    }
  }
  return best;
}

template <int BM, bool kDx>
cudaError_t launch_tile(const TileArgs& a, int P, cudaStream_t s) {
  const int cols = kDx ? a.in : a.out;
  const int64_t ct = (cols + kBN - 1) / kBN, bt = (a.B + BM - 1) / BM;
  const int split = tile_split(ct * bt * P, kDx ? a.out : a.in);
  return launch_pdl(k_tile_f32<BM, kDx>, dim3(static_cast<unsigned>(ct * split), static_cast<unsigned>(bt), P),
                    dim3(kThreads), tile_smem(BM), s, false, split, a, split);
}

// Samples per tile: the smallest that holds the batch, up to 64 (B > 64: tiles of 64).
template <bool kDx>
cudaError_t launch_tile_any(const TileArgs& a, int P, cudaStream_t s) {
  if (a.B <= 8) return launch_tile<8, kDx>(a, P, s);
  if (a.B <= 16) return launch_tile<16, kDx>(a, P, s);
  if (a.B <= 32) return launch_tile<32, kDx>(a, P, s);
  return launch_tile<64, kDx>(a, P, s);
}

template <int BM, bool kDx>
cudaError_t tile_configure() {
  return cudaFuncSetAttribute(k_tile_f32<BM, kDx>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              tile_smem(BM));
}

}  // namespace

cudaError_t fp32_configure() {
  cudaError_t e = cudaSuccess;
  for (cudaError_t r : {tile_configure<8, false>(), tile_configure<16, false>(), tile_configure<32, false>(),
                        tile_configure<64, false>(), tile_configure<8, true>(), tile_configure<16, true>(),
                        tile_configure<32, true>(), tile_configure<64, true>(),
                        cudaFuncSetAttribute(k_dw_f32<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmem),
                        cudaFuncSetAttribute(k_dw_f32<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmem),
                        cudaFuncSetAttribute(k_head_f32, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kHeadSmemMax)})
    if (e == cudaSuccess) e = r;
  return e;
}

cudaError_t launch_fwd_f32(const F32Rows& h, const float* W, const float* bias, int64_t ld, int in,
                           int out, int B, int relu, float* out_act, int P, cudaStream_t s) {
  TileArgs a{};
  a.act = h.base;
  a.act_stride = h.stride;
  a.N = h.N;
  a.row0 = h.row0;
  a.W = W;
  a.ld = ld;
  a.in = in;
  a.out = out;
  a.B = B;
  a.vec_act = in % 4 == 0 && aligned16(h.base);
  a.vec_w = in % 4 == 0;
  a.bias = bias;
  a.relu = relu;
  a.y = out_act;
  return launch_tile_any<false>(a, P, s);
}

cudaError_t launch_dx_f32(const float* dZ, const float* W, int64_t ld, const float* Hprev, int in,
                          int out, int B, float* dZprev, int P, cudaStream_t s) {
  TileArgs a{};
  a.act = dZ;
  a.act_stride = static_cast<int64_t>(B) * out;
  a.N = B;
  a.W = W;
  a.ld = ld;
  a.in = in;
  a.out = out;
  a.B = B;
  a.vec_act = out % 4 == 0;
  a.vec_w = in % 4 == 0;
  a.mask = Hprev;
  a.y = dZprev;
  return launch_tile_any<true>(a, P, s);
}

cudaError_t launch_xent_f32(const float* Z, const int32_t* y, int64_t N, int64_t row0, int B,
                            int C, float* dZ, float* loss, int P, cudaStream_t s) {
  if (static_cast<int64_t>(B) * C >= kXentSpread) {
    const int per = (B + kXentRanks - 1) / kXentRanks, ranks = (B + per - 1) / per;
    return launch_pdl(k_xent_f32_cluster, dim3(ranks, P), dim3(kXentcThreads), static_cast<size_t>(per) * 16, s,
                      false, ranks, Z, y, N, row0, B, C, per, dZ, loss);
  }
  return launch_pdl(k_xent_f32, dim3(P), dim3(kXentThreads), static_cast<size_t>(B) * sizeof(float), s,
                    false, 1, Z, y, N, row0, B, C, dZ, loss);
}

cudaError_t launch_dw_update_f32(const float* dZ, const F32Rows& h, float* W, float* bias, int64_t ld,
                                 int in, int out, int B, float lr, int P, cudaStream_t s) {
  DwArgs a{};
  a.dZ = dZ;
  a.H = h.base;
  a.h_stride = h.stride;
  a.N = h.N;
  a.row0 = h.row0;
  a.W = W;
  a.bias = bias;
  a.ld = ld;
  a.in = in;
  a.out = out;
  a.B = B;
  a.lr = lr;
  a.vec_z = out % 4 == 0;
  const dim3 grid((in + kDwI - 1) / kDwI, (out + kDwO - 1) / kDwO, P);
  if (in % 4 == 0 && aligned16(h.base))
    return launch_pdl(k_dw_f32<true>, grid, dim3(kDwThreads), kDwSmem, s, false, 1, a);
  return launch_pdl(k_dw_f32<false>, grid, dim3(kDwThreads), kDwSmem, s, false, 1, a);
}

bool head32_supported(int C, int in, int B) {
  return C <= kHeadC && B <= kHeadB && head32_slice(in) <= 4 * kThreads &&
         head32_smem(in, B, 1) <= kHeadSmemMax;
}

cudaError_t launch_head_f32(const Head32Args& args, int P, cudaStream_t s) {
  Head32Args a = args;
  a.bufs = a.steps > 1 && head32_smem(a.in, a.B, 2) <= kHeadSmemMax ? 2 : 1;
  a.vec = a.in % 4 == 0 && aligned16(a.H);
  const int F = head32_slice(a.in), S = (a.in + F - 1) / F;
  return launch_pdl(k_head_f32, dim3(S, P), dim3(kThreads), head32_smem(a.in, a.B, a.bufs), s, false, S, a);
}

}  // namespace ha
