// Whole local steps of a small net in one launch (Algorithm 1 inner loop, Sec. 3.1): forward,
// softmax cross-entropy, backward and update of every layer, for one or several consecutive
// steps.  One cluster of eight CTAs per learner; CTA s owns a slice of every layer's inputs:
// features [s F, s F + F) of the batch rows, of each hidden layer, and the same columns of the
// weights that read them, which stay in its shared memory across the launch's steps.
//   forward    partial products of its slice for all outputs; after a cluster barrier each CTA
//              adds the eight partials of its own neurons in rank order (distributed shared
//              memory), adds the bias and applies the ReLU
//   logits     every CTA adds all of them and forms the whole gradient, so nothing is sent
//   backward   dZ of its own neurons from the whole dZ of the next layer and its own columns,
//              sent to the others while the columns are updated (arrive ... update ... wait)
// So a step costs 2 L - 1 cluster barriers and no launch between them.  What bounds it is
// latency (barriers, phases of under a microsecond on 8 of the SMs per learner); products run
// as FFMA on 4 x 4 outputs per thread.  bf16 operands are rounded to bf16 values held in fp32,
// whose products are exact in fp32.
// (264-136-200-13, P = 6, B = 20: 18.5 us per step of a round, 22.5 by step(), 5 cluster barriers and
// some 15 phases of 1000 to 5000 cycles; 512 threads instead of 256 took as long.  The weights
// come by cp.async, all layers in flight, and leave from the last update: 29 us by step() with
// plain loads, a pass of its own for the stores and dZ rows on the same banks.  Up to 16 classes
// take 16 lanes per sample, and b_L and the loss are the last warp's while the others go on:
// 784-40-10, B = 64 21 -> 18.5 us per step.)
#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace ha {
namespace {

constexpr int kT = 256;                 // threads
constexpr int kR = 8;                   // CTAs of a cluster
constexpr int kSmallSmemMax = 200 * 1024;

__host__ __device__ constexpr int slice(int d) { return ((d + kR - 1) / kR + 3) / 4 * 4; }
// Row pitch of a slice: an odd number of 16-byte quads, so that consecutive rows fall on
// distinct bank groups.
__host__ __device__ constexpr int pitch(int F) { return (F / 4 | 1) * 4; }

inline int round4(int n) { return (n + 3) / 4 * 4; }

SmallLayout small_layout(const int* dims, int L, int B, bool bf16) {
  SmallLayout s{};
  int at = 0;
  auto take = [&](int n) {
    const int o = at;
    at += round4(n);
    return o;
  };
  const int B4 = round4(B);
  for (int l = 0; l < L; ++l) {
    const int p = pitch(slice(dims[l]));
    s.w[l] = take(dims[l + 1] * p);
    s.wq[l] = bf16 ? take(dims[l + 1] * p) : s.w[l];
    s.h[l] = take(B4 * p);
    s.bias[l] = take(l + 1 < L ? slice(dims[l + 1]) : dims[L]);
    const int op = kR * slice(dims[l + 1]);
    s.wide = op > s.wide ? op : s.wide;
  }
  s.z[0] = take(B4 * s.wide);
  s.z[1] = take(B4 * s.wide);
  s.dz = take(B4 * (s.wide + 4));
  s.own[0] = take(B4 * (s.wide / kR));
  s.own[1] = take(B4 * (s.wide / kR));
  s.g = take(B4 * kSmallC);
  s.loss = take(B4);
  s.labels = take(2 * B4);
  s.raw = take(bf16 ? (B * slice(dims[0]) + 1) / 2 : B * slice(dims[0]));
  s.total = at;
  return s;
}

__device__ __forceinline__ float4 fma4(float s, float4 v, float4 a) {
  return make_float4(fmaf(s, v.x, a.x), fmaf(s, v.y, a.y), fmaf(s, v.z, a.z), fmaf(s, v.w, a.w));
}
__device__ __forceinline__ float dot4(float4 a, float4 b, float c) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
  return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
}
template <bool kBf16>
__device__ __forceinline__ float rnd(float v) {
  return kBf16 ? __bfloat162float(__float2bfloat16_rn(v)) : v;
}
template <bool kBf16>
__device__ __forceinline__ float4 rnd4(float4 v) {
  return make_float4(rnd<kBf16>(v.x), rnd<kBf16>(v.y), rnd<kBf16>(v.z), rnd<kBf16>(v.w));
}
__device__ __forceinline__ float upd(float w, float lr, float g) { return __fsub_rn(w, __fmul_rn(lr, g)); }

// i / d for i * d < 2^32.
struct Div {
  uint32_t d, m;
  __device__ __forceinline__ explicit Div(int n) : d(n), m(n == 1 ? 0u : 0xffffffffu / n + 1u) {}
  __device__ __forceinline__ int operator()(int i) const { return d == 1 ? i : static_cast<int>(__umulhi(i, m)); }
};

// Partial products z[b][n] = sum_f h[b][f] w[n][f] of a slice: 4 samples (b, b + nb, ...) x 4
// outputs (n, n + no, ...), so that neighbouring lanes' rows fall on distinct banks, per KS
// neighbouring lanes, which take every KS-th quad of features and then share out the 16 sums.
template <int KS>
__device__ __forceinline__ void forward_slice(const float* h, const float* w, float* z, int F, int p, int op,
                                              int nb, int out, int t) {
  const int no = (out + 3) / 4, tiles = nb * no, part = t & (KS - 1);
  const Div dno(no);
  for (int base = 0; base < tiles; base += kT / KS) {
    const int id = base + t / KS;
    if (KS > 1 ? base + (t & ~31) / KS >= tiles : id >= tiles) break;   // (whole warps shuffle)
    const int tile = id < tiles ? id : tiles - 1;
    const int bb = dno(tile), n = tile - bb * no;
    float acc[16] = {};
    const float* wr[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) wr[e] = w + (n + e * no < out ? n + e * no : n) * p;
    const float* hr = h + bb * p;
#pragma unroll 2
    for (int f = 4 * part; f < F; f += 4 * KS) {
      float4 hv[4], wv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) hv[i] = *reinterpret_cast<const float4*>(hr + i * nb * p + f);
#pragma unroll
      for (int e = 0; e < 4; ++e) wv[e] = *reinterpret_cast<const float4*>(wr[e] + f);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[4 * i + e] = dot4(hv[i], wv[e], acc[4 * i + e]);
    }
    if constexpr (KS > 1) __syncwarp();
#pragma unroll
    for (int off = KS / 2, half = 8; off > 0; off >>= 1, half >>= 1) {
      const bool up = t & off;
#pragma unroll
      for (int i = 0; i < half; ++i) {
        const float send = up ? acc[i] : acc[i + half], keep = up ? acc[i + half] : acc[i];
        acc[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, off));
      }
    }
    if (id >= tiles) continue;
#pragma unroll
    for (int k = 0; k < 16 / KS; ++k) {
      const int v = part * (16 / KS) + k, i = v >> 2, c = n + (v & 3) * no;
      if (c < out) z[(bb + i * nb) * op + c] = acc[k];
    }
  }
}

// Logits (the ranks' partials in order, then b_L) and softmax cross-entropy of the whole batch,
// LC lanes per sample, every turn's remote loads in flight: dz (rounded), g and the samples' losses.
template <bool kBf16, int LC>
__device__ __forceinline__ void cross_entropy(const float* z, int op, const float* bias, const int* y, float* dz,
                                              float* g, float* loss, int B, int C, int t) {
  constexpr int kTurn = kT / LC;
  float zv[64 / kTurn];
#pragma unroll
  for (int i = 0; i < 64 / kTurn; ++i) {
    const int b = i * kTurn + t / LC, c = t % LC;
    zv[i] = 0.f;
    if (b >= B || c >= C) continue;
    float v[kR];
#pragma unroll
    for (int r = 0; r < kR; ++r) v[r] = ld_cluster_f1(z + b * op + c, r);
#pragma unroll
    for (int r = 1; r < kR; ++r) v[0] = __fadd_rn(v[0], v[r]);
    zv[i] = __fadd_rn(v[0], bias[c]);
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 64 / kTurn; ++i) {
    if (i * kTurn >= B) break;
    const int b = i * kTurn + t / LC, c = t % LC;
    const bool live = b < B && c < C;
    float m = live ? zv[i] : -INFINITY;
#pragma unroll
    for (int off = 1; off < LC; off <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    const float ex = live ? expf(zv[i] - m) : 0.f;
    float sum = ex;
#pragma unroll
    for (int off = 1; off < LC; off <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (live) {
      const float gv = __fdiv_rn(__fsub_rn(__fdiv_rn(ex, sum), c == y[b] ? 1.f : 0.f), static_cast<float>(B));
      if (c == y[b]) loss[b] = logf(sum) + m - zv[i];
      dz[b * (op + 4) + c] = rnd<kBf16>(gv);
      g[b * kSmallC + c] = gv;
    }
  }
}

template <bool kBf16>
__global__ void __launch_bounds__(kT, 2) k_small(const SmallArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int t = threadIdx.x, s = blockIdx.x, L = a.L, B = a.B, C = a.dims[a.L];
  const int64_t j = blockIdx.y;
  const int B4 = (B + 3) / 4 * 4, nb = B4 / 4;
  const SmallLayout& o = a.lay;
  float* const P = a.params + j * a.ld;
  float* const dzg = sm + o.dz;
  float* const rl = sm + o.loss;
  int* const ys = reinterpret_cast<int*>(sm + o.labels);
  const int64_t N = a.N;

  // (Samples from B on and outputs beyond a layer's are computed in partly filled tiles and
  // never read; features beyond a slice's are zeros in H and W.)
  using T = std::conditional_t<kBf16, __nv_bfloat16, float>;
  T* const raw = reinterpret_cast<T*>(sm + o.raw);
  // the batch's features of this slice into raw [B][F], asynchronously
  auto load_batch = [&](int step) {
    const int F = slice(a.dims[0]), in = a.dims[0], k0 = s * F;
    const int64_t r0 = a.row0 + static_cast<int64_t>(step) * B;
    const T* X = static_cast<const T*>(a.X) + j * N * in + k0;
    if (a.vec) {
      const Div dq(F / 4);
      for (int idx = t; idx < B * (F / 4); idx += kT) {
        const int b = dq(idx), f = 4 * (idx - b * (F / 4));
        const bool ok = k0 + f < in;
        const T* src = ok ? X + wrap_row(r0 + b, N) * in + f : static_cast<const T*>(a.X);
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(raw + b * F + f)), "l"(src),
                     "n"(4 * sizeof(T)), "r"(ok ? static_cast<int>(4 * sizeof(T)) : 0)
                     : "memory");
      }
    } else if constexpr (!kBf16) {     // (rows off 16 bytes)
      const Div df(F);
      for (int idx = t; idx < B * F; idx += kT) {
        const int b = df(idx), f = idx - b * F;
        const bool ok = k0 + f < in;
        const T* src = ok ? X + wrap_row(r0 + b, N) * in + f : static_cast<const T*>(a.X);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(raw + b * F + f)), "l"(src),
                     "r"(ok ? 4 : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (t < B) ys[(step & 1) * B4 + t] = a.y[j * N + wrap_row(r0 + t, N)];
  };

  grid_dep_wait();
  load_batch(0);
  for (int l = 0; l < L; ++l) {
    const int F = slice(a.dims[l]), p = pitch(F), in = a.dims[l], out = a.dims[l + 1], k0 = s * F;
    const float* W = P + a.woff[l] + k0;
    auto copy = [&](int at, const float* src, int n, auto bytes) {   // n floats of it, then zeros
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(sm + o.w[l] + at)),
                   "l"(n > 0 ? src : P), "n"(decltype(bytes)::value), "r"(4 * n)
                   : "memory");
    };
    if (in % 4 == 0) {
      const Div dq(F / 4);
#pragma unroll 4
      for (int idx = t; idx < out * (F / 4); idx += kT) {
        const int r = dq(idx), f = 4 * (idx - r * (F / 4));
        copy(r * p + f, W + r * in + f, k0 + f < in ? 4 : 0, std::integral_constant<int, 16>{});
      }
    } else {
      const Div df(F);
      for (int idx = t; idx < out * F; idx += kT) {
        const int r = df(idx), f = idx - r * F;
        copy(r * p + f, W + r * in + f, k0 + f < in ? 1 : 0, std::integral_constant<int, 4>{});
      }
    }
    const float* bias = P + a.boff[l];
    if (l + 1 < L) {
      const int Fo = slice(out);
      for (int n = t; n < Fo; n += kT) sm[o.bias[l] + n] = s * Fo + n < out ? bias[s * Fo + n] : 0.f;
    } else {
      for (int n = t; n < out; n += kT) sm[o.bias[l] + n] = bias[n];
    }
  }

  asm volatile("cp.async.commit_group;" ::: "memory");

  int ph = 0;                           // which z buffer the next forward phase writes
  for (int step = 0; step < a.steps; ++step) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (kBf16 && step == 0) {           // the weights have arrived too
      for (int l = 0; l < L; ++l) {
        const int q = pitch(slice(a.dims[l])) / 4 * a.dims[l + 1];
        for (int idx = t; idx < q; idx += kT)
          reinterpret_cast<float4*>(sm + o.wq[l])[idx] =
              rnd4<true>(reinterpret_cast<const float4*>(sm + o.w[l])[idx]);
      }
    }
    {
      const int F = slice(a.dims[0]), p = pitch(F);
      const Div dq(F / 4);
      for (int idx = t; idx < B * (F / 4); idx += kT) {
        const int b = dq(idx), f = 4 * (idx - b * (F / 4));
        const T* src = raw + b * F + f;
        float4 v;
        if constexpr (kBf16) {
          const float2 lo = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(src)[0]);
          const float2 hi = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(src)[1]);
          v = make_float4(lo.x, lo.y, hi.x, hi.y);
        } else {
          v = *reinterpret_cast<const float4*>(src);
        }
        *reinterpret_cast<float4*>(sm + o.h[0] + b * p + f) = v;
      }
    }
    __syncthreads();
    // the next batch loads during this step
    if (step + 1 < a.steps) load_batch(step + 1);
    const int* const yb = ys + (step & 1) * B4;
    // ---------------------------------------------------------------- forward
    for (int l = 0; l < L; ++l, ph ^= 1) {
      const int F = slice(a.dims[l]), p = pitch(F), out = a.dims[l + 1];
      const int Fo = slice(out), op = kR * Fo, po = l + 1 < L ? pitch(Fo) : 0;
      const float *h = sm + o.h[l], *w = sm + o.wq[l];
      float* z = sm + o.z[ph];
      // lanes per tile: as many as leave every tile a thread, two quads each at least
      const int tiles = nb * ((out + 3) / 4), q2 = F / 8;
      if (8 * tiles <= kT && q2 >= 8) forward_slice<8>(h, w, z, F, p, op, nb, out, t);
      else if (4 * tiles <= kT && q2 >= 4) forward_slice<4>(h, w, z, F, p, op, nb, out, t);
      else if (2 * tiles <= kT && q2 >= 2) forward_slice<2>(h, w, z, F, p, op, nb, out, t);
      else forward_slice<1>(h, w, z, F, p, op, nb, out, t);
      // One barrier per phase: the buffers alternate, and a rank writes this one again only
      // after the next phase's barrier, which follows every rank's reads here.
      cluster_sync_all();
      if (l + 1 < L) {
        float* hn = sm + o.h[l + 1];
        const int q4 = Fo / 4;
        const Div dq(q4);
        for (int idx = t; idx < B * q4; idx += kT) {
          const int b = dq(idx), q = idx - b * q4, n = s * Fo + 4 * q;
          float4 v[kR];
#pragma unroll
          for (int r = 0; r < kR; ++r) v[r] = ld_cluster_f4(z + b * op + n, r);
#pragma unroll
          for (int r = 1; r < kR; ++r) v[0] = add4(v[0], v[r]);
          const float4 c = add4(v[0], *reinterpret_cast<const float4*>(sm + o.bias[l] + 4 * q));
          float4 hv = make_float4(n < out ? fmaxf(c.x, 0.f) : 0.f, n + 1 < out ? fmaxf(c.y, 0.f) : 0.f,
                                  n + 2 < out ? fmaxf(c.z, 0.f) : 0.f, n + 3 < out ? fmaxf(c.w, 0.f) : 0.f);
          *reinterpret_cast<float4*>(hn + b * po + 4 * q) = rnd4<kBf16>(hv);
        }
        __syncthreads();
      } else {
        if (C <= 16)
          cross_entropy<kBf16, 16>(z, op, sm + o.bias[l], yb, dzg, sm + o.g, rl, B, C, t);
        else
          cross_entropy<kBf16, kSmallC>(z, op, sm + o.bias[l], yb, dzg, sm + o.g, rl, B, C, t);
        __syncthreads();
        // the last warp adds b_L's gradient and the loss while the others go on
        if (t >= kT - 32 && t - (kT - 32) < C) {
          const int c = t - (kT - 32);
          float db = 0.f;
#pragma unroll 8
          for (int b = 0; b < B; ++b) db = __fadd_rn(db, sm[o.g + b * kSmallC + c]);
          sm[o.bias[l] + c] = upd(sm[o.bias[l] + c], a.lr, db);
        }
        if (s == 0 && t == kT - 33 && step + 1 == a.steps) {
          float x = 0.f;
#pragma unroll 8
          for (int b = 0; b < B; ++b) x += rl[b];
          a.loss[j] = x / B;
        }
      }
    }
    // ---------------------------------------------------------------- backward
    for (int l = L - 1; l >= 0; --l) {
      const int F = slice(a.dims[l]), p = pitch(F), out = a.dims[l + 1], q4 = F / 4;
      const int dp = kR * slice(out) + 4;       // pitch of dZ: rows on distinct bank groups
      const float* h = sm + o.h[l];
      const Div dq(q4);
      float* own = sm + o.own[l & 1];
      if (l > 0) {
        // dZ_l of the own neurons: tiles of 4 samples (b, b + nb, ...) x 4 neurons, the sum
        // over the outputs split over ng groups of threads whose partials meet in the free z
        // buffer
        const float* w = sm + o.wq[l];
        float* part = sm + o.z[ph];
        const int tiles = nb * q4;
        int ng = kT / tiles;
        ng = ng < 1 ? 1 : ng > kR ? kR : ng;
        ng = ng * F > o.wide ? o.wide / F : ng;
        const int per = (out + ng - 1) / ng;
        const Div dt(tiles);
        for (int id = t; id < tiles * ng; id += kT) {
          const int g = dt(id), tile = id - g * tiles, bb = dq(tile), q = tile - bb * q4;
          const int o1 = (g + 1) * per < out ? (g + 1) * per : out;
          float4 acc[4] = {};
          const float* d = dzg + bb * dp;
#pragma unroll 4
          for (int r = g * per; r < o1; ++r) {
            const float4 wv = *reinterpret_cast<const float4*>(w + r * p + 4 * q);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = fma4(d[i * nb * dp + r], wv, acc[i]);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4*>(part + (g * B4 + bb + i * nb) * F + 4 * q) = acc[i];
        }
        __syncthreads();
        for (int idx = t; idx < B * q4; idx += kT) {
          const int b = dq(idx), q = idx - b * q4;
          float4 v = *reinterpret_cast<const float4*>(part + b * F + 4 * q);
#pragma unroll 4
          for (int g = 1; g < ng; ++g)
            v = add4(v, *reinterpret_cast<const float4*>(part + (g * B4 + b) * F + 4 * q));
          const float4 hv = *reinterpret_cast<const float4*>(h + b * p + 4 * q);
          v = make_float4(hv.x > 0.f ? v.x : 0.f, hv.y > 0.f ? v.y : 0.f, hv.z > 0.f ? v.z : 0.f,
                          hv.w > 0.f ? v.w : 0.f);
          *reinterpret_cast<float4*>(own + b * F + 4 * q) = rnd4<kBf16>(v);
          if (kBf16) *reinterpret_cast<float4*>(part + b * F + 4 * q) = v;   // unrounded, for the bias
        }
        cluster_arrive();
        __syncthreads();
        for (int n = t; n < F; n += kT) {
          const float* src = kBf16 ? part : own;
          float db = 0.f;
#pragma unroll 8
          for (int b = 0; b < B; ++b) db = __fadd_rn(db, src[b * F + n]);
          sm[o.bias[l - 1] + n] = upd(sm[o.bias[l - 1] + n], a.lr, db);
        }
      }
      // W_l of the own columns: 4 outputs x 4 inputs per thread, samples in ascending order; the
      // last step writes it out
      const int in = a.dims[l], k0 = s * F;
      const bool last = step + 1 == a.steps;
      const int no = (out + 3) / 4;
      for (int id = t; id < no * q4; id += kT) {
        const int n = dq(id), q = id - n * q4;
        float4 acc[4] = {};
#pragma unroll 4
        for (int b = 0; b < B; ++b) {
          const float4 d = *reinterpret_cast<const float4*>(dzg + b * dp + 4 * n);
          const float4 hv = *reinterpret_cast<const float4*>(h + b * p + 4 * q);
          acc[0] = fma4(d.x, hv, acc[0]);
          acc[1] = fma4(d.y, hv, acc[1]);
          acc[2] = fma4(d.z, hv, acc[2]);
          acc[3] = fma4(d.w, hv, acc[3]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (4 * n + e >= out) break;
          const int at = (4 * n + e) * p + 4 * q;
          float4 w = *reinterpret_cast<const float4*>(sm + o.w[l] + at);
          w = make_float4(upd(w.x, a.lr, acc[e].x), upd(w.y, a.lr, acc[e].y), upd(w.z, a.lr, acc[e].z),
                          upd(w.w, a.lr, acc[e].w));
          if (!last) {
            *reinterpret_cast<float4*>(sm + o.w[l] + at) = w;
            if constexpr (kBf16) *reinterpret_cast<float4*>(sm + o.wq[l] + at) = rnd4<true>(w);
            continue;
          }
          const int left = in - k0 - 4 * q;
          float* dst = P + a.woff[l] + (4 * n + e) * in + k0 + 4 * q;
          if (in % 4 == 0) {
            if (left > 0) *reinterpret_cast<float4*>(dst) = w;
          } else {
            if (left > 0) dst[0] = w.x;
            if (left > 1) dst[1] = w.y;
            if (left > 2) dst[2] = w.z;
            if (left > 3) dst[3] = w.w;
          }
        }
      }
      __syncthreads();                  // dZ_{l+1} has been read
      if (l > 0) {
        cluster_wait();
        const int dp1 = kR * F + 4;
        const Div dc(kR * q4);
        for (int idx = t; idx < B * kR * q4; idx += kT) {
          const int b = dc(idx), c = idx - b * kR * q4, r = dq(c), q = c - r * q4;
          *reinterpret_cast<float4*>(dzg + b * dp1 + 4 * c) = ld_cluster_f4(own + b * F + 4 * q, r);
        }
        __syncthreads();
      }
    }
  }

  for (int l = 0; l < L; ++l) {
    const int out = a.dims[l + 1];
    float* bias = P + a.boff[l];
    if (l + 1 < L) {
      const int Fo = slice(out);
      for (int n = t; n < Fo; n += kT)
        if (s * Fo + n < out) bias[s * Fo + n] = sm[o.bias[l] + n];
    } else if (s == 0) {
      for (int n = t; n < out; n += kT) bias[n] = sm[o.bias[l] + n];
    }
  }
  cluster_sync_all();                   // what the others read here has been read
}

}  // namespace

// Nets that take these steps.  One wave of clusters: 15 of one CTA per SM, 19 where two fit an
// SM (784-32-10 bf16, B = 64, a round of 8 steps: P = 16 366 -> 182 us, P = 64 209 -> 466).  Up
// to 2 M multiply-adds per learner and forward.  Time here over that of the kernels per layer,
// rounds of 8 steps | loops of 4 single steps: 0.7 to 1.4 M, P = 2 0.5-0.9 | 0.55-1.0, P = 16 0.45-1.0 |
// 0.5-1.15; 2 to 2.8 M, P = 2 0.53-1.0 | 0.6-1.1; 4 M, P = 2 0.6-1.0 | 0.66-1.14, so past the line fewer
// and fewer nets gain, and single steps of some lose.  (784-40-10 bf16, P = 2, B = 64, just below
// it: 213 -> 148 us; 264-136-200-13, P = 6, B = 20, 1.3 M: 145 -> 82 us for 4 steps; fp32 100-37-10,
// P = 4, B = 7: 49 -> 37 us; 512-96-80-10, P = 2, B = 32, 1.8 M, 8 steps: 271 -> 151 us; two of
// 216 lose, single steps of fp32 784-128-10 and 1024-64-10, P = 16, B = 16: loops 74 -> 85 and 65 ->
// 69 us, their rounds 151 -> 141 and 132 -> 114.)  One layer of up to 16 classes stays with the head
// kernels (784-10 bf16, P = 16, B = 64, 28 steps: 308 against 388 us here).
constexpr int kSmallClusters = 15;       // of eight CTAs that fill an SM each
constexpr int kSmallSmemHalf = 112 * 1024;
constexpr int64_t kSmallWork = int64_t(1) << 21;

bool small_supported(const int* dims, int L, int B, int P, bool bf16) {
  if (L > kSmallLayers || dims[L] > kSmallC || B > 64 || P * kR > kSms) return false;
  int64_t w = 0;
  for (int l = 0; l < L; ++l) w += static_cast<int64_t>(dims[l]) * dims[l + 1];
  if (w * B > kSmallWork) return false;
  const int smem = small_layout(dims, L, B, bf16).total * 4;
  return smem <= (P <= kSmallClusters ? kSmallSmemMax : kSmallSmemHalf);
}

cudaError_t small_configure() {
  const cudaError_t e =
      cudaFuncSetAttribute(k_small<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmemMax);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_small<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmemMax);
}

cudaError_t launch_small(const SmallArgs& args, bool bf16, int P, cudaStream_t s) {
  SmallArgs a = args;
  a.lay = small_layout(a.dims, a.L, a.B, bf16);
  a.vec = a.dims[0] % 4 == 0 && reinterpret_cast<uintptr_t>(a.X) % 16 == 0;
  return launch_pdl(bf16 ? k_small<true> : k_small<false>, dim3(kR, P), dim3(kT),
                    static_cast<size_t>(a.lay.total) * 4, s, false, kR, a);
}

}  // namespace ha
