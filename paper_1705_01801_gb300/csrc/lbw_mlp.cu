// lbw_mlp.cu -- a small multilayer perceptron, trained and evaluated on the device, used as a
// surrogate from ensemble geometry parameters to the lowest mode frequencies the batched
// lattice-Boltzmann runs measure (the paper has no counterpart; the LBM stays the reference).
//
// Network: depth weight layers, in -> hidden -> ... -> hidden -> out, tanh after every layer
// but the last (linear).  Loss: mean over samples and outputs of (y - t)^2.  Parameters are one
// FP32 vector: for each layer W (out x in, row-major) then b (out).  Training: Adam on
// minibatches whose order comes from the caller.  Inference also exists with weights stored
// in BF16 (FP32 accumulation).  All arithmetic runs in the kernels below: training in one launch
// (train_kernel) where the network suits it; otherwise a tiled FP32 GEMM (C = op(A) op(B) with
// transposes for the backward pass), bias / activation / loss kernels, a column-sum reduction for
// bias gradients and the Adam update.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <algorithm>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "lbw_internal.h"
#include "lbw_mlp_forward.cuh"

namespace lbw {
namespace {

constexpr int TM = 64, TN = 64, TK = 16;  // GEMM tile; 256 threads, 4 x 4 outputs each

// C[m x n] = op(A) op(B) (+ bias[n]); op(A) is m x k (A stored k x m when ta), op(B) is k x n
// (B stored n x k when tb).  Leading dimensions are the stored row lengths.
template <typename WB>
__global__ void __launch_bounds__(256) gemm_kernel(const float* __restrict__ A, int lda, bool ta,
                                                   const WB* __restrict__ B, int ldb, bool tb,
                                                   float* __restrict__ C, int ldc, int m, int n, int k,
                                                   const float* __restrict__ bias, bool accumulate) {
  __shared__ float As[TK][TM + 1];
  __shared__ float Bs[TK][TN + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int row0 = blockIdx.y * TM, col0 = blockIdx.x * TN;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < k; k0 += TK) {
    for (int e = threadIdx.x; e < TM * TK; e += 256) {
      const int r = e / TK, c = e % TK;  // tile row (m), tile col (k)
      const int gm = row0 + r, gk = k0 + c;
      float v = 0.f;
      if (gm < m && gk < k) v = ta ? A[(size_t)gk * lda + gm] : A[(size_t)gm * lda + gk];
      As[c][r] = v;
    }
    for (int e = threadIdx.x; e < TN * TK; e += 256) {
      const int r = e / TK, c = e % TK;  // tile col (n), k index
      const int gn = col0 + r, gk = k0 + c;
      float v = 0.f;
      if (gn < n && gk < k) v = (float)(tb ? B[(size_t)gn * ldb + gk] : B[(size_t)gk * ldb + gn]);
      Bs[c][r] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gm = row0 + ty * 4 + i, gn = col0 + tx * 4 + j;
      if (gm < m && gn < n) {
        float v = acc[i][j] + (bias ? bias[gn] : 0.f);
        if (accumulate) v += C[(size_t)gm * ldc + gn];
        C[(size_t)gm * ldc + gn] = v;
      }
    }
}

__global__ void bias_act_kernel(float* __restrict__ Y, const float* __restrict__ b, int m, int n, bool act) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * n; e += gridDim.x * blockDim.x) {
    float v = Y[e] + b[e % n];
    Y[e] = act ? tanhf(v) : v;
  }
}

// dY = 2 (y - t) / (m n); loss partial sums per block
__global__ void mse_kernel(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ dy,
                           int count, float* __restrict__ loss) {
  __shared__ float red[256];
  float s = 0.f;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x) {
    const float d = y[e] - t[e];
    dy[e] = 2.f * d / (float)count;
    s += d * d;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(loss, red[0] / (float)count);
}

// dZ = dY (1 - y^2) through tanh, in place on dY
__global__ void tanh_back_kernel(float* __restrict__ d, const float* __restrict__ y, int count) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x)
    d[e] *= 1.f - y[e] * y[e];
}

// db[j] = sum_i dZ[i, j]
__global__ void colsum_kernel(const float* __restrict__ d, int m, int n, float* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  float s = 0.f;
  for (int i = 0; i < m; ++i) s += d[(size_t)i * n + j];
  out[j] = s;
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                            float* __restrict__ m2, int count, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x) {
    const float gi = g[e];
    const float a = b1 * m1[e] + (1.f - b1) * gi;
    const float v = b2 * m2[e] + (1.f - b2) * gi * gi;
    m1[e] = a;
    m2[e] = v;
    p[e] -= lr * (a / c1) / (sqrtf(v / c2) + eps);
  }
}

// ---------------------------------------------------------------- training in one launch ---
//
// A minibatch of the surrogate (64 rows through 7 -> 256 -> 256 -> 256 -> 8) is 53 MFLOP: under a
// microsecond of the chip's FP32 rate, but some thirty launches when every product, bias, tanh and
// update is one (340 us per step).  train_kernel runs a whole sequence of Adam steps: each CTA owns
// NPC neurons of every hidden layer (and at most one output neuron), keeps their weight rows in
// shared memory, and exchanges activations and deltas with the others through the L2.  Per step a
// CTA
//   forward   reads the layer's input (all rows), forms its neurons' outputs, publishes them;
//   output    forms all outputs and their deltas itself (out is small), then its neurons' deltas;
//   backward  reads the deltas of the layer above and its columns of that layer's weights;
//   update    sums its rows' gradients over the batch and applies Adam to its own parameters,
// with one barrier after each published layer (2 depth - 3 per step) and the gradient sums of the
// layer above between arriving at it and waiting for the others.  Updated parameters go to the
// other of two parameter buffers, so a slower CTA still reads this step's columns.  The launch is
// cooperative and every wait is bounded (*err is raised).  Measured, 400 steps of the network above:
// 340 -> 21 us per step with 64 rows, 17 with 16; about half of it is the exchange (a release, an
// arrival and an acquire take 2500 cycles, the layer's 64 KB from the L2 another 1000).  Two neurons
// per CTA (128 CTAs): four (64 CTAs) take 5 us longer.
constexpr int kTrainThreads = 512;
constexpr int kTrainMaxDepth = 16, kTrainMaxIn = 64, kTrainMaxOut = 16;

struct TrainArgs {
  int depth, in, hidden, out, rows;
  int steps, keep;                          // keep: shared memory holds the hidden layers' inputs
  unsigned woff[kTrainMaxDepth], boff[kTrainMaxDepth];
  const float *x, *t;                       // all samples
  const int* order;                         // steps x rows
  const float2* corr;                       // bias corrections of each step
  float lr;
  float *p[2], *m1, *m2;                    // p[0] holds the parameters before the first step
  float* act[kTrainMaxDepth];               // act[l]: 2 x rows x hidden, l = 1 .. depth - 1
  float* delta[kTrainMaxDepth];             // delta[l]: dL/dz of weight layer l, l = 1 .. depth - 2
  float* curve;
  unsigned* bar;
  int* err;
};

// Shared memory in floats: the inputs of weight layers 1 .. depth - 2 (keep), partial gradient
// sums, the CTA's parameters and their two moments, columns of a layer's weights, the output layer's weights, two
// minibatches of inputs and targets, output deltas, the CTA's activations of every layer and its
// deltas of one.
struct TrainSmem {
  int slot, red, own, own_n, vec, wout, x0, t0, y, ax, dz, total;
};

__host__ __device__ inline TrainSmem train_smem(int depth, int in, int hidden, int out, int rows, int npc, bool keep) {
  TrainSmem s;
  s.slot = 0;
  s.red = s.slot + (keep ? depth - 2 : 0) * rows * hidden;
  s.own = s.red + kTrainThreads * npc;
  s.own_n = (npc * (in + 1) + 3) / 4 * 4 + (depth - 2) * (npc * hidden + 4) + hidden + 4;
  s.vec = s.own + 3 * s.own_n;
  s.wout = s.vec + npc * hidden;
  s.x0 = s.wout + (out <= 4 ? (out + 3) / 4 * 4 : (out + 7) / 8 * 8) * hidden;
  s.t0 = s.x0 + 2 * rows * in;
  s.y = s.t0 + 2 * rows * out;
  s.ax = s.y + rows * out;
  s.dz = s.ax + (depth - 1) * rows * npc;
  s.total = s.dz + rows * npc;
  return s;
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float acc) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}

// Sums of V values over the warp (V a power of two up to 32): lane l ends with the sum of value
// l >> (5 - log2 V).
template <int V>
__device__ __forceinline__ float warp_sums(float (&a)[V]) {
  const int lane = threadIdx.x & 31;
  int off = 16;
#pragma unroll
  for (int h = V / 2; h >= 1; h /= 2, off /= 2) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float keep = up ? a[i + h] : a[i], send = up ? a[i] : a[i + h];
      a[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  for (; off >= 1; off /= 2) a[0] += __shfl_xor_sync(0xffffffffu, a[0], off);
  return a[0];
}

// Neurons per CTA and hidden layer NPC, float4 per lane and row J (hidden <= 128 J).
template <int NPC, int J>
__global__ void __launch_bounds__(kTrainThreads, 1) train_kernel(const TrainArgs a) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int bad;
  constexpr int WARPS = kTrainThreads / 32, RB = J == 4 ? 2 : 4;  // rows of a warp at a time
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = blockIdx.x, ncta = gridDim.x;
  const int L = a.depth - 1, H = a.hidden, rows = a.rows, k4 = H / 4;
  const TrainSmem S = train_smem(a.depth, a.in, H, a.out, rows, NPC, a.keep);
  float* const red = sm + S.red;
  float* const vec = sm + S.vec;
  float* const wout = sm + S.wout;
  float* const ax = sm + S.ax;
  float* const dz = sm + S.dz;
  float* const y = sm + S.y;
  const int n0 = cta * NPC;                  // first neuron of every hidden layer
  const int oj = ncta - 1 - cta;             // output neuron, if below a.out
  const bool has_out = oj < a.out;
  auto width = [&](int l) { return l == 0 ? a.in : H; };  // inputs of weight layer l
  // own parameters: per hidden weight layer NPC rows, then NPC biases (padded to float4); then the
  // output neuron's row and bias
  auto own_at = [&](int l) { return sm + S.own + (l == 0 ? 0 : (NPC * (a.in + 1) + 3) / 4 * 4 + (l - 1) * (NPC * H + 4)); };

  for (int l = 0; l <= L; ++l) {
    const int w = width(l), cnt = l == L ? (has_out ? 1 : 0) : NPC;
    for (int e = tid; e < cnt * (w + 1); e += kTrainThreads) {
      const int n = e % cnt, k = e / cnt, o = l == L ? oj : n0 + n;  // k == w: the bias
      float* const own = own_at(l) + (k == w ? cnt * w + n : n * w + k);
      if (l == L || o < H) {
        const size_t at = k == w ? a.boff[l] + o : a.woff[l] + (size_t)o * w + k;
        own[0] = a.p[0][at];
        own[S.own_n] = a.m1[at];
        own[2 * S.own_n] = a.m2[at];
      } else {
        own[0] = 0.f;
      }
    }
  }
  auto fetch = [&](int s) {  // minibatch s into its half of the input and target buffers
    if (s >= a.steps) return;
    float* x = sm + S.x0 + (s & 1) * rows * a.in;
    float* t = sm + S.t0 + (s & 1) * rows * a.out;
    const int* idx = a.order + (size_t)s * rows;
    // a few threads per row: its index is read once, its values one after the other
    const int per = kTrainThreads / rows, r = tid / per, q = tid % per;
    if (r < rows) {
      const size_t i = idx[r];
      for (int e = q; e < a.in; e += per) x[r * a.in + e] = a.x[i * a.in + e];
      for (int e = q; e < a.out; e += per) t[r * a.out + e] = a.t[i * a.out + e];
    }
  };
  fetch(0);
  for (int e = tid; e < S.x0 - S.vec; e += kTrainThreads) vec[e] = 0.f;
  if (tid == 0) bad = 0;
  __syncthreads();

  unsigned want = 0;
  auto arrive = [&]() {
    __syncthreads();
    want += ncta;
    if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(a.bar) : "memory");
  };
  auto wait = [&]() -> bool {
    if (tid == 0) {
      unsigned v;
      long long n = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(a.bar) : "memory");
        if (++n > (1LL << 21)) {
          *a.err = 1;
          bad = 1;
          break;
        }
      } while (v < want);
    }
    __syncthreads();
    return bad == 0;
  };
  // dots of every row of `src` (rows x H, published by all CTAs) with the C vectors at v (H each):
  // the warp's rows come straight from the L2 into registers, RB at a time (and into `slot`);
  // emit(row, c, sum) runs on one lane per sum
  auto row_dots = [&](auto count, const float* src, const float* v, float* slot, auto&& emit) {
    constexpr int C = decltype(count)::value, V = RB * C;
    for (int r0 = warp * RB; r0 < rows; r0 += WARPS * RB) {
      float4 x[RB][J];
#pragma unroll
      for (int i = 0; i < RB; ++i)
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const int c4 = lane + 32 * j;
          x[i][j] = r0 + i < rows && c4 < k4 ? __ldcg(reinterpret_cast<const float4*>(src) + (size_t)(r0 + i) * k4 + c4)
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      float acc[V] = {};
#pragma unroll
      for (int c = 0; c < C; ++c)
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const int c4 = lane + 32 * j;
          const float4 w = c4 < k4 ? reinterpret_cast<const float4*>(v + c * H)[c4] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int i = 0; i < RB; ++i) acc[i * C + c] = dot4(x[i][j], w, acc[i * C + c]);
        }
      if (slot) {
#pragma unroll
        for (int i = 0; i < RB; ++i)
#pragma unroll
          for (int j = 0; j < J; ++j)
            if (r0 + i < rows && lane + 32 * j < k4)
              reinterpret_cast<float4*>(slot)[(r0 + i) * k4 + lane + 32 * j] = x[i][j];
      }
      const float s = warp_sums<V>(acc);
      constexpr int PER = 32 / V;
      const int e = lane / PER, r = r0 + e / C;
      if (lane % PER == 0 && r < rows) emit(r, e % C, s);
    }
  };
  using One = std::integral_constant<int, 1>;
  using Own = std::integral_constant<int, NPC>;
  using Four = std::integral_constant<int, 4>;
  using Eight = std::integral_constant<int, 8>;

  for (int s = 0; s < a.steps; ++s) {
    const float* const pc = a.p[s & 1];
    float* const pn = a.p[(s + 1) & 1];
    const float* const x0 = sm + S.x0 + (s & 1) * rows * a.in;
    const float* const tgt = sm + S.t0 + (s & 1) * rows * a.out;
    const float2 corr = a.corr[s];
    // two sets in turn: a slower CTA may still read the last step's
    auto act = [&](int l) { return a.act[l] + (size_t)(s & 1) * rows * H; };
    auto slot = [&](int l) { return a.keep && l < L ? sm + S.slot + (l - 1) * rows * H : nullptr; };
    auto adam = [&](float* own, size_t at, float g) {
      const float b1 = 0.9f, b2 = 0.999f;
      const float m = b1 * own[S.own_n] + (1.f - b1) * g;
      const float v = b2 * own[2 * S.own_n] + (1.f - b2) * g * g;
      own[S.own_n] = m;
      own[2 * S.own_n] = v;
      const float q = *own - a.lr * (m / corr.x) / (sqrtf(v / corr.y) + 1e-8f);
      *own = q;
      pn[at] = q;
    };
    // gradients of the CTA's rows of weight layer l (C deltas a row, `stride` apart), summed over the
    // batch by groups of threads, and the update
    auto update = [&](auto count, int l, const float* d, int stride) {
      constexpr int C = decltype(count)::value;
      const int w = width(l), wp = min(kTrainThreads, (w + 31) / 32 * 32), groups = kTrainThreads / wp;
      const int o0 = l == L ? oj : n0, group = tid / wp, kt = tid - group * wp;
      float* own = own_at(l);
      if (warp == WARPS - 1) {  // biases
        float g[C] = {};
        for (int r = lane; r < rows; r += 32)
#pragma unroll
          for (int n = 0; n < C; ++n) g[n] += d[r * stride + n];
        const float sum = warp_sums<C>(g);
        const int n = lane / (32 / C);
        if (lane % (32 / C) == 0 && (l == L || o0 + n < H)) adam(own + C * w + n, a.boff[l] + o0 + n, sum);
      }
      for (int kb = 0; kb < w; kb += wp) {
        const int k = kb + kt;
        const bool in_row = k < w && group < groups;
        float g[C] = {};
        auto sums = [&](auto&& value) {
#pragma unroll 8
          for (int r = group; r < rows; r += groups) {
            const float v = value(r);
#pragma unroll
            for (int n = 0; n < C; ++n) g[n] = fmaf(d[r * stride + n], v, g[n]);
          }
        };
        if (in_row) {
          if (const float* in = l == 0 ? x0 : slot(l)) sums([&](int r) { return in[r * w + k]; });
          else sums([&](int r) { return __ldcg(act(l) + (size_t)r * w + k); });
#pragma unroll
          for (int n = 0; n < C; ++n) red[(group * C + n) * wp + kt] = g[n];
        }
        __syncthreads();
#pragma unroll
        for (int n = 0; n < C; ++n) {
          const int q = group + n * groups;
          if (in_row && q < C && (l == L || o0 + q < H)) {
            float sum = 0.f;
            for (int p = 0; p < groups; ++p) sum += red[(p * C + q) * wp + kt];
            adam(own + q * w + k, a.woff[l] + (size_t)(o0 + q) * w + k, sum);
          }
        }
        __syncthreads();
      }
    };

    // first layer: few inputs, one output per thread
    for (int e = tid; e < rows * NPC; e += kTrainThreads) {
      const int r = e / NPC, n = e % NPC;
      const float* w = own_at(0) + n * a.in;
      float v = 0.f;
      for (int k = 0; k < a.in; ++k) v = fmaf(x0[r * a.in + k], w[k], v);
      v = tanhf(v + own_at(0)[NPC * a.in + n]);
      ax[e] = v;
      if (n0 + n < H) act(1)[(size_t)r * H + n0 + n] = v;
    }
    arrive();
    fetch(s + 1);
    if (!wait()) return;
    // the output layer's weights: their owners wrote them before arriving at the barrier just passed
    auto load_wout = [&]() {
      for (int e = tid; e < a.out * H; e += kTrainThreads) wout[e] = __ldcg(pc + a.woff[L] + e);
    };
    if (L == 1) {
      load_wout();
      __syncthreads();
    }
    for (int l = 1; l < L; ++l) {
      row_dots(Own{}, act(l), own_at(l), slot(l), [&](int r, int n, float v) {
        v = tanhf(v + own_at(l)[NPC * H + n]);
        ax[(l * rows + r) * NPC + n] = v;
        if (n0 + n < H) act(l + 1)[(size_t)r * H + n0 + n] = v;
      });
      arrive();
      if (l == 1) load_wout();
      if (!wait()) return;
    }
    // all outputs and their deltas
    for (int j = 0; j < a.out;) {
      auto emit = [&](int r, int c, float v) {
        if (j + c < a.out) y[r * a.out + j + c] = v + __ldcg(pc + a.boff[L] + j + c) - tgt[r * a.out + j + c];
      };
      if (a.out - j > 4) {  // rows of wout past the last output hold zeros
        row_dots(Eight{}, act(L), wout + j * H, nullptr, emit);
        j += 8;
      } else if (a.out - j > 1) {
        row_dots(Four{}, act(L), wout + j * H, nullptr, emit);
        j += 4;
      } else {
        row_dots(One{}, act(L), wout + j * H, nullptr, emit);
        ++j;
      }
    }
    const float inv = (float)(rows * a.out);
    __syncthreads();
    if (cta == 0 && warp == WARPS - 1) {  // the loss
      float sum = 0.f;
      for (int e = lane; e < rows * a.out; e += 32) sum += y[e] * y[e];
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
      if (lane == 0) a.curve[s] = sum / inv;
    }
    for (int e = tid; e < rows * NPC; e += kTrainThreads) {
      const int r = e / NPC, n = e % NPC;
      float v = 0.f;
      if (n0 + n < H)
        for (int j = 0; j < a.out; ++j) v = fmaf(2.f * y[r * a.out + j] / inv, wout[j * H + n0 + n], v);
      const float h = ax[(L - 1) * rows * NPC + e];
      v *= 1.f - h * h;
      dz[e] = v;
      if (L > 1 && n0 + n < H) a.delta[L - 1][(size_t)r * H + n0 + n] = v;
    }
    for (int l = L - 1; l >= 0; --l) {
      // dz holds the CTA's deltas of weight layer l, published for l >= 1
      if (l >= 1) arrive();
      else __syncthreads();
      if (l >= 1)
        for (int e = tid; e < NPC * H; e += kTrainThreads) {  // its neurons' columns of weight layer l
          const int o = e / NPC, n = e % NPC;
          vec[n * H + o] = n0 + n < H ? __ldcg(pc + a.woff[l] + (size_t)o * H + n0 + n) : 0.f;
        }
      if (l == L - 1 && has_out) {
        for (int r = tid; r < rows; r += kTrainThreads) y[r * a.out + oj] = 2.f * y[r * a.out + oj] / inv;
        __syncthreads();
        update(One{}, L, y + oj, a.out);
      }
      update(Own{}, l, dz, NPC);
      if (l == 0) break;
      if (!wait()) return;
      row_dots(Own{}, a.delta[l], vec, nullptr, [&](int r, int n, float v) {
        const float h = ax[((l - 1) * rows + r) * NPC + n];
        v *= 1.f - h * h;
        dz[r * NPC + n] = v;
        if (l > 1 && n0 + n < H) a.delta[l - 1][(size_t)r * H + n0 + n] = v;
      });
    }
    __syncthreads();
  }
  for (int l = 0; l <= L; ++l) {  // the moments go back
    const int w = width(l), cnt = l == L ? (has_out ? 1 : 0) : NPC;
    for (int e = tid; e < cnt * (w + 1); e += kTrainThreads) {
      const int n = e % cnt, k = e / cnt, o = l == L ? oj : n0 + n;
      const float* const own = own_at(l) + (k == w ? cnt * w + n : n * w + k);
      if (l == L || o < H) {
        const size_t at = k == w ? a.boff[l] + o : a.woff[l] + (size_t)o * w + k;
        a.m1[at] = own[S.own_n];
        a.m2[at] = own[2 * S.own_n];
      }
    }
  }
}

__global__ void gather_rows_kernel(const float* __restrict__ src, const int* __restrict__ idx, int rows,
                                   int cols, float* __restrict__ dst) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols; e += gridDim.x * blockDim.x)
    dst[e] = src[(size_t)idx[e / cols] * cols + e % cols];
}

__global__ void to_bf16_kernel(const float* __restrict__ p, __nv_bfloat16* __restrict__ q, int count) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x)
    q[e] = __float2bfloat16_rn(p[e]);
}

}  // namespace
}  // namespace lbw

using namespace lbw;

struct lbw_mlp {
  int in = 0, hidden = 0, depth = 0, out = 0;
  std::vector<int> dims;         // depth + 1 layer widths
  std::vector<size_t> woff, boff;  // parameter offsets of each layer
  size_t nparam = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float *p = nullptr, *g = nullptr, *m1 = nullptr, *m2 = nullptr;
  __nv_bfloat16* pb = nullptr;   // BF16 copy for inference
  bool pb_valid = false;
  long long adam_t = 0;
  // work buffers for up to cap rows
  int cap = 0;
  std::vector<float*> act;       // activations per layer (depth + 1), cap x width
  float *delta = nullptr, *delta2 = nullptr, *target = nullptr, *loss = nullptr;
  int* idx = nullptr;
  float *data_x = nullptr, *data_t = nullptr;
  int data_n = 0;
  // training in one launch: the second parameter buffer, exchanged layers, barrier and error words
  float *p2 = nullptr, *xch = nullptr;
  size_t xch_size = 0;
  unsigned* sync = nullptr;
  // inference in one launch: transposed weights in FP32 / BF16 (valid since the last change of the
  // parameters) and the rows' inputs and outputs
  float* wt = nullptr;
  __nv_bfloat16* wtb = nullptr;
  bool wt_valid = false, wtb_valid = false;
  float* io = nullptr;
  size_t io_size = 0;
};

namespace {

// the rounded and transposed copies of the weights are stale
void params_changed(lbw_mlp* q) { q->pb_valid = q->wt_valid = q->wtb_valid = false; }

void free_work(lbw_mlp* q) {
  for (float* a : q->act)
    if (a) cudaFreeAsync(a, q->stream);
  q->act.clear();
  float** bufs[] = {&q->delta, &q->delta2, &q->target, &q->loss};
  for (float** b : bufs)
    if (*b) { cudaFreeAsync(*b, q->stream); *b = nullptr; }
  if (q->idx) { cudaFreeAsync(q->idx, q->stream); q->idx = nullptr; }
  q->cap = 0;
}

lbw_status ensure_work(lbw_mlp* q, int rows) {
  if (rows <= q->cap) return LBW_OK;
  free_work(q);
  int maxw = 0;
  for (int w : q->dims) maxw = std::max(maxw, w);
  q->act.assign(q->dims.size(), nullptr);
  for (size_t l = 0; l < q->dims.size(); ++l)
    LBW_CUDA(cudaMallocAsync((void**)&q->act[l], sizeof(float) * rows * q->dims[l], q->stream));
  LBW_CUDA(cudaMallocAsync((void**)&q->delta, sizeof(float) * rows * maxw, q->stream));
  LBW_CUDA(cudaMallocAsync((void**)&q->delta2, sizeof(float) * rows * maxw, q->stream));
  LBW_CUDA(cudaMallocAsync((void**)&q->target, sizeof(float) * rows * q->out, q->stream));
  LBW_CUDA(cudaMallocAsync((void**)&q->loss, sizeof(float), q->stream));
  LBW_CUDA(cudaMallocAsync((void**)&q->idx, sizeof(int) * rows, q->stream));
  q->cap = rows;
  return LBW_OK;
}

dim3 gemm_grid(int m, int n) { return dim3((n + TN - 1) / TN, (m + TM - 1) / TM); }

// forward through all layers for act[0] (rows x in) already on the device
template <typename WB>
void forward(lbw_mlp* q, int rows, const WB* params) {
  for (int l = 0; l < q->depth; ++l) {
    const int in = q->dims[l], out = q->dims[l + 1];
    gemm_kernel<WB><<<gemm_grid(rows, out), 256, 0, q->stream>>>(q->act[l], in, false, params + q->woff[l], in,
                                                                  true, q->act[l + 1], out, rows, out, in,
                                                                  nullptr, false);
    bias_act_kernel<<<152 * 4, 256, 0, q->stream>>>(q->act[l + 1], q->p + q->boff[l], rows, out, l + 1 < q->depth);
  }
}

// loss and parameter gradient (into q->g) for act[0] and target on the device
void backward(lbw_mlp* q, int rows) {
  const int last = q->depth;
  const int cnt = rows * q->out;
  cudaMemsetAsync(q->loss, 0, sizeof(float), q->stream);
  mse_kernel<<<152, 256, 0, q->stream>>>(q->act[last], q->target, q->delta, cnt, q->loss);
  for (int l = q->depth - 1; l >= 0; --l) {
    const int in = q->dims[l], out = q->dims[l + 1];
    if (l + 1 < q->depth) tanh_back_kernel<<<152 * 4, 256, 0, q->stream>>>(q->delta, q->act[l + 1], rows * out);
    // dW = dZ^T X  (out x in)
    gemm_kernel<float><<<gemm_grid(out, in), 256, 0, q->stream>>>(q->delta, out, true, q->act[l], in, false,
                                                                   q->g + q->woff[l], in, out, in, rows,
                                                                   nullptr, false);
    colsum_kernel<<<(out + 255) / 256, 256, 0, q->stream>>>(q->delta, rows, out, q->g + q->boff[l]);
    if (l > 0) {
      // dX = dZ W  (rows x in)
      gemm_kernel<float><<<gemm_grid(rows, in), 256, 0, q->stream>>>(q->delta, out, false, q->p + q->woff[l], in,
                                                                      false, q->delta2, in, rows, in, out,
                                                                      nullptr, false);
      std::swap(q->delta, q->delta2);
    }
  }
}

template <typename WB, int RB>
cudaError_t launch_forward(lbw_mlp* q, const FwdArgs& a, const WB* wt) {
  const size_t smem = fwd_smem<RB>(a.dims, a.depth);
  const cudaError_t e =
      cudaFuncSetAttribute(forward_kernel<WB, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  forward_kernel<WB, RB><<<(a.n + RB - 1) / RB, kFwdThreads, smem, q->stream>>>(a, wt);
  return cudaGetLastError();
}

template <typename WB>
cudaError_t launch_forward_rows(lbw_mlp* q, const FwdArgs& a, const WB* wt) {
  int widest = 0, units = 0;
  for (int l = 0; l <= a.depth; ++l) widest = std::max(widest, a.dims[l]);
  for (int l = 1; l <= a.depth; ++l) units = std::max(units, fwd_pad(a.dims[l]));
  // a thread per unit; too few blocks to fill the SMs split the rows further
  const int threads = a.n >= 8 * 152 * kFwdRows ? units : std::max(units, std::min(256, 4 * units));
  bool splits = false;
  for (int l = 0; l < a.depth; ++l) splits |= fwd_splits(a.dims[l], a.dims[l + 1], threads);
  const size_t smem = sizeof(float) * kFwdRows * (2 * widest + (splits ? kFwdThreads : 0));
  const cudaError_t e =
      cudaFuncSetAttribute(forward_rows_kernel<WB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  forward_rows_kernel<WB><<<(a.n + kFwdRows - 1) / kFwdRows, threads, smem, q->stream>>>(a, wt);
  return cudaGetLastError();
}

bool fits_forward(const lbw_mlp* q) {
  for (int w : q->dims)
    if (w > kFwdMaxWidth) return false;
  return q->depth <= kFwdMaxDepth;
}

// n rows through the network in one launch, host to host; WB the weights' storage.
template <typename WB>
lbw_status forward_fused(lbw_mlp* q, const float* host_x, int n, float* host_y, WB*& wt, bool& valid) {
  FwdArgs a{};
  a.depth = q->depth;
  a.n = n;
  a.bias = q->p;
  size_t at = 0;
  for (int l = 0; l <= q->depth; ++l) a.dims[l] = q->dims[l];
  for (int l = 0; l < q->depth; ++l) {
    a.woff[l] = (unsigned)at;
    a.boff[l] = (unsigned)q->boff[l];
    at += (size_t)a.dims[l] * fwd_pad(a.dims[l + 1]);
  }
  if (!wt) LBW_CUDA(cudaMallocAsync((void**)&wt, sizeof(WB) * at, q->stream));
  const size_t nx = (size_t)n * q->in, ny = (size_t)n * q->out;
  if (nx + ny > q->io_size) {
    if (q->io) cudaFreeAsync(q->io, q->stream);
    q->io = nullptr;
    q->io_size = 0;
    LBW_CUDA(cudaMallocAsync((void**)&q->io, sizeof(float) * (nx + ny), q->stream));
    q->io_size = nx + ny;
  }
  a.x = q->io;
  a.y = q->io + nx;
  LBW_CUDA(cudaMemcpyAsync(q->io, host_x, sizeof(float) * nx, cudaMemcpyHostToDevice, q->stream));
  if (!valid) {
    for (int l = 0; l < q->depth; ++l)
      pack_kernel<WB><<<dim3((a.dims[l] + 31) / 32, fwd_pad(a.dims[l + 1]) / 32), dim3(32, 8), 0, q->stream>>>(
          q->p + q->woff[l], a.dims[l], a.dims[l + 1], wt + a.woff[l]);
    LBW_CUDA(cudaGetLastError());
    valid = true;
  }
  // rows per CTA: more rows share a read of the weights, fewer fill the SMs
  const cudaError_t e = n <= 4 * 152       ? launch_forward<WB, 4>(q, a, wt)
                        : n <= 8 * 2 * 152 ? launch_forward<WB, 8>(q, a, wt)
                                           : launch_forward_rows<WB>(q, a, wt);
  if (e != cudaSuccess) return cuda_fail(e, "mlp forward");
  LBW_CUDA(cudaMemcpyAsync(host_y, a.y, sizeof(float) * ny, cudaMemcpyDeviceToHost, q->stream));
  LBW_CUDA(cudaStreamSynchronize(q->stream));
  return LBW_OK;
}

// Launch shape of train_kernel.
struct TrainPlan {
  int npc = 0, ctas = 0;
  bool keep = false;
  size_t smem = 0;
};

template <int NPC, typename F>
cudaError_t with_train_width(int hidden, F&& f) {
  return hidden <= 128 ? f(train_kernel<NPC, 1>) : hidden <= 256 ? f(train_kernel<NPC, 2>) : f(train_kernel<NPC, 4>);
}

template <typename F>
cudaError_t with_train_kernel(int npc, int hidden, F&& f) {
  return npc == 1 ? with_train_width<1>(hidden, f) : npc == 2 ? with_train_width<2>(hidden, f)
                                                              : with_train_width<4>(hidden, f);
}

// npc = 0: the network or the batch does not suit it (wide layers, rows that do not fit shared
// memory, widths that are no multiple of 4).
TrainPlan train_plan(const lbw_mlp* q, int rows) {
  TrainPlan t;
  int dev = 0, sms = 0, smem_max = 0, coop = 0;
  if (q->depth < 2 || q->hidden % 4 != 0 || q->hidden > 512 || q->in > kTrainMaxIn || q->out > kTrainMaxOut || rows > kTrainThreads)
    return t;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
    cudaGetLastError();
    return t;
  }
  for (int npc = 1; npc <= 4; npc *= 2) {
    const int ctas = (q->hidden + npc - 1) / npc;
    if (ctas > sms || q->out > ctas) continue;
    for (int keep = 1; keep >= 0; --keep) {
      const size_t bytes = sizeof(float) * (size_t)train_smem(q->depth, q->in, q->hidden, q->out, rows, npc, keep).total;
      if (bytes + 64 > (size_t)smem_max) continue;
      int per = 0;
      const cudaError_t e = with_train_kernel(npc, q->hidden, [&](auto kern) {
        cudaError_t f = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (f == cudaSuccess) f = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kTrainThreads, bytes);
        return f;
      });
      if (e != cudaSuccess || per < 1) {
        cudaGetLastError();
        continue;
      }
      t.npc = npc;
      t.ctas = ctas;
      t.keep = keep;
      t.smem = bytes;
      return t;
    }
  }
  return t;
}

// Device memory of one call, given back on every way out.
struct Temporary {
  void* p = nullptr;
  cudaStream_t stream;
  explicit Temporary(cudaStream_t s) : stream(s) {}
  Temporary(const Temporary&) = delete;
  ~Temporary() {
    if (p) cudaFreeAsync(p, stream);
  }
  template <typename T> T* as() const { return static_cast<T*>(p); }
};

// n_steps Adam steps on train_kernel; order, corrections and the loss curve on the device.  adam_t counts
// the steps launched.
lbw_status train_fused(lbw_mlp* q, const TrainPlan& t, const int* d_order, const float2* d_corr, int n_steps, int rows,
                       float lr, float* d_curve) {
  const size_t layer = (size_t)rows * q->hidden, need = layer * (2 * (q->depth - 1) + q->depth);
  if (!q->p2) LBW_CUDA(cudaMallocAsync((void**)&q->p2, sizeof(float) * q->nparam, q->stream));
  if (!q->sync) LBW_CUDA(cudaMallocAsync((void**)&q->sync, 2 * sizeof(unsigned), q->stream));
  if (need > q->xch_size) {
    if (q->xch) cudaFreeAsync(q->xch, q->stream);
    q->xch = nullptr;
    q->xch_size = 0;
    LBW_CUDA(cudaMallocAsync((void**)&q->xch, sizeof(float) * need, q->stream));
    q->xch_size = need;
  }
  TrainArgs a{};
  a.depth = q->depth;
  a.in = q->in;
  a.hidden = q->hidden;
  a.out = q->out;
  a.rows = rows;
  a.keep = t.keep;
  for (int l = 0; l < q->depth; ++l) {
    a.woff[l] = (unsigned)q->woff[l];
    a.boff[l] = (unsigned)q->boff[l];
    a.act[l] = l > 0 ? q->xch + (size_t)(l - 1) * 2 * layer : nullptr;
    a.delta[l] = q->xch + (size_t)(q->depth - 1) * 2 * layer + l * layer;
  }
  a.x = q->data_x;
  a.t = q->data_t;
  a.lr = lr;
  a.m1 = q->m1;
  a.m2 = q->m2;
  a.bar = q->sync;
  a.err = reinterpret_cast<int*>(q->sync + 1);
  LBW_CUDA(cudaMemsetAsync(q->sync, 0, 2 * sizeof(unsigned), q->stream));
  const int chunk = 1024;  // steps per launch: some 15 ms
  for (int s = 0; s < n_steps; s += chunk) {
    a.steps = std::min(chunk, n_steps - s);
    a.order = d_order + (size_t)s * rows;
    a.corr = d_corr + s;
    a.curve = d_curve + s;
    a.p[0] = q->p;
    a.p[1] = q->p2;
    if (s > 0) LBW_CUDA(cudaMemsetAsync(q->sync, 0, sizeof(unsigned), q->stream));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(t.ctas);
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = t.smem;
    cfg.stream = q->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    LBW_CUDA(with_train_kernel(t.npc, q->hidden, [&](auto kern) { return cudaLaunchKernelEx(&cfg, kern, a); }));
    if (a.steps & 1) std::swap(q->p, q->p2);
    q->adam_t += a.steps;
    params_changed(q);
  }
  return LBW_OK;
}

unsigned long long splitmix(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ULL;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
  return x ^ (x >> 31);
}

}  // namespace

extern "C" {

lbw_status lbw_mlp_create(int32_t in_dim, int32_t hidden, int32_t depth, int32_t out_dim, uint64_t seed,
                          void* stream, lbw_mlp** out) {
  if (!out) return fail(LBW_EINVAL, "out is NULL");
  *out = nullptr;
  if (in_dim < 1 || in_dim > 4096 || hidden < 1 || hidden > 4096 || out_dim < 1 || out_dim > 4096 ||
      depth < 1 || depth > 16)
    return fail(LBW_EINVAL, "dimensions out of range (1..4096, depth 1..16)");
  lbw_mlp* q = new (std::nothrow) lbw_mlp();
  if (!q) return fail(LBW_ENOMEM, "host allocation failed");
  q->in = in_dim; q->hidden = hidden; q->depth = depth; q->out = out_dim;
  q->dims.push_back(in_dim);
  for (int l = 0; l + 1 < depth; ++l) q->dims.push_back(hidden);
  q->dims.push_back(out_dim);
  size_t off = 0;
  for (int l = 0; l < depth; ++l) {
    q->woff.push_back(off);
    off += (size_t)q->dims[l + 1] * q->dims[l];
    q->boff.push_back(off);
    off += q->dims[l + 1];
  }
  q->nparam = off;
  q->stream = reinterpret_cast<cudaStream_t>(stream);
  if (!q->stream) {
    if (cudaStreamCreate(&q->stream) != cudaSuccess) {
      delete q;
      return fail(LBW_ECUDA, "cudaStreamCreate failed");
    }
    q->own_stream = true;
  }
  // uniform(-s, s) with s = sqrt(6 / (fan_in + fan_out)) from a counter-based generator
  std::vector<float> h(q->nparam, 0.f);
  for (int l = 0; l < depth; ++l) {
    const double s = std::sqrt(6.0 / (q->dims[l] + q->dims[l + 1]));
    for (size_t e = 0; e < (size_t)q->dims[l + 1] * q->dims[l]; ++e) {
      const double u = (splitmix(seed ^ (q->woff[l] + e) * 0x2545F4914F6CDD1DULL) >> 11) * (1.0 / 9007199254740992.0);
      h[q->woff[l] + e] = (float)((2.0 * u - 1.0) * s);
    }
  }
  cudaError_t e = cudaMallocAsync((void**)&q->p, sizeof(float) * q->nparam, q->stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&q->g, sizeof(float) * q->nparam, q->stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&q->m1, sizeof(float) * q->nparam, q->stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&q->m2, sizeof(float) * q->nparam, q->stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&q->pb, sizeof(__nv_bfloat16) * q->nparam, q->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(q->p, h.data(), sizeof(float) * q->nparam, cudaMemcpyHostToDevice, q->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(q->m1, 0, sizeof(float) * q->nparam, q->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(q->m2, 0, sizeof(float) * q->nparam, q->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(q->stream);
  if (e != cudaSuccess) {
    lbw_mlp_destroy(q);
    return cuda_fail(e, "mlp create");
  }
  *out = q;
  return LBW_OK;
}

void lbw_mlp_destroy(lbw_mlp* q) {
  if (!q) return;
  free_work(q);
  if (q->sync) cudaFreeAsync(q->sync, q->stream);
  if (q->wtb) cudaFreeAsync(q->wtb, q->stream);
  float* bufs[] = {q->p, q->g, q->m1, q->m2, q->data_x, q->data_t, q->p2, q->xch, q->wt, q->io};
  for (float* b : bufs)
    if (b) cudaFreeAsync(b, q->stream);
  if (q->pb) cudaFreeAsync(q->pb, q->stream);
  cudaStreamSynchronize(q->stream);
  if (q->own_stream) cudaStreamDestroy(q->stream);
  delete q;
}

lbw_status lbw_mlp_param_count(lbw_mlp* q, int64_t* n) {
  if (!q || !n) return fail(LBW_EINVAL, "NULL argument");
  *n = (int64_t)q->nparam;
  return LBW_OK;
}

lbw_status lbw_mlp_get_params(lbw_mlp* q, float* host_params) {
  if (!q || !host_params) return fail(LBW_EINVAL, "NULL argument");
  LBW_CUDA(cudaMemcpyAsync(host_params, q->p, sizeof(float) * q->nparam, cudaMemcpyDeviceToHost, q->stream));
  LBW_CUDA(cudaStreamSynchronize(q->stream));
  return LBW_OK;
}

lbw_status lbw_mlp_set_params(lbw_mlp* q, const float* host_params) {
  if (!q || !host_params) return fail(LBW_EINVAL, "NULL argument");
  LBW_CUDA(cudaMemcpyAsync(q->p, host_params, sizeof(float) * q->nparam, cudaMemcpyHostToDevice, q->stream));
  LBW_CUDA(cudaMemsetAsync(q->m1, 0, sizeof(float) * q->nparam, q->stream));
  LBW_CUDA(cudaMemsetAsync(q->m2, 0, sizeof(float) * q->nparam, q->stream));
  LBW_CUDA(cudaStreamSynchronize(q->stream));
  q->adam_t = 0;
  params_changed(q);
  return LBW_OK;
}

lbw_status lbw_mlp_forward(lbw_mlp* q, const float* host_x, int32_t n, float* host_y) {
  if (!q || !host_x || !host_y || n < 1) return fail(LBW_EINVAL, "bad argument");
  if (fits_forward(q)) return forward_fused<float>(q, host_x, n, host_y, q->wt, q->wt_valid);
  lbw_status st = ensure_work(q, n);
  if (st != LBW_OK) return st;
  LBW_CUDA(cudaMemcpyAsync(q->act[0], host_x, sizeof(float) * n * q->in, cudaMemcpyHostToDevice, q->stream));
  forward<float>(q, n, q->p);
  LBW_CUDA(cudaGetLastError());
  LBW_CUDA(cudaMemcpyAsync(host_y, q->act[q->depth], sizeof(float) * n * q->out, cudaMemcpyDeviceToHost, q->stream));
  LBW_CUDA(cudaStreamSynchronize(q->stream));
  return LBW_OK;
}

lbw_status lbw_mlp_predict_bf16(lbw_mlp* q, const float* host_x, int32_t n, float* host_y) {
  if (!q || !host_x || !host_y || n < 1) return fail(LBW_EINVAL, "bad argument");
  if (fits_forward(q)) return forward_fused<__nv_bfloat16>(q, host_x, n, host_y, q->wtb, q->wtb_valid);
  lbw_status st = ensure_work(q, n);
  if (st != LBW_OK) return st;
  if (!q->pb_valid) {
    to_bf16_kernel<<<152 * 4, 256, 0, q->stream>>>(q->p, q->pb, (int)q->nparam);
    q->pb_valid = true;
  }
  LBW_CUDA(cudaMemcpyAsync(q->act[0], host_x, sizeof(float) * n * q->in, cudaMemcpyHostToDevice, q->stream));
  forward<__nv_bfloat16>(q, n, q->pb);
  LBW_CUDA(cudaGetLastError());
  LBW_CUDA(cudaMemcpyAsync(host_y, q->act[q->depth], sizeof(float) * n * q->out, cudaMemcpyDeviceToHost, q->stream));
  LBW_CUDA(cudaStreamSynchronize(q->stream));
  return LBW_OK;
}

lbw_status lbw_mlp_grad(lbw_mlp* q, const float* host_x, const float* host_t, int32_t n, float* host_grad,
                        float* host_loss) {
  if (!q || !host_x || !host_t || n < 1) return fail(LBW_EINVAL, "bad argument");
  lbw_status st = ensure_work(q, n);
  if (st != LBW_OK) return st;
  LBW_CUDA(cudaMemcpyAsync(q->act[0], host_x, sizeof(float) * n * q->in, cudaMemcpyHostToDevice, q->stream));
  LBW_CUDA(cudaMemcpyAsync(q->target, host_t, sizeof(float) * n * q->out, cudaMemcpyHostToDevice, q->stream));
  forward<float>(q, n, q->p);
  backward(q, n);
  LBW_CUDA(cudaGetLastError());
  if (host_grad)
    LBW_CUDA(cudaMemcpyAsync(host_grad, q->g, sizeof(float) * q->nparam, cudaMemcpyDeviceToHost, q->stream));
  if (host_loss) LBW_CUDA(cudaMemcpyAsync(host_loss, q->loss, sizeof(float), cudaMemcpyDeviceToHost, q->stream));
  LBW_CUDA(cudaStreamSynchronize(q->stream));
  return LBW_OK;
}

lbw_status lbw_mlp_adam_step(lbw_mlp* q, const float* host_grad, float lr) {
  if (!q || !host_grad) return fail(LBW_EINVAL, "NULL argument");
  LBW_CUDA(cudaMemcpyAsync(q->g, host_grad, sizeof(float) * q->nparam, cudaMemcpyHostToDevice, q->stream));
  ++q->adam_t;
  const float b1 = 0.9f, b2 = 0.999f;
  adam_kernel<<<152 * 4, 256, 0, q->stream>>>(q->p, q->g, q->m1, q->m2, (int)q->nparam, lr, b1, b2, 1e-8f,
                                               (float)(1.0 - std::pow(0.9, (double)q->adam_t)),
                                               (float)(1.0 - std::pow(0.999, (double)q->adam_t)));
  LBW_CUDA(cudaGetLastError());
  LBW_CUDA(cudaStreamSynchronize(q->stream));
  params_changed(q);
  return LBW_OK;
}

lbw_status lbw_mlp_train(lbw_mlp* q, const float* host_x, const float* host_t, int32_t n,
                         const int32_t* host_order, int32_t n_steps, int32_t batch, float lr, float* host_loss) {
  if (!q || !host_x || !host_t || !host_order || n < 1 || n_steps < 0 || batch < 1 || batch > n)
    return fail(LBW_EINVAL, "bad argument");
  for (long long e = 0; e < (long long)n_steps * batch; ++e)
    if (host_order[e] < 0 || host_order[e] >= n) return fail(LBW_EINVAL, "host_order holds an index outside [0, n)");
  const TrainPlan plan = train_plan(q, batch);
  lbw_status st = plan.npc ? LBW_OK : ensure_work(q, batch);
  if (st != LBW_OK) return st;
  if (q->data_n != n) {
    if (q->data_x) cudaFreeAsync(q->data_x, q->stream);
    if (q->data_t) cudaFreeAsync(q->data_t, q->stream);
    q->data_x = q->data_t = nullptr;
    q->data_n = 0;
    LBW_CUDA(cudaMallocAsync((void**)&q->data_x, sizeof(float) * n * q->in, q->stream));
    LBW_CUDA(cudaMallocAsync((void**)&q->data_t, sizeof(float) * n * q->out, q->stream));
    q->data_n = n;
  }
  LBW_CUDA(cudaMemcpyAsync(q->data_x, host_x, sizeof(float) * n * q->in, cudaMemcpyHostToDevice, q->stream));
  LBW_CUDA(cudaMemcpyAsync(q->data_t, host_t, sizeof(float) * n * q->out, cudaMemcpyHostToDevice, q->stream));
  Temporary order(q->stream), curve(q->stream);
  LBW_CUDA(cudaMallocAsync(&order.p, sizeof(int) * (size_t)n_steps * batch, q->stream));
  LBW_CUDA(cudaMemcpyAsync(order.p, host_order, sizeof(int) * (size_t)n_steps * batch, cudaMemcpyHostToDevice,
                           q->stream));
  LBW_CUDA(cudaMallocAsync(&curve.p, sizeof(float) * std::max(1, n_steps), q->stream));
  const int* const d_order = order.as<int>();
  float* const d_curve = curve.as<float>();
  if (plan.npc) {
    std::vector<float2> corr(std::max(1, n_steps));
    for (int s = 0; s < n_steps; ++s) {
      const double t = (double)(q->adam_t + s + 1);
      corr[s] = make_float2((float)(1.0 - std::pow(0.9, t)), (float)(1.0 - std::pow(0.999, t)));
    }
    Temporary d_corr(q->stream);
    int err = 0;
    LBW_CUDA(cudaMallocAsync(&d_corr.p, sizeof(float2) * corr.size(), q->stream));
    LBW_CUDA(cudaMemcpyAsync(d_corr.p, corr.data(), sizeof(float2) * corr.size(), cudaMemcpyHostToDevice, q->stream));
    st = train_fused(q, plan, d_order, d_corr.as<float2>(), n_steps, batch, lr, d_curve);
    if (st != LBW_OK) return st;
    LBW_CUDA(cudaMemcpyAsync(&err, q->sync + 1, sizeof(int), cudaMemcpyDeviceToHost, q->stream));
    if (host_loss && n_steps > 0)
      LBW_CUDA(cudaMemcpyAsync(host_loss, d_curve, sizeof(float) * n_steps, cudaMemcpyDeviceToHost, q->stream));
    LBW_CUDA(cudaStreamSynchronize(q->stream));
    if (err) return fail(LBW_ETIMEOUT, "a training step's bounded wait ran out; the parameters are undefined until "
                                       "lbw_mlp_set_params");
    return LBW_OK;
  }
  const float b1 = 0.9f, b2 = 0.999f;
  for (int s = 0; s < n_steps; ++s) {
    gather_rows_kernel<<<64, 256, 0, q->stream>>>(q->data_x, d_order + (size_t)s * batch, batch, q->in, q->act[0]);
    gather_rows_kernel<<<64, 256, 0, q->stream>>>(q->data_t, d_order + (size_t)s * batch, batch, q->out, q->target);
    forward<float>(q, batch, q->p);
    backward(q, batch);
    cudaMemcpyAsync(d_curve + s, q->loss, sizeof(float), cudaMemcpyDeviceToDevice, q->stream);
    ++q->adam_t;
    adam_kernel<<<152 * 4, 256, 0, q->stream>>>(q->p, q->g, q->m1, q->m2, (int)q->nparam, lr, b1, b2, 1e-8f,
                                                 (float)(1.0 - std::pow(0.9, (double)q->adam_t)),
                                                 (float)(1.0 - std::pow(0.999, (double)q->adam_t)));
  }
  params_changed(q);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && host_loss && n_steps > 0)
    e = cudaMemcpyAsync(host_loss, d_curve, sizeof(float) * n_steps, cudaMemcpyDeviceToHost, q->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(q->stream);
  if (e != cudaSuccess) return cuda_fail(e, "mlp train");
  return LBW_OK;
}

}  // extern "C"
