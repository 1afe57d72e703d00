// lbw_mlp_forward.cuh -- forward pass of the surrogate network in one launch (lbw_mlp.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

namespace lbw {
namespace {

// Layer by layer, a forward pass was a product and a bias / tanh launch per layer (eight for the
// surrogate) with the activations going through memory.  forward_kernel takes RB rows through all
// layers: the activations stay in shared memory ([unit][row], so the rows of a unit are one
// broadcast vector), each thread forms one unit's outputs for all RB rows over a share of the
// inputs, and the shares are added through shared memory.  The weights are read from the L2, in a
// transposed copy ([input][unit], rounded up to 32 units) so that a warp reads one line; the copy
// is made when the parameters have changed.  RB grows with the number of rows (fewer reads of
// the weights per row) as long as the SMs stay filled.  Measured on 7 -> 256 -> 256 -> 256 -> 8,
// whole calls with the copies of inputs and outputs: 1 row 134 -> 45 us, 400 rows 177 -> 47 us.  More
// than 2432 rows go through forward_rows_kernel: 4000 rows 216 -> 92 us, 20,000 rows 464 -> 270.
constexpr int kFwdThreads = 512;
constexpr int kFwdMaxWidth = 512;  // wider layers re-read their weights too often: tiled products
constexpr int kFwdMaxDepth = 16;

struct FwdArgs {
  int depth, n;
  int dims[kFwdMaxDepth + 1];
  unsigned woff[kFwdMaxDepth];   // transposed weights of each layer
  unsigned boff[kFwdMaxDepth];   // biases in the parameter vector
  const float* bias;
  const float* x;
  float* y;
};

__host__ __device__ inline int fwd_pad(int w) { return (w + 31) / 32 * 32; }

template <int RB>
inline size_t fwd_smem(const int* dims, int depth) {
  int w = 0;
  for (int l = 0; l <= depth; ++l) w = dims[l] > w ? dims[l] : w;
  return sizeof(float) * ((size_t)2 * w * RB + (size_t)kFwdThreads * RB);
}

template <int RB>  // RB consecutive floats in shared memory
__device__ __forceinline__ void load_rows(const float* p, float (&v)[RB]) {
#pragma unroll
  for (int i = 0; i < RB; i += 4) {
    const float4 t = *reinterpret_cast<const float4*>(p + i);
    v[i] = t.x; v[i + 1] = t.y; v[i + 2] = t.z; v[i + 3] = t.w;
  }
}

template <typename WB, int RB>
__global__ void __launch_bounds__(kFwdThreads) forward_kernel(const FwdArgs a, const WB* __restrict__ wt) {
  extern __shared__ __align__(16) float sm[];
  int maxw = 0;
  for (int l = 0; l <= a.depth; ++l) maxw = max(maxw, a.dims[l]);
  float* cur = sm;
  float* nxt = sm + maxw * RB;
  float* const red = sm + 2 * maxw * RB;
  const int tid = threadIdx.x, r0 = blockIdx.x * RB;
  for (int e = tid; e < a.dims[0] * RB; e += kFwdThreads) {
    const int r = e / a.dims[0], k = e % a.dims[0];
    cur[k * RB + r] = r0 + r < a.n ? a.x[(size_t)(r0 + r) * a.dims[0] + k] : 0.f;
  }
  __syncthreads();
  for (int l = 0; l < a.depth; ++l) {
    const int in = a.dims[l], out = a.dims[l + 1], wp = fwd_pad(out), groups = kFwdThreads / wp;
    const int group = tid / wp, j = tid - group * wp;
    const int len = (in + groups - 1) / groups, k0 = group * len, k1 = min(in, k0 + len);
    if (group < groups) {
      float acc[RB] = {};
      const WB* w = wt + a.woff[l] + j;
#pragma unroll 8
      for (int k = k0; k < k1; ++k) {
        const float c = (float)w[(size_t)k * wp];
        float v[RB];
        load_rows<RB>(cur + k * RB, v);
#pragma unroll
        for (int i = 0; i < RB; ++i) acc[i] = fmaf(c, v[i], acc[i]);
      }
#pragma unroll
      for (int i = 0; i < RB; ++i) red[(group * RB + i) * wp + j] = acc[i];
    }
    __syncthreads();
    const bool last = l + 1 == a.depth;
    for (int e = tid; e < wp * RB; e += kFwdThreads) {
      const int u = e % wp, r = e / wp;
      if (u >= out) continue;
      float s = red[r * wp + u];
      for (int g = 1; g < groups; ++g) s += red[(g * RB + r) * wp + u];
      s += a.bias[a.boff[l] + u];
      if (!last) nxt[u * RB + r] = tanhf(s);
      else if (r0 + r < a.n) a.y[(size_t)(r0 + r) * out + u] = s;
    }
    __syncthreads();
    float* t = cur;
    cur = nxt;
    nxt = t;
  }
}

// Many rows: each thread forms its unit's outputs for some of the block's rows over all inputs, so
// no sums go through shared memory and a layer ends with one barrier.  The additions are those of
// forward_kernel (a partial sum per share of the inputs, added in order), hence the results too.
// Launched with as many threads as the widest layer has units, so that several blocks fit an SM; a
// narrower layer's threads split the rows, and one narrower by four or more (the outputs) the shares of
// the inputs, which shortens its chain.  Splitting the inputs of every layer, with 512 threads, cost 16
// additions through shared memory for every product of a narrow network: 200,000 rows of 7 ->
// 16 -> 16 -> 16 -> 8 564 -> 264 us (layer by layer 332), 20,000 of a network 256 wide 392 -> 270,
// 300 wide 677 -> 366 (590).
constexpr int kFwdRows = 16;  // rows per block

// whether a layer's threads split its inputs (their sums take kFwdThreads x kFwdRows floats)
__host__ __device__ inline bool fwd_splits(int in, int out, int threads) {
  return threads >= 4 * fwd_pad(out) && in >= 32;
}

template <int RT>  // RT consecutive floats in shared memory
__device__ __forceinline__ void load_some(const float* p, float (&v)[RT]) {
  if constexpr (RT >= 4) {
    load_rows<RT>(p, v);
  } else if constexpr (RT == 2) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    v[0] = t.x; v[1] = t.y;
  } else {
    v[0] = *p;
  }
}

template <typename WB>
__global__ void __launch_bounds__(kFwdThreads, 2) forward_rows_kernel(const FwdArgs a, const WB* __restrict__ wt) {
  constexpr int RB = kFwdRows;
  extern __shared__ __align__(16) float sm[];
  int maxw = 0;
  for (int l = 0; l <= a.depth; ++l) maxw = max(maxw, a.dims[l]);
  float* cur = sm;
  float* nxt = sm + maxw * RB;
  float* const red = sm + 2 * maxw * RB;
  const int tid = threadIdx.x, nthr = blockDim.x, r0 = blockIdx.x * RB;
  for (int e = tid; e < a.dims[0] * RB; e += nthr) {
    const int r = e / a.dims[0], k = e % a.dims[0];
    cur[k * RB + r] = r0 + r < a.n ? a.x[(size_t)(r0 + r) * a.dims[0] + k] : 0.f;
  }
  __syncthreads();
  for (int l = 0; l < a.depth; ++l) {
    const int in = a.dims[l], out = a.dims[l + 1], wp = fwd_pad(out);
    const int parts = kFwdThreads / wp, len = (in + parts - 1) / parts, group = tid / wp, j = tid - group * wp;
    const bool last = l + 1 == a.depth;
    const WB* w = wt + a.woff[l] + j;
    auto layer = [&](auto count) {  // rows group RT .. group RT + RT - 1 of unit j
      constexpr int RT = decltype(count)::value;
      if (group >= RB / RT || j >= out) return;
      const float* x = cur + group * RT;
      float s[RT] = {};
      auto term = [&](int k, float (&acc)[RT]) {
        const float c = (float)w[(size_t)k * wp];
        float v[RT];
        load_some<RT>(x + k * RB, v);
#pragma unroll
        for (int i = 0; i < RT; ++i) acc[i] = fmaf(c, v[i], acc[i]);
      };
      if (len == 1) {  // narrow layers: each product is a share of its own
#pragma unroll 8
        for (int k = 0; k < in; ++k) {
          float acc[RT] = {};
          term(k, acc);
#pragma unroll
          for (int i = 0; i < RT; ++i) s[i] += acc[i];
        }
      } else {
        for (int k0 = 0; k0 < in; k0 += len) {
          const int k1 = min(in, k0 + len);
          float acc[RT] = {};
#pragma unroll 8
          for (int k = k0; k < k1; ++k) term(k, acc);
#pragma unroll
          for (int i = 0; i < RT; ++i) s[i] = k0 == 0 ? acc[i] : s[i] + acc[i];
        }
      }
      const float b = a.bias[a.boff[l] + j];
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const int r = group * RT + i;
        const float v = s[i] + b;
        if (!last) nxt[j * RB + r] = tanhf(v);
        else if (r0 + r < a.n) a.y[(size_t)(r0 + r) * out + j] = v;
      }
    };
    const int groups = nthr / wp;
    if (fwd_splits(in, out, nthr)) {
      for (int p = group; p < parts && group < groups; p += groups) {
        const int k1 = min(in, (p + 1) * len);
        float acc[RB] = {};
#pragma unroll 4
        for (int k = p * len; k < k1; ++k) {
          const float c = (float)w[(size_t)k * wp];
          float v[RB];
          load_rows<RB>(cur + k * RB, v);
#pragma unroll
          for (int i = 0; i < RB; ++i) acc[i] = fmaf(c, v[i], acc[i]);
        }
#pragma unroll
        for (int i = 0; i < RB; ++i) red[(p * RB + i) * wp + j] = acc[i];
      }
      __syncthreads();
      for (int e = tid; e < wp * RB; e += nthr) {
        const int u = e % wp, r = e / wp;
        if (u >= out) continue;
        float s = red[r * wp + u];
        for (int p = 1; p < parts; ++p) s += red[(p * RB + r) * wp + u];
        s += a.bias[a.boff[l] + u];
        if (!last) nxt[u * RB + r] = tanhf(s);
        else if (r0 + r < a.n) a.y[(size_t)(r0 + r) * out + u] = s;
      }
    } else if (groups >= 16) layer(std::integral_constant<int, 1>{});
    else if (groups >= 8) layer(std::integral_constant<int, 2>{});
    else if (groups >= 4) layer(std::integral_constant<int, 4>{});
    else if (groups >= 2) layer(std::integral_constant<int, 8>{});
    else layer(std::integral_constant<int, 16>{});
    __syncthreads();
    float* t = cur;
    cur = nxt;
    nxt = t;
  }
}

template <typename WB> __device__ __forceinline__ WB to_weight(float v);
template <> __device__ __forceinline__ float to_weight<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 to_weight<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// The weights of one layer (out x in, FP32) transposed to [in][out padded], zeros in the padding.
template <typename WB>
__global__ void pack_kernel(const float* __restrict__ p, int in, int out, WB* __restrict__ wt) {
  __shared__ float tile[32][33];
  const int k0 = blockIdx.x * 32, u0 = blockIdx.y * 32, wp = fwd_pad(out);
  for (int i = threadIdx.y; i < 32; i += 8)
    tile[i][threadIdx.x] =
        u0 + i < out && k0 + (int)threadIdx.x < in ? p[(size_t)(u0 + i) * in + k0 + threadIdx.x] : 0.f;
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8)
    if (k0 + i < in) wt[(size_t)(k0 + i) * wp + u0 + threadIdx.x] = to_weight<WB>(tile[threadIdx.x][i]);
}

}  // namespace
}  // namespace lbw
