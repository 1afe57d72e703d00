// lbw_mlp_forward.cuh -- forward pass of the surrogate network in one launch (lbw_mlp.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

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
// whole calls with the copies of inputs and outputs: 1 row 134 -> 45 us, 400 rows 177 -> 47 us, 4000
// rows 216 -> 93 us, 20,000 rows 464 -> 390 us (shared-memory reads of the rows bound the last).
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
