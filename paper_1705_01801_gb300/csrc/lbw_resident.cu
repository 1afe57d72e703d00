// lbw_resident.cu -- many time steps of small lattices in one launch.
//
// A lattice (or an ensemble of them) of a few hundred thousand nodes steps faster than a kernel
// can be launched: one step of a 128 x 128 FP64 disk moves 1.8 MB that never leave the L2, and
// of its 10.6 us nearly all went to launch, prologue and pipeline fill.  Here every CTA owns one box of one
// lattice for a whole launch of up to kResChunk steps: node offsets, face flags and the force
// coefficients are set up once, and a step costs the loads and stores of its populations (L2
// hits) and one barrier among the CTAs of the lattice.  Per step a thread pulls the seven
// populations of its K nodes and of a share of the box's one-node halo (whose populations
// other CTAs own), puts their post-stream rho into shared memory, and after one __syncthreads
// collides its nodes (the populations stay in registers) and stores them to the other buffer.
// Measured per step, a launch per step -> here: disk 10.6 -> 3.2 us, the paper's 20 x 200 x 30
// torus in FP64 with a ring source 29.3 -> 10.5 us, 41 pipes of 10,000 FP32 nodes with sources
// 176 -> 9.5 us (38 + 3 of them in two turns).  What bounds it: 2.0 us of barrier and load
// latency for the smallest lattices, the FP64 pipe for FP64, load latency beyond a few hundred
// nodes per CTA (25 % of the issue slots busy).
//
// Sources that impose P replace the node's outputs as they are stored, from values that the last
// threads compute (an FP64 sine) while thread 0 waits at the barrier; other sources take a pass
// through memory behind one more __syncthreads (which cost 5 us per step when all did).
//
// One CTA per SM, of as many threads as leave the populations in registers (kResShapes; 1024
// threads of two or three nodes spilled and were 10 to 30 % slower).
//
// The launch is cooperative, so all CTAs are resident and the barrier (one arrival counter per
// lattice, cleared before each launch) completes; its wait is bounded like every device wait
// of the step kernels and raises counters[3].
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "lbw_internal.h"
#include "lbw_march.cuh"
#include "lbw_resident.h"
#include "lbw_tma.cuh"

namespace lbw {
namespace {

using namespace dev;

constexpr int kResMaxSlots = 1 << 14, kResMaxRows = 1 << 10;  // fields of a node's packed word
constexpr long long kResWaitLimit = 1LL << 21;                // tries of under a microsecond

template <typename S>
struct ResArgs {
  StepArgs<S> one;                 // the lattice (members == nullptr)
  const StepArgs<S>* members;      // or an ensemble's, for source buffer 0
  const ResItem* items;            // one per CTA
  unsigned* bars;                  // arrival counters, 32 words apart
  unsigned long long* counters;
  const unsigned long long* stall;  // injected-timeout request (nullptr: none)
  S* base[2];                      // population buffers of all lattices (sources)
  const SourceEntry* src;
  const int* src_order;
  int src_kind;
  double src_amp;
  int cur, steps, nprobe;
  long long cap;
  int last_group;                  // this launch advances the step and sample counters
};

// plain loads: other CTAs write these values during the launch, so neither the read-only
// path nor a compiler's assumption of constancy may be used
template <typename S> __device__ __forceinline__ typename Store<S>::R ld_pop(const S* p) {
  return Store<S>::ld_smem(p);
}

// Strides of the populations and of the q1 and q3 axes, in elements.
struct Strides {
  int ps, s1, s3;
};
// Per face, the source of the population that streams in through it (relative to the node) and
// the factor it arrives with.  In shared memory: most nodes need neither.
template <typename R>
struct Faces {
  int off[6];
  R m[6];
};

// Pull streaming of the seven populations into the node at element x (flag bit 2 axis + side:
// the node lies on that face), in two parts: the loads, which have no branches, so that those of
// all of a thread's nodes are in flight together, then the factors of the walls it lies on.
template <typename S>
__device__ __forceinline__ void load_node(const S* f, int x, unsigned fl, const Strides& F,
                                          const Faces<typename Store<S>::R>& faces, typename Store<S>::R (&v)[7]) {
  const int o[6] = {F.ps - F.s1, 2 * F.ps + F.s1, 3 * F.ps - 1, 4 * F.ps + 1, 5 * F.ps - F.s3, 6 * F.ps + F.s3};
  v[0] = ld_pop(f + x);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    int d = o[i];
    if ((fl >> i) & 1) d = faces.off[i];
    v[i + 1] = ld_pop(f + (x + d));
  }
}

// `walls`: the faces whose factor is not 1.
template <typename S, bool TILE>
__device__ __forceinline__ void finish_node(unsigned fl, unsigned walls, const Faces<typename Store<S>::R>& faces,
                                            const typename Store<S>::R (&wt)[2], typename Store<S>::R (&v)[7]) {
  if constexpr (Store<S>::kScaled && !TILE) {
    v[0] *= wt[0];
#pragma unroll
    for (int i = 1; i < 7; ++i) v[i] *= wt[1];
  }
  if (fl & walls) {
#pragma unroll
    for (int i = 0; i < 6; ++i)
      if ((fl >> i) & 1) v[i + 1] *= faces.m[i];
  }
}

// rho of the pulled populations, in the summation order of the kernel that advances a lattice
// of this kind step by step (TILE: the TMA tile kernels; otherwise lbw_march.cuh)
template <typename S, bool TILE>
__device__ __forceinline__ typename Store<S>::R rho_of(const typename Store<S>::R (&v)[7],
                                                       const typename Store<S>::R (&wt)[2]) {
  if constexpr (Store<S>::kScaled && TILE) {
    const float s = __fadd_rn(__fadd_rn(__fadd_rn(v[1], v[2]), __fadd_rn(v[3], v[4])), __fadd_rn(v[5], v[6]));
    return __fmaf_rn(wt[0], v[0], __fmul_rn(wt[1], s));
  } else {
    return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + v[6]);
  }
}

// Collision of one node: v holds its pulled populations and receives the post-collision ones;
// X13: the metric couples q1 and q3 (FP64; otherwise those coefficients are zero).
// 64-bit storage: with h^a half the forcing term, j^a = f_a+ - f_a- + h^a, so
// f*_a+ = e + j^a - f_a+ = (e + h^a) - f_a- and f*_a- = (e - h^a) - f_a+: 28 to 32 operations a
// node where forming j^a takes 46, which is what FP64 (2 a cycle and SM) is bound by
// (120k nodes: 14.0 -> 10.2 us per step).  The rows then hold half the coefficients, signed,
// and the node's own in one (coef_row).  32- and 16-bit storage repeats the operations of the
// kernels that step once per launch, so the results do not depend on which of them runs.
template <typename S, bool TILE, bool X13>
__device__ __forceinline__ void collide_node(const typename Store<S>::R (&c)[T_SLOTS],
                                             typename Store<S>::R cs2, typename Store<S>::R two_w0,
                                             typename Store<S>::R rho, typename Store<S>::R ru,
                                             typename Store<S>::R rd, typename Store<S>::R rr,
                                             typename Store<S>::R rl, typename Store<S>::R rn,
                                             typename Store<S>::R rp, typename Store<S>::R (&v)[7]) {
  using R = typename Store<S>::R;
  if constexpr (sizeof(R) == 8) {
    R h1 = c[T_MG1] * rho + c[T_A1P] * ru + c[T_A1M] * rd;
    R h3 = c[T_MG3] * rho + c[T_C33P] * rn + c[T_C33M] * rp;
    if constexpr (X13) {
      h1 = h1 + c[T_C13P] * rn + c[T_C13M] * rp;
      h3 = h3 + c[T_B13P] * ru + c[T_B13M] * rd;
    }
    const R h2 = c[T_H22] * (rr - rl);
    const R e = cs2 * rho;
    const R a1 = (e + h1) - v[2], a2 = (e - h1) - v[1], a3 = (e + h2) - v[4], a4 = (e - h2) - v[3],
            a5 = (e + h3) - v[6], a6 = (e - h3) - v[5];
    v[0] = two_w0 * rho - v[0];
    v[1] = a1; v[2] = a2; v[3] = a3; v[4] = a4; v[5] = a5; v[6] = a6;
  } else if constexpr (TILE) {
    constexpr bool SC = Store<S>::kScaled;
    const float half = SC ? 1.f / cs2 : 0.5f;
    float nD1 = __fmaf_rn(c[T_A1M], rd, __fmul_rn(-c[T_A1P], ru));
    float nD3 = __fmaf_rn(c[T_B13M], rd, __fmul_rn(-c[T_B13P], ru));
    nD1 = __fmaf_rn(-c[T_S1], rho, __fmaf_rn(c[T_C13M], rp, __fmaf_rn(-c[T_C13P], rn, nD1)));
    nD3 = __fmaf_rn(-c[T_S3], rho, __fmaf_rn(c[T_C33M], rp, __fmaf_rn(-c[T_C33P], rn, nD3)));
    const float D2 = __fmul_rn(c[T_H22], __fsub_rn(rr, rl));
    const float j1 = __fmaf_rn(half, __fmaf_rn(c[T_MG1], rho, nD1), __fsub_rn(v[1], v[2]));
    const float j2 = __fmaf_rn(-half, D2, __fsub_rn(v[3], v[4]));
    const float j3 = __fmaf_rn(half, __fmaf_rn(c[T_MG3], rho, nD3), __fsub_rn(v[5], v[6]));
    const float e = SC ? __fadd_rn(rho, rho) : __fmul_rn(cs2, rho);
    v[0] = SC ? __fsub_rn(e, v[0]) : __fsub_rn(__fmul_rn(two_w0, rho), v[0]);
    v[1] = __fsub_rn(__fadd_rn(e, j1), v[1]);
    v[2] = __fsub_rn(__fsub_rn(e, j1), v[2]);
    v[3] = __fsub_rn(__fadd_rn(e, j2), v[3]);
    v[4] = __fsub_rn(__fsub_rn(e, j2), v[4]);
    v[5] = __fsub_rn(__fadd_rn(e, j3), v[5]);
    v[6] = __fsub_rn(__fsub_rn(e, j3), v[6]);
  } else {
    const R D1 = c[T_A1P] * ru - c[T_A1M] * rd + c[T_C13P] * rn - c[T_C13M] * rp + c[T_S1] * rho;
    const R D3 = c[T_B13P] * ru - c[T_B13M] * rd + c[T_C33P] * rn - c[T_C33M] * rp + c[T_S3] * rho;
    const R D2 = c[T_H22] * (rr - rl);
    const R half = R(0.5);
    const R j1 = (v[1] - v[2]) + half * (c[T_MG1] * rho - D1);
    const R j2 = (v[3] - v[4]) - half * D2;
    const R j3 = (v[5] - v[6]) + half * (c[T_MG3] * rho - D3);
    const R e = cs2 * rho;
    v[0] = two_w0 * rho - v[0];
    v[1] = e + j1 - v[1];
    v[2] = e - j1 - v[2];
    v[3] = e + j2 - v[3];
    v[4] = e - j2 - v[4];
    v[5] = e + j3 - v[5];
    v[6] = e - j3 - v[6];
  }
}

// A row of the coefficient table as collide_node takes it (64-bit storage: h^a's signed
// coefficients; halving is exact).
template <typename S>
__device__ __forceinline__ typename Store<S>::R coef_row(const typename Store<S>::R* t, int k) {
  using R = typename Store<S>::R;
  if constexpr (sizeof(R) == 4) return t[k];
  const R v = t[k], h = R(0.5);
  switch (k) {
    case T_A1P: case T_B13P: case T_C13P: case T_C33P: case T_H22: return -h * v;
    case T_A1M: case T_B13M: case T_C13M: case T_C33M: return h * v;
    case T_MG1: return h * (v - t[T_S1]);
    case T_MG3: return h * (v - t[T_S3]);
    default: return v;
  }
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(p) : "memory");
}

// Shared memory: rho of the box with a one-node border ((bx + 2) (by + 2) (bz + 2)), the
// coefficient rows of the box (by bz), and per halo node its element and packed word.
template <typename S, bool TILE, int NT, int K, bool X13>
__global__ void __launch_bounds__(NT, 1) resident_kernel(const ResArgs<S> ra) {
  using R = typename Store<S>::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) StepArgs<S> A;
  __shared__ Faces<R> faces;
  __shared__ int probe_x[kMaxProbes], probe_id[kMaxProbes];
  __shared__ int probe_cnt, halo_cnt, bad;
  // kind 0 sources of the box (P imposed; up to kNear): element and this step's populations at
  // rest and in motion, stored in place of the node's own; the others go through memory
  constexpr int kNear = 64;
  __shared__ int near_x[kNear];
  __shared__ R near_v[kNear][2];
  __shared__ double near_sg[kNear], near_om[kNear], near_cs2;
  // The others of a lattice have one frequency: 32- and 16-bit storage takes the sine of the first once
  // (far_v) instead of one per source, which bound plates of them (a plane of 128 x 128, FP32: 18.7 ->
  // 14.2 us a step).  FP64 is bound by its nodes, and the share would cost them registers.
  constexpr bool kShare = sizeof(S) < 8;
  __shared__ int ntimed;  // sources whose sine is taken here: the near ones, or the first
  __shared__ double far_v;
  const int tid = threadIdx.x, nthr = blockDim.x;
  // what only the prologue, the edges and thread 0 need stays in shared memory: 1024 threads have
  // 64 registers each
  __shared__ ResItem it;
  __shared__ unsigned long long t0, sample0;
  if (tid == 0) {
    it = ra.items[blockIdx.x];
    t0 = ra.counters[0];
    sample0 = ra.counters[1];
  }
  __syncthreads();
  {
    const unsigned* from = reinterpret_cast<const unsigned*>(ra.members ? ra.members + it.member : &ra.one);
    unsigned* to = reinterpret_cast<unsigned*>(&A);
    for (int k = tid; k < (int)(sizeof(StepArgs<S>) / 4); k += nthr) to[k] = from[k];
  }
  if (tid == 0) {
    probe_cnt = halo_cnt = 0;
    bad = ra.counters[3] != 0ull;  // an earlier step timed out: nothing to advance
  }
  const int px = it.bx + 2, pxy = px * (it.by + 2), nslot = pxy * (it.bz + 2);
  R* const rho = reinterpret_cast<R*>(smem_raw);
  R* const tab = rho + (nslot + 3) / 4 * 4;
  int2* const halo = reinterpret_cast<int2*>(tab + it.by * it.bz * T_SLOTS);
  for (int k = tid; k < nslot; k += nthr) rho[k] = R(0);  // ghosts beyond walls stay zero
  __syncthreads();

  const int n1 = A.n1, n2 = A.n2, n3 = A.n3;
  const Strides F{(int)A.ps, A.pitch, n1 * A.pitch};
  const R wt[2] = {A.w[0], A.w[1]};
  if (tid < 6) {
    const int b = A.bc[tid], opp = tid & 1 ? tid : tid + 2;  // the population reflected into pop tid + 1
    const int wrap = tid >> 1 == 0 ? (n1 - 1) * F.s1 : tid >> 1 == 1 ? n2 - 1 : (n3 - 1) * F.s3;
    faces.off[tid] = b == LBW_BC_PERIODIC ? (tid + 1) * F.ps + (tid & 1 ? -wrap : wrap)
                     : b == LBW_BC_FREE   ? (tid + 1) * F.ps : opp * F.ps;
    faces.m[tid] = b == LBW_BC_BOUNCE ? A.damping : (b == LBW_BC_ANTIBOUNCE ? R(-1) : R(1));
  }
  __syncthreads();
  unsigned walls = 0;
  for (int i = 0; i < 6; ++i) walls |= faces.m[i] != R(1) ? 1u << i : 0u;
  const bool p1 = A.bc[0] == LBW_BC_PERIODIC, p2 = A.bc[2] == LBW_BC_PERIODIC, p3 = A.bc[4] == LBW_BC_PERIODIC;
  auto flags_of = [&](int q1, int q2, int q3) -> unsigned {
    return (q1 == 0) | (q1 == n1 - 1) << 1 | (q2 == 0) << 2 | (q2 == n2 - 1) << 3 | (q3 == 0) << 4 |
           (q3 == n3 - 1) << 5;
  };
  auto elem_of = [&](int q1, int q2, int q3) { return (q3 * n1 + q1) * F.s1 + A.col0 + q2; };

  for (int s = tid; s < A.nprobe; s += nthr) {
    const int q1 = A.probe_q[3 * s], q2 = A.probe_q[3 * s + 1], q3 = A.probe_q[3 * s + 2];
    if (q1 >= it.y0 && q1 < it.y0 + it.by && q2 >= it.x0 && q2 < it.x0 + it.bx && q3 >= it.z0 && q3 < it.z0 + it.bz) {
      const int at = atomicAdd(&probe_cnt, 1);
      probe_x[at] = elem_of(q1, q2, q3);
      probe_id[at] = s;
    }
  }
  __syncthreads();

  // own nodes: element and packed word (flags | probe << 6 | source << 7 | slot << 8 | row << 22)
  const int nbox = it.bx * it.by * it.bz;
  int xe[K];
  unsigned pk[K];
  const int own = tid < nbox ? (nbox - tid - 1) / nthr + 1 : 0;  // the thread's nodes
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int id = k < own ? tid + k * nthr : 0;  // past them the box's first node is loaded and dropped
    const int ix = id % it.bx, r = id / it.bx, iy = r % it.by, iz = r / it.by;
    const int q2 = it.x0 + ix, q1 = it.y0 + iy, q3 = it.z0 + iz;
    xe[k] = elem_of(q1, q2, q3);
    pk[k] = flags_of(q1, q2, q3) | (unsigned)((iz + 1) * pxy + (iy + 1) * px + ix + 1) << 8 | (unsigned)r << 22;
    for (int s = 0; s < probe_cnt; ++s)
      if (probe_x[s] == xe[k]) pk[k] |= 1u << 6;
  }
  for (int k = tid; k < it.by * it.bz * T_SLOTS; k += nthr) {
    const int r = k / T_SLOTS, q1 = it.y0 + r % it.by, q3 = it.z0 + r / it.by;
    tab[k] = coef_row<S>(A.tab + ((long long)q3 * n1 + q1) * T_SLOTS, k % T_SLOTS);
  }
  // halo nodes: the box's six faces, except along an axis that the box spans (its periodic wrap
  // is served by the border copies below) and beyond walls
  const bool sx = it.bx == n2, sy = it.by == n1, sz = it.bz == n3;
  {
    const int nx = sx ? 0 : it.by * it.bz, ny = sy ? 0 : it.bx * it.bz, nz = sz ? 0 : it.bx * it.by;
    for (int h = tid; h < 2 * (nx + ny + nz); h += nthr) {
      int ix, iy, iz;
      if (h < 2 * nx) {
        const int u = h >> 1;
        ix = h & 1 ? it.bx : -1; iy = u % it.by; iz = u / it.by;
      } else if (h < 2 * (nx + ny)) {
        const int e = h - 2 * nx, u = e % ny;
        iy = e >= ny ? it.by : -1; ix = u % it.bx; iz = u / it.bx;
      } else {
        const int e = h - 2 * (nx + ny), u = e % nz;
        iz = e >= nz ? it.bz : -1; ix = u % it.bx; iy = u / it.bx;
      }
      const int q1 = resolve(it.y0 + iy, n1, p1), q2 = resolve(it.x0 + ix, n2, p2), q3 = resolve(it.z0 + iz, n3, p3);
      if (q1 >= 0 && q2 >= 0 && q3 >= 0)
        halo[atomicAdd(&halo_cnt, 1)] = make_int2(
            elem_of(q1, q2, q3), (int)(flags_of(q1, q2, q3) | (unsigned)((iz + 1) * pxy + (iy + 1) * px + ix + 1) << 8));
    }
  }
  __syncthreads();
  const int nhalo = halo_cnt, npr = probe_cnt;

  // along a spanned periodic axis the first and the last nodes' rho also go to the border
  const unsigned img = (sy && p1 ? 3u : 0u) | (sx && p2 ? 12u : 0u) | (sz && p3 ? 48u : 0u);

  S* const buf[2] = {const_cast<S*>(A.fin), A.fout};
  const int nsrc = it.src_hi - it.src_lo;
  const bool near = nsrc <= kNear && ra.src_kind == 0;
  if (tid == 0) ntimed = near ? nsrc : kShare && nsrc > 0;
  auto source_entry = [&](int e) { return ra.src[ra.src_order[it.src_lo + e]]; };
  // near source `mine`'s populations at time t, as impose_source writes them; the last threads
  // compute them, thread 0 waits at the barrier meanwhile
  const int mine = nthr - 1 - tid;
  __syncthreads();
  auto set_near = [&](unsigned long long t) {
    const double v = ra.src_amp * sin(near_om[mine] * (double)t), rho = near_sg[mine] * v;
    if (kShare && mine == 0) far_v = v;
    const double w0 = 1.0 - 3.0 * near_cs2, w1 = 0.5 * near_cs2;
    double rest = w0 * rho, moving = w1 * rho;
    if (Store<S>::kScaled) {
      rest /= w0;
      moving /= w1;
    }
    near_v[mine][0] = (R)rest;
    near_v[mine][1] = (R)moving;
  };
  if (mine < ntimed) {
    const SourceEntry e = source_entry(mine);
    near_x[mine] = (int)(e.off - (A.fin - ra.base[0]));  // relative to the lattice's own buffer
    near_sg[mine] = e.sg;
    near_om[mine] = e.omega;
    near_cs2 = e.cs2;
  }
  __syncthreads();
  if (mine < ntimed) set_near(t0 + 1);
  __syncthreads();
  if (near && nsrc > 0) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      for (int e = 0; e < nsrc; ++e)
        if (near_x[e] == xe[k]) pk[k] |= 1u << 7;
  }
  bool ok = bad == 0;
  if (ok && ra.stall && *ra.stall) {  // injected timeout: a bounded wait that nothing completes
    if (tid == 0) {
      int n = 0;
      while (ld_acquire(ra.bars + 32 * it.group) != 0xffffffffu && ++n < kStallTries) {}
      ra.counters[3] = 1;
    }
    ok = false;
  }

  // FP32 values land in the registers they stay in, so all of a thread's loads go out first (204,800
  // nodes 5.9 -> 4.9 us per step); 16-bit values need a conversion each and FP64 twice the
  // registers, and node by node is faster (240,000 nodes: FP16 7.1 -> 5.5 us)
  constexpr bool kTogether = sizeof(S) == 4;
  int cur = ra.cur;
  for (int s = 0; ok && s < ra.steps; ++s) {
    const S* const f = buf[cur];
    S* const g = buf[1 - cur];
    R v[K][7];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if constexpr (kTogether) {
        load_node(f, xe[k], pk[k], F, faces, v[k]);
      } else if (k < own) {
        load_node(f, xe[k], pk[k], F, faces, v[k]);
        finish_node<S, TILE>(pk[k], walls, faces, wt, v[k]);
      }
    }
    for (int h = nthr - 1 - tid; h < nhalo; h += nthr) {  // threads without a last node first
      const int2 e = halo[h];
      R u[7];
      load_node(f, e.x, (unsigned)e.y, F, faces, u);
      finish_node<S, TILE>((unsigned)e.y, walls, faces, wt, u);
      rho[(unsigned)e.y >> 8] = rho_of<S, TILE>(u, wt);
    }
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (k < own) {
        if constexpr (kTogether) finish_node<S, TILE>(pk[k], walls, faces, wt, v[k]);
        const int slot = (pk[k] >> 8) & (kResMaxSlots - 1);
        const R r = rho_of<S, TILE>(v[k], wt);
        rho[slot] = r;
        const unsigned edge = pk[k] & img;
        if (edge) {
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const int shift = a == 0 ? it.by * px : a == 1 ? it.bx : it.bz * pxy;
            if (edge & (1u << (2 * a))) rho[slot + shift] = r;
            if (edge & (2u << (2 * a))) rho[slot - shift] = r;
          }
        }
      }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (k < own) {
        const int slot = (pk[k] >> 8) & (kResMaxSlots - 1);
        const R* T = tab + (pk[k] >> 22) * T_SLOTS;
        R c[T_SLOTS];
#pragma unroll
        for (int q = 0; q < T_SLOTS; q += 4) {
          if (sizeof(R) == 4) {
            const float4 t = *reinterpret_cast<const float4*>(T + q);
            c[q] = t.x; c[q + 1] = t.y; c[q + 2] = t.z; c[q + 3] = t.w;
          } else {
            const double2 t = *reinterpret_cast<const double2*>(T + q), t2 = *reinterpret_cast<const double2*>(T + q + 2);
            c[q] = t.x; c[q + 1] = t.y; c[q + 2] = t2.x; c[q + 3] = t2.y;
          }
        }
        const R r = rho[slot];
        R rl = rho[slot - 1], rr = rho[slot + 1];
        if (!p2) {
          if (pk[k] & 4u) rl = A.s2lo * r;
          if (pk[k] & 8u) rr = A.s2hi * r;
        }
        collide_node<S, TILE, X13>(c, A.cs2, A.two_w0, r, rho[slot + px], rho[slot - px], rr, rl, rho[slot + pxy],
                              rho[slot - pxy], v[k]);
#pragma unroll
        for (int i = 0; i < 7; ++i)
          if (Store<S>::kScaled && !TILE) v[k][i] *= i == 0 ? A.inv_w[0] : A.inv_w[1];
        if (pk[k] & 128u) {
          int e = 0;
          while (near_x[e] != xe[k]) ++e;
#pragma unroll
          for (int i = 0; i < 7; ++i) v[k][i] = near_v[e][i > 0];
        }
#pragma unroll
        for (int i = 0; i < 7; ++i) Store<S>::st(g + (xe[k] + i * F.ps), v[k][i]);
        if (pk[k] & 64u) {
          const unsigned long long t = sample0 + s;
          if (t < (unsigned long long)A.cap)
            for (int q = 0; q < npr; ++q)
              if (probe_x[q] == xe[k]) A.series[(long long)probe_id[q] * A.cap + t] = (double)r * (double)c[T_INVSG];
        }
      }
    if (nsrc > 0 && !near) {  // harmonic sources on the state just written (as source_kernel does)
      __syncthreads();
      for (int e = tid; e < nsrc; e += nthr) {
        const SourceEntry se = source_entry(e);
        impose_source<S, false>(ra.base[1 - cur], se, ra.src_kind, kShare ? far_v : ra.src_amp * sin(se.omega * (double)(t0 + s + 1)));
      }
    }
    cur ^= 1;
    if (s + 1 == ra.steps) break;
    __syncthreads();
    if (tid == 0) red_release(ra.bars + 32 * it.group);
    // the next step's source values, while the other CTAs arrive
    if (mine < ntimed) set_near(t0 + s + 2);
    if (tid == 0) {
      const unsigned want = (unsigned)(s + 1) * (unsigned)it.group_size;
      long long n = 0;
      const unsigned* const bar = ra.bars + 32 * it.group;
      while (ld_acquire(bar) < want) {
        if (++n > kResWaitLimit) {
          ra.counters[3] = 1;
          bad = 1;
          break;
        }
      }
    }
    __syncthreads();
    ok = bad == 0;
  }

  __syncthreads();
  if (tid == 0 && ra.last_group) {
    __threadfence();
    const unsigned ticket = atomicAdd(reinterpret_cast<unsigned*>(&ra.counters[2]), 1u);
    if (ticket == gridDim.x - 1) {
      ra.counters[0] = t0 + ra.steps;
      const unsigned long long t = sample0 + ra.steps;
      if (ra.nprobe > 0) ra.counters[1] = t < (unsigned long long)ra.cap ? t : (unsigned long long)ra.cap;
      ra.counters[2] = 0;
      __threadfence();
    }
  }
}


// Threads and nodes per thread of a box of `own` nodes.
struct ResShape {
  int threads, k;
};
constexpr ResShape kResShapes[] = {{512, 1}, {512, 2}, {768, 2}, {768, 3}, {768, 4}, {1024, 4}};

int shape_of(int own) {
  int i = 0;
  while (kResShapes[i].threads * kResShapes[i].k < own) ++i;
  return i;
}

template <typename S, bool TILE, bool X13, typename F>
auto with_shape(int own, F&& f) {
  switch (shape_of(own)) {
    case 0: return f(resident_kernel<S, TILE, 512, 1, X13>);
    case 1: return f(resident_kernel<S, TILE, 512, 2, X13>);
    case 2: return f(resident_kernel<S, TILE, 768, 2, X13>);
    case 3: return f(resident_kernel<S, TILE, 768, 3, X13>);
  }
  if constexpr (sizeof(S) < 8) {
    if (shape_of(own) == 4) return f(resident_kernel<S, TILE, 768, 4, X13>);
    return f(resident_kernel<S, TILE, 1024, 4, X13>);
  } else {
    return f(resident_kernel<S, TILE, 768, 3, X13>);
  }
}

// The kernel for (storage, arithmetic form, coupled axes, nodes per box): f(kernel).
template <typename S, typename F>
auto with_kernel(bool tile, bool x13, int own, F&& f) {
  if constexpr (sizeof(S) == 8) {
    if (x13) return with_shape<S, true, true>(own, f);
  } else {
    if (!tile) return with_shape<S, false, false>(own, f);
  }
  return with_shape<S, true, false>(own, f);
}

template <typename F>
auto with_prec(int prec, F&& f) {
  switch (prec) {
    case LBW_F64: return f(double());
    case LBW_F32: return f(float());
    case LBW_F16S: return f(__half());
    default: return f(__nv_bfloat16());
  }
}

int max_box(int prec) { return prec == LBW_F64 ? 2048 : 4096; }

int round32(long long n) { return (int)((n + 31) / 32 * 32); }

struct Box {
  int b[3] = {0, 0, 0};  // q1, q2, q3 extent
  long long count = 0;   // boxes in the lattice
  int own = 0, halo = 0, smem = 0;
  double cost = 1e300;
};

// Best box for a lattice on at most `budget` CTAs: the least work per CTA.  A halo node costs a
// pull and a sum but no collision; one across a q2 face also brings a sector per value.
Box best_box(const lbw_grid_desc& d, int budget, int prec) {
  const int rs = prec == LBW_F64 ? 8 : 4, own_max = max_box(prec);
  Box best;
  auto ceil_div = [](int a, int b) { return (a + b - 1) / b; };
  for (int c2 = 1; c2 <= std::min(d.n[1], budget); ++c2) {
    const int b2 = ceil_div(d.n[1], c2);
    if (c2 > 1 && ceil_div(d.n[1], b2) != c2) continue;
    for (int c1 = 1; c1 <= std::min(d.n[0], budget / c2); ++c1) {
      const int b1 = ceil_div(d.n[0], c1);
      if (c1 > 1 && ceil_div(d.n[0], b1) != c1) continue;
      // the most q3 splits give the smallest boxes
      for (int c3 = std::min(d.n[2], budget / (c1 * c2)); c3 >= 1; --c3) {
        const int b3 = ceil_div(d.n[2], c3);
        const long long own = (long long)b1 * b2 * b3, slots = (b1 + 2LL) * (b2 + 2) * (b3 + 2);
        if (own > own_max || slots > kResMaxSlots || (long long)b1 * b3 > kResMaxRows) break;
        const int h2 = b2 < d.n[1] ? 2 * b1 * b3 : 0, h1 = b1 < d.n[0] ? 2 * b2 * b3 : 0,
                  h3 = b3 < d.n[2] ? 2 * b1 * b2 : 0;
        const long long smem = (slots + 3) / 4 * 4 * rs + (long long)b1 * b3 * T_SLOTS * rs + 8LL * (h1 + h2 + h3);
        if (smem > 200 * 1024) break;
        const double cost = round32(own) + 0.6 * round32(h1 + h3) + 1.5 * h2;
        if (cost < best.cost) {
          best.b[0] = b1; best.b[1] = b2; best.b[2] = b3;
          best.count = (long long)ceil_div(d.n[0], b1) * ceil_div(d.n[1], b2) * ceil_div(d.n[2], b3);
          best.own = (int)own;
          best.halo = h1 + h2 + h3;
          best.smem = (int)smem;
          best.cost = cost;
        }
        if (ceil_div(d.n[2], b3) < c3) c3 = ceil_div(d.n[2], b3);
      }
    }
  }
  return best;
}

template <typename S>
cudaError_t launch_t(const Resident* r, const Resident::Launch& L, const StepArgs<S>* one, const void* members,
                     const ResState& st, int steps, bool last) {
  ResArgs<S> ra;
  if (one) ra.one = *one;
  else std::memset(&ra.one, 0, sizeof(ra.one));
  ra.members = one ? nullptr : reinterpret_cast<const StepArgs<S>*>(members);
  ra.items = r->items + L.first;
  ra.bars = r->bars;
  ra.counters = st.counters;
  ra.stall = st.stall;
  ra.base[0] = reinterpret_cast<S*>(st.f[0]);
  ra.base[1] = reinterpret_cast<S*>(st.f[1]);
  ra.src = st.src;
  ra.src_order = r->src_order;
  ra.src_kind = st.src_kind;
  ra.src_amp = st.src_amp;
  ra.cur = st.cur;
  ra.steps = steps;
  ra.nprobe = st.nprobe;
  ra.cap = st.cap;
  ra.last_group = last;
  cudaError_t e = cudaMemsetAsync(r->bars, 0, sizeof(unsigned) * 32 * L.groups, st.stream);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(L.count);
  cfg.blockDim = dim3(L.threads);
  cfg.dynamicSmemBytes = L.smem;
  cfg.stream = st.stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return with_kernel<S>(r->tile, r->x13, L.own, [&](auto kern) { return cudaLaunchKernelEx(&cfg, kern, ra); });
}

}  // namespace

lbw_status resident_create(const Grid* const* lattices, int n, int prec, bool tile, long long max_nodes,
                           cudaStream_t stream, Resident** out) {
  *out = nullptr;
  long long total = 0;
  for (int m = 0; m < n; ++m) total += lattices[m]->nn;
  if (total > max_nodes) return LBW_OK;
  int dev = 0, sms = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
    cudaGetLastError();
    return LBW_OK;
  }
  const int own_max = max_box(prec);
  std::vector<ResItem> items;
  Resident r;
  r.prec = prec;
  r.tile = tile;
  r.nodes = total;
  for (int m = 0; m < n; ++m) r.x13 |= lattices[m]->d.kind == LBW_TRUMPET;
  for (int first = 0; first < n;) {
    // the lattices of one launch: as many as the SMs hold at the most nodes per thread
    long long nodes = 0;
    int end = first, need = 0;
    for (; end < n; ++end) {
      const lbw_grid_desc& d = lattices[end]->d;
      if (7 * pop_stride(lattices[end]) >= (1LL << 31)) return LBW_OK;
      const int want = (int)((lattices[end]->nn * 5 / 4 + own_max - 1) / own_max);
      if (end > first && need + want > sms) break;
      if (lattices[end]->nn > (long long)own_max * sms || d.geom_mode != LBW_GEOM_AUTO) return LBW_OK;
      need += want;
      nodes += lattices[end]->nn;
    }
    Resident::Launch L;
    L.first = (int)items.size();
    L.groups = end - first;
    int own = 0, halo = 0;
    for (int m = first; m < end; ++m) {
      const Grid* g = lattices[m];
      const int share = std::max(1, (int)((double)sms * g->nn / nodes));
      const Box b = best_box(g->d, share, prec);
      if (b.count == 0) return LBW_OK;
      ResItem it{};
      it.member = m;
      it.group = m - first;
      it.group_size = (int)b.count;
      for (it.z0 = 0; it.z0 < g->d.n[2]; it.z0 += b.b[2])
        for (it.y0 = 0; it.y0 < g->d.n[0]; it.y0 += b.b[0])
          for (it.x0 = 0; it.x0 < g->d.n[1]; it.x0 += b.b[1]) {
            it.by = std::min(b.b[0], g->d.n[0] - it.y0);
            it.bx = std::min(b.b[1], g->d.n[1] - it.x0);
            it.bz = std::min(b.b[2], g->d.n[2] - it.z0);
            items.push_back(it);
          }
      own = std::max(own, b.own);
      halo = std::max(halo, b.halo);
      L.smem = std::max(L.smem, b.smem);
    }
    L.count = (int)items.size() - L.first;
    if (L.count > sms) return LBW_OK;
    const ResShape shape = kResShapes[shape_of(own)];
    L.own = own;
    L.threads = std::min(shape.threads, std::max(64, round32((own + shape.k - 1) / shape.k + (shape.k == 1 ? halo : 0))));
    int per = 0;
    const cudaError_t e = with_prec(prec, [&](auto tag) {
      return with_kernel<decltype(tag)>(tile, r.x13, own, [&](auto kern) {
        cudaError_t f = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (f == cudaSuccess) f = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, L.threads, L.smem);
        return f;
      });
    });
    if (e != cudaSuccess || per < 1) {
      cudaGetLastError();
      return LBW_OK;
    }
    r.launches.push_back(L);
    first = end;
  }
  int groups = 1;
  for (const Resident::Launch& L : r.launches) groups = std::max(groups, L.groups);
  r.host_items = items;
  Resident* p = new (std::nothrow) Resident(r);
  if (!p) return fail(LBW_ENOMEM, "host allocation failed");
  // one allocation: the barriers, then the boxes
  const size_t bars = sizeof(unsigned) * 32 * groups;
  cudaError_t e = cudaMallocAsync((void**)&p->bars, bars + sizeof(ResItem) * items.size(), stream);
  if (e == cudaSuccess) {
    p->items = reinterpret_cast<ResItem*>(reinterpret_cast<unsigned char*>(p->bars) + bars);
    e = cudaMemcpyAsync(p->items, items.data(), sizeof(ResItem) * items.size(), cudaMemcpyHostToDevice, stream);
  }
  if (e != cudaSuccess) {
    resident_destroy(p, stream);
    if (e != cudaErrorMemoryAllocation) return cuda_fail(e, "resident step kernel: upload");
    cudaGetLastError();
    return LBW_OK;  // a launch per step needs no memory of its own
  }
  *out = p;
  return LBW_OK;
}

void resident_destroy(Resident* r, cudaStream_t stream) {
  if (!r) return;
  if (r->bars) cudaFreeAsync(r->bars, stream);
  if (r->src_order) cudaFreeAsync(r->src_order, stream);
  delete r;
}

lbw_status resident_sources(Resident* r, const int32_t* host_q, int per_lattice, cudaStream_t stream) {
  // boxes of a lattice are regular and listed with q2 fastest, then q1, then q3
  std::vector<ResItem> items = r->host_items;
  std::vector<int> box_of, first_of, nx_of, ny_of;
  for (size_t k = 0; k < items.size(); ++k) {
    const ResItem& it = items[k];
    if (it.x0 == 0 && it.y0 == 0 && it.z0 == 0) {
      first_of.push_back((int)k);
      nx_of.push_back(0);
      ny_of.push_back(0);
    }
    if (it.y0 == 0 && it.z0 == 0) ++nx_of.back();
    if (it.x0 == 0 && it.z0 == 0) ++ny_of.back();
    items[k].src_lo = items[k].src_hi = 0;
  }
  for (size_t m = 0; m < first_of.size(); ++m) {
    const ResItem& b = items[first_of[m]];
    for (int k = 0; k < per_lattice; ++k) {
      const int32_t* q = host_q + 3 * (m * per_lattice + k);
      box_of.push_back(first_of[m] + ((q[2] / b.bz) * ny_of[m] + q[0] / b.by) * nx_of[m] + q[1] / b.bx);
      ++items[box_of.back()].src_hi;
    }
  }
  int at = 0;
  for (ResItem& it : items) {
    const int count = it.src_hi;
    it.src_lo = it.src_hi = at;
    at += count;
  }
  std::vector<int> order(box_of.size());
  for (size_t e = 0; e < box_of.size(); ++e) order[items[box_of[e]].src_hi++] = (int)e;
  // the new order first: where it cannot be had, the boxes stay as they are
  int* d_order = nullptr;
  if (!order.empty()) {
    LBW_CUDA(cudaMallocAsync((void**)&d_order, sizeof(int) * order.size(), stream));
    LBW_CUDA(cudaMemcpyAsync(d_order, order.data(), sizeof(int) * order.size(), cudaMemcpyHostToDevice, stream));
  }
  LBW_CUDA(cudaMemcpyAsync(r->items, items.data(), sizeof(ResItem) * items.size(), cudaMemcpyHostToDevice, stream));
  if (r->src_order) cudaFreeAsync(r->src_order, stream);
  r->src_order = d_order;
  r->most = 0;
  for (const ResItem& it : items) r->most = std::max(r->most, it.src_hi - it.src_lo);
  r->host_items.swap(items);
  return LBW_OK;  // pageable copies have left the host arrays; callers synchronise
}

// Up to kFewSources sources in a box never decide.  Beyond, ns a step as measured: a node of the largest
// box and a source of the fullest here (kind 0, 1), a node of all lattices where a step is a launch
// (tile kernels, others); FP32 with four planes of P sources here / launched: 64 x 128 x 70 31 / 19 us, 64 x 64
// x 100 20 / 15; with one plane 17 / 18, 12 / 15.
bool resident_pays(const Resident* r, int src_kind) {
  constexpr int kFewSources = 256;
  if (r->most <= kFewSources) return true;
  struct Cost {
    double node, source[2], launched[2];
  };
  const Cost c = r->prec == LBW_F64   ? Cost{10.2, {9.2, 7.0}, {0.12, 0.19}}
                 : r->prec == LBW_F32 ? Cost{3.3, {8.5, 14.5}, {0.010, 0.030}}
                                      : Cost{3.5, {25.0, 31.0}, {0.008, 0.050}};
  double here = r->most * c.source[src_kind != 0];
  for (const Resident::Launch& L : r->launches) here += 2000.0 + L.own * c.node;
  return here < 10500.0 + r->nodes * c.launched[r->tile ? 0 : 1];
}

cudaError_t resident_run(const Resident* r, const Grid* one, const void* members, const ResState& st, int steps) {
  for (size_t l = 0; l < r->launches.size(); ++l) {
    const cudaError_t e = with_prec(r->prec, [&](auto tag) {
      using S = decltype(tag);
      if (one) {
        const StepArgs<S> a = step_args<S>(*one, 0);
        return launch_t<S>(r, r->launches[l], &a, nullptr, st, steps, l + 1 == r->launches.size());
      }
      return launch_t<S>(r, r->launches[l], nullptr, members, st, steps, l + 1 == r->launches.size());
    });
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace lbw
