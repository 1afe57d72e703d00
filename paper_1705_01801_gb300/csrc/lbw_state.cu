// lbw_state.cu -- initial state and read-out: everything that touches the whole state outside the
// time steps.
//
// Initial state.  A Gaussian pulse is below 2e-35 of its amplitude beyond e = 80, 12.6 sigma away,
// so most (q1, q3) rows of a lattice see no pulse at all.  A row's nodes share their distance from
// the axis and their height (X = (a cos, a sin, z) for every kind but the Cartesian one), which
// gives the nearest a pulse can come to the row: rows that none reaches keep the zeros of one
// memset, the others evaluate the embedding from tables of the trigonometric functions along q2
// and q3.  FP64 (2 operations a cycle and SM) bounded the former pass, which took sincos and
// every pulse's distance at every node: torus 192 x 1024 x 256 8.3 -> 0.45 ms, 48 trumpets with
// twelve pulses each 33 -> 8.5 ms.
//
// Read-out.  The values go through the population buffer that the next step overwrites, so large
// lattices need no device memory for it; whether they are finite is decided where they are computed (a host
// loop over the field took 23 of the 39 ms of the torus's snapshot, first touches of the caller's
// array 13; now 6 ms).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <unistd.h>

#include <algorithm>
#include <cmath>
#include <thread>
#include <vector>

#include "lbw_internal.h"
#include "lbw_march.cuh"

namespace lbw {
namespace {

using namespace dev;

template <typename F>
cudaError_t dispatch(int prec, F&& fn) {
  switch (prec) {
    case LBW_F64: return fn(double());
    case LBW_F32: return fn(float());
    case LBW_F16S: return fn(__half());
    default: return fn(__nv_bfloat16());
  }
}

// ---------------------------------------------------------------- initial state ----------

struct InitGeom {
  int kind, profile, n1, n2, n3;
  double h[3], x0[3], geom[4];
};

// A pulse on the device: centre, sigma, amplitude, the centre's distance from the z axis and the
// squared distance beyond which it is left out, with a margin for the rows' test.
struct Pulse {
  double x[3], sigma, amp, axis, cut;
};

// Scratch of one initialisation: cos and sin along q2 (unused on Cartesian lattices), per q3
// the flare (or cos u3), u3 (or sin u3), one byte per row: some pulse reaches it.
struct InitScratch {
  double *c2, *s2, *a3, *b3;
  unsigned char* near;
};

inline InitScratch carve_init(void* base, int n2, int n3) {
  InitScratch s;
  s.c2 = static_cast<double*>(base);
  s.s2 = s.c2 + n2;
  s.a3 = s.s2 + n2;
  s.b3 = s.a3 + n3;
  s.near = reinterpret_cast<unsigned char*>(s.b3 + n3);
  return s;
}
size_t scratch_bytes(const lbw_grid_desc& d) {
  return sizeof(double) * 2 * ((size_t)d.n[1] + d.n[2]) + (size_t)d.n[0] * d.n[2];
}
size_t scratch_offset(const Grid& g) { return ((size_t)g.nn * (g.elem == 8 ? 8 : 4) + 15) / 16 * 16; }

// Position of row q3's nodes along the axis: the flare (or cos u3), and u3 (or sin u3).
__device__ __forceinline__ void plane_terms(const InitGeom& G, int q3, double& a, double& b) {
  const double u3 = G.x0[2] + (q3 + 0.5) * G.h[2];
  a = 1.0;
  b = u3;
  if (G.kind == LBW_TRUMPET) {
    if (G.profile == 0) a = pow(G.geom[0] - u3, -G.geom[1]);
    else a = (G.geom[0] + G.geom[1] * exp(G.geom[2] * u3)) / (G.geom[0] + G.geom[1]);
  } else if (G.kind == LBW_TOROIDAL) {
    sincos(u3, &b, &a);
  }
}

__device__ __forceinline__ void column_terms(const InitGeom& G, int q2, double& c, double& s) {
  const double u2 = G.x0[1] + (q2 + 0.5) * G.h[1];
  s = 0.0;
  c = u2;
  if (G.kind != LBW_CARTESIAN) sincos(u2, &s, &c);
}

__global__ void axis_kernel(const InitGeom G, InitScratch t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < G.n2) {
    if (G.kind != LBW_CARTESIAN) column_terms(G, i, t.c2[i], t.s2[i]);
  } else if (i < G.n2 + G.n3) {
    plane_terms(G, i - G.n2, t.a3[i - G.n2], t.b3[i - G.n2]);
  }
}

// What a warp takes at a time: `rows` whole rows of up to 16 nodes side by side in its lanes, or
// `cols` columns (a multiple of 32) of one row.  Whole rows repeat the test of the pulses least
// often, but a lattice of few rows needs their parts to fill the SMs: with a warp per row,
// one of 1,048,576 nodes took 43 ms, 4 x 4 of 65,536 4.0, and 300,000 of three nodes 0.33; now
// 121, 111 and 87 us (a thread per node that tests every pulse: 151, 146, 137).
struct InitUnits {
  int rows, cols, parts;
  long long count;
};

InitUnits init_units(int n1, int n2, int n3) {
  InitUnits u;
  const long long rows = (long long)n1 * n3, warps = 152LL * 64;
  u.rows = n2 <= 16 ? 32 / n2 : 1;
  u.parts = u.rows > 1 ? 1 : (int)std::max(1LL, std::min<long long>((n2 + 31) / 32, warps / rows));
  u.cols = (n2 + 32 * u.parts - 1) / (32 * u.parts) * 32;
  u.parts = (n2 + u.cols - 1) / u.cols;
  u.count = (rows + u.rows - 1) / u.rows * u.parts;
  return u;
}

// A lane's place in a unit: its row (of `rows` from `first` on) and its columns c0, c0 + 32, ... below c1.
struct InitLane {
  long long first, row;
  int rows, sub, c0, c1;
  __device__ InitLane(const InitUnits& U, long long unit, long long all_rows, int n2) {
    const int lane = threadIdx.x & 31, part = (int)(unit % U.parts);
    first = unit / U.parts * U.rows;
    rows = (int)min((long long)U.rows, all_rows - first);
    sub = U.rows > 1 ? lane / n2 : 0;
    const bool in = sub < rows;  // lanes past the unit's last row repeat its first and store nothing
    if (!in) sub = 0;
    row = first + sub;
    c0 = U.rows > 1 ? (in ? lane % n2 : n2) : part * U.cols + lane;
    c1 = U.rows > 1 ? n2 : min(n2, (part + 1) * U.cols);
  }
};

// Adds a pulse's value at (X0, X1, z) to P0.
__device__ __forceinline__ void add_pulse(const Pulse& p, double X0, double X1, double z, double& P0) {
  const double d2 = (X0 - p.x[0]) * (X0 - p.x[0]) + (X1 - p.x[1]) * (X1 - p.x[1]) + (z - p.x[2]) * (z - p.x[2]);
  if (d2 > p.cut) return;
  const double e = d2 / (2.0 * p.sigma * p.sigma);
  if (e < 80.0) P0 += p.amp * exp(-e);  // beyond: below 2e-35 of the amplitude
}

// rho0 = sqrt(g) P0, P0 a sum of Gaussian pulses in the embedding distance (FP64 math), on the rows
// that a pulse reaches.
template <typename R>
__global__ void init_rho_kernel(const InitGeom G, const InitScratch t, const InitUnits U,
                                const Pulse* __restrict__ pulses, int npulse, const R* __restrict__ tab,
                                R* __restrict__ rho0) {
  const int lane = threadIdx.x & 31, n2 = G.n2;
  const long long all_rows = (long long)G.n1 * G.n3, warps = (long long)gridDim.x * (blockDim.x >> 5);
  const bool flat = G.kind == LBW_CARTESIAN;
  for (long long unit = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); unit < U.count; unit += warps) {
    const InitLane L(U, unit, all_rows, n2);
    const int q3 = (int)(L.row / G.n1), q1 = (int)(L.row - (long long)q3 * G.n1);
    const double u1 = G.x0[0] + (q1 + 0.5) * G.h[0];
    // the row's nodes sit at (a c2, a s2, z), or (u1, u2, u3) on a Cartesian lattice
    double a = u1, z = t.b3[q3];
    if (G.kind == LBW_TRUMPET) a = u1 * t.a3[q3];
    if (G.kind == LBW_TOROIDAL) {
      a = G.geom[0] + u1 * t.a3[q3];
      z = u1 * t.b3[q3];
    }
    auto reaches = [&](const Pulse& p, double as, double zs) -> bool {
      const double da = flat ? as - p.x[0] : fabs(as) - p.axis, dz = zs - p.x[2];
      return !(da * da + dz * dz > p.cut);
    };
    // which of the pulses first .. first + 31 reach row s of the unit (a lane per pulse)
    auto reach = [&](int first, int s) -> unsigned {
      const double as = __shfl_sync(0xffffffffu, a, s * n2 & 31), zs = __shfl_sync(0xffffffffu, z, s * n2 & 31);
      return __ballot_sync(0xffffffffu, first + lane < npulse && reaches(pulses[min(first + lane, npulse - 1)], as, zs));
    };
    // fewer pulses than rows: every lane tests its own row instead
    const bool few = npulse < L.rows;
    unsigned hit = 0;  // the rows that some pulse reaches
    bool any = false;
    if (few) {
      for (int k = 0; k < npulse; ++k) any |= reaches(pulses[k], a, z);
      hit = __ballot_sync(0xffffffffu, any);
    } else {
      for (int s = 0; s < L.rows; ++s)
        for (int first = 0; first < npulse && !(hit >> s & 1); first += 32)
          if (reach(first, s)) hit |= 1u << s;
      any = hit >> L.sub & 1;
    }
    if (L.c0 == 0) t.near[L.row] = any;
    if (!hit) continue;
    const double sg = (double)tab[L.row * T_SLOTS + T_SG];
    const int steps = U.rows > 1 ? 1 : (L.c1 - (L.c0 - lane) + 31) / 32;  // the same for every lane
    for (int k = 0, q2 = L.c0; k < steps; ++k, q2 += 32) {
      const bool in = q2 < L.c1 && any;
      double c2 = 0.0, s2 = 0.0;
      if (in) {
        c2 = flat ? G.x0[1] + (q2 + 0.5) * G.h[1] : t.c2[q2];
        s2 = flat ? 0.0 : t.s2[q2];
      }
      const double X0 = flat ? a : a * c2, X1 = flat ? c2 : a * s2;
      double P0 = 0.0;
      if (few) {
        if (in)
          for (int j = 0; j < npulse; ++j) add_pulse(pulses[j], X0, X1, z, P0);
      } else {
        for (int first = 0; first < npulse; first += 32) {
          unsigned left = 0;
          for (int s = 0; s < L.rows; ++s) left |= reach(first, s);
          for (; left; left &= left - 1) add_pulse(pulses[first + __ffs(left) - 1], X0, X1, z, P0);
        }
      }
      if (in) rho0[L.row * n2 + q2] = (R)(sg * P0);
    }
  }
}

// The same for small lattices and few pulses: a thread per node tests every pulse and evaluates the
// terms of its axes itself, which costs less than the launch that tabulates them and the tests of the
// rows (3000 members of 512 nodes, a launch each: 54 -> 40 ms).
template <typename R>
__global__ void init_rho_small_kernel(const InitGeom G, unsigned char* __restrict__ near,
                                      const Pulse* __restrict__ pulses, int npulse, const R* __restrict__ tab,
                                      R* __restrict__ rho0) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, row = x / G.n2, q2 = x - row * G.n2;
  if (row >= G.n1 * G.n3) return;
  const int q3 = row / G.n1, q1 = row - q3 * G.n1;
  const double u1 = G.x0[0] + (q1 + 0.5) * G.h[0];
  double a3, z, c2, s2, a = u1;
  plane_terms(G, q3, a3, z);
  column_terms(G, q2, c2, s2);
  if (G.kind == LBW_TRUMPET) a = u1 * a3;
  if (G.kind == LBW_TOROIDAL) {
    a = G.geom[0] + u1 * a3;
    z = u1 * z;
  }
  const bool flat = G.kind == LBW_CARTESIAN;
  const double X0 = flat ? a : a * c2, X1 = flat ? c2 : a * s2;
  double P0 = 0.0;
  for (int k = 0; k < npulse; ++k) add_pulse(pulses[k], X0, X1, z, P0);
  rho0[x] = (R)((double)tab[(long long)row * T_SLOTS + T_SG] * P0);
  if (q2 == 0) near[row] = 1;
}

// Post-collision state at rest, f*_i = f_i^eq(rho0, F(rho0) / 2) with F from the same table, on the
// rows that a pulse reaches and their neighbours; the others are zero (`all`: written here).
template <typename S>
__global__ void init_f_kernel(const StepArgs<S> a, const unsigned char* __restrict__ near, const InitUnits U, bool all,
                              const typename Store<S>::R* __restrict__ rho0) {
  using R = typename Store<S>::R;
  const bool p1 = a.bc[0] == LBW_BC_PERIODIC, p2 = a.bc[2] == LBW_BC_PERIODIC, p3 = a.bc[4] == LBW_BC_PERIODIC;
  const int n1 = a.n1, n2 = a.n2;
  const long long all_rows = (long long)n1 * a.n3, warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long unit = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); unit < U.count; unit += warps) {
    const InitLane lane(U, unit, all_rows, n2);
    const long long row = lane.row;
    const int q3 = (int)(row / n1), q1 = (int)(row - (long long)q3 * n1);
    // rho0 of a row, or nullptr where it is zero (or a ghost)
    auto line = [&](int r1, int r3) -> const R* {
      r1 = resolve(r1, n1, p1);
      r3 = resolve(r3, a.n3, p3);
      if (r1 < 0 || r3 < 0) return nullptr;
      const long long r = (long long)r3 * n1 + r1;
      return near[r] ? rho0 + r * n2 : nullptr;
    };
    const R *Lc = line(q1, q3), *Lu = line(q1 + 1, q3), *Ld = line(q1 - 1, q3), *Ln = line(q1, q3 + 1), *Lp = line(q1, q3 - 1);
    if (!all && !Lc && !Lu && !Ld && !Ln && !Lp) continue;
    auto at = [](const R* l, int q2) -> R { return l ? l[q2] : R(0); };
    const R* c = a.tab + row * T_SLOTS;
    for (int q2 = lane.c0; q2 < lane.c1; q2 += 32) {
      const R rho = at(Lc, q2), ru = at(Lu, q2), rd = at(Ld, q2), rn = at(Ln, q2), rp = at(Lp, q2);
      const int ql = q2 == 0 ? n2 - 1 : q2 - 1, qr = q2 == n2 - 1 ? 0 : q2 + 1;
      R rr = at(Lc, qr), rl = at(Lc, ql);
      if (q2 == 0 && !p2) rl = a.s2lo * rho;
      if (q2 == n2 - 1 && !p2) rr = a.s2hi * rho;
      const R D1 = c[T_A1P] * ru - c[T_A1M] * rd + c[T_C13P] * rn - c[T_C13M] * rp + c[T_S1] * rho;
      const R D3 = c[T_B13P] * ru - c[T_B13M] * rd + c[T_C33P] * rn - c[T_C33M] * rp + c[T_S3] * rho;
      const R D2 = c[T_H22] * (rr - rl);
      const R j1 = R(0.5) * (c[T_MG1] * rho - D1), j2 = R(-0.5) * D2,
              j3 = R(0.5) * (c[T_MG3] * rho - D3);
      const R e = R(0.5) * a.cs2 * rho;
      R o[7] = {R(0.5) * a.two_w0 * rho, e + R(0.5) * j1, e - R(0.5) * j1, e + R(0.5) * j2,
                e - R(0.5) * j2, e + R(0.5) * j3, e - R(0.5) * j3};
      const long long px = row * a.pitch + a.col0 + q2;
      // ghost copy of a node near the periodic wrap (padded storage only)
      int gq = -1;
      if (a.col0 > 0 && p2) gq = q2 < a.col0 ? a.col0 + n2 + q2 : (q2 >= n2 - a.col0 ? q2 - n2 + a.col0 : -1);
#pragma unroll
      for (int i = 0; i < 7; ++i) {
        R v = o[i];
        if (Store<S>::kScaled) v *= a.inv_w[i];
        Store<S>::st(a.fout + (long long)i * a.ps + px, v);
        if (gq >= 0) Store<S>::st(a.fout + (long long)i * a.ps + (px - a.col0 - q2) + gq, v);
      }
    }
  }
}

// Lattices of up to kInitAll nodes have every node written by the last kernel instead of a memset
// before it; those of up to kInitSmall with at most kInitFew pulses take the kernel for them.
constexpr long long kInitAll = 1 << 20, kInitSmall = 1 << 16;
constexpr int kInitFew = 16;

template <typename S>
cudaError_t launch_init_t(Grid* g, const void* d_pulses, int npulse, void* d_scratch) {
  using R = typename Store<S>::R;
  InitGeom G;
  G.kind = g->d.kind;
  G.profile = g->d.horn_profile;
  G.n1 = g->d.n[0];
  G.n2 = g->d.n[1];
  G.n3 = g->d.n[2];
  for (int a = 0; a < 3; ++a) { G.h[a] = g->d.h[a]; G.x0[a] = g->d.x0[a]; }
  for (int k = 0; k < 4; ++k) G.geom[k] = g->d.geom[k];
  // rho0 goes to the other population buffer (>= N values of R), and the scratch behind it where it fits
  R* rho0 = reinterpret_cast<R*>(g->f[1 - g->cur]);
  if (init_scratch_bytes(*g) == 0) d_scratch = static_cast<unsigned char*>(g->f[1 - g->cur]) + scratch_offset(*g);
  const InitScratch t = carve_init(d_scratch, G.n2, G.n3);
  const bool all = g->nn <= kInitAll && npulse > 0;
  cudaError_t e = cudaSuccess;
  if (!all) e = cudaMemsetAsync(g->f[g->cur], 0, (size_t)7 * pop_stride(g) * g->elem, g->stream);
  if (e != cudaSuccess || npulse == 0) return e;
  const InitUnits U = init_units(G.n1, G.n2, G.n3);
  const int warps = U.count < 152 * 16 ? 2 : 8;  // per block: few units spread over the SMs
  const int blocks = (int)std::min<long long>((U.count + warps - 1) / warps, 152LL * 16);
  const Pulse* pulses = static_cast<const Pulse*>(d_pulses);
  const R* tab = reinterpret_cast<const R*>(g->table);
  if (g->nn <= kInitSmall && npulse <= kInitFew) {
    init_rho_small_kernel<R><<<(int)(g->nn + 127) / 128, 128, 0, g->stream>>>(G, t.near, pulses, npulse, tab, rho0);
  } else {
    axis_kernel<<<(G.n2 + G.n3 + 127) / 128, 128, 0, g->stream>>>(G, t);
    init_rho_kernel<R><<<blocks, 32 * warps, 0, g->stream>>>(G, t, U, pulses, npulse, tab, rho0);
  }
  StepArgs<S> a = step_args<S>(*g, 1 - g->cur);  // fout = current buffer
  init_f_kernel<S><<<blocks, 32 * warps, 0, g->stream>>>(a, t.near, U, all, rho0);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- read-out ---------------

// Storage address of dense node x (q2 fastest) in a possibly padded layout; I: an index type that
// holds every node.
template <typename I>
struct Pad {
  I n2, pitch, col0;
  __device__ long long at(I x) const {
    if (pitch == n2) return x;
    const I row = x / n2;
    return (long long)row * pitch + col0 + (x - row * n2);
  }
};

// P = rho / sqrt(g); *bad becomes 1 when a value is not finite
template <typename S, typename I>
__global__ void field_kernel(const S* __restrict__ f, I nn, long long ps, Pad<I> pad,
                             const typename Store<S>::R* __restrict__ tab, double w0, double w1,
                             double* __restrict__ P, unsigned long long* bad) {
  bool ok = true;
  for (I x = blockIdx.x * (I)blockDim.x + threadIdx.x; x < nn; x += (I)gridDim.x * blockDim.x) {
    const I row = x / pad.n2;
    const long long px = (long long)row * pad.pitch + pad.col0 + (x - row * pad.n2);
    double r = 0.0;
    for (int i = 0; i < 7; ++i) {
      double v = (double)Store<S>::ld(f + (long long)i * ps + px);
      if (Store<S>::kScaled) v *= (i == 0 ? w0 : w1);
      r += v;
    }
    const double p = r * (double)tab[(long long)row * T_SLOTS + T_INVSG];
    ok &= isfinite(p);
    P[x] = p;
  }
  if (!ok) *bad = 1;
}

// populations i0 .. i0 + gridDim.y - 1 as doubles
template <typename S, typename I>
__global__ void to_double_kernel(const S* __restrict__ f, int i0, I nn, long long ps, Pad<I> pad, double w0, double w1,
                                 double* __restrict__ out) {
  const int i = i0 + blockIdx.y;
  f += i * ps;
  out += (long long)blockIdx.y * nn;
  for (I x = blockIdx.x * (I)blockDim.x + threadIdx.x; x < nn; x += (I)gridDim.x * blockDim.x) {
    double v = (double)Store<S>::ld(f + pad.at(x));
    if (Store<S>::kScaled) v *= (i == 0 ? w0 : w1);
    out[x] = v;
  }
}

// Dense doubles into storage; padded storage also gets the ghost copies of a periodic q2.
template <typename S, typename I>
__global__ void from_double_kernel(const double* __restrict__ in, int i0, I nn, long long ps, Pad<I> pad, bool p2,
                                   double w0, double w1, S* __restrict__ f) {
  const int i = i0 + blockIdx.y;
  f += i * ps;
  in += (long long)blockIdx.y * nn;
  for (I x = blockIdx.x * (I)blockDim.x + threadIdx.x; x < nn; x += (I)gridDim.x * blockDim.x) {
    double v = in[x];
    if (Store<S>::kScaled) v /= (i == 0 ? w0 : w1);
    const long long px = pad.at(x);
    const typename Store<S>::R r = (typename Store<S>::R)v;
    Store<S>::st(f + px, r);
    if (pad.col0 > 0 && p2) {
      const I q2 = x % pad.n2;
      const long long row = px - (long long)pad.col0 - (long long)q2;
      if (q2 < pad.col0) Store<S>::st(f + row + pad.col0 + pad.n2 + q2, r);
      if (q2 >= pad.n2 - pad.col0) Store<S>::st(f + row + q2 - pad.n2 + pad.col0, r);
    }
  }
}

// f(element tag, index tag) for a lattice: 32-bit indices where they hold every node
template <typename F>
cudaError_t with_types(const Grid* g, F&& f) {
  return dispatch(g->d.prec, [&](auto tag) {
    return g->nn < (1LL << 30) ? f(tag, unsigned()) : f(tag, (unsigned long long)0);
  });
}

template <typename I>
Pad<I> pad_of(const Grid* g) {
  return Pad<I>{(I)g->d.n[1], (I)(g->pitch ? g->pitch : g->d.n[1]), (I)g->col0};
}

constexpr int kReadThreads = 256, kReadBlocks = 152 * 8;

unsigned read_blocks(const Grid* g) {
  return (unsigned)std::min<long long>((g->nn + kReadThreads - 1) / kReadThreads, kReadBlocks);
}

// Room for `per` planes of doubles on the device: the other population buffer, which holds 1 to 7, or
// a temporary of all seven (up to `limit` bytes, where it can be had), as every turn costs a launch and
// a copy of its own and a large temporary is slow to map.  FP32, through the buffer / a temporary: read
// 64 nodes 68 / 31 us, 262,144 488 / 375, 512,000 930 / 815, 1e6 2320 / 2560; written 28 / 19, 133 / 115,
// 210 / 305, 390 / 545.
struct Planes {
  Grid* g;
  double* d;
  int per;
  bool own = false;
  Planes(Grid* grid, long long limit) : g(grid), d(static_cast<double*>(grid->f[1 - grid->cur])) {
    const long long all = 7LL * 8 * g->nn;
    per = (int)std::max<long long>(1, std::min<long long>(7, 7 * pop_stride(g) * (long long)g->elem / (8 * g->nn)));
    void* t = nullptr;
    if (per == 7 || all > limit) return;
    if (cudaMallocAsync(&t, (size_t)all, g->stream) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    d = static_cast<double*>(t);
    per = 7;
    own = true;
  }
  ~Planes() {
    if (own) cudaFreeAsync(d, g->stream);
  }
};

}  // namespace

size_t init_scratch_bytes(const Grid& g) {
  return scratch_offset(g) + scratch_bytes(g.d) <= (size_t)7 * pop_stride(&g) * g.elem ? 0 : scratch_bytes(g.d);
}

size_t pulse_bytes(int n) { return sizeof(Pulse) * std::max(1, n); }

void pack_pulses(const lbw_pulse* p, int n, void* out) {
  Pulse* q = static_cast<Pulse*>(out);
  for (int k = 0; k < n; ++k) {
    for (int a = 0; a < 3; ++a) q[k].x[a] = p[k].x[a];
    q[k].sigma = p[k].sigma;
    q[k].amp = p[k].amp;
    q[k].axis = std::sqrt(p[k].x[0] * p[k].x[0] + p[k].x[1] * p[k].x[1]);
    // distances round to some 1e-16 of the coordinates: leave a wide margin around e = 80
    const double r = 13.0 * p[k].sigma + 1e-9 * (q[k].axis + std::fabs(p[k].x[2]));
    q[k].cut = r * r;
  }
}

cudaError_t launch_init(Grid* g, const void* d_pulses, int npulse, void* d_scratch) {
  return dispatch(g->d.prec, [&](auto tag) { return launch_init_t<decltype(tag)>(g, d_pulses, npulse, d_scratch); });
}

// First touches of a large host array by several threads: the kernel maps its pages an order
// faster than the copy that would otherwise take the faults one after the other (403 MB: 13 -> 4 ms).
void touch_pages(void* p, size_t bytes) {
  const size_t page = (size_t)sysconf(_SC_PAGESIZE), least = (size_t)4 << 20;
  // smaller arrays come from pages that the allocator keeps mapped as a rule, and asking for the number
  // of cores alone takes 20 us
  if (bytes < 8 * least) return;
  const int n = (int)std::min<size_t>({bytes / least, 8, std::max(1u, std::thread::hardware_concurrency())});
  if (n < 2) return;
  std::vector<std::thread> threads;
  volatile unsigned char* b = static_cast<unsigned char*>(p);
  auto part = [=](int k) {
    for (size_t i = bytes / n * k; i < (k + 1 == n ? bytes : bytes / n * (k + 1)); i += page) b[i] = 0;
  };
  try {
    threads.reserve(n);
    for (int k = 1; k < n; ++k) threads.emplace_back(part, k);
    part(0);
  } catch (...) {  // no memory or no more threads: the copy touches the rest itself
  }
  for (std::thread& t : threads) t.join();
}

cudaError_t read_field(Grid* g, double* host_P, unsigned long long* d_bad) {
  double* d = static_cast<double*>(g->f[1 - g->cur]);  // 14 to 56 bytes per node
  const cudaError_t e = with_types(g, [&](auto tag, auto index) {
    using S = decltype(tag);
    using I = decltype(index);
    field_kernel<S, I><<<read_blocks(g), kReadThreads, 0, g->stream>>>(
        static_cast<const S*>(g->f[g->cur]), (I)g->nn, pop_stride(g), pad_of<I>(g),
        static_cast<const typename Store<S>::R*>(g->table), g->w0, g->w1, d, d_bad);
    return cudaGetLastError();
  });
  if (e != cudaSuccess) return e;
  touch_pages(host_P, sizeof(double) * g->nn);
  return cudaMemcpyAsync(host_P, d, sizeof(double) * g->nn, cudaMemcpyDeviceToHost, g->stream);
}

cudaError_t read_populations(Grid* g, double* host_f) {
  const Planes p(g, 32 << 20);
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 7 && e == cudaSuccess; i += p.per) {
    const int n = std::min(p.per, 7 - i);
    e = with_types(g, [&](auto tag, auto index) {
      using S = decltype(tag);
      using I = decltype(index);
      to_double_kernel<S, I><<<dim3(read_blocks(g), n), kReadThreads, 0, g->stream>>>(
          static_cast<const S*>(g->f[g->cur]), i, (I)g->nn, pop_stride(g), pad_of<I>(g), g->w0, g->w1, p.d);
      return cudaGetLastError();
    });
    if (i == 0) touch_pages(host_f, sizeof(double) * 7 * g->nn);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(host_f + (size_t)i * g->nn, p.d, sizeof(double) * n * g->nn, cudaMemcpyDeviceToHost, g->stream);
  }
  return e;
}

cudaError_t write_populations(Grid* g, const double* host_f) {
  const Planes p(g, 16 << 20);
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 7 && e == cudaSuccess; i += p.per) {
    const int n = std::min(p.per, 7 - i);
    e = cudaMemcpyAsync(p.d, host_f + (size_t)i * g->nn, sizeof(double) * n * g->nn, cudaMemcpyHostToDevice, g->stream);
    if (e != cudaSuccess) break;
    e = with_types(g, [&](auto tag, auto index) {
      using S = decltype(tag);
      using I = decltype(index);
      from_double_kernel<S, I><<<dim3(read_blocks(g), n), kReadThreads, 0, g->stream>>>(
          p.d, i, (I)g->nn, pop_stride(g), pad_of<I>(g), g->d.bc[2] == LBW_BC_PERIODIC, g->w0, g->w1,
          static_cast<S*>(g->f[g->cur]));
      return cudaGetLastError();
    });
  }
  return e;
}

}  // namespace lbw
