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
// Read-out.  The values go through the population buffer that the next step overwrites, so no
// device memory is allocated; whether they are finite is decided where they are computed (a host
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

// Scratch of one initialisation: cos and sin along q2 (u2 and nothing for Cartesian lattices), per
// q3 the flare (or cos u3), u3 (or sin u3), one byte per row: some pulse reaches it.
struct InitScratch {
  double *c2, *s2, *a3, *b3;
  unsigned char* near;
};

__host__ __device__ inline InitScratch carve_init(void* base, int n1, int n2, int n3) {
  InitScratch s;
  s.c2 = static_cast<double*>(base);
  s.s2 = s.c2 + n2;
  s.a3 = s.s2 + n2;
  s.b3 = s.a3 + n3;
  s.near = reinterpret_cast<unsigned char*>(s.b3 + n3);
  (void)n1;
  return s;
}

__global__ void axis_kernel(const InitGeom G, InitScratch t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < G.n2) {
    const double u2 = G.x0[1] + (i + 0.5) * G.h[1];
    if (G.kind == LBW_CARTESIAN) t.c2[i] = u2;
    else sincos(u2, &t.s2[i], &t.c2[i]);
  } else if (i < G.n2 + G.n3) {
    const int q3 = i - G.n2;
    const double u3 = G.x0[2] + (q3 + 0.5) * G.h[2];
    double a = 1.0, b = u3;
    if (G.kind == LBW_TRUMPET) {
      if (G.profile == 0) a = pow(G.geom[0] - u3, -G.geom[1]);
      else a = (G.geom[0] + G.geom[1] * exp(G.geom[2] * u3)) / (G.geom[0] + G.geom[1]);
    } else if (G.kind == LBW_TOROIDAL) {
      sincos(u3, &b, &a);
    }
    t.a3[q3] = a;
    t.b3[q3] = b;
  }
}

// rho0 = sqrt(g) P0, P0 a sum of Gaussian pulses in the embedding distance (FP64 math), on the rows
// that a pulse reaches.  One warp per row.
template <typename R>
__global__ void init_rho_kernel(const InitGeom G, const InitScratch t, const Pulse* __restrict__ pulses, int npulse,
                                const R* __restrict__ tab, R* __restrict__ rho0) {
  const int lane = threadIdx.x & 31;
  const long long rows = (long long)G.n1 * G.n3, warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long row = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); row < rows; row += warps) {
    const int q3 = (int)(row / G.n1), q1 = (int)(row - (long long)q3 * G.n1);
    const double u1 = G.x0[0] + (q1 + 0.5) * G.h[0];
    const bool flat = G.kind == LBW_CARTESIAN;
    // the row's nodes sit at (a c2, a s2, z), or (u1, u2, u3) on a Cartesian lattice
    double a = u1, z = t.b3[q3];
    if (G.kind == LBW_TRUMPET) a = u1 * t.a3[q3];
    if (G.kind == LBW_TOROIDAL) {
      a = G.geom[0] + u1 * t.a3[q3];
      z = u1 * t.b3[q3];
    }
    auto reach = [&](int first) -> unsigned {  // which of the pulses first .. first + 31 reach the row
      bool near = false;
      if (first + lane < npulse) {
        const Pulse& p = pulses[first + lane];
        const double da = flat ? a - p.x[0] : fabs(a) - p.axis, dz = z - p.x[2];
        near = !(da * da + dz * dz > p.cut);
      }
      return __ballot_sync(0xffffffffu, near);
    };
    bool any = false;
    for (int first = 0; first < npulse && !any; first += 32) any = reach(first) != 0;
    if (lane == 0) t.near[row] = any;
    if (!any) continue;
    const double sg = (double)tab[row * T_SLOTS + T_SG];
    for (int base = 0; base < G.n2; base += 32) {
      const int q2 = base + lane;
      const bool in = q2 < G.n2;
      const double c2 = in ? t.c2[q2] : 0.0, s2 = in && !flat ? t.s2[q2] : 0.0;
      const double X0 = flat ? a : a * c2, X1 = flat ? c2 : a * s2;
      double P0 = 0.0;
      for (int first = 0; first < npulse; first += 32)
        for (unsigned left = reach(first); left; left &= left - 1) {
          const Pulse& p = pulses[first + __ffs(left) - 1];
          const double d2 = (X0 - p.x[0]) * (X0 - p.x[0]) + (X1 - p.x[1]) * (X1 - p.x[1]) + (z - p.x[2]) * (z - p.x[2]);
          if (d2 > p.cut) continue;
          const double e = d2 / (2.0 * p.sigma * p.sigma);
          if (e < 80.0) P0 += p.amp * exp(-e);  // beyond: below 2e-35 of the amplitude
        }
      if (in) rho0[row * G.n2 + q2] = (R)(sg * P0);
    }
  }
}

// Post-collision state at rest on the rows that a pulse reaches and their neighbours (elsewhere it
// is zero): f*_i = f_i^eq(rho0, F(rho0) / 2), F from the same table.  One warp per row.
template <typename S>
__global__ void init_f_kernel(const StepArgs<S> a, const unsigned char* __restrict__ near,
                              const typename Store<S>::R* __restrict__ rho0) {
  using R = typename Store<S>::R;
  const bool p1 = a.bc[0] == LBW_BC_PERIODIC, p2 = a.bc[2] == LBW_BC_PERIODIC, p3 = a.bc[4] == LBW_BC_PERIODIC;
  const int lane = threadIdx.x & 31, n1 = a.n1, n2 = a.n2;
  const long long rows = (long long)n1 * a.n3, warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long row = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); row < rows; row += warps) {
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
    if (!Lc && !Lu && !Ld && !Ln && !Lp) continue;
    auto at = [](const R* l, int q2) -> R { return l ? l[q2] : R(0); };
    const R* c = a.tab + row * T_SLOTS;
    for (int q2 = lane; q2 < n2; q2 += 32) {
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
  const InitScratch t = carve_init(d_scratch, G.n1, G.n2, G.n3);
  // rho0 goes to the scratch bytes of the other population buffer (>= N values of R)
  R* rho0 = reinterpret_cast<R*>(g->f[1 - g->cur]);
  cudaError_t e = cudaMemsetAsync(g->f[g->cur], 0, (size_t)7 * pop_stride(g) * g->elem, g->stream);
  if (e != cudaSuccess || npulse == 0) return e;
  const long long rows = (long long)G.n1 * G.n3;
  const int blocks = (int)std::min<long long>((rows + 7) / 8, 152LL * 16);
  axis_kernel<<<(G.n2 + G.n3 + 127) / 128, 128, 0, g->stream>>>(G, t);
  init_rho_kernel<R><<<blocks, 256, 0, g->stream>>>(G, t, static_cast<const Pulse*>(d_pulses), npulse,
                                                    reinterpret_cast<const R*>(g->table), rho0);
  StepArgs<S> a = step_args<S>(*g, 1 - g->cur);  // fout = current buffer
  init_f_kernel<S><<<blocks, 256, 0, g->stream>>>(a, t.near, rho0);
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

// populations per turn through the other buffer: as many planes of doubles as it holds
int planes_per_turn(const Grid* g) {
  return (int)std::max<long long>(1, std::min<long long>(7, 7 * pop_stride(g) * (long long)g->elem / (8 * g->nn)));
}

}  // namespace

size_t init_scratch_bytes(const lbw_grid_desc& d) {
  return sizeof(double) * 2 * ((size_t)d.n[1] + d.n[2]) + (size_t)d.n[0] * d.n[2];
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
  cudaError_t e = cudaMemsetAsync(d_bad, 0, sizeof(*d_bad), g->stream);
  if (e == cudaSuccess)
    e = with_types(g, [&](auto tag, auto index) {
      using S = decltype(tag);
      using I = decltype(index);
      field_kernel<S, I><<<kReadBlocks, kReadThreads, 0, g->stream>>>(
          static_cast<const S*>(g->f[g->cur]), (I)g->nn, pop_stride(g), pad_of<I>(g),
          static_cast<const typename Store<S>::R*>(g->table), g->w0, g->w1, d, d_bad);
      return cudaGetLastError();
    });
  if (e != cudaSuccess) return e;
  touch_pages(host_P, sizeof(double) * g->nn);
  return cudaMemcpyAsync(host_P, d, sizeof(double) * g->nn, cudaMemcpyDeviceToHost, g->stream);
}

cudaError_t read_populations(Grid* g, double* host_f) {
  double* d = static_cast<double*>(g->f[1 - g->cur]);
  const int per = planes_per_turn(g);
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 7 && e == cudaSuccess; i += per) {
    const int n = std::min(per, 7 - i);
    e = with_types(g, [&](auto tag, auto index) {
      using S = decltype(tag);
      using I = decltype(index);
      to_double_kernel<S, I><<<dim3(kReadBlocks, n), kReadThreads, 0, g->stream>>>(
          static_cast<const S*>(g->f[g->cur]), i, (I)g->nn, pop_stride(g), pad_of<I>(g), g->w0, g->w1, d);
      return cudaGetLastError();
    });
    if (i == 0) touch_pages(host_f, sizeof(double) * 7 * g->nn);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(host_f + (size_t)i * g->nn, d, sizeof(double) * n * g->nn, cudaMemcpyDeviceToHost, g->stream);
  }
  return e;
}

cudaError_t write_populations(Grid* g, const double* host_f) {
  double* d = static_cast<double*>(g->f[1 - g->cur]);
  const int per = planes_per_turn(g);
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 7 && e == cudaSuccess; i += per) {
    const int n = std::min(per, 7 - i);
    e = cudaMemcpyAsync(d, host_f + (size_t)i * g->nn, sizeof(double) * n * g->nn, cudaMemcpyHostToDevice, g->stream);
    if (e != cudaSuccess) break;
    e = with_types(g, [&](auto tag, auto index) {
      using S = decltype(tag);
      using I = decltype(index);
      from_double_kernel<S, I><<<dim3(kReadBlocks, n), kReadThreads, 0, g->stream>>>(
          d, i, (I)g->nn, pop_stride(g), pad_of<I>(g), g->d.bc[2] == LBW_BC_PERIODIC, g->w0, g->w1,
          static_cast<S*>(g->f[g->cur]));
      return cudaGetLastError();
    });
  }
  return e;
}

}  // namespace lbw
