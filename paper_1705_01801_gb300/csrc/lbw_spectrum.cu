// lbw_spectrum.cu -- mode frequencies of probe series, on the device, in FP64.
//
// The paper reads normal modes off driven frequency sweeps (Sec. IV.A, Fig. Fig.Frequencies;
// Sec. IV.C, Fig. FreqTorus).  For a pulse-excited run the same modes are the peaks of the
// probe signal's spectrum, estimated here:
//   1. mean removed, Hann window w_t = 1/2 - 1/2 cos(2 pi t / (T - 1));
//   2. zero padding to M = smallest power of two >= 4 T; the real series as one complex
//      Stockham FFT of M / 2 points (even samples real, odd samples imaginary), sixteen points
//      per thread and pass;
//   3. |X_j|^2, local maxima above 1e-3 of the largest bin; the k strongest are chosen with
//      warp-shuffle arg-max reductions (ties: lower bin) and sorted by frequency;
//   4. each peak is refined by a parabola through log-power at j-1, j, j+1 and 40
//      golden-section steps on the windowed DTFT over +-1 bin.  Over that range the DTFT is a
//      power series in omega - omega_0 whose coefficients are moments of the series, so the
//      series is read once per peak and not once per evaluation.
//
// All estimates of a call (the series of lbw_spectrum_series, the members of an ensemble) run in
// the same launches, grid.y of them.  FP64 arithmetic (2 operations a cycle and SM) is what
// bounds the estimator: a radix-2 pass with a sincospi per butterfly takes 50 operations a
// point, a radix-16 pass about 20 and does the work of four; golden section on the sums takes
// 81 x 8 a sample and peak, the moments about 40, spread over all SMs instead of one CTA per peak.
// Measured, 16 host series of 20,000 samples with 8 peaks each, one after the other -> here:
// 62.2 -> 1.07 ms a call (0.86 in the kernels: moments 0.30, four FFT passes 0.17, search 0.10,
// selection 0.08, power 0.06);
// one series of 20,000: 4.1 -> 0.46 ms, of 256: 0.97 -> 0.41 ms.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "lbw_internal.h"

namespace lbw {
namespace {

constexpr double kGolden = 0.6180339887498949;
constexpr double kPi = 3.141592653589793238462643383279502884;
constexpr int kParts = 64;   // partial sums of a series' mean
constexpr int kSegs = 64;    // segments of a series in the refinement
constexpr int kSegQ = 7;     // moments about a segment's centre: |dw (t - tc)| <= pi / 256, so
                             // the first neglected term is below 1e-17 of the sum of |x|
constexpr int kMom = 18;     // moments about the series' centre: |dw (t - T / 2)| <= pi / 4

// Device arrays of the estimates of one call: estimate e's slice of each begins at e times the
// length given here.
struct Work {
  double* xw;               // T      summed, then windowed series
  double* part;             // kParts partial sums
  double2 *A, *B;           // M / 2  FFT ping-pong
  double* P;                // M / 2 + 1
  long long* cand;          // M / 4 + 1
  unsigned long long* count;  // 2: candidates, largest power (bits)
  long long* chosen;        // 64
  double2* mom;             // k x kSegs x kSegQ
  double* res;              // kRes: number of peaks, mean, 64 frequencies, 64 amplitudes
};
constexpr int kRes = 2 + 2 * 64;

// sum of the nser series (stride apart) of each estimate, and partial sums for the mean
__global__ void sum_kernel(const double* __restrict__ x, long long T, int nser, long long stride,
                           long long est_stride, Work w) {
  __shared__ double red[32];
  const double* src = x + blockIdx.y * est_stride;
  double* dst = w.xw + blockIdx.y * T;
  const long long len = (T + gridDim.x - 1) / gridDim.x, t0 = blockIdx.x * len, t1 = min(T, t0 + len);
  double s = 0.0;
  for (long long t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
    double v = 0.0;
    for (int p = 0; p < nser; ++p) v += src[(long long)p * stride + t];
    dst[t] = v;
    s += v;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += red[k];
    w.part[blockIdx.y * kParts + blockIdx.x] = v;
  }
}

// xw_t = w_t (x_t - mean) in place
__global__ void window_kernel(long long T, int parts, Work w) {
  __shared__ double mean;
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < parts; ++k) s += w.part[blockIdx.y * kParts + k];
    mean = s / (double)T;
    if (blockIdx.x == 0) w.res[blockIdx.y * kRes + 1] = mean;
  }
  __syncthreads();
  double* x = w.xw + blockIdx.y * T;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < T; t += (long long)gridDim.x * blockDim.x)
    x[t] = (0.5 - 0.5 * cospi(2.0 * (double)t / (double)(T - 1))) * (x[t] - mean);
}

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 mul_mi(double2 a) { return make_double2(a.y, -a.x); }  // a (-i)

// forward DFTs of R values in registers, natural order
template <int R> __device__ __forceinline__ void dft(double2 (&v)[R]);
template <> __device__ __forceinline__ void dft<2>(double2 (&v)[2]) {
  const double2 a = v[0];
  v[0] = cadd(a, v[1]);
  v[1] = csub(a, v[1]);
}
template <> __device__ __forceinline__ void dft<4>(double2 (&v)[4]) {
  const double2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = mul_mi(csub(v[1], v[3]));
  v[0] = cadd(a, c);
  v[1] = cadd(b, d);
  v[2] = csub(a, c);
  v[3] = csub(b, d);
}
template <> __device__ __forceinline__ void dft<8>(double2 (&v)[8]) {
  constexpr double h = 0.70710678118654752440;  // cos(pi / 4)
  double2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
  dft<4>(e);
  dft<4>(o);
  o[1] = make_double2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
  o[2] = mul_mi(o[2]);
  o[3] = make_double2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = cadd(e[k], o[k]);
    v[k + 4] = csub(e[k], o[k]);
  }
}
template <> __device__ __forceinline__ void dft<16>(double2 (&v)[16]) {
  constexpr double h = 0.70710678118654752440, c = 0.92387953251128675613, s = 0.38268343236508977173;  // pi / 8
  const double2 w[10] = {{1, 0}, {c, -s}, {h, -h}, {s, -c}, {0, -1}, {0, 0}, {-h, -h}, {0, 0}, {0, 0}, {-c, s}};
  double2 t[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    double2 u[4] = {v[a], v[a + 4], v[a + 8], v[a + 12]};
    dft<4>(u);
#pragma unroll
    for (int b = 0; b < 4; ++b) t[b][a] = a * b == 0 ? u[b] : (a * b == 4 ? mul_mi(u[b]) : cmul(u[b], w[a * b]));
  }
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    dft<4>(t[b]);
#pragma unroll
    for (int a = 0; a < 4; ++a) v[b + 4 * a] = t[b][a];
  }
}

// One Stockham pass: R sub-transforms of size ns are combined into one of R ns.  The first pass
// (FIRST, ns = 1) reads the windowed series, zero past its end.
template <int R, bool FIRST>
__global__ void __launch_bounds__(128) stockham_kernel(const double2* __restrict__ in, double2* __restrict__ out,
                                                       const double* __restrict__ xw, long long T, long long N,
                                                       long long ns) {
  const long long part = N / R;
  out += blockIdx.y * N;
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < part; j += (long long)gridDim.x * blockDim.x) {
    double2 v[R];
    if constexpr (FIRST) {
      const double* x = xw + blockIdx.y * T;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const long long t = 2 * (j + q * part);
        v[q] = make_double2(t < T ? x[t] : 0.0, t + 1 < T ? x[t + 1] : 0.0);
      }
    } else {
      const double2* src = in + blockIdx.y * N;
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = src[j + q * part];
    }
    const long long k = j & (ns - 1);
    if constexpr (!FIRST) {
      double s, c;
      sincospi(2.0 * (double)k / (double)(ns * R), &s, &c);
      double2 w[R];  // e^{-2 pi i k q / (R ns)}, powers by halving
      w[1] = make_double2(c, -s);
#pragma unroll
      for (int q = 2; q < R; ++q) w[q] = cmul(w[q / 2], w[q - q / 2]);
#pragma unroll
      for (int q = 1; q < R; ++q) v[q] = cmul(v[q], w[q]);
    }
    dft<R>(v);
    const long long d = (j - k) * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) out[d + q * ns] = v[q];
  }
}

// |X_k|^2 of the real series for k = 0 .. N from the packed transform Z (N points), two bins per
// thread: X_k = E + w O and X_{N-k} = conj(E - w O) with E = (Z_k + conj Z_{N-k}) / 2,
// O = -i (Z_k - conj Z_{N-k}) / 2, w = e^{-i pi k / N}; and the largest power past bin 0.
__global__ void power_kernel(const double2* __restrict__ Zall, long long N, Work w) {
  __shared__ double red[32];
  const double2* Z = Zall + blockIdx.y * N;
  double* P = w.P + blockIdx.y * (N + 1);
  double m = 0.0;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k <= N / 2; k += (long long)gridDim.x * blockDim.x) {
    const double2 a = Z[k], b = Z[k == 0 ? 0 : N - k];
    const double2 E = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
    const double2 O = make_double2(0.5 * (a.y + b.y), -0.5 * (a.x - b.x));
    double s, c;
    sincospi((double)k / (double)N, &s, &c);
    const double2 r = cmul(make_double2(c, -s), O);
    const double2 p = cadd(E, r), q = csub(E, r);
    const double pk = p.x * p.x + p.y * p.y, pn = q.x * q.x + q.y * q.y;
    P[k] = pk;
    P[N - k] = pn;
    if (k > 0) m = fmax(m, pk);
    m = fmax(m, pn);
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) m = fmax(m, red[k]);
    // non-negative doubles are ordered like their bits
    atomicMax(w.count + 2 * blockIdx.y + 1, (unsigned long long)__double_as_longlong(m));
  }
}

__global__ void candidates_kernel(long long N, double thresh, Work w) {
  const double* P = w.P + blockIdx.y * (N + 1);
  unsigned long long* count = w.count + 2 * blockIdx.y;
  const double lim = thresh * __longlong_as_double((long long)count[1]);
  long long* cand = w.cand + blockIdx.y * (N / 2 + 1);
  for (long long j = 1 + blockIdx.x * (long long)blockDim.x + threadIdx.x; j < N; j += (long long)gridDim.x * blockDim.x) {
    const double p = P[j];
    if (p > P[j - 1] && p >= P[j + 1] && p >= lim) cand[atomicAdd(count, 1ULL)] = j;
  }
}

// better(a, b): higher power wins, equal power -> lower bin
__device__ __forceinline__ bool better(double pa, long long ja, double pb, long long jb) {
  return pa > pb || (pa == pb && ja < jb);
}

// lowest-frequency selection: the lower bin wins
__device__ __forceinline__ bool lower(double, long long ja, double, long long jb) { return ja < jb; }

// k rounds of a block-wide arg-max over the candidate list (warp shuffles), then sort; the
// winner of a round is the strongest candidate, or with `lowest` the lowest-frequency one
__global__ void select_kernel(long long N, int k, bool lowest, Work w) {
  const double* P = w.P + blockIdx.x * (N + 1);
  long long* cand = w.cand + blockIdx.x * (N / 2 + 1);
  long long* chosen = w.chosen + blockIdx.x * 64;
  auto wins = [&](double pa, long long ja, double pb, long long jb) {
    return lowest ? lower(pa, ja, pb, jb) : better(pa, ja, pb, jb);
  };
  __shared__ double sp[32];
  __shared__ long long sj[32];
  __shared__ long long pick[64];
  const long long n = (long long)w.count[2 * blockIdx.x];
  int got = 0;
  for (int r = 0; r < k; ++r) {
    double bp = -1.0;
    long long bj = -1;
    for (long long i = threadIdx.x; i < n; i += blockDim.x) {
      const long long j = cand[i];
      if (j < 0) continue;
      if (bj < 0 || wins(P[j], j, bp, bj)) { bp = P[j]; bj = j; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double op = __shfl_down_sync(0xffffffffu, bp, o);
      const long long oj = __shfl_down_sync(0xffffffffu, bj, o);
      if (oj >= 0 && (bj < 0 || wins(op, oj, bp, bj))) { bp = op; bj = oj; }
    }
    if ((threadIdx.x & 31) == 0) { sp[threadIdx.x >> 5] = bp; sj[threadIdx.x >> 5] = bj; }
    __syncthreads();
    if (threadIdx.x < 32) {
      bp = threadIdx.x < (blockDim.x >> 5) ? sp[threadIdx.x] : -1.0;
      bj = threadIdx.x < (blockDim.x >> 5) ? sj[threadIdx.x] : -1;
      for (int o = 16; o > 0; o >>= 1) {
        const double op = __shfl_down_sync(0xffffffffu, bp, o);
        const long long oj = __shfl_down_sync(0xffffffffu, bj, o);
        if (oj >= 0 && (bj < 0 || wins(op, oj, bp, bj))) { bp = op; bj = oj; }
      }
      if (threadIdx.x == 0) sj[0] = bj;
    }
    __syncthreads();
    const long long win = sj[0];
    __syncthreads();
    if (win < 0) break;
    for (long long i = threadIdx.x; i < n; i += blockDim.x)
      if (cand[i] == win) cand[i] = -1;
    if (threadIdx.x == 0) pick[got] = win;
    ++got;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    for (int a = 1; a < got; ++a) {  // insertion sort by frequency
      long long v = pick[a];
      int b = a - 1;
      while (b >= 0 && pick[b] > v) { pick[b + 1] = pick[b]; --b; }
      pick[b + 1] = v;
    }
    for (int a = 0; a < got; ++a) chosen[a] = pick[a];
    w.res[blockIdx.x * kRes] = (double)got;
  }
}

// Frequency of the parabola through log-power about bin j: the centre of the refinement.
__device__ __forceinline__ double parabola(const double* P, long long j, long long M) {
  const double la = log(P[j - 1]), lb = log(P[j]), lc = log(P[j + 1]);
  const double den = la - 2.0 * lb + lc;
  double delta = (den < 0.0) ? 0.5 * (la - lc) / den : 0.0;
  if (!isfinite(delta)) delta = 0.0;
  return 2.0 * kPi * ((double)j + delta) / (double)M;
}

// Moments sum_t xw_t e^{-i omega_0 (t - T/2)} ((t - tc) 2 / T)^q, q = 0 .. kSegQ - 1, of each
// segment (centre tc) of the series, about the parabola's omega_0 of each chosen peak.  One warp
// per segment; grid (kSegs / 8, peaks, estimates).
__global__ void __launch_bounds__(256) moments_kernel(long long T, long long N, int k, Work w) {
  const int lane = threadIdx.x & 31, seg = blockIdx.x * 8 + (threadIdx.x >> 5), peak = blockIdx.y, est = blockIdx.z;
  if (peak >= (int)w.res[est * kRes]) return;
  const double om = parabola(w.P + est * (N + 1), w.chosen[est * 64 + peak], 2 * N);
  const long long len = (T + kSegs - 1) / kSegs, t0 = min(T, seg * len), t1 = min(T, t0 + len);
  const double* x = w.xw + est * T;
  const double mid = 0.5 * (double)T, tc = (double)t0 + 0.5 * (double)(len - 1), sc = 2.0 / (double)T;
  double re[kSegQ] = {}, im[kSegQ] = {};
  if (t0 + lane < t1) {
    double s, c, ds, dc;
    sincos(om * ((double)(t0 + lane) - mid), &s, &c);
    sincos(om * 32.0, &ds, &dc);
    for (long long t = t0 + lane; t < t1; t += 32) {
      const double v = x[t], u = ((double)t - tc) * sc;
      double pr = v * c, pi = v * s;  // the imaginary part's sign goes in at the end
#pragma unroll
      for (int q = 0; q < kSegQ; ++q) {
        re[q] += pr;
        im[q] += pi;
        pr *= u;
        pi *= u;
      }
      const double cn = c * dc - s * ds;
      s = s * dc + c * ds;
      c = cn;
    }
  }
  double2* out = w.mom + (((size_t)est * k + peak) * kSegs + seg) * kSegQ;
#pragma unroll
  for (int q = 0; q < kSegQ; ++q) {
    for (int o = 16; o > 0; o >>= 1) {
      re[q] += __shfl_down_sync(0xffffffffu, re[q], o);
      im[q] += __shfl_down_sync(0xffffffffu, im[q], o);
    }
    if (lane == 0) out[q] = make_double2(re[q], -im[q]);
  }
}

// 40 golden-section steps on |X(omega)|^2 over omega_0 +- 1 bin, with
// X(omega_0 + y 2 / T) e^{i omega T / 2} = sum_m (-i y)^m / m! G_m and G_m the moments about the
// centre of the series.  One warp per peak: the lanes shift the segments' moments to the centre
// (binomially) and add them up; every lane then runs the same search.
__global__ void __launch_bounds__(32) refine_kernel(long long T, long long N, int k, Work w) {
  const int lane = threadIdx.x, peak = blockIdx.x, est = blockIdx.y;
  if (peak >= (int)w.res[est * kRes]) return;
  const double om = parabola(w.P + est * (N + 1), w.chosen[est * 64 + peak], 2 * N);
  const long long len = (T + kSegs - 1) / kSegs;
  const double sc = 2.0 / (double)T;
  const double2* mom = w.mom + ((size_t)est * k + peak) * kSegs * kSegQ;
  double re[kMom] = {}, im[kMom] = {};
  for (int seg = lane; seg < kSegs; seg += 32) {
    const double v = ((double)min(T, seg * len) + 0.5 * (double)(len - 1) - 0.5 * (double)T) * sc;
    // add mom_q C(m, q) v^(m - q) to every G_m: row q starts at m = q and grows by v (m + 1) / (m + 1 - q)
#pragma unroll
    for (int q = 0; q < kSegQ; ++q) {
      double ar = mom[seg * kSegQ + q].x, ai = mom[seg * kSegQ + q].y;
#pragma unroll
      for (int m = q; m < kMom; ++m) {
        re[m] += ar;
        im[m] += ai;
        const double g = v * ((double)(m + 1) / (double)(m + 1 - q));
        ar *= g;
        ai *= g;
      }
    }
  }
  double fact = 1.0;
#pragma unroll
  for (int m = 0; m < kMom; ++m) {
    for (int o = 16; o > 0; o >>= 1) {
      re[m] += __shfl_xor_sync(0xffffffffu, re[m], o);
      im[m] += __shfl_xor_sync(0xffffffffu, im[m], o);
    }
    if (m > 0) fact /= (double)m;
    // times (-i)^m / m!
    const double a = re[m] * fact, b = im[m] * fact;
    re[m] = m % 4 == 0 ? a : m % 4 == 1 ? b : m % 4 == 2 ? -a : -b;
    im[m] = m % 4 == 0 ? b : m % 4 == 1 ? -a : m % 4 == 2 ? -b : a;
  }
  auto power = [&](double omega) {
    const double y = (omega - om) * (0.5 * (double)T), y2 = y * y;
    double r[2], i[2];  // even and odd powers, two short chains each
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      double a = re[kMom - 2 + h], b = im[kMom - 2 + h];
#pragma unroll
      for (int m = kMom - 4 + h; m >= 0; m -= 2) {
        a = fma(a, y2, re[m]);
        b = fma(b, y2, im[m]);
      }
      r[h] = a;
      i[h] = b;
    }
    const double x = fma(r[1], y, r[0]), z = fma(i[1], y, i[0]);
    return x * x + z * z;
  };
  const double halfw = kPi / (double)N;
  double a = om - halfw, b = om + halfw;
  double c = b - kGolden * (b - a), d = a + kGolden * (b - a);
  double fc = power(c), fd = power(d);
  for (int it = 0; it < 40; ++it) {
    if (fc > fd) {
      b = d; d = c; fd = fc;
      c = b - kGolden * (b - a);
      fc = power(c);
    } else {
      a = c; c = d; fc = fd;
      d = a + kGolden * (b - a);
      fd = power(d);
    }
  }
  if (lane == 0) {
    const double o = 0.5 * (a + b);
    w.res[est * kRes + 2 + peak] = o;
    // the Hann weights add up to (T - 1) / 2
    w.res[est * kRes + 2 + 64 + peak] = 2.0 * sqrt(power(o)) / (0.5 * (double)(T - 1));
  }
}

constexpr size_t round16(size_t n) { return (n + 15) / 16 * 16; }

// Workspace for `count` estimates of T samples, transforms of M points and k peaks.
constexpr size_t workspace_bytes(size_t M, size_t T, size_t count, size_t k) {
  return round16(count * T * 8) + round16(count * kParts * 8) + 2 * (count * (M / 2) * 16) +
         round16(count * (M / 2 + 1) * 8) + round16(count * (M / 4 + 1) * 8) + round16(count * 16) +
         round16(count * 64 * 8) + count * k * kSegs * kSegQ * 16 + round16(count * kRes * 8);
}

Work carve(unsigned char* base, size_t M, size_t T, size_t count, size_t k) {
  unsigned char* p = base;
  auto take = [&](size_t n) { unsigned char* q = p; p += round16(n); return q; };
  Work w;
  w.xw = (double*)take(count * T * 8);
  w.part = (double*)take(count * kParts * 8);
  w.A = (double2*)take(count * (M / 2) * 16);
  w.B = (double2*)take(count * (M / 2) * 16);
  w.P = (double*)take(count * (M / 2 + 1) * 8);
  w.cand = (long long*)take(count * (M / 4 + 1) * 8);
  w.count = (unsigned long long*)take(count * 16);
  w.chosen = (long long*)take(count * 64 * 8);
  w.mom = (double2*)take(count * k * kSegs * kSegQ * 16);
  w.res = (double*)take(count * kRes * 8);
  return w;
}

// The estimator's launches on stream s for `count` estimates, and the copy of their results
// (kRes values each) to the host (synchronous).  Every workspace value is written before it is
// read except the candidate counters, which are cleared here, so a workspace may hold anything
// from an earlier call.
cudaError_t run_estimator(const Work& w, const double* d_x, int64_t T, int count, int64_t est_stride, int nser,
                          int64_t stride_series, int32_t k, bool lowest, double rel_power, cudaStream_t s,
                          std::vector<double>& res) {
  long long M = 1;
  while (M < 4 * T) M <<= 1;
  const long long N = M / 2;
  // a launch error left behind by an unrelated earlier runtime call on this thread would
  // otherwise be read back below as this call's failure
  (void)cudaGetLastError();
  cudaError_t e = cudaMemsetAsync(w.count, 0, 16 * (size_t)count, s);
  auto blocks = [](long long n, int per) { return (unsigned)std::max(1LL, std::min((n + per - 1) / per, 152LL * 8)); };
  if (e == cudaSuccess) {
    const int parts = (int)std::min<long long>(kParts, (T + 1023) / 1024);
    sum_kernel<<<dim3(parts, count), 256, 0, s>>>(d_x, T, nser, stride_series, est_stride, w);
    window_kernel<<<dim3(blocks(T, 256), count), 256, 0, s>>>(T, parts, w);
    double2 *in = w.A, *out = w.B;
    for (long long ns = 1; ns < N;) {
      // radix 16 passes, the first one taking what is left over (N >= 8)
      int bits = 0;
      while ((ns << bits) < N) ++bits;
      const int r = ns == 1 && bits % 4 != 0 ? 1 << (bits % 4) : 16;
      const dim3 grid(blocks(N / r, 128), count);
      if (ns > 1) stockham_kernel<16, false><<<grid, 128, 0, s>>>(in, out, w.xw, T, N, ns);
      else if (r == 16) stockham_kernel<16, true><<<grid, 128, 0, s>>>(in, out, w.xw, T, N, ns);
      else if (r == 8) stockham_kernel<8, true><<<grid, 128, 0, s>>>(in, out, w.xw, T, N, ns);
      else if (r == 4) stockham_kernel<4, true><<<grid, 128, 0, s>>>(in, out, w.xw, T, N, ns);
      else stockham_kernel<2, true><<<grid, 128, 0, s>>>(in, out, w.xw, T, N, ns);
      ns *= r;
      std::swap(in, out);
    }
    power_kernel<<<dim3(blocks(N / 2 + 1, 256), count), 256, 0, s>>>(in, N, w);
    candidates_kernel<<<dim3(blocks(N, 256), count), 256, 0, s>>>(N, rel_power, w);
    select_kernel<<<count, 256, 0, s>>>(N, k, lowest, w);
    moments_kernel<<<dim3(kSegs / 8, k, count), 256, 0, s>>>(T, N, k, w);
    refine_kernel<<<dim3(k, count), 32, 0, s>>>(T, N, k, w);
    e = cudaGetLastError();
  }
  res.resize((size_t)count * kRes);
  if (e == cudaSuccess) e = cudaMemcpyAsync(res.data(), w.res, 8 * res.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e;
}

// Estimate e's results to the caller's arrays; false when its series' mean is not finite (a NaN
// or infinity in the series: an unstable run).
bool put_result(const std::vector<double>& res, int e, double* freq, double* amp, int32_t* n) {
  const double* r = res.data() + (size_t)e * kRes;
  if (!std::isfinite(r[1])) return false;
  *n = (int32_t)r[0];
  std::copy(r + 2, r + 2 + *n, freq);
  std::copy(r + 2 + 64, r + 2 + 64 + *n, amp);
  return true;
}

}  // namespace

lbw_status spectrum_device(const double* d_x, int64_t T, int32_t count, int64_t est_stride, int32_t n_sum,
                           int64_t stride_series, int32_t k, cudaStream_t s, double* h_freq, double* h_amp,
                           int32_t* h_n, bool lowest, double rel_power) {
  size_t M = 1;
  while (M < 4 * (size_t)T) M <<= 1;
  // as many estimates per pass as fit in 256 MB of workspace, or in what there is
  int per = (int)std::max<size_t>(1, std::min<size_t>(std::min(count, 4096), (256u << 20) / workspace_bytes(M, (size_t)T, 1, k)));
  unsigned char* base = nullptr;
  while (cudaMallocAsync((void**)&base, workspace_bytes(M, (size_t)T, per, k), s) != cudaSuccess) {
    const cudaError_t e = cudaGetLastError();
    if (e != cudaErrorMemoryAllocation || per == 1) return cuda_fail(e, "spectrum workspace");
    per = (per + 1) / 2;
  }
  const Work w = carve(base, M, (size_t)T, per, k);
  std::vector<double> res;
  cudaError_t e = cudaSuccess;
  bool finite = true;
  for (int first = 0; first < count && e == cudaSuccess && finite; first += per) {
    const int n = std::min(per, count - first);
    e = run_estimator(w, d_x + (size_t)first * est_stride, T, n, est_stride, n_sum, stride_series, k, lowest, rel_power,
                      s, res);
    for (int j = 0; j < n && e == cudaSuccess && finite; ++j)
      finite = put_result(res, j, h_freq + (size_t)(first + j) * k, h_amp + (size_t)(first + j) * k, h_n + first + j);
  }
  cudaFreeAsync(base, s);
  if (e != cudaSuccess) return cuda_fail(e, "spectrum");
  if (!finite) return fail(LBW_EUNSTABLE, "spectrum: the series holds a non-finite value (unstable run)");
  return LBW_OK;
}

}  // namespace lbw

// ---------------------------------------------------------------- no-allocation variant -----
//
// lbw_spectrum_series_static: the estimator above on a caller-owned device series, with all of
// its workspace in one file-scope device array instead of stream-ordered allocations, for
// callers that must not allocate device memory.  The array is sized for series of up to
// kStaticMaxT samples and is held by every GPU that loads the library until the process exits.

namespace lbw {
namespace {
constexpr int64_t kStaticMaxT = 16384;
constexpr size_t kStaticMaxM = 4 * (size_t)kStaticMaxT;  // a power of two: M of the largest T
}  // namespace
}  // namespace lbw

// The workspace.  In host code this name is only a host-side handle: its device address comes
// from cudaGetSymbolAddress, looked up once per device context (static_workspace below).
static __device__ __align__(256) unsigned char
    g_spectrum_scratch[lbw::workspace_bytes(lbw::kStaticMaxM, lbw::kStaticMaxT, 1, 64)];

namespace {

typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

// Unique ID of the calling thread's current context (0 when there is none or the driver does
// not say).  IDs are never reused within a process, so a context created after a device reset
// never matches an ID cached before it.
unsigned long long current_context_id() {
  static CtxGetCurrentFn get_current = nullptr;
  static CtxGetIdFn get_id = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<CtxGetCurrentFn>(fn);
    fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<CtxGetIdFn>(fn);
    (void)cudaGetLastError();
  });
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx) return 0;
  if (get_id(ctx, &id) != CUDA_SUCCESS) return 0;
  return id;
}

struct StaticAddr {
  unsigned long long ctx_id = 0;
  void* ptr = nullptr;
};
std::mutex g_static_mu;
StaticAddr g_static_addr[256];

// Device address of the workspace on the current device.  Set-up, with that device current:
// cudaGetSymbolAddress, once per device context; the address is cached under the context's ID
// and looked up again when the device's context has changed (after cudaDeviceReset).
cudaError_t static_workspace(int dev, unsigned char** out) {
  std::lock_guard<std::mutex> lock(g_static_mu);
  StaticAddr& a = g_static_addr[dev];
  const unsigned long long id = current_context_id();
  if (id == 0 || a.ptr == nullptr || a.ctx_id != id) {
    void* ptr = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&ptr, g_spectrum_scratch);
    if (e != cudaSuccess) return e;
    a.ptr = ptr;
    a.ctx_id = current_context_id();  // the look-up makes the device's primary context current
  }
  *out = static_cast<unsigned char*>(a.ptr);
  return cudaSuccess;
}

}  // namespace

extern "C" lbw_status lbw_spectrum_series_static(const double* dev_x, int64_t T, int32_t k,
                                                 void* stream, double* host_freq, double* host_amp,
                                                 int32_t* host_n_found) {
  using namespace lbw;
  if (!dev_x || !host_freq || !host_amp || !host_n_found) return fail(LBW_EINVAL, "NULL argument");
  if (T < 4 || T > kStaticMaxT)
    return fail(LBW_EINVAL, "lbw_spectrum_series_static: T must be in [4, " + std::to_string(kStaticMaxT) +
                                "] (the fixed workspace holds " + std::to_string(kStaticMaxT) + " samples)");
  if (k < 1 || k > 64) return fail(LBW_EINVAL, "1 <= k <= 64");
  int dev = 0;
  LBW_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 256) return fail(LBW_EINVAL, "device ordinal out of range");
  unsigned char* base = nullptr;
  cudaError_t e = static_workspace(dev, &base);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_spectrum_scratch)");
  size_t M = 1;
  while (M < 4 * (size_t)T) M <<= 1;
  std::vector<double> res;
  e = run_estimator(carve(base, M, (size_t)T, 1, k), dev_x, T, 1, T, 1, T, k, false, 1e-3,
                    reinterpret_cast<cudaStream_t>(stream), res);
  if (e != cudaSuccess) return cuda_fail(e, "lbw_spectrum_series_static");
  int32_t nfound = 0;
  if (!put_result(res, 0, host_freq, host_amp, &nfound))
    return fail(LBW_EUNSTABLE, "spectrum: the series holds a non-finite value");
  *host_n_found = nfound;
  return LBW_OK;
}
