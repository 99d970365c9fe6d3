// fc_noise: the random solenoidal no-slip perturbation of App. A, built on
// the device from caller-supplied uniform draws.
//
//   q = curl curl(phi z_hat) + curl(psi z_hat)
//     = (d_x d_z phi + d_y psi, d_y d_z phi - d_x psi, -(d_xx + d_yy) phi),
//   phi = sum a e^{i(kx x + ky y)} g_m(z'),  psi = sum b e^{i(kx x + ky y)} sin(m pi (z' + 1/2)),
//   z' = z/Lz - 1/2,  g_m the Chandrasekhar-Reid functions (cosh/cos for odd
//   m, sinh/sin for even m) with lambda_m from g_m'(+-1/2) = 0,
//   a = k^slope_phi e^{2 pi i u_a}, b = k^slope_psi e^{2 pi i u_b},
//   k^2 = kx^2 + ky^2 + lambda_m^2, over the half plane of horizontal modes in
//   the annulus kperp2_min <= kx^2 + ky^2 <= kperp2_max and m_min <= m <= m_max;
//   the real part, scaled to a largest component magnitude of `amplitude`.
//
// The sums are separable: the vertical profiles of every horizontal mode (sum
// over m), then per (z, y) row the sums over the modes that share |kx|, then a
// real Fourier sum over n = |kx| Lx / 2 pi per point:
//   r(x) = sum_n A_n cos(n x) - B_n sin(n x),
//   A_n = Re(Q_n + Q_-n), B_n = Im(Q_n - Q_-n), Q_n = sum_l P_nl e^{i l y}.
// The cosine and sine sums of even and of odd n, taken once for a point i,
// give the four points i, Nx - i, Nx/2 + i, Nx/2 - i by additions (Nx a
// multiple of four; else the two points i and Nx - i).  What bounds the sums
// is arithmetic: taken point by point over +-n they kept the float64 pipe
// (1/74 of the float32 rate here) 88 % busy.
//
// float64 output: all of it in float64: 2 multiply-adds per n and four points
// and component instead of 4 per n and point; the largest magnitude is taken
// as the rows are written, and one pass scales them.
// float32 output: from the profiles (float64) on, every factor is a pair of
// floats (48 bits) and every sum a compensated one on the float32 pipe, which
// makes a second evaluation cheaper than a second and third trip through
// memory: the first run over the rows takes the largest magnitude and writes
// nothing, the second writes every value scaled and rounded once.
#include "internal.hpp"

#include <cmath>
#include <cstring>

namespace fcns {
namespace {

constexpr int kMaxM = 64;

// the two arithmetics of the row sums: a value V, a complex factor W
// (re, im) and s += a b over W's components
struct NoiseF64 {
  using T = double;
  using V = double;
  struct W { double re, im; };
  static __device__ __forceinline__ W pack(double re, double im) { return {re, im}; }
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ V re(const W& w) { return w.re; }
  static __device__ __forceinline__ V neg(V a) { return -a; }
  static __device__ __forceinline__ V add(V a, V b) { return a + b; }
  static __device__ __forceinline__ W join(V re, V im) { return {re, im}; }
  // s += Re(a) Re(b), s += Im(a) Im(b), ... (component pairs named by the suffix)
  static __device__ __forceinline__ void mrr(V& s, const W& a, const W& b) { s = fma(a.re, b.re, s); }
  static __device__ __forceinline__ void mii(V& s, const W& a, const W& b) { s = fma(a.im, b.im, s); }
  static __device__ __forceinline__ void mri(V& s, const W& a, const W& b) { s = fma(a.re, b.im, s); }
  static __device__ __forceinline__ void mir(V& s, const W& a, const W& b) { s = fma(a.im, b.re, s); }
};
// pairs of floats: hi + lo, |lo| of the order of ulp(hi)
struct NoiseF32 {
  using T = float;
  struct V { float hi, lo; };
  struct __align__(16) W { float rh, rl, ih, il; };
  static __device__ __forceinline__ W pack(double re, double im) {
    W w;
    w.rh = (float)re; w.rl = (float)(re - (double)w.rh);
    w.ih = (float)im; w.il = (float)(im - (double)w.ih);
    return w;
  }
  static __device__ __forceinline__ V zero() { return {0.f, 0.f}; }
  static __device__ __forceinline__ V re(const W& w) { return {w.rh, w.rl}; }
  static __device__ __forceinline__ V neg(V a) { return {-a.hi, -a.lo}; }
  // (Knuth two-sum of the high parts)
  static __device__ __forceinline__ V add(V a, V b) {
    const float s = __fadd_rn(a.hi, b.hi), z = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, z)), __fsub_rn(b.hi, z));
    return {s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
  }
  static __device__ __forceinline__ W join(V re, V im) {   // renormalised: hi = fl(hi + lo)
    W w;
    w.rh = __fadd_rn(re.hi, re.lo); w.rl = __fsub_rn(re.lo, __fsub_rn(w.rh, re.hi));
    w.ih = __fadd_rn(im.hi, im.lo); w.il = __fsub_rn(im.lo, __fsub_rn(w.ih, im.hi));
    return w;
  }
  // s += (ah + al)(bh + bl): the high product exactly (multiply, then the
  // fused remainder), the cross terms in float
  static __device__ __forceinline__ void mac(V& s, float ah, float al, float bh, float bl) {
    const float p = __fmul_rn(ah, bh);
    const float e = __fmaf_rn(al, bh, __fmaf_rn(ah, bl, __fmaf_rn(ah, bh, -p)));
    const float t = __fadd_rn(s.hi, p), z = __fsub_rn(t, s.hi);
    const float r = __fadd_rn(__fsub_rn(s.hi, __fsub_rn(t, z)), __fsub_rn(p, z));
    s.hi = t;
    s.lo = __fadd_rn(s.lo, __fadd_rn(r, e));
  }
  static __device__ __forceinline__ void mrr(V& s, const W& a, const W& b) { mac(s, a.rh, a.rl, b.rh, b.rl); }
  static __device__ __forceinline__ void mii(V& s, const W& a, const W& b) { mac(s, a.ih, a.il, b.ih, b.il); }
  static __device__ __forceinline__ void mri(V& s, const W& a, const W& b) { mac(s, a.rh, a.rl, b.ih, b.il); }
  static __device__ __forceinline__ void mir(V& s, const W& a, const W& b) { mac(s, a.ih, a.il, b.rh, b.rl); }
};

// P[(h * Nz + s) * 3 + c]: the z-profile of component c of horizontal mode h
template <class A>
__global__ void noise_profiles(int H, int nm, int m_min, int Nz, double Lz, const double2* __restrict__ kxy,
                               const double2* __restrict__ ab, const double* __restrict__ lam,
                               typename A::W* __restrict__ P) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)H * Nz) return;
  const int h = (int)(idx / Nz), s = (int)(idx % Nz);
  const double zp = (double)(2 * s - (Nz - 1)) / (double)(2 * (Nz - 1));
  const double kx = kxy[h].x, ky = kxy[h].y, kp2 = kx * kx + ky * ky;
  double2 pu = make_double2(0, 0), pv = make_double2(0, 0), pw = make_double2(0, 0);
  for (int mi = 0; mi < nm; ++mi) {
    const int m = m_min + mi;
    const double L = lam[mi];
    double g, dg;
    if (m & 1) {
      const double ch = cosh(0.5 * L), co = cos(0.5 * L);
      g = cosh(L * zp) / ch - cos(L * zp) / co;
      dg = L * (sinh(L * zp) / ch + sin(L * zp) / co);
    } else {
      const double sh = sinh(0.5 * L), si = sin(0.5 * L);
      g = sinh(L * zp) / sh - sin(L * zp) / si;
      dg = L * (cosh(L * zp) / sh - cos(L * zp) / si);
    }
    const double dgdz = dg / Lz;
    // sin(m pi (z' + 1/2)) = sin(pi m s / (Nz - 1)), reduced exactly modulo 2
    const long long num = ((long long)m * s) % (2LL * (Nz - 1));
    const double sn = sinpi((double)num / (double)(Nz - 1));
    const double2 a = ab[2 * (h * nm + mi)], b = ab[2 * (h * nm + mi) + 1];
    // i c = (-c.y, c.x)
    pu.x += -kx * a.y * dgdz - ky * b.y * sn;
    pu.y += kx * a.x * dgdz + ky * b.x * sn;
    pv.x += -ky * a.y * dgdz + kx * b.y * sn;
    pv.y += ky * a.x * dgdz - kx * b.x * sn;
    pw.x += kp2 * a.x * g;
    pw.y += kp2 * a.y * g;
  }
  P[idx * 3 + 0] = A::pack(pu.x, pu.y);
  P[idx * 3 + 1] = A::pack(pv.x, pv.y);
  P[idx * 3 + 2] = A::pack(pw.x, pw.y);
}

// Ex[n * ni + i] = e^{2 pi i n i / Nx} (n = 0..nmax, i < ni), Ey[l * Ny + j] =
// e^{2 pi i l j / Ny}: the phase taken modulo 2 pi in integers
template <class A>
__global__ void noise_phases(int nmax, int lmax, int Nx, int ni, int Ny, typename A::W* __restrict__ Ex,
                             typename A::W* __restrict__ Ey) {
  const long long nx = (long long)(nmax + 1) * ni, ny = (long long)(lmax + 1) * Ny;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= nx + ny) return;
  const bool inx = idx < nx;
  const long long k = inx ? idx : idx - nx;
  const int per = inx ? ni : Ny, N = inx ? Nx : Ny;
  const long long r = ((k / per) * (k % per)) % N;
  double sv, cv;
  sincospi(2.0 * (double)r / (double)N, &sv, &cv);
  (inx ? Ex : Ey)[k] = A::pack(cv, sv);
}

// the larger of two magnitudes; the float32 one keeps its low part, so that
// the scale factor carries the pairs' precision
struct NoiseMax {
  double d = 0.0;
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void take(double v) { d = fmax(d, fabs(v)); }
  __device__ __forceinline__ void take(NoiseF32::V v) {
    const float h = fabsf(v.hi), l = v.hi < 0.f ? -v.lo : v.lo;
    if (h > hi || (h == hi && l > lo)) { hi = h; lo = l; }
  }
  __device__ __forceinline__ double value() const { return fmax(d, (double)hi + (double)lo); }
};

// value v scaled by f: float64 output is scaled by a pass of its own
__device__ __forceinline__ double noise_out(double v, float2) { return v; }
__device__ __forceinline__ float noise_out(NoiseF32::V v, float2 f) {
  const float p = __fmul_rn(v.hi, f.x);
  return __fadd_rn(p, __fmaf_rn(v.lo, f.x, __fmaf_rn(v.hi, f.y, __fmaf_rn(v.hi, f.x, -p))));
}

constexpr int kNoiseThreads = 128;

// One block per (z, group of `rows` y rows).  First the folded sums (A_n, B_n)
// of the group's rows into shared memory, one (row, component, n) per thread;
// then one point i of one row per thread, all three components: 2 sums per n
// for QUARTER four (else two) points.  Measured at 512 x 512 x 257, float32
// output, whole call: 1.09 ms, against 16.0 ms for one float64 sum over +-n
// per point and passes of their own for the maximum and the scaling; error
// against 64 bits 2.5e-8 (before: 3.7e-8, two roundings).
template <class A, bool QUARTER, bool MAX, bool WRITE, bool SHIFT = false>
__global__ void __launch_bounds__(kNoiseThreads) noise_rows(int nmax, int Nx, int ni, int Ny, int Nz, int rows,
                                                            const int* __restrict__ start, const int* __restrict__ ml,
                                                            const typename A::W* __restrict__ P,
                                                            const typename A::W* __restrict__ Ex,
                                                            const typename A::W* __restrict__ Ey,
                                                            typename A::T* __restrict__ out, unsigned long long* word,
                                                            double amplitude) {
  using W = typename A::W;
  using V = typename A::V;
  extern __shared__ __align__(16) unsigned char noise_sm[];
  W* Q = reinterpret_cast<W*>(noise_sm);   // [rows][nmax + 1][3]
  const int groups = (Ny + rows - 1) / rows;
  const int s = (int)(blockIdx.x / groups), j0 = (int)(blockIdx.x % groups) * rows;
  const int nr = min(rows, Ny - j0), NN = nmax + 1;
  for (int t = threadIdx.x; t < nr * NN * 3; t += kNoiseThreads) {
    const int c = t % 3, n = (t / 3) % NN, j = j0 + t / (3 * NN);
    V a = A::zero(), b = A::zero();
    for (int sg = n > 0 ? 0 : 1; sg < 2; ++sg) {   // modes of -n, then of +n
      V re = A::zero(), rm = A::zero(), im = A::zero();
      const int k = sg == 0 ? nmax - n : nmax + n;
      for (int h = start[k]; h < start[k + 1]; ++h) {
        const W p = P[((long long)h * Nz + s) * 3 + c], e = Ey[(long long)ml[h] * Ny + j];
        A::mrr(re, p, e);
        A::mii(rm, p, e);
        A::mri(im, p, e);
        A::mir(im, p, e);
      }
      a = A::add(a, A::add(re, A::neg(rm)));
      b = A::add(b, sg == 0 ? A::neg(im) : im);
    }
    Q[t] = A::join(a, b);
  }
  __syncthreads();
  float2 f = make_float2(0.f, 0.f);
  int shift = 0;
  if constexpr (WRITE && !MAX) {
    const double mx = __longlong_as_double((long long)*word);
    double fd = mx > 0.0 ? amplitude / mx : 1.0;
    if constexpr (SHIFT) {   // the exponent apart
      int ea = 0, em = 0;
      fd = mx > 0.0 ? frexp(amplitude, &ea) / frexp(mx, &em) : 1.0;
      shift = ea - em;
    }
    f.x = (float)fd;
    f.y = (float)(fd - (double)f.x);
  }
  const long long plane = (long long)Nz * Ny * Nx;
  NoiseMax m;
  for (int t = threadIdx.x; t < nr * ni; t += kNoiseThreads) {
    const int r = t / ni, i = t % ni;
    // sums over even n (0) and odd n (1) of A_n cos (C) and B_n sin (S)
    V Cs[3][2], Ss[3][2];
    const W* q = Q + (long long)r * NN * 3;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      Cs[c][0] = A::re(q[c]);   // n = 0
      Cs[c][1] = Ss[c][0] = Ss[c][1] = A::zero();
    }
    for (int n = 1; n < NN; n += 2) {
#pragma unroll
      for (int o = 1; o >= 0; --o) {   // odd n, then even n + 1
        const int nn = n + 1 - o;
        if (o == 1 || nn < NN) {
          const W e = Ex[(long long)nn * ni + i];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const W w = q[nn * 3 + c];
            A::mrr(Cs[c][QUARTER ? o : 0], w, e);
            A::mii(Ss[c][QUARTER ? o : 0], w, e);
          }
        }
      }
    }
    typename A::T* row = out + ((long long)s * Ny + j0 + r) * Nx;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      typename A::T* o = row + c * plane;
      auto put = [&](int x, V v) {
        if constexpr (MAX) m.take(v);
        if constexpr (WRITE) o[x] = SHIFT ? (typename A::T)ldexp(noise_out(v, f), shift) : noise_out(v, f);
      };
      if constexpr (QUARTER) {
        // cos n(pi -+ x) = (-1)^n cos nx, sin n(pi - x) = -(-1)^n sin nx
        const V cp = A::add(Cs[c][0], Cs[c][1]), cm = A::add(Cs[c][0], A::neg(Cs[c][1]));
        const V sp = A::add(Ss[c][0], Ss[c][1]), sm = A::add(Ss[c][0], A::neg(Ss[c][1]));
        put(i, A::add(cp, A::neg(sp)));
        put(Nx / 2 + i, A::add(cm, A::neg(sm)));
        if (i > 0 && 4 * i != Nx) {   // (i = 0 and i = Nx / 4 are two points only)
          put(Nx - i, A::add(cp, sp));
          put(Nx / 2 - i, A::add(cm, sm));
        }
      } else {
        put(i, A::add(Cs[c][0], A::neg(Ss[c][0])));
        if (i > 0 && 2 * i != Nx) put(Nx - i, A::add(Cs[c][0], Ss[c][0]));
      }
    }
  }
  if constexpr (MAX) {   // bits of a non-negative double: their unsigned order is the numeric order
    __shared__ double red[kNoiseThreads / 32];
    double v = m.value();
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 1; k < kNoiseThreads / 32; ++k) v = fmax(v, red[k]);
      atomicMax(word, (unsigned long long)__double_as_longlong(v));
    }
  }
}

__global__ void noise_scale(double* __restrict__ out, long long n, const unsigned long long* word, double amplitude) {
  const double mx = __longlong_as_double((long long)*word);
  if (!(mx > 0.0)) return;
  const double f = amplitude / mx;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = out[i] * f;
}

struct NoiseGrid {
  int H, nm, m_min, nmax, lmax, Nx, Ny, Nz, ni, sms;
  double Lz, amplitude;
};
struct NoiseDev {
  unsigned long long* word;
  double2 *kxy, *ab;
  double* lam;
  int *start, *ml;
  void *P, *Ex, *Ey;
};

template <class A, bool QUARTER>
void noise_launch(const NoiseGrid& g, const NoiseDev& d, typename A::T* out, cudaStream_t st) {
  using W = typename A::W;
  W *P = static_cast<W*>(d.P), *Ex = static_cast<W*>(d.Ex), *Ey = static_cast<W*>(d.Ey);
  const long long np = (long long)g.H * g.Nz;
  noise_profiles<A><<<(unsigned)((np + 127) / 128), 128, 0, st>>>(g.H, g.nm, g.m_min, g.Nz, g.Lz, d.kxy, d.ab, d.lam, P);
  const long long ne = (long long)(g.nmax + 1) * g.ni + (long long)(g.lmax + 1) * g.Ny;
  noise_phases<A><<<(unsigned)((ne + 255) / 256), 256, 0, st>>>(g.nmax, g.lmax, g.Nx, g.ni, g.Ny, Ex, Ey);
  // eight rows per block (their sums fill the block's threads once or twice for a few modes), fewer when the
  // folded sums would pass 24 KB
  const size_t per = sizeof(W) * 3 * (g.nmax + 1);
  const int rows = (int)std::max<size_t>(1, std::min<size_t>(8, 24 * 1024 / per));
  const unsigned grid = (unsigned)((long long)g.Nz * ((g.Ny + rows - 1) / rows));
  if constexpr (std::is_same_v<A, NoiseF32>) {
    noise_rows<A, QUARTER, true, false><<<grid, kNoiseThreads, per * rows, st>>>(
        g.nmax, g.Nx, g.ni, g.Ny, g.Nz, rows, d.start, d.ml, P, Ex, Ey, out, d.word, g.amplitude);
    // amplitude / max has to stay in float's range as a pair (the sums are near 1); far amplitudes have their exponent apart
    // (for all of them, ldexp on every value would cost 5 %)
    const double amp = std::fabs(g.amplitude);
    auto kern = amp > 0.0 && (amp < 0x1p-60 || amp > 0x1p60) ? noise_rows<A, QUARTER, false, true, true>
                                                            : noise_rows<A, QUARTER, false, true, false>;
    kern<<<grid, kNoiseThreads, per * rows, st>>>(
        g.nmax, g.Nx, g.ni, g.Ny, g.Nz, rows, d.start, d.ml, P, Ex, Ey, out, d.word, g.amplitude);
  } else {
    noise_rows<A, QUARTER, true, true><<<grid, kNoiseThreads, per * rows, st>>>(
        g.nmax, g.Nx, g.ni, g.Ny, g.Nz, rows, d.start, d.ml, P, Ex, Ey, out, d.word, g.amplitude);
    const long long n = 3LL * g.Nz * g.Ny * g.Nx;
    const unsigned gb = (unsigned)std::max(1LL, std::min<long long>((n + 255) / 256, (long long)std::max(g.sms, 1) * 8));
    noise_scale<<<gb, 256, 0, st>>>(out, n, d.word, g.amplitude);
  }
}

// lambda_m: root of tanh t + tan t (odd m) or tanh t - tan t (even m), t = lambda/2,
// on the m-th bracket; bisection to adjacent doubles
double cr_lambda(int m) {
  const double pi = 3.14159265358979323846;
  const bool odd = (m & 1) != 0;
  const int j = odd ? (m + 1) / 2 : m / 2;
  double lo = odd ? j * pi - pi / 2 : j * pi, hi = odd ? j * pi : j * pi + pi / 2;
  lo += 1e-9;
  hi -= 1e-9;
  auto f = [odd](double t) { return odd ? std::tanh(t) + std::tan(t) : std::tanh(t) - std::tan(t); };
  const double flo = f(lo);
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    const double fm = f(mid);
    if (fm == 0.0) return 2.0 * mid;
    if ((fm < 0) == (flo < 0)) lo = mid;
    else hi = mid;
  }
  return std::fabs(f(lo)) <= std::fabs(f(hi)) ? 2.0 * lo : 2.0 * hi;
}

struct NoiseModes {
  int nmax = 0, lmax = 0;
  std::vector<int2> nl;        // horizontal modes (n, l), enumeration order
  std::vector<double2> kxy;    // their (kx, ky)
};

fc_status check_params(const fc_noise_params* p) {
  if (!p) {
    set_error("fc_noise: NULL parameters");
    return FC_ERR_ARG;
  }
  const bool ok = std::isfinite(p->Lx) && std::isfinite(p->Ly) && std::isfinite(p->Lz) && p->Lx > 0 && p->Ly > 0 &&
                  p->Lz > 0 && std::isfinite(p->kperp2_min) && std::isfinite(p->kperp2_max) && p->kperp2_min >= 0 &&
                  p->kperp2_max >= p->kperp2_min && p->kperp2_max * p->Lx * p->Lx < 4e8 &&
                  p->kperp2_max * p->Ly * p->Ly < 4e8 && p->m_min >= 1 && p->m_max >= p->m_min &&
                  p->m_max <= kMaxM && std::isfinite(p->slope_phi) && std::isfinite(p->slope_psi) &&
                  std::isfinite(p->amplitude);
  if (!ok) {
    set_error("fc_noise: need Lx, Ly, Lz > 0, 0 <= kperp2_min <= kperp2_max (kperp2_max Lx^2, kperp2_max Ly^2 < 4e8), "
              "1 <= m_min <= m_max <= 64, finite slopes and amplitude");
    return FC_ERR_ARG;
  }
  return FC_OK;
}

NoiseModes enumerate_modes(const fc_noise_params& p) {
  const double pi = 3.14159265358979323846;
  NoiseModes r;
  const int nmax = (int)std::floor(std::sqrt(p.kperp2_max) * p.Lx / (2 * pi)) + 1;
  const int lmax = (int)std::floor(std::sqrt(p.kperp2_max) * p.Ly / (2 * pi)) + 1;
  for (int n = -nmax; n <= nmax; ++n)
    for (int l = 0; l <= lmax; ++l) {
      if (l == 0 && n <= 0) continue;
      const double kx = 2 * pi * n / p.Lx, ky = 2 * pi * l / p.Ly, kp2 = kx * kx + ky * ky;
      if (!(p.kperp2_min * (1 - 1e-12) <= kp2 && kp2 <= p.kperp2_max * (1 + 1e-12))) continue;
      r.nl.push_back(make_int2(n, l));
      r.kxy.push_back(make_double2(kx, ky));
      r.nmax = std::max(r.nmax, n < 0 ? -n : n);
      r.lmax = std::max(r.lmax, l);
    }
  return r;
}

}  // namespace
}  // namespace fcns

using namespace fcns;

extern "C" fc_status fc_noise_params_default(fc_noise_params* p) {
  if (!p) {
    set_error("fc_noise_params_default: NULL");
    return FC_ERR_ARG;
  }
  p->Lx = p->Ly = 2 * 3.14159265358979323846;
  p->Lz = 1.0;
  p->kperp2_min = 4.0;
  p->kperp2_max = 25.0;
  p->m_min = 2;
  p->m_max = 5;
  p->slope_phi = -4.0;
  p->slope_psi = -3.0;
  p->amplitude = 1.0;
  return FC_OK;
}

extern "C" fc_status fc_noise_modes(const fc_noise_params* p, int* count) {
  if (fc_status s = check_params(p)) return s;
  if (!count) {
    set_error("fc_noise_modes: NULL count");
    return FC_ERR_ARG;
  }
  *count = (int)enumerate_modes(*p).nl.size() * (p->m_max - p->m_min + 1);
  return FC_OK;
}

extern "C" fc_status fc_noise(const fc_noise_params* p, fc_dtype dtype, int Nx, int Ny, int Nz, const double* draws,
                              int ndraws, void* out, fc_stream_t stream) {
  if (fc_status inj = injected("fc_noise")) return inj;
  if (fc_status s = check_params(p)) return s;
  if ((dtype != FC_F32 && dtype != FC_F64) || Nx < 1 || Ny < 1 || Nz < 2 || !out || !draws) {
    set_error("fc_noise: dtype must be FC_F32 or FC_F64, Nx, Ny >= 1, Nz >= 2, draws and out non-NULL");
    return FC_ERR_ARG;
  }
  const NoiseModes md = enumerate_modes(*p);
  const int H = (int)md.nl.size(), nm = p->m_max - p->m_min + 1;
  if (H == 0) {
    set_error("fc_noise: no horizontal mode in the annulus");
    return FC_ERR_ARG;
  }
  if ((long long)ndraws != 2LL * H * nm) {
    set_error("fc_noise: ndraws must be 2 x fc_noise_modes()");
    return FC_ERR_ARG;
  }
  if (Nx <= 2 * md.nmax || Ny <= 2 * md.lmax) {
    set_error("fc_noise: the grid must resolve every mode (Nx > 2 max|n|, Ny > 2 max l)");
    return FC_ERR_ARG;
  }
  if (2 * md.nmax + 1 > 1024) {   // the synthesis keeps a row's 3 x (nmax + 1) sums in 24 KB of shared memory
    set_error("fc_noise: at most 511 kx indices on each side of the annulus");
    return FC_ERR_UNSUPPORTED;
  }
  if ((long long)Nz * Ny > 0x7fffffffLL || 3LL * Nz * Ny * Nx > (1LL << 40)) {
    set_error("fc_noise: grid too large");
    return FC_ERR_ARG;
  }
  for (int i = 0; i < ndraws; ++i)
    if (!std::isfinite(draws[i])) {
      set_error("fc_noise: non-finite draw");
      return FC_ERR_ARG;
    }
  // host side: lambda_m and the complex amplitudes a, b of every (n, l, m) mode
  const double pi = 3.14159265358979323846;
  std::vector<double> lam(nm);
  for (int mi = 0; mi < nm; ++mi) lam[mi] = cr_lambda(p->m_min + mi);
  std::vector<double2> ab(2 * (size_t)H * nm);
  for (int h = 0; h < H; ++h)
    for (int mi = 0; mi < nm; ++mi) {
      const double kx = md.kxy[h].x, ky = md.kxy[h].y;
      const double k = std::sqrt(kx * kx + ky * ky + lam[mi] * lam[mi]);
      const size_t j = (size_t)h * nm + mi;
      const double ra = std::pow(k, p->slope_phi), rb = std::pow(k, p->slope_psi);
      ab[2 * j] = make_double2(ra * std::cos(2 * pi * draws[2 * j]), ra * std::sin(2 * pi * draws[2 * j]));
      ab[2 * j + 1] = make_double2(rb * std::cos(2 * pi * draws[2 * j + 1]), rb * std::sin(2 * pi * draws[2 * j + 1]));
    }
  // the largest magnitude is scaled away at the end: keep the vertical profiles (g_m and g_m' / lambda_m are below about 2)
  // near 1 by a power of two, whatever the slopes and the box
  double big = 0.0;
  for (int h = 0; h < H; ++h)
    for (int mi = 0; mi < nm; ++mi) {
      const double2 a = ab[2 * ((size_t)h * nm + mi)], b = ab[2 * ((size_t)h * nm + mi) + 1];
      const double kx = md.kxy[h].x, ky = md.kxy[h].y, kp = std::sqrt(kx * kx + ky * ky);
      big = std::max(big, std::hypot(a.x, a.y) * std::max(kp * kp, kp * lam[mi] / p->Lz));
      big = std::max(big, std::hypot(b.x, b.y) * kp);
    }
  if (big > 0.0 && std::isfinite(big)) {
    const int e = std::ilogb(big);
    for (double2& v : ab) v = make_double2(std::ldexp(v.x, -e), std::ldexp(v.y, -e));
  }
  // the modes of one n are contiguous in the enumeration: [start[n + nmax], start[n + nmax + 1])
  std::vector<int> start(2 * md.nmax + 2, 0), ml(H);
  for (int h = 0; h < H; ++h) {
    ++start[md.nl[h].x + md.nmax + 1];
    ml[h] = md.nl[h].y;
  }
  for (size_t k = 1; k < start.size(); ++k) start[k] += start[k - 1];
  // points of a row that are summed: a quarter and one more (Nx a multiple of four), else a half
  const bool quarter = Nx % 4 == 0;
  const int ni = quarter ? Nx / 4 + 1 : Nx / 2 + 1;
  // one device block of scratch: tables, profiles, phase tables, max word (a
  // float pair per component and a double per component take the same 16 bytes)
  const size_t nEx = (size_t)(md.nmax + 1) * ni, nEy = (size_t)(md.lmax + 1) * Ny;
  const size_t nP = (size_t)H * Nz * 3;
  static_assert(sizeof(NoiseF32::W) == 16 && sizeof(NoiseF64::W) == 16, "factor size");
  size_t off = 0;
  auto take = [&off](size_t bytes) { const size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
  const size_t o_word = take(sizeof(unsigned long long)), o_kxy = take(sizeof(double2) * H),
               o_start = take(sizeof(int) * start.size()), o_ml = take(sizeof(int) * H),
               o_ab = take(sizeof(double2) * ab.size()), o_lam = take(sizeof(double) * nm), o_P = take(16 * nP),
               o_Ex = take(16 * nEx), o_Ey = take(16 * nEy);
  const size_t host_bytes = o_P;  // everything before the profiles comes from the host
  std::vector<unsigned char> h(host_bytes, 0);
  std::memcpy(h.data() + o_kxy, md.kxy.data(), sizeof(double2) * H);
  std::memcpy(h.data() + o_start, start.data(), sizeof(int) * start.size());
  std::memcpy(h.data() + o_ml, ml.data(), sizeof(int) * H);
  std::memcpy(h.data() + o_ab, ab.data(), sizeof(double2) * ab.size());
  std::memcpy(h.data() + o_lam, lam.data(), sizeof(double) * nm);

  cudaStream_t st = (cudaStream_t)stream;
  unsigned char* buf = nullptr;
  const cudaError_t ae = cudaMallocAsync((void**)&buf, off, st);
  if (ae == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    set_error("fc_noise: cudaMallocAsync of the scratch failed");
    return FC_ERR_NOMEM;
  }
  fc_status s = cuda_status(ae, "cudaMallocAsync");
  if (s) return s;
  // pageable source: the call returns once the bytes are staged, so `h` may go
  s = cuda_status(cudaMemcpyAsync(buf, h.data(), host_bytes, cudaMemcpyHostToDevice, st), "cudaMemcpyAsync");
  if (!s) {
    NoiseDev d;
    d.word = reinterpret_cast<unsigned long long*>(buf + o_word);
    d.kxy = reinterpret_cast<double2*>(buf + o_kxy);
    d.ab = reinterpret_cast<double2*>(buf + o_ab);
    d.lam = reinterpret_cast<double*>(buf + o_lam);
    d.start = reinterpret_cast<int*>(buf + o_start);
    d.ml = reinterpret_cast<int*>(buf + o_ml);
    d.P = buf + o_P;
    d.Ex = buf + o_Ex;
    d.Ey = buf + o_Ey;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const NoiseGrid g = {H, nm, p->m_min, md.nmax, md.lmax, Nx, Ny, Nz, ni, sms, p->Lz, p->amplitude};
    if (dtype == FC_F32) {
      quarter ? noise_launch<NoiseF32, true>(g, d, static_cast<float*>(out), st)
              : noise_launch<NoiseF32, false>(g, d, static_cast<float*>(out), st);
    } else {
      quarter ? noise_launch<NoiseF64, true>(g, d, static_cast<double*>(out), st)
              : noise_launch<NoiseF64, false>(g, d, static_cast<double*>(out), st);
    }
    s = cuda_status(cudaGetLastError(), "fc_noise launch");
  }
  const fc_status s2 = cuda_status(cudaFreeAsync(buf, st), "cudaFreeAsync");
  return s ? s : s2;
}
