// FC-Gram continuation of the lines of a CTA (Sec. 3), shared by the z kernels.
#pragma once
#include "engine.cuh"

namespace fcns {

#if defined(__CUDACC__)
#define FC_NOINLINE __host__ __device__ __noinline__
#else
#define FC_NOINLINE
#endif

constexpr int DMAX = 10;
constexpr int CMAX = 64;

// C continuation value jj (point Nz + jj) of a complex line from its first /
// last d values (Sec. 3 continuation formula; right matrix M_r, left matrix
// its row/column reversal), with compensated sums: float-float products in
// float32, double-double in float64 (the weights reach 4e3 and cancel).
// D > 0: d = D at compile time.
template <class T, int D>
FC_HD cx<T> continuation_sum(int jj, const cx<T>* first, const cx<T>* last, int d, int Cc, const double* Ms,
                             const float2* Ms2) {
  const int n = D > 0 ? D : d;
  if constexpr (sizeof(T) == 4) {
    float2 h = make_float2(0.f, 0.f), l = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float2 m1 = Ms2[jj * n + i];
      const float2 m2 = Ms2[(Cc - 1 - jj) * n + (n - 1 - i)];
      ff_fma2(h, l, m1.x, m1.y, last[i]);
      ff_fma2(h, l, m2.x, m2.y, first[i]);
    }
    return cadd(h, l);
  } else {
    dd re{0.0, 0.0}, im{0.0, 0.0};
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const double m1 = Ms[jj * n + i];
      const double m2 = Ms[(Cc - 1 - jj) * n + (n - 1 - i)];
      dd_fma(re, m1, last[i].x);
      dd_fma(im, m1, last[i].y);
      dd_fma(re, m2, first[i].x);
      dd_fma(im, m2, first[i].y);
    }
    return mk<T>((T)dd_round(re), (T)dd_round(im));
  }
}
// d = 5 (the default continuation) inline, any other d through one copy of the code
template <class T>
FC_NOINLINE cx<T> continuation_any(int jj, const cx<T>* first, const cx<T>* last, int d, int Cc, const double* Ms,
                                   const float2* Ms2) {
  return continuation_sum<T, 0>(jj, first, last, d, Cc, Ms, Ms2);
}
template <class T>
FC_HD cx<T> continuation_value(int jj, const cx<T>* first, const cx<T>* last, int d, int Cc, const double* Ms,
                               const float2* Ms2) {
  return d == 5 ? continuation_sum<T, 5>(jj, first, last, d, Cc, Ms, Ms2)
                : continuation_any<T>(jj, first, last, d, Cc, Ms, Ms2);
}
// The continuation of a CTA's lines, f(jj, li, value): one (point, line) pair
// per thread and turn, whatever thread holds those rows otherwise (where each
// thread continued the rows it holds, a few lanes of every warp did all the
// sums, twice: the stage combine of 256^2 x 257 x 4 went 734 -> 675 us).
// A thread's items are all of line li = tid % LINES (THREADS is a multiple of
// LINES), so a thread of an absent or unused line may leave the call out.
// Ev: [LINES][stride] with the first d values, then (at DMAX) the last d.
template <class T, int LINES, int THREADS, class F>
FC_HD void continue_lines(int tid, const cx<T>* Ev, int stride, int d, int Cc, const double* Ms, const float2* Ms2, F&& f) {
  for (int i = tid; i < Cc * LINES; i += THREADS) {
    const int jj = i / LINES, li = i % LINES;
    const cx<T>* e = Ev + li * stride;
    f(jj, li, continuation_value<T>(jj, e, e + DMAX, d, Cc, Ms, Ms2));
  }
}

}  // namespace fcns
