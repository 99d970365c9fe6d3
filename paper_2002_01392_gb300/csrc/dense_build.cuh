// Blocks of the dense z operators from the derivative kernels of the
// N'-periodic unit grid: what one thread writes, shared by the kernels that
// build the blocks on the device (k_dense.cu, k_dense64.cu) and the CPU checks.
//
// A plan keeps the kernels alone (two orders of N' values) and the blocks,
// 0.1 to 2.7 MB of float16, are built where they are used: built on the host
// and copied they cost fc_setup up to 80 ms and a plan's first call up to 165 us.
#pragma once
#include <cuda_fp16.h>

#include "dense64.hpp"

namespace fcns {

// entry (jo, ji) of part q's block: the sum over the distinct rows n of orbit ji of sign(n) c(n0(jo) - n),
// sign = 1, m, s, s m for the four members (q & 1: m = -1, q & 2: s = -1)
template <class V>
FC_DG V dense_entry(const DenseGeom& g, int q, int jo, int ji, const V* c) {
  const int n0 = dense_row(g, jo, 0);
  int rows[4];
  V v = 0;
  for (int i = 0; i < g.NQ; ++i) {
    rows[i] = dense_row(g, ji, i);
    bool seen = false;
    for (int k = 0; k < i; ++k) seen = seen || rows[k] == rows[i];
    if (seen) continue;
    const V x = c[n0 - rows[i] + (n0 < rows[i] ? g.Np : 0)];
    v += ((q & i & 1) + ((q & i) >> 1)) & 1 ? -x : x;
  }
  return v;
}

// Float32 blocks of one order: per output chunk, part and contraction slab the
// high values and then the low values, each as groups of eight contraction
// indexes x NC outputs (the shared-memory image that the kernel copies).
// One thread: two adjacent contraction indexes of one output; entries c / NQ 2^e.
FC_DG long long dense_pairs(const DenseGeom& g) { return (long long)g.chunks * g.NQ * (g.KQ / 8) * g.NC * 4; }
FC_DG void dense_pair(const DenseGeom& g, const double* c, int e, long long i, __half* order) {
  const int p = (int)(i % 4), r = (int)(i / 4 % g.NC), kc = (int)(i / 4 / g.NC % (g.KQ / 8)), cq = (int)(i / 4 / g.NC / (g.KQ / 8));
  const int q = cq % g.NQ, jo = cq / g.NQ * g.NC + r, s = kc / (2 * g.per), n = dense_slab(g, s);
  __half* hi = order + (long long)cq * 2 * g.KQ * g.NC + (long long)s * g.per * 32 * g.NC + ((kc - 2 * s * g.per) * g.NC + r) * 8 + 2 * p;
  const double sc = ldexp(1.0, e) / g.NQ;
  __half2 h, l;
  auto put = [&](int k, __half* hv, __half* lv) {
    const int ji = kc * 8 + 2 * p + k;
    const double v = jo < g.No && ji < g.No ? sc * dense_entry(g, q, jo, ji, c) : 0.0;
    *hv = __double2half(v);
    *lv = __double2half(v - (double)__half2float(*hv));
  };
  put(0, &h.x, &l.x);
  put(1, &h.y, &l.y);
  *reinterpret_cast<__half2*>(hi) = h;
  *reinterpret_cast<__half2*>(hi + n * 16 * g.NC) = l;
}

// Float64 blocks of one order: per output tile of 16 orbits, part, 16-step and
// digit the operand fragment of the matrix instruction (32 lanes x 8 halves).
// One thread: two adjacent halves of one lane, all digits; the kernels c are whole numbers.
FC_DG long long dense64_pairs(const DenseGeom& g) { return (long long)(g.KQ / 16) * g.NQ * (g.KQ / 16) * 128; }
FC_DG void dense64_pair(const DenseGeom& g, const long long* c, long long i, __half* order) {
  const int KT = g.KQ / 16, p = (int)(i % 4), lane = (int)(i / 4 % 32), ks = (int)(i / 128 % KT), q = (int)(i / 128 / KT % g.NQ),
            jt = (int)(i / 128 / KT / g.NQ);
  __half* out = order + (i / 128) * kD64Digits * 256 + lane * 8 + 2 * p;
  // (the inverse of d64_b_index)
  const int jo = jt * 16 + lane / 4 + 8 * (p >> 1), ji = ks * 16 + 2 * (lane % 4) + 8 * (p & 1);
  unsigned long long w[2];
  for (int h = 0; h < 2; ++h) w[h] = d64_bias(jo < g.No && ji + h < g.No ? dense_entry(g, q, jo, ji + h, c) : 0);
  for (int d = 0; d < kD64Digits; ++d) {
    __half2 v;
    v.x = __int2half_rn(d64_field(w[0], d) - 128);
    v.y = __int2half_rn(d64_field(w[1], d) - 128);
    *reinterpret_cast<__half2*>(out + d * 256) = v;
  }
}

}  // namespace fcns
