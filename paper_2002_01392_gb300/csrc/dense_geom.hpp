// Geometry of the dense z operators (dense_z.cuh), shared by the kernel, the
// table builder and the CPU checks.
//
// A z operator of the N'-periodic continued grid is a circular convolution
// with a kernel that is even (d2/dz2) or odd (d/dz).  It commutes, up to that
// sign, with the mirror n -> Nz - 1 - n, and when N' is even it commutes with
// the half shift n -> n + N'/2.  The group these generate (NQ = 2 or 4
// elements) splits a line into NQ parts, one per sign pattern, and the
// operator into NQ blocks of about N'/NQ each: NQ times fewer multiplies than
// the N' x N' matrix.  Orbit j has the rows
//   n0 = floor(Nz / 2) + j,  n1 = Nz - 1 - n0  [, n2 = n0 + N'/2, n3 = n1 + N'/2]
// modulo N'; part (s, m) of a line is x0 + m x1 + s (x2 + m x3) per orbit.
#pragma once

#if defined(__CUDACC__)
#define FC_DG __host__ __device__ __forceinline__
#else
#define FC_DG inline
#endif

namespace fcns {

constexpr int kDenseLines = 128;     // lines per tile: the rows of one tensor-core tile
constexpr int kDenseSlabSteps = 9;   // 16-steps of a slab at most
constexpr int kDenseMaxK = 576;      // NQ * KQ: the split line has to fit tensor memory and shared memory

struct DenseGeom {
  int Nz = 0, Np = 0;
  int NQ = 0;        // 4 (N' even) or 2
  int No = 0;        // orbits
  int KQ = 0;        // No rounded up to 16: the contraction length of a block
  int NC = 0;        // orbits per output chunk (a multiple of 16)
  int chunks = 0;    // NC * chunks >= No
  int slabs = 0;     // pieces of the contraction that a block is loaded in,
  int per = 0;       // of this many 16-steps each (the last one the rest)
};

// row of member i (0..NQ-1) of orbit j
FC_DG int dense_row(const DenseGeom& g, int j, int i) {
  int n = g.Nz / 2 + j;
  if (i & 1) n = g.Nz - 1 - n;
  if (n < 0) n += g.Np;
  if (i & 2) {
    n += g.Np / 2;
    if (n >= g.Np) n -= g.Np;
  }
  return n;
}
// 16-steps of slab s
FC_DG int dense_slab(const DenseGeom& g, int s) {
  const int left = g.KQ / 16 - s * g.per;
  return left < g.per ? left : g.per;
}

// geometry for (Nz, N'); false where the split line does not fit
inline bool dense_geom(int Nz, int Np, DenseGeom* o) {
  DenseGeom g;
  g.Nz = Nz;
  g.Np = Np;
  g.NQ = Np % 2 == 0 ? 4 : 2;
  const int m = g.NQ == 4 ? Np / 2 : Np;                       // orbits of the mirror modulo m
  const int fixed = m % 2 ? 1 : (Nz % 2 ? 2 : 0);              // solutions of 2 n = Nz - 1 (mod m)
  g.No = (m + fixed) / 2;
  g.KQ = (g.No + 15) / 16 * 16;
  if (g.NQ * g.KQ > kDenseMaxK) return false;
  const int most = 48;   // accumulator columns: NQ * NC, twice that for NQ = 2 (dense_z.cuh), up to 192
  g.chunks = (g.No + most - 1) / most;
  g.NC = ((g.No + g.chunks - 1) / g.chunks + 15) / 16 * 16;
  const int kt = g.KQ / 16, fit = 9 * 48 / g.NC;  // slabs of at most 27 KB
  const int most_steps = fit < kDenseSlabSteps ? fit : kDenseSlabSteps;
  g.slabs = (kt + most_steps - 1) / most_steps;
  g.per = (kt + g.slabs - 1) / g.slabs;
  *o = g;
  return true;
}
// halves of one slab's high (or low) part, of a block, and of one order
FC_DG long long dense_block_halves(const DenseGeom& g) { return 2LL * g.KQ * g.NC; }
FC_DG long long dense_order_halves(const DenseGeom& g) { return dense_block_halves(g) * g.chunks * g.NQ; }
// largest slab in bytes
FC_DG int dense_slab_bytes(const DenseGeom& g) { return (g.per < g.KQ / 16 ? g.per : g.KQ / 16) * 16 * g.NC * 4; }

// shared memory of the kernel (byte offsets) with `stages` slabs in the ring
constexpr int kDenseBars = 28;   // barriers: full[8], empty[8], accumulators full[4], free[4], A ready, scouts full, free, end
constexpr int kDenseSmemMax = 227 * 1024;
struct DenseSmem {
  int lo, ring, cont, scale, lmax, mr, bars, total;
};
inline DenseSmem dense_smem(const DenseGeom& g, int d, int C, int stages) {
  DenseSmem s;
  s.lo = 0;
  s.ring = g.NQ * g.KQ * 2 * kDenseLines;
  s.cont = s.ring + stages * dense_slab_bytes(g);
  s.scale = s.cont + C * kDenseLines * 4;
  s.lmax = s.scale + 2 * kDenseLines * 4;
  s.mr = s.lmax + kDenseLines * 4 + 16;
  s.bars = (s.mr + C * d * 8 + 15) / 16 * 16;
  s.total = s.bars + 8 * kDenseBars + 16;
  return s;
}
// slabs that fit (at most 8)
inline int dense_stages(const DenseGeom& g, int d, int C) {
  const int n = (kDenseSmemMax - dense_smem(g, d, C, 0).total) / dense_slab_bytes(g);
  return n < 8 ? n : 8;
}
// geometry of a plan: the ring needs two slabs, and the continuation of d, C takes shared memory too (with N' above 510
// and C from 48 on there is room for one only: such plans have no dense operators)
inline bool dense_plan(int Nz, int d, int C, DenseGeom* o) {
  DenseGeom g;
  if (!dense_geom(Nz, Nz + C, &g) || dense_stages(g, d, C) < 2) return false;
  *o = g;
  return true;
}

}  // namespace fcns
