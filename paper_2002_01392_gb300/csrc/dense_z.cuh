// Dense z operators on the tensor cores (float32 lines).
//
// The derivative operators of one continued line are NQ small dense blocks
// per order (dense_geom.hpp).  A tile is 128 lines; for every block the tile's
// part (128 x KQ) is multiplied by the block (KQ x KQ) with tcgen05.mma, lines
// on the M axis (one line per tensor-memory lane), output orbits on N.
//
// Precision: every float32 operand is split into two float16 values, high and
// low (22 bits and a sign, of a line scaled by a power of two into float16's
// range: from a sample of the line, checked against every value), and the
// products high x high, high x low and low x high are accumulated in float32,
// the small ones first (of NQ = 2, whose blocks come in several slabs, apart
// from the large ones) and, where the contraction is short and the time of a
// tile is its loads (KQ <= 48), low x low too.  Error of d/dz against the
// transforms', 2-norm over rough lines: 0.33 to 0.97 for N' from 125 to 575
// (1.01 and 0.92 at N' = 384); with the small products of NQ = 2 added to the
// large sums it was up to 1.16.
//
// On-chip memory sets the shape: the split tile takes 4 bytes per value, 128 x
// 576 x 4 = 288 KB, more than the 227 KB of shared memory, so the high parts
// stay in tensor memory (two per 32-bit column: KQ NQ / 2 <= 288 columns; they
// are the A operand of two of the three products) and the low parts in shared
// memory (147 KB); the accumulators of a chunk of NC output orbits take NQ NC
// <= 192 columns, and the blocks stream from L2 through a ring of slabs (27 KB,
// bulk copies).
//
// Roles (20 warps, 96 registers a thread; one CTA per SM, persistent over tiles):
//   warps 0-15  workers: load and split a tile (four threads per line), then
//               per chunk read the accumulators, combine the parts and store
//   warps 16-17 scouts: scale and continuation values of the next tile's lines,
//               and its rows into L2
//   warp 18     issues the MMAs;  warp 19 issues the bulk copies
// Measured, d/dz and d2/dz2 of 3 x 512^2 x 513 float32: 1.69 ms (0.42 of the
// measured HBM rate), against 2.91 ms for the length-1080 transforms, whose
// arithmetic alone is bounded at 1.25 ms; error against 64 bits 2.1e-6 (2.7e-6).
// A tile takes about 45 us on its SM: 13 us of loading and splitting (latency
// of L2 at 64 KB in flight), then six chunks of 4 us, of which the tensor pipe
// is busy for 1.7 (648 MMAs of 24 to 44 cycles): what is left is the hand-over
// between slabs (about 400 cycles of waits and pipe restart per 27 MMAs).
// Slabs of 27 KB beat 15 KB (1.99 ms) and 9 KB (2.06) for that reason; the
// bulk copies do not bound it (they reach 85 bytes per cycle and SM).
// Streaming hints on the stores and on the tile's loads keep the next tile's
// rows in L2 (1.97 -> 1.70 together with the sampled scale, which saves a
// second pass over the tile).
//
// Every wait is bounded (dz::mbar_wait): after one that runs out the outputs are
// NaN, and the error word is set, which the plan's next call reports.
#pragma once
#include <cuda_fp16.h>

#include "dense_geom.hpp"
#include "engine.cuh"

namespace fcns {

struct DenseArgs {
  DenseGeom g;
  int d, Cc, stages, resident, low_low, orders;   // orders: bit 0 d/dz, bit 1 d2/dz2
  long long per;           // lines of one field: adjacent in memory; the z stride
  long long outer;         // elements between fields
  long long lines;         // all lines
  long long tiles;
  const float* in;
  float* out1;
  float* out2;
  const __half* B;         // blocks of both orders
  long long order_halves;
  const float2* Mr2;
  float f[2];              // output factors (grid spacing and the blocks' scale): a number in [1, 2) times 2^fe
  int fe[2];
  unsigned* err;           // error word (managed memory), may be null
};

#if defined(__CUDACC__) && !defined(FC_HOSTCHECK)

constexpr int kDenseWorkers = 512, kDenseScouts = 64, kDenseThreads = 640;

constexpr float kDenseLimit = 8192.f;    // largest scaled magnitude: a part is a sum of four values, below 2^15
constexpr int kDenseSampleTo = 6;        // the sampled maximum is scaled to [2^6, 2^7): true maxima may be 64 times larger

namespace dz {
__device__ __forceinline__ void workers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kDenseWorkers) : "memory"); }
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// powers of two s1, s2 (s2 = 1 but for tiny lines) that bring a line of largest magnitude mx to [2^to, 2^(to + 1))
__device__ __forceinline__ void line_scale(float mx, int to, float& s1, float& s2) {
  int k = 126;   // a sample of zeros: see the check after the load
  if (mx > 0.f) k = to - (mx < 3.4e38f ? ilogbf(mx) : 128);
  const int k1 = k > 126 ? 126 : k;
  s1 = ldexpf(1.f, k1);
  s2 = ldexpf(1.f, k - k1);
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// bounded wait of a whole warp.  One that runs out (2^24 polls or two seconds) puts its id into the abort flag; once the
// flag is up every wait gives up after 256 polls, so that all roles run their loops to the end (on values that no longer
// mean anything, within the same buffers) and the kernel ends with the error word set.  No loop leaves early: the loops'
// control flow stays uniform, which the operands of the MMAs need.  A failed poll returns at once, in about 15 cycles:
// the many warps that can wait a little sleep between polls, so as not to take the issue slots of the one that feeds the
// tensor cores.
template <int SLEEP = 0>
__device__ __forceinline__ void mbar_wait(unsigned bar, unsigned parity, volatile int* abort, int id, bool leave = true) {
  unsigned long long t0 = 0;
  bool done = mbar_try(bar, parity);
  for (int i = 1; !done && i < (1 << 24); ++i) {
    if (SLEEP) __nanosleep(SLEEP);
    done = mbar_try(bar, parity);
    if ((i & 255) == 0) {
      const unsigned long long t = now_ns();
      if (!t0) t0 = t;
      if ((leave && *abort) || t - t0 > 2000000000ull) break;
    }
  }
  if (!done && !*abort) *abort = id;
  __syncwarp();
}
__device__ __forceinline__ void bulk_g2s(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// one lane of a converged warp
__device__ __forceinline__ bool elect() {
  unsigned p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void mma_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// descriptor of a shared-memory operand, K-major, no swizzle: core matrices of 8 rows x 16 bytes, `lbo` bytes apart
// along K and 128 bytes apart along the rows (low word: address and lbo in 16-byte units; high word: 128 bytes, version)
__device__ __forceinline__ unsigned desc_lo(unsigned addr, unsigned lbo) { return ((addr >> 4) & 0x3fff) | ((lbo >> 4) << 16); }
constexpr unsigned kDescHi = (128u >> 4) | (1u << 14);
// d (+)= a b, issued by one thread; acc = 0 overwrites d.  A from shared memory (ss) or tensor memory (ts), operands as
// low descriptor words
__device__ __forceinline__ void mma_ss(unsigned d, unsigned a, unsigned b, unsigned idesc, unsigned acc) {
  asm volatile(
      "{\n.reg .pred p;\n.reg .b64 da, db;\nsetp.ne.u32 p, %4, 0;\nmov.b64 da, {%1, %5};\nmov.b64 db, {%2, %5};\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}" ::"r"(d),
      "r"(a), "r"(b), "r"(idesc), "r"(acc), "r"(kDescHi)
      : "memory");
}
__device__ __forceinline__ void mma_ts(unsigned d, unsigned a, unsigned b, unsigned idesc, unsigned acc) {
  asm volatile(
      "{\n.reg .pred p;\n.reg .b64 db;\nsetp.ne.u32 p, %4, 0;\nmov.b64 db, {%2, %5};\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n}" ::"r"(d),
      "r"(a), "r"(b), "r"(idesc), "r"(acc), "r"(kDescHi)
      : "memory");
}
// the products of one slab of n 16-steps (straight-line code: what one lane issues per MMA has to stay below the 31 cycles
// it takes): the small ones, low x high and high x low (and low x low where LL), into ds, then high x high into d, which may
// be the same; then the arrivals on barriers be (slab read) and ba (accumulators done), where not 0
template <int n, bool LL>
__device__ __forceinline__ void issue_slab(unsigned d, unsigned ds, unsigned as, unsigned at, unsigned bh, unsigned bl,
                                           unsigned inc, unsigned idesc, unsigned acc, unsigned be, unsigned ba) {
  if (elect()) {
    if (LL) {
#pragma unroll
      for (int k = 0; k < n; ++k) mma_ss(ds, as + k * (kDenseLines * 2), bl + k * inc, idesc, k > 0 ? 1 : acc);
    }
#pragma unroll
    for (int k = 0; k < n; ++k) mma_ss(ds, as + k * (kDenseLines * 2), bh + k * inc, idesc, LL || k > 0 ? 1 : acc);
#pragma unroll
    for (int k = 0; k < n; ++k) mma_ts(ds, at + 8 * k, bl + k * inc, idesc, 1);
#pragma unroll
    for (int k = 0; k < n; ++k) mma_ts(d, at + 8 * k, bh + k * inc, idesc, k > 0 || d == ds ? 1 : acc);
    if (be) mma_commit(be);
    if (ba) mma_commit(ba);
  }
}
template <bool LL>
__device__ __forceinline__ void issue_slab(int n, unsigned d, unsigned ds, unsigned as, unsigned at, unsigned bh, unsigned bl,
                                           unsigned inc, unsigned idesc, unsigned acc, unsigned be, unsigned ba) {
  switch (n) {
    case 1: issue_slab<1, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
    case 2: issue_slab<2, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
    case 3: issue_slab<3, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
    case 4: issue_slab<4, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
    case 5: issue_slab<5, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
    case 6: issue_slab<6, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
    case 7: issue_slab<7, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
    case 8: issue_slab<8, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
    default: issue_slab<9, LL>(d, ds, as, at, bh, bl, inc, idesc, acc, be, ba); break;
  }
}
__device__ __forceinline__ void tmem_st4(unsigned addr, const unsigned (&v)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[0]), "r"(v[1]),
               "r"(v[2]), "r"(v[3])
               : "memory");
}
__device__ __forceinline__ void tmem_ld4(unsigned addr, float* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
// (h + l) += (m.x + m.y) x for two values of x: the float-float sum of fft_reg.cuh (ff_fma), packed
__device__ __forceinline__ void ff2_fma(float2& h, float2& l, float2 m, float2 x) {
  const float2 mh = make_float2(m.x, m.x), p = __fmul2_rn(mh, x);
  const float2 e = __ffma2_rn(mh, x, make_float2(-p.x, -p.y));
  const float2 t = add2(h, p), z = sub2(t, h);
  const float2 r = add2(sub2(h, sub2(t, z)), sub2(p, z));
  h = t;
  l = add2(l, add2(add2(r, e), __fmul2_rn(make_float2(m.y, m.y), x)));
}
// s as two pairs of float16: high and low parts of two K-adjacent values
__device__ __forceinline__ void split2(float2 s, unsigned& hi, unsigned& lo) {
  const __half2 h = __float22half2_rn(s);
  const __half2 l = __float22half2_rn(sub2(s, __half22float2(h)));
  hi = *reinterpret_cast<const unsigned*>(&h);
  lo = *reinterpret_cast<const unsigned*>(&l);
}
}  // namespace dz

template <int NQ, int D>
__global__ void __launch_bounds__(kDenseThreads, 1) dense_z_kernel(const __grid_constant__ DenseArgs a, const DenseSmem so) {
  extern __shared__ __align__(128) unsigned char sm[];
  const DenseGeom& g = a.g;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const unsigned smb = dz::smem_u32(sm);
  const unsigned bfull = smb + so.bars, bempty = bfull + 64, bAcc = bempty + 64, bFree = bAcc + 32, bA = bFree + 32,
                 bSf = bA + 8, bSe = bA + 16, bEnd = bA + 24;
  volatile int* abort = reinterpret_cast<int*>(sm + so.bars + 8 * kDenseBars);
  unsigned* tmem_slot = reinterpret_cast<unsigned*>(sm + so.bars + 8 * kDenseBars + 8);
  float* cont = reinterpret_cast<float*>(sm + so.cont);
  float* scale = reinterpret_cast<float*>(sm + so.scale);   // power of two per line, and a second one (1 but for tiny lines)
  float2* mr = reinterpret_cast<float2*>(sm + so.mr);
  int* lmax = reinterpret_cast<int*>(sm + so.lmax);         // per line, used by a second load only
  volatile int* redo = lmax + kDenseLines;                  // tile `it` of this CTA is loaded again (slot it & 1)
  if (tid == 0) {
    *abort = 0;
    for (int i = 0; i < 8; ++i) {
      dz::mbar_init(bfull + 8 * i, 1);
      dz::mbar_init(bempty + 8 * i, 1);
    }
    for (int q = 0; q < 4; ++q) {
      dz::mbar_init(bAcc + 8 * q, 1);
      dz::mbar_init(bFree + 8 * q, kDenseWorkers);
    }
    dz::mbar_init(bA, kDenseWorkers);
    dz::mbar_init(bSf, kDenseScouts);
    dz::mbar_init(bSe, kDenseWorkers);
    dz::mbar_init(bEnd, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < a.Cc * a.d; i += kDenseThreads) mr[i] = a.Mr2[i];
  if (tid < kDenseLines + 4) lmax[tid] = 0;
  if (warp == 18) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(dz::smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  dz::fence_before();
  __syncthreads();
  dz::fence_after();
  const unsigned tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const unsigned hiw = (unsigned)(NQ * g.KQ / 2);          // columns of the high parts; the accumulators follow
  const int nord = (a.orders & 1) + (a.orders >> 1);
  const int slabB = dense_slab_bytes(g);
  // Of NQ = 2, the small products have accumulators of their own: added to the large sums of the slabs before, they would
  // lose what the tensor cores cut off (not rounded) below 2^-24 of the sum.  A block of NQ = 4 is one slab.
  constexpr int acc_sets = NQ == 2 ? 2 : 1;

  if (warp < 16) {
    // ------------------------------------------------------------- workers
    const int line = (warp & 3) * 32 + lane, sub = warp >> 2;
    const unsigned tl = tmem + ((unsigned)((warp & 3) * 32) << 16);
    unsigned step = 0;
    int it = 0;
    for (long long tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, ++it) {
      const long long L = tile * kDenseLines + line;
      const bool valid = L < a.lines;
      const long long grp = valid ? L / a.per : 0, off = valid ? L % a.per : 0;
      const float* in = a.in + grp * a.outer + off;
      dz::mbar_wait<64>(bSf, it & 1, abort, 1);
      float s1 = scale[line], s2 = scale[kDenseLines + line];
      bool tiny = __any_sync(0xffffffffu, s2 != 1.f);
      float mx = 0.f;
      // --- load, form the parts and split: groups of 8 orbits, every fourth one
      float x[NQ][8];
      auto fetch = [&](int q8) {
        const int j0 = q8 * 8;
        bool pure = j0 + 8 <= g.No;
        int r0[NQ];
#pragma unroll
        for (int i = 0; i < NQ; ++i) {   // rows move by one per orbit: the group's ends (and a wrap between them)
          r0[i] = dense_row(g, j0, i);
          const int r1 = dense_row(g, j0 + 7, i);
          pure = pure && r0[i] < g.Nz && r1 < g.Nz && (r1 - r0[i] == 7 || r0[i] - r1 == 7);
        }
        if (pure) {
#pragma unroll
          for (int i = 0; i < NQ; ++i) {
            const float* p = in + (long long)r0[i] * a.per;
            const long long st = (i & 1) ? -a.per : a.per;
#pragma unroll
            for (int k = 0; k < 8; ++k, p += st) x[i][k] = __ldcs(p);
          }
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
              const int r = dense_row(g, j0 + k, i);
              float v = 0.f;
              if (j0 + k < g.No) v = r < g.Nz ? __ldcg(in + (long long)r * a.per) : cont[(r - g.Nz) * kDenseLines + line];
              x[i][k] = v;
            }
        }
      };
      auto load_tile = [&] {
      for (int q8 = sub; q8 < g.KQ / 8; q8 += 4) {
        fetch(q8);
#pragma unroll
        for (int i = 0; i < NQ; ++i)
#pragma unroll
          for (int k = 0; k < 8; ++k) mx = fmaxf(mx, fabsf(x[i][k]));
        unsigned hi[NQ][4], lo[NQ][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float2 v[NQ];
#pragma unroll
          for (int i = 0; i < NQ; ++i) {
            v[i] = __fmul2_rn(make_float2(x[i][2 * k], x[i][2 * k + 1]), make_float2(s1, s1));
            if (tiny) v[i] = __fmul2_rn(v[i], make_float2(s2, s2));
          }
          const float2 p = dz::add2(v[0], v[1]), m = dz::sub2(v[0], v[1]);   // mirror sums and differences
          if constexpr (NQ == 4) {
            const float2 p2 = dz::add2(v[2], v[3]), m2 = dz::sub2(v[2], v[3]);
            dz::split2(dz::add2(p, p2), hi[0][k], lo[0][k]);
            dz::split2(dz::add2(m, m2), hi[1][k], lo[1][k]);
            dz::split2(dz::sub2(p, p2), hi[2][k], lo[2][k]);
            dz::split2(dz::sub2(m, m2), hi[3][k], lo[3][k]);
          } else {
            dz::split2(p, hi[0][k], lo[0][k]);
            dz::split2(m, hi[1][k], lo[1][k]);
          }
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          dz::tmem_st4(tl + (unsigned)(q * (g.KQ / 2) + q8 * 4), hi[q]);
          *reinterpret_cast<uint4*>(sm + so.lo + ((size_t)(q * (g.KQ / 8) + q8) * kDenseLines + line) * 16) =
              make_uint4(lo[q][0], lo[q][1], lo[q][2], lo[q][3]);
        }
      }
      };
      load_tile();
      // the scale came from a sample of the line: where a value passes the limit all the same (the float16 parts of the
      // sums have to stay below 2^16), the tile is loaded again, that line with the scale of its true maximum
      auto too_large = [&](float m) { return m * s1 * s2 > kDenseLimit || (m > 0.f && s1 == 0x1p126f && s2 == 1.f); };
      if (tid == 0) redo[(it + 1) & 1] = 0;
      if (too_large(mx)) redo[it & 1] = 1;
      dz::workers_sync();
      if (redo[it & 1]) {
        atomicMax(lmax + line, __float_as_int(mx));   // (non-negative floats order like their bits)
        // the first pass's tensor-memory stores are asynchronous and go to the columns the second one writes again
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        dz::workers_sync();
        // only the lines that passed it get another scale: a line's bits do not depend on its neighbours in the tile
        const float all = __int_as_float(lmax[line]);
        if (too_large(all)) dz::line_scale(all, 12, s1, s2);
        tiny = __any_sync(0xffffffffu, s2 != 1.f);
        load_tile();
        dz::workers_sync();
        if (sub == 0) lmax[line] = 0;
      }
      const int scaled = (__float_as_int(s1) >> 23) + (__float_as_int(s2) >> 23) - 254;   // the line is scaled by 2^scaled
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      dz::fence_before();
      dz::mbar_arrive(bSe);
      dz::mbar_arrive(bA);
      // --- outputs, chunk by chunk
      const int ng = g.NC / 16;   // groups of 4 orbits of this thread's quarter of a chunk
      constexpr int MG = 3;
      for (int o = 0; o < 2; ++o) {
        if (!(a.orders >> o & 1)) continue;
        float* out = (o == 0 ? a.out1 : a.out2) + grp * a.outer + off;
        // the factor undoes the line's scale: a.f 2^K.  Where that or a part times it could leave float's range, the
        // accumulators take most of it first (by 1 for the other lines of the warp: a line's bits do not depend on them)
        const int K = a.fe[o] - scaled, K1 = min(max(K, -100), 100);
        const bool far = K < -80 || K > 80;
        const bool steps = __any_sync(0xffffffffu, far);
        const float fa = far ? __int_as_float((min(max(K - K1, -126), 127) + 127) << 23) : __int_as_float(__float_as_int(a.f[o]) + (K << 23));
        const float par = o == 0 ? -1.f : 1.f;
        for (int c = 0; c < g.chunks; ++c, ++step) {
          // each part's accumulators are handed back as soon as they are read, so that the MMAs of the next chunk
          // follow those of this one without a gap
          float y[MG][NQ][4];
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            dz::mbar_wait<32>(bAcc + 8 * q, step & 1, abort, 2);
            dz::fence_after();
#pragma unroll
            for (int k = 0; k < MG; ++k)
              if (k < ng) dz::tmem_ld4(tl + hiw + (unsigned)(q * acc_sets * g.NC + (sub * ng + k) * 4), y[k][q]);
            float small[MG][4];
            if constexpr (acc_sets == 2) {
#pragma unroll
              for (int k = 0; k < MG; ++k)
                if (k < ng) dz::tmem_ld4(tl + hiw + (unsigned)((2 * q + 1) * g.NC + (sub * ng + k) * 4), small[k]);
            }
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if constexpr (acc_sets == 2) {
#pragma unroll
              for (int k = 0; k < MG; ++k)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  asm volatile("" : "+f"(y[k][q][e]), "+f"(small[k][e]));   // (the sum stays behind the wait)
                  if (k < ng) y[k][q][e] += small[k][e];
                }
            }
            dz::fence_before();
            dz::mbar_arrive(bFree + 8 * q);
          }
          // (a role that gives up sets the flag before it goes on, so what came of it is read behind it)
          const float fb = *abort ? __int_as_float(0x7fc00000) : fa;
          if (steps) {
            const int K = a.fe[o] - scaled;
            const float f1 = K < -80 || K > 80 ? a.f[o] * __int_as_float((min(max(K, -100), 100) + 127) << 23) : 1.f;
#pragma unroll
            for (int k = 0; k < MG; ++k)
#pragma unroll
              for (int q = 0; q < NQ; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if (k < ng) y[k][q][e] *= f1;
          }
          if (!valid) continue;
#pragma unroll
          for (int k = 0; k < MG; ++k) {
            const int j0 = c * g.NC + (sub * ng + k) * 4;
            if (k < ng && j0 < g.No) {
              // the members' values, in place
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                float(&Y)[NQ][4] = y[k];
                if constexpr (NQ == 4) {
                  const float P = (Y[0][e] + Y[2][e]) * fb, M = (Y[0][e] - Y[2][e]) * fb;
                  const float R = Y[1][e] + Y[3][e], S = Y[1][e] - Y[3][e];
                  Y[0][e] = fmaf(R, fb, P);
                  Y[1][e] = par * fmaf(-R, fb, P);
                  Y[2][e] = fmaf(S, fb, M);
                  Y[3][e] = par * fmaf(-S, fb, M);
                } else {
                  const float P = Y[0][e] * fb, R = Y[1][e];
                  Y[0][e] = fmaf(R, fb, P);
                  Y[1][e] = par * fmaf(-R, fb, P);
                }
              }
#pragma unroll
              for (int i = 0; i < NQ; ++i) {
                const int w0 = dense_row(g, j0, i), w1 = dense_row(g, j0 + 3, i);
                if (j0 + 4 <= g.No && w0 < g.Nz && w1 < g.Nz && (w1 - w0 == 3 || w0 - w1 == 3)) {
                  float* p = out + (long long)w0 * a.per;
                  const long long st = (i & 1) ? -a.per : a.per;
#pragma unroll
                  for (int e = 0; e < 4; ++e, p += st) __stcs(p, y[k][i][e]);
                } else {
#pragma unroll
                  for (int e = 0; e < 4; ++e) {
                    const int r = dense_row(g, j0 + e, i);
                    if (j0 + e < g.No && r < g.Nz) __stcs(out + (long long)r * a.per, y[k][i][e]);
                  }
                }
              }
            }
          }
        }
      }
    }
  } else if (warp < 18) {
    // ------------------------------------------------ scouts (two lines each)
    const int line0 = (warp - 16) * 32 + lane;
    int it = 0;
    for (long long tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, ++it) {
      const float* in[2];
      bool valid[2];
      float mx[2] = {0.f, 0.f};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const long long L = tile * kDenseLines + line0 + 64 * u;
        valid[u] = L < a.lines;
        in[u] = a.in + (valid[u] ? (L / a.per) * a.outer + L % a.per : 0);   // (an absent line reads the first one)
      }
      // this tile's rows into L2 while the workers are busy with the one before: a prefetch per 128 bytes, eight rows at
      // a time
      const long long Ln = tile * kDenseLines + 32 * (lane & 3);
      if (Ln < a.lines) {
        const float* nx = a.in + (Ln / a.per) * a.outer + Ln % a.per;
        for (int n = (warp - 16) * 8 + (lane >> 2); n < g.Nz; n += 16) prefetch_l2(nx + (long long)n * a.per);
      }
      // a sample of the line for its scale: at most 32 rows
      const int every = (g.Nz + 31) / 32;
      const long long skip = a.per * every;
      const float *p0 = in[0], *p1 = in[1];
#pragma unroll 16
      for (int n = 0; n < g.Nz; n += every, p0 += skip, p1 += skip) {
        mx[0] = fmaxf(mx[0], fabsf(__ldcg(p0)));
        mx[1] = fmaxf(mx[1], fabsf(__ldcg(p1)));
      }
      if (it > 0) dz::mbar_wait<64>(bSe, (it - 1) & 1, abort, 3);
      // continuation (Sec. 3): M_r f_last + its mirror on f_first, in float
      // pairs, both lines in one packed operation; values jj and C - 1 - jj
      // share their matrix entries
      constexpr int DM = D > 0 ? D : 10;
      const int d = D > 0 ? D : a.d;
      float2 first[DM], last[DM];
#pragma unroll
      for (int i = 0; i < DM; ++i) {
        const long long of = (long long)i * a.per, ol = (long long)(g.Nz - d + i) * a.per;
        first[i] = i < d ? make_float2(__ldcg(in[0] + of), __ldcg(in[1] + of)) : make_float2(0.f, 0.f);
        last[i] = i < d ? make_float2(__ldcg(in[0] + ol), __ldcg(in[1] + ol)) : make_float2(0.f, 0.f);
      }
      for (int jj = 0; 2 * jj < a.Cc; ++jj) {
        float2 h[2] = {}, l[2] = {};   // value jj and its mirror: high and low sums
#pragma unroll
        for (int i = 0; i < DM; ++i)
          if (i < d) {
            const float2 m1 = mr[jj * d + i], m2 = mr[(a.Cc - 1 - jj) * d + (d - 1 - i)];
            const float2 n1 = mr[(a.Cc - 1 - jj) * d + i], n2 = mr[jj * d + (d - 1 - i)];
            dz::ff2_fma(h[0], l[0], m1, last[i]);
            dz::ff2_fma(h[1], l[1], n1, last[i]);
            dz::ff2_fma(h[0], l[0], m2, first[i]);
            dz::ff2_fma(h[1], l[1], n2, first[i]);
          }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float2 v = dz::add2(h[u], l[u]);
          const int row = u == 0 ? jj : a.Cc - 1 - jj;
          mx[0] = fmaxf(mx[0], fabsf(v.x));
          mx[1] = fmaxf(mx[1], fabsf(v.y));
          cont[row * kDenseLines + line0] = v.x;
          cont[row * kDenseLines + line0 + 64] = v.y;
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float s1, s2;
        dz::line_scale(mx[u], kDenseSampleTo, s1, s2);
        scale[line0 + 64 * u] = s1;
        scale[kDenseLines + line0 + 64 * u] = s2;
      }
      dz::mbar_arrive(bSf);
    }
  } else if (warp == 18) {
    // ----------------------------------------------------------------- MMA
    // the whole warp runs the loops (votes keep them uniform, so that operands stay in uniform registers: a lane that
    // loops by itself issued an MMA every 70 cycles, against 31 for the tensor pipe itself); the elected lane issues
    const unsigned idesc = (1u << 4) | ((unsigned)(g.NC >> 3) << 17) | ((unsigned)(kDenseLines >> 4) << 24);
    const unsigned kstep = 32u * (unsigned)g.NC, lbo = 16u * (unsigned)g.NC, inc = kstep >> 4;
    unsigned step = 0, st = 0, ph = 0;
    int it = 0;
    for (long long tile = blockIdx.x; tile < a.tiles; tile += gridDim.x, ++it) {
      dz::mbar_wait(bA, it & 1, abort, 4);
      if (a.resident) st = 0;
      for (int oc = 0; oc < nord * g.chunks; ++oc, ++step) {
        unsigned dcol = tmem + hiw, ahi = tmem, alo = smb + so.lo;
        for (int q = 0; q < NQ; ++q) {
          unsigned acc = 0;
          if (step > 0) dz::mbar_wait(bFree + 8 * q, (step - 1) & 1, abort, 5);
          for (int s = 0; s < g.slabs; ++s) {
            if (!a.resident || it == 0) dz::mbar_wait(bfull + 8 * st, ph, abort, 6);
            dz::fence_after();
            const int n = dense_slab(g, s);
            const unsigned bh = smb + so.ring + st * slabB, bl = bh + (unsigned)n * kstep;
            const unsigned da = dz::desc_lo(alo, kDenseLines * 16), dh = dz::desc_lo(bh, lbo), dl = dz::desc_lo(bl, lbo);
            const unsigned ds = dcol + (NQ == 2 ? (unsigned)g.NC : 0u);
            const unsigned be = a.resident ? 0u : bempty + 8 * st, ba = s == g.slabs - 1 ? bAcc + 8 * q : 0u;
            if (NQ == 4 && a.low_low) dz::issue_slab<true>(n, dcol, ds, da, ahi, dh, dl, inc, idesc, acc, be, ba);
            else dz::issue_slab<false>(n, dcol, ds, da, ahi, dh, dl, inc, idesc, acc, be, ba);
            __syncwarp();
            acc = 1;
            alo += (unsigned)n * (2 * kDenseLines * 16);
            ahi += 8 * (unsigned)n;
            if (++st == (unsigned)a.stages && !a.resident) {
              st = 0;
              ph ^= 1;
            }
          }
          dcol += (unsigned)(acc_sets * g.NC);
        }
      }
    }
    // nothing of this CTA's tensor work is in flight when its memory goes
    if (dz::elect()) dz::mma_commit(bEnd);
    __syncwarp();
    dz::mbar_wait(bEnd, 0, abort, 7, false);
  } else {
    // ---------------------------------------------------------- bulk copies
    unsigned st = 0, round = 0, use = 0;
    const long long ntiles = a.resident ? blockIdx.x + 1 : a.tiles;   // a resident block set is loaded for the first tile only
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      for (int o = 0; o < 2; ++o) {
        if (!(a.orders >> o & 1)) continue;
        const __half* b = a.B + o * a.order_halves;
        for (int cq = 0; cq < g.chunks * NQ; ++cq)
          for (int s = 0; s < g.slabs; ++s) {
            const unsigned bytes = (unsigned)(dense_slab(g, s) * 16 * g.NC * 4);
            if (round > 0) dz::mbar_wait(bempty + 8 * st, (round - 1) & 1, abort, 8);
            if (dz::elect()) {
              dz::mbar_expect(bfull + 8 * st, bytes);
              dz::bulk_g2s(smb + so.ring + st * slabB, b, bytes, bfull + 8 * st);
            }
            __syncwarp();
            b += bytes / 2;
            ++use;
            if (++st == (unsigned)a.stages) {
              st = 0;
              ++round;
            }
          }
      }
    }
    // the last copies have landed
    const unsigned first = use > (unsigned)a.stages ? use - (unsigned)a.stages : 0;
    for (unsigned u = first; u < use; ++u)
      dz::mbar_wait(bfull + 8 * (u % (unsigned)a.stages), (u / (unsigned)a.stages) & 1, abort, 9, false);
  }
  dz::fence_before();
  __syncthreads();
  dz::fence_after();
  if (warp == 18) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  if (tid == 0 && *abort && a.err) {
    *a.err = (unsigned)*abort;   // which wait gave up first
    __threadfence_system();
  }
}

#endif  // __CUDACC__

}  // namespace fcns
