// fc_deriv_z in float64 by the dense operators (dense64.hpp): the exact integer
// products run on the tensor cores instead of transforms on the float64 pipe,
// which does 1.8 operations per cycle and SM and bounds the transform kernel.
#include <atomic>
#include <cmath>

#include <cuda_fp16.h>

#include "dense64.hpp"
#include "dense_build.cuh"
#include "internal.hpp"

namespace fcns {
namespace {

constexpr int kD64Threads = 256;

struct Dense64Args {
  DenseGeom g;
  int d, Cc, orders;          // orders: bit 0 d/dz, bit 1 d2/dz2
  long long per, outer;       // lines per field, values per field
  long long lines, tiles;     // all lines
  const double* in;
  double* out[2];
  const uint4* B;             // fragments of both orders
  long long order_words;      // uint4 per order
  const double* Mr;
  double f[2];                // scale factor mantissa and exponent (with the operator's and the sums' units)
  int k[2];
  int sh[2];
};

// One CTA walks tiles of 16 lines.  Bound: the tensor pipe (36 products of 16 x
// 8 x 16 per fragment pair), then the operators' fragments out of L2 (2.65 MB per
// tile at N' = 538).  16 lines because the digits of all NQ parts have to be in
// shared memory together (an output row is a sum over the parts): 147 KB, beside
// the line itself (69 KB), into which the next tile is copied while the products run.
// A warp owns 16 orbits of one order: eight float32 sums of 16 x 16 values, and
// 4 x 8 whole numbers per thread for the rows of its orbits.
// mma.sync, not tcgen05: the eight sums and the digits of 128 lines would need
// four times the tensor memory of an SM.
// Measured, 3 x 256^2 x 513: transforms 24.4 ms, this 8.36; 513 x 32k lines 4104
// -> 1467 us (with seven digits, where the error exceeded the transform's,
// 1309, the tensor pipe 48 % busy; without the next step's fragments read ahead
// 1410).  The rest: splitting the line into digits, which overlaps nothing (15
// %), 18 items over 8 warps (10 %), the issue distance of two warps per
// scheduler.  Error 3 to 30 times below the transform's.
template <int NQ>
__global__ void __launch_bounds__(kD64Threads, 1) dense64_kernel(const __grid_constant__ Dense64Args a) {
  extern __shared__ __align__(16) unsigned char sm[];
  const DenseGeom& g = a.g;
  const int KT = g.KQ / 16, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint4* A = reinterpret_cast<uint4*>(sm);                                    // [NQ][KT][8][32]
  unsigned long long* X = reinterpret_cast<unsigned long long*>(A + NQ * KT * kD64Digits * 32);   // [N'][16]
  double* scale = reinterpret_cast<double*>(X + g.Np * kD64Lines);            // [2][2][16]
  unsigned* top = reinterpret_cast<unsigned*>(scale + 4 * kD64Lines);         // [16] largest high word
  int* slow = reinterpret_cast<int*>(top + kD64Lines);
  const int li = tid & 15, r0 = tid >> 4;

  auto copy_in = [&](long long tile) {
    const long long ln = tile * kD64Lines + li;
    const bool ok = ln < a.lines;
    const double* src = a.in + (ok ? ln / a.per * a.outer + ln % a.per : 0);
    const unsigned dst = (unsigned)__cvta_generic_to_shared(X + li), bytes = ok ? 8 : 0;
    for (int n = r0; n < g.Nz; n += kD64Threads / 16)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst + n * kD64Lines * 8),
                   "l"(src + (ok ? n * a.per : 0)), "r"(bytes)
                   : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  copy_in(blockIdx.x);
  for (long long tile = blockIdx.x; tile < a.tiles; tile += gridDim.x) {
    if (tid < kD64Lines) top[tid] = 1u << 20;
    if (tid == 0) *slow = 0;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // largest magnitude of every line, by the high words
    unsigned most = 0;
    for (int n = r0; n < g.Nz; n += kD64Threads / 16)
      most = max(most, (unsigned)(X[n * kD64Lines + li] >> 32) & 0x7fffffffu);
    // ... and of its continuation (Sec. 3)
    for (int jj = r0; jj < a.Cc; jj += kD64Threads / 16) {
      const unsigned long long v =
          d64_continuation(jj, a.d, a.Cc, a.Mr, X + li, X + (g.Nz - a.d) * kD64Lines + li, kD64Lines);
      X[(g.Nz + jj) * kD64Lines + li] = v;
      most = max(most, (unsigned)(v >> 32) & 0x7fffffffu);
    }
    most = max(most, __shfl_xor_sync(0xffffffffu, most, 16));
    if (lane < 16) atomicMax(top + li, most);
    __syncthreads();
    if (tid < 2 * kD64Lines) {   // scale of the outputs; a line with Inf or NaN gives NaN
      const int o = tid >> 4, E = (int)(top[li] >> 20);
      const int k = a.k[o] + E, k1 = min(max(k, -960), 900), k2 = min(max(k - k1, -1022), 1023);
      scale[o * 32 + li] = E == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
                                      : a.f[o] * __longlong_as_double((long long)(k1 + 1023) << 52);
      scale[o * 32 + 16 + li] = __longlong_as_double((long long)(k2 + 1023) << 52);
      if (k2) *slow = 1;
    }
    // parts and digits, two orbits of one line per thread and turn
    {
      const int E = (int)(top[li] >> 20);
      __half2* Ah = reinterpret_cast<__half2*>(A);
      for (int jp = r0; jp < g.KQ / 2; jp += kD64Threads / 16) {
        long long u[2][NQ];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int j = 2 * jp + h;
          long long x[NQ];
#pragma unroll
          for (int i = 0; i < NQ; ++i)
            x[i] = j < g.No && E < 0x7ff ? d64_fixed(X[dense_row(g, j, i) * kD64Lines + li], E) : 0;
          const long long p0 = x[0] + x[1], p1 = x[0] - x[1];
          if constexpr (NQ == 4) {
            const long long s0 = x[2] + x[3], s1 = x[2] - x[3];
            u[h][0] = p0 + s0;
            u[h][1] = p1 + s1;
            u[h][2] = p0 - s0;
            u[h][3] = p1 - s1;
          } else {
            u[h][0] = p0;
            u[h][1] = p1;
          }
        }
        const int at = d64_a_index(li, 2 * jp & 15) / 2, ks = jp >> 3;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const unsigned long long w0 = d64_bias(u[0][q]), w1 = d64_bias(u[1][q]);
#pragma unroll
          for (int i = 0; i < kD64Digits; ++i) {
            // 1024 + field as float16 bits, less 1152: exact
            const unsigned bits = 0x64006400u | (unsigned)d64_field(w0, i) | (unsigned)d64_field(w1, i) << 16;
            Ah[((q * KT + ks) * kD64Digits + i) * 128 + at] =
                __hsub2(*reinterpret_cast<const __half2*>(&bits), __half2half2(__ushort_as_half(0x6480)));
          }
        }
      }
    }
    __syncthreads();
    if (tile + gridDim.x < a.tiles) copy_in(tile + gridDim.x);

    // lines of this thread's outputs: lane / 4 and 8 more
    long long at[2];
    bool there[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const long long ln = tile * kD64Lines + (lane >> 2) + 8 * h;
      there[h] = ln < a.lines;
      at[h] = there[h] ? ln / a.per * a.outer + ln % a.per : 0;
    }
    const int first = a.orders & 1 ? 0 : KT, last = a.orders & 2 ? 2 * KT : KT;
    for (int item = first + blockIdx.y + gridDim.y * warp; item < last; item += gridDim.y * (kD64Threads / 32)) {
      const int o = item >= KT, nt = item - o * KT;
      const uint4* B = a.B + o * a.order_words + (long long)nt * NQ * KT * kD64Digits * 32 + lane;
      long long row[NQ][8] = {};
      // fragments of the next step are read as soon as the registers of this
      // one's are free; they follow one another over q and ks
      const uint4* Af = A + lane;
      uint4 x[kD64Digits], b[kD64Digits];
#pragma unroll
      for (int i = 0; i < kD64Digits; ++i) {
        b[i] = __ldg(B + i * 32);
        x[i] = Af[i * 32];
      }
#pragma unroll 1
      for (int q = 0; q < NQ; ++q) {
        float c[kD64Sums][8] = {};
#pragma unroll 1
        for (int ks = 0; ks < KT; ++ks) {
          const int step = q < NQ - 1 || ks < KT - 1 ? kD64Digits * 32 : 0;   // (the last step reads its own again)
          B += step;
          Af += step;
#pragma unroll
          for (int j = 0; j < kD64Digits; ++j) {
            // digits x[1] and x[0] come last: theirs are the youngest loads
#pragma unroll
            for (int i = kD64Sums - 1 - j; i >= 0; --i) {
              float* s = c[i + j];
              asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                  : "+f"(s[0]), "+f"(s[1]), "+f"(s[2]), "+f"(s[3])
                  : "r"(x[i].x), "r"(x[i].y), "r"(x[i].z), "r"(x[i].w), "r"(b[j].x), "r"(b[j].y));
              asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                  : "+f"(s[4]), "+f"(s[5]), "+f"(s[6]), "+f"(s[7])
                  : "r"(x[i].x), "r"(x[i].y), "r"(x[i].z), "r"(x[i].w), "r"(b[j].z), "r"(b[j].w));
            }
            b[j] = __ldg(B + j * 32);
            x[kD64Sums - 1 - j] = Af[(kD64Sums - 1 - j) * 32];
          }
        }
        // signs of the rows of an orbit: part q and the operator's own parity
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          int s[kD64Sums];
#pragma unroll
          for (int i = 0; i < kD64Sums; ++i) s[i] = __float2int_rn(c[i][v]);
          const long long y = d64_combine(s, a.sh[o]);
#pragma unroll
          for (int i = 0; i < NQ; ++i) {
            const int neg = (__popc(q & i) + (o == 0 ? i : 0)) & 1;
            row[i][v] += neg ? -y : y;
          }
        }
      }
      double* out = a.out[o];
      const bool two = *slow;
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const int h = (v >> 1) & 1, l = (lane >> 2) + 8 * h;
        const int j = nt * 16 + 8 * (v >> 2) + 2 * (lane & 3) + (v & 1);
        if (!there[h] || j >= g.No) continue;
        const double sc = scale[o * 32 + l], sc2 = scale[o * 32 + 16 + l];
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
          const int n = dense_row(g, j, i);
          if (n >= g.Nz) continue;
          double y = (double)row[i][v] * sc;
          if (two) y *= sc2;
          __stcs(out + at[h] + n * a.per, y);
        }
      }
    }
    __syncthreads();
  }
}

__global__ void dense64_build_kernel(const __grid_constant__ DenseGeom g, const long long* __restrict__ c, __half* out) {
  const long long n = dense64_pairs(g), i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * n) return;
  const int o = i >= n;
  dense64_pair(g, c + o * g.Np, i - o * n, out + o * dense64_order_halves(g));
}

}  // namespace

fc_status launch_deriv_dense64(const DerivDevTables& t, const PlanData& p, int batch, long long lines, double Lz,
                               const void* f, void* df, void* d2f, cudaStream_t stream) {
  Dense64Args a = {};
  a.g = p.dense64;
  a.d = p.d;
  a.Cc = p.C;
  a.orders = (df ? 1 : 0) | (d2f ? 2 : 0);
  a.per = lines;
  a.outer = lines * p.Nz;
  a.lines = lines * batch;
  a.tiles = (a.lines + kD64Lines - 1) / kD64Lines;
  a.in = static_cast<const double*>(f);
  a.out[0] = static_cast<double*>(df);
  a.out[1] = static_cast<double*>(d2f);
  a.B = static_cast<const uint4*>(t.dense64);
  a.order_words = dense64_order_halves(a.g) / 8;
  a.Mr = t.Mr;
  const double dz = Lz / (p.Nz - 1), s[2] = {1.0 / dz, 1.0 / (dz * dz)};
  for (int o = 0; o < 2; ++o) {
    int e = 0;
    a.f[o] = std::frexp(s[o], &e);
    a.sh[o] = p.kern.sh[o];
    a.k[o] = 56 + a.sh[o] - 1082 - p.kern.e64[o] + e;
  }
  const size_t smem = (size_t)a.g.NQ * (a.g.KQ / 16) * kD64Digits * 512 + (size_t)a.g.Np * kD64Lines * 8 + 6 * kD64Lines * 8;
  auto kern = a.g.NQ == 4 ? dense64_kernel<4> : dense64_kernel<2>;
  static std::atomic<unsigned long long> attr_set[2];
  static std::atomic<int> sm_count[64];
  int dev = 0;
  cudaGetDevice(&dev);
  std::atomic<unsigned long long>& attr = attr_set[a.g.NQ == 4];
  if (dev >= 64 || !(attr.load() >> dev & 1ull)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute(dense z, float64)");
    if (dev < 64) attr.fetch_or(1ull << dev);
  }
  int sms = dev < 64 ? sm_count[dev].load() : 0;
  if (!sms) {
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_status(e, "cudaDeviceGetAttribute");
    if (dev < 64) sm_count[dev].store(sms);
  }
  // fewer tiles than SMs: the orbits of a tile over several CTAs (each reads and splits the lines for itself), down to
  // one warp per quarter of an SM.  513 x 512 lines: 114 -> 59 us (seven digits)
  const int items = ((df ? 1 : 0) + (d2f ? 1 : 0)) * (a.g.KQ / 16);
  const long long most = (items + 3) / 4, room = a.tiles < sms ? sms / a.tiles : 1;
  const dim3 grid((unsigned)(a.tiles < sms ? a.tiles : sms), (unsigned)(room < most ? room : most));
  kern<<<grid, kD64Threads, smem, stream>>>(a);
  return cuda_status(cudaGetLastError(), "dense z launch (float64)");
}

fc_status launch_dense64_build(const PlanData& p, const long long* c, void* out, cudaStream_t stream) {
  const long long n = 2 * dense64_pairs(p.dense64);
  dense64_build_kernel<<<(unsigned)((n + 127) / 128), 128, 0, stream>>>(p.dense64, c, static_cast<__half*>(out));
  return cuda_status(cudaGetLastError(), "dense z blocks launch (float64)");
}

}  // namespace fcns
