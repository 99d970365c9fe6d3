// Host-check library: runs the kernel phase functions on the CPU, one block
// after another, so that tests without a GPU can compare the kernels' index
// arithmetic and data flow with the oracle.  Not part of libfcns and never
// loaded by the product path.
#define FC_HOSTCHECK 1
#include <cuda_fp16.h>

#include <chrono>
#include <complex>
#include <vector>

#include "deriv_kernel.cuh"
#include "dense_build.cuh"
#include "host_tables.hpp"
#include "slabs.hpp"

namespace fcns {

template <class T, int L1, int L2, int LINES, int JN, bool SYM, int JI = 0, bool FULL = false>
static int emu_deriv_k(const double* Mr, int d, int Cc, int Nz, int batch, long long lines, double Lz,
                       const T* f, T* df, T* d2f) {
  using K = DerivPair<T, L1, L2, LINES, JN, SYM, JI, FULL>;
  const int L = L1 * L2;
  std::vector<std::complex<double>> H1, H2, tw;
  deriv_conv_spectra(Nz, Nz + Cc, L, &H1, &H2);
  engine_twiddles(L1, L2, &tw);
  std::vector<cx<T>> H1t(L), H2t(L), twt(2 * L);
  for (int i = 0; i < L; ++i) {
    H1t[i] = mk<T>((T)H1[i].real(), (T)H1[i].imag());
    H2t[i] = mk<T>((T)H2[i].real(), (T)H2[i].imag());
  }
  for (int i = 0; i < 2 * L; ++i) twt[i] = mk<T>((T)tw[i].real(), (T)tw[i].imag());
  typename K::Args a;
  a.f = f; a.df = df; a.d2f = d2f;
  a.Nz = Nz; a.Np = Nz + Cc; a.d = d; a.Cc = Cc;
  a.lines = lines; a.pairs = (lines + 1) / 2; a.tiles = (a.pairs + LINES - 1) / LINES;
  a.zstride = lines; a.bstride = lines * Nz;
  const double dz = Lz / (Nz - 1);
  a.s1 = T(1.0 / dz); a.s2 = T(1.0 / (dz * dz));
  std::vector<float2> Mr2(Cc * d);
  for (int i = 0; i < Cc * d; ++i) { Mr2[i].x = (float)Mr[i]; Mr2[i].y = (float)(Mr[i] - (double)Mr2[i].x); }
  a.Mr = Mr; a.Mr2 = Mr2.data(); a.H1 = H1t.data(); a.H2 = H2t.data(); a.tw = twt.data();

  a.nblocks = a.tiles * batch;
  a.pf_dist = 3;
  a.vec = lines % 2 == 0 ? 1 : 0;
  phased_emulate<K>(a, a.tiles * batch, K::smem_bytes);
  return 0;
}

// the variant fc_deriv_z launches: symmetric kernel spectra when L >= 2 N' - 1 or L = N'
template <class T, int L1, int L2, int LINES, int JN>
static int emu_deriv(const double* Mr, int d, int Cc, int Nz, int batch, long long lines, double Lz,
                     const T* f, T* df, T* d2f) {
  const int L = L1 * L2, Np = Nz + Cc;
  // the interior-row form fc_deriv_z runs for float32 at L = 1080, Nz >= 481
  if constexpr (sizeof(T) == 4 && L1 == 30 && L2 == 36 && JN == 16)
    if (L >= 2 * Np - 1 && Nz >= 481)
      return lines % 8 == 0 ? emu_deriv_k<T, L1, L2, LINES, JN, true, 13, true>(Mr, d, Cc, Nz, batch, lines, Lz, f, df, d2f)
                            : emu_deriv_k<T, L1, L2, LINES, JN, true, 13>(Mr, d, Cc, Nz, batch, lines, Lz, f, df, d2f);
  if (L == Np || L >= 2 * Np - 1)
    return emu_deriv_k<T, L1, L2, LINES, JN, true>(Mr, d, Cc, Nz, batch, lines, Lz, f, df, d2f);
  return emu_deriv_k<T, L1, L2, LINES, JN, false>(Mr, d, Cc, Nz, batch, lines, Lz, f, df, d2f);
}

}  // namespace fcns

using namespace fcns;

// The slab plan of fc_deriv_z_host: out[3 i + 0..2] = field, first y row, rows
// of slab i (at most max slabs); returns the staging rows, *n the slab count.
extern "C" long long fchc_slab_plan(int batch, long long Ny, size_t yrow, size_t slab_bytes, long long* out, int max,
                                    int* n) {
  std::vector<Slab> sl;
  const long long Yc = plan_slabs(batch, Ny, yrow, slab_bytes, &sl);
  *n = (int)sl.size();
  for (int i = 0; i < (int)sl.size() && i < max; ++i) {
    out[3 * i] = sl[i].b;
    out[3 * i + 1] = sl[i].y0;
    out[3 * i + 2] = sl[i].yc;
  }
  return Yc;
}

// Emulate fc_deriv_z for transform length L (must be one of the compiled
// shapes and >= N' + Nz - 1).  dtype 0 = float, 1 = double.
extern "C" int fchc_deriv_z(int dtype, int L, const double* Mr, int d, int Cc, int Nz, int batch, int Nx,
                            int Ny, double Lz, const void* f, void* df, void* d2f) {
  const long long lines = (long long)Nx * Ny;
#define HC(LL, A, B, LF, LD)                                                                                 \
  if (L == LL) {                                                                                            \
    if (Nz + Cc <= B * (A / 2 + 1)) {                                                                       \
      if (dtype == 0)                                                                                       \
        return emu_deriv<float, A, B, LF, A / 2 + 1>(Mr, d, Cc, Nz, batch, lines, Lz, (const float*)f, (float*)df, (float*)d2f); \
      return emu_deriv<double, A, B, LD, A / 2 + 1>(Mr, d, Cc, Nz, batch, lines, Lz, (const double*)f, (double*)df, (double*)d2f); \
    }                                                                                                       \
    if (dtype == 0)                                                                                         \
      return emu_deriv<float, A, B, LF, A>(Mr, d, Cc, Nz, batch, lines, Lz, (const float*)f, (float*)df, (float*)d2f); \
    return emu_deriv<double, A, B, LD, A>(Mr, d, Cc, Nz, batch, lines, Lz, (const double*)f, (double*)df, (double*)d2f); \
  }
  HC(64, 8, 8, 16, 8)
  HC(96, 8, 12, 16, 8)
  HC(160, 10, 16, 16, 8)
  HC(288, 16, 18, 16, 8)
  HC(1080, 30, 36, 4, 2)
#undef HC
  return -1;
}

// ---------------------------------------------------------------------------
// Navier-Stokes simulation run on the CPU with the same kernel sequence
// (NsCore with an emulating backend; host memory throughout).
// ---------------------------------------------------------------------------
#include <cstdlib>
#include <cstring>
#if defined(__SANITIZE_ADDRESS__)
#include <sanitizer/asan_interface.h>
#endif

#include "ns_core.hpp"

namespace fcns {
void set_error(const std::string&) {}
fc_status cuda_status(cudaError_t, const char*) { return FC_OK; }

struct EmuBK {
  template <class K>
  fc_status run(const typename K::Args& a, long long grid, void*) {
    phased_emulate<K>(a, grid, K::smem_bytes);
    return FC_OK;
  }
  fc_status alloc(void** p, size_t b) { *p = std::calloc(1, b); return *p ? FC_OK : FC_ERR_NOMEM; }
  void free(void* p) { std::free(p); }
  fc_status h2d(void* d, const void* s, size_t b) { std::memcpy(d, s, b); return FC_OK; }
  fc_status d2d(void* d, const void* s, size_t b, void*) { std::memmove(d, s, b); return FC_OK; }
  fc_status memset(void* d, int v, size_t b, void*) { std::memset(d, v, b); return FC_OK; }
  fc_status d2d_2d(void* dst, size_t dp, const void* src, size_t sp, size_t w, size_t rows, void*) {
    for (size_t r = 0; r < rows; ++r) std::memmove((char*)dst + r * dp, (const char*)src + r * sp, w);
    return FC_OK;
  }
  fc_status sync(void*) { return FC_OK; }
  int sms() { return 1; }
  fc_status d2h(void* d, const void* s, size_t b, void*) { std::memcpy(d, s, b); return FC_OK; }
  // host wall time of the emulated launches (lets the autotuner's logic run on the CPU)
  template <class F>
  fc_status time_ms(F&& f, void*, float* ms) {
    const auto t0 = std::chrono::steady_clock::now();
    const fc_status s = f();
    *ms = std::chrono::duration<float, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return s;
  }
};
}  // namespace fcns

extern "C" {
void* fchc_ns_create(const ns_params* p) {
  auto* c = new NsCore<EmuBK>();
  if (c->create(*p, nullptr, 0)) { c->destroy(); delete c; return nullptr; }
#if FC_LAYOUT_GUARD && defined(__SANITIZE_ADDRESS__)
  // the guard bands between the workspace arrays become unaddressable: a
  // kernel or copy that strays out of its array is reported by the sanitizer
  for (auto& g : c->l.guards) {
    const size_t b = (g.first + 7) / 8 * 8;
    if (g.second > b) ASAN_POISON_MEMORY_REGION(c->ws + b, g.second - b);
  }
#endif
  return c;
}
void fchc_ns_destroy(void* h) {
  auto* c = (NsCore<EmuBK>*)h;
#if FC_LAYOUT_GUARD && defined(__SANITIZE_ADDRESS__)
  ASAN_UNPOISON_MEMORY_REGION(c->ws, c->l.total);
#endif
  c->destroy();
  delete c;
}
int fchc_ns_set_fields(void* h, const void* phys) { return ((NsCore<EmuBK>*)h)->set_fields_any(phys, nullptr); }
int fchc_ns_get_fields(void* h, void* phys) { return ((NsCore<EmuBK>*)h)->get_fields_any(phys, nullptr); }
int fchc_ns_rhs(void* h, const void* in, void* out) { return ((NsCore<EmuBK>*)h)->rhs_any(in, out, nullptr); }
int fchc_ns_project(void* h, double dt, const void* in, void* out, void* gp) {
  return ((NsCore<EmuBK>*)h)->project_any(dt, in, out, gp, nullptr);
}
int fchc_ns_step(void* h, double dt) { return ((NsCore<EmuBK>*)h)->step_any(dt, nullptr); }
int fchc_ns_set_tiles(void* h, const int* tiles) {
  auto* c = (NsCore<EmuBK>*)h;
  for (int k = 0; k < NsCore<EmuBK>::TK_N; ++k) c->tile[k] = tiles[k] & c->variant_mask(k);
  return 0;
}
int fchc_ns_profiles_raw(void* h, double* out) { return ((NsCore<EmuBK>*)h)->profiles_any(out, nullptr); }
int fchc_ns_interpolate(void* dst, void* src) {
  return ((NsCore<EmuBK>*)dst)->interpolate_from_any(*(NsCore<EmuBK>*)src, nullptr);
}
int fchc_ns_diag_raw(void* h, double* acc6) { return ((NsCore<EmuBK>*)h)->diagnostics_any(acc6, nullptr); }
int fchc_ns_get_state(void* h, void* out) {
  auto* c = (NsCore<EmuBK>*)h;
  std::memcpy(out, c->ws + c->l.X[c->cur], c->state_bytes());
  return 0;
}
int fchc_ns_put_state(void* h, const void* in) {
  auto* c = (NsCore<EmuBK>*)h;
  std::memcpy(c->ws + c->l.X[c->cur], in, c->state_bytes());
  return c->mean_init_any(nullptr);
}
int fchc_ns_count_nonfinite(void* h, long long* count) {
  auto* c = (NsCore<EmuBK>*)h;
  fc_status s = c->count_nonfinite_any(true, nullptr);
  unsigned long long n = 0;
  if (!s) s = c->bk.d2h(&n, c->ws + c->l.nfin, sizeof(n), nullptr);
  *count = (long long)n;
  return s;
}
// ns_tune mode 1 on the CPU: every variant timed by host wall clock; the
// choice is written to tiles (5 ints)
int fchc_ns_autotune(void* h, int* tiles) {
  auto* c = (NsCore<EmuBK>*)h;
  const fc_status s = c->autotune_any(nullptr);
  for (int k = 0; k < NsCore<EmuBK>::TK_N; ++k) tiles[k] = c->tile[k];
  return s;
}
// geometry of the dense z operators for (Nz, N'): out = NQ, No, KQ, NC, chunks, slabs; 1 where there is none
int fchc_dense_geom(int Nz, int Np, int* out) {
  DenseGeom g;
  if (!dense_geom(Nz, Np, &g)) return 1;
  const int v[6] = {g.NQ, g.No, g.KQ, g.NC, g.chunks, g.slabs};
  for (int i = 0; i < 6; ++i) out[i] = v[i];
  return 0;
}
// slabs in the ring of a plan's kernel and its shared memory in bytes; 0 where the plan has no dense operators
int fchc_dense_plan(int Nz, int d, int C, int* smem) {
  DenseGeom g;
  if (!dense_plan(Nz, d, C, &g)) return 0;
  const int n = dense_stages(g, d, C);
  *smem = dense_smem(g, d, C, n).total;
  return n;
}
int fchc_dense_row(int Nz, int Np, int j, int i) {
  DenseGeom g;
  return dense_geom(Nz, Np, &g) ? dense_row(g, j, i) : -1;
}
int fchc_dense_slab(int Nz, int Np, int s) {
  DenseGeom g;
  return dense_geom(Nz, Np, &g) ? dense_slab(g, s) : -1;
}
// blocks of derivative order 1 or 2 (float16 bits, as the kernel copies them) and their scale exponent
int fchc_dense_blocks(int Nz, int Np, int order, unsigned short* halves, int* exponent) {
  DenseGeom g;
  if (!dense_geom(Nz, Np, &g)) return 1;
  DenseKernels k;
  dense_kernels(g, &k);
  *exponent = k.e[order - 1];
  for (long long i = 0; i < dense_pairs(g); ++i)
    dense_pair(g, k.c.data() + (order - 1) * Np, k.e[order - 1], i, reinterpret_cast<__half*>(halves));
  return 0;
}
static void dense64_order(const DenseGeom& g, const DenseKernels& k, int order, std::vector<__half>* out) {
  out->resize(dense64_order_halves(g));
  for (long long i = 0; i < dense64_pairs(g); ++i) dense64_pair(g, k.ci.data() + (order - 1) * g.Np, i, out->data());
}
// The sums of digit products that the float64 kernel adds in float32 are exact: the largest possible magnitude of one, for
// line digits of at most 128, over all outputs, parts and weights of an order; 0 where there is no geometry.
long long fchc_dense64_largest_sum(int Nz, int Np, int order) {
  DenseGeom g;
  if (!dense64_geom(Nz, Np, &g)) return 0;
  DenseKernels k;
  dense_kernels(g, &k);
  long long most = 0;
  for (int jo = 0; jo < g.No; ++jo)
    for (int q = 0; q < g.NQ; ++q) {
      long long by_digit[kD64Digits] = {};
      for (int ji = 0; ji < g.No; ++ji) {
        const unsigned long long w = d64_bias(dense_entry(g, q, jo, ji, k.ci.data() + (order - 1) * Np));
        for (int i = 0; i < kD64Digits; ++i) by_digit[i] += std::abs(d64_field(w, i) - 128);
      }
      long long sum = 0;   // the last weight has all digits
      for (int i = 0; i < kD64Digits; ++i) sum += 128 * by_digit[i];
      most = std::max(most, sum);
    }
  return most;
}
// Float64 derivative of order 1 or 2 (unit spacing) of a tile of 16 lines x
// [Nz][16] by the dense operators, y [Nz][16]: the kernel's own tables, index
// maps and number formats, the products and sums in 64-bit integers.  Returns
// 1 where there is no geometry, 3 where a digit sum left 2^24.
int fchc_dense64_tile(int Nz, int d, int C, const double* Mr, int order, const double* x, double* y) {
  DenseGeom g;
  if (!dense64_geom(Nz, Nz + C, &g)) return 1;
  DenseKernels kern;
  dense_kernels(g, &kern);
  const int ex = kern.e64[order - 1], sh = kern.sh[order - 1];
  std::vector<__half> blocks;
  dense64_order(g, kern, order, &blocks);
  const int KT = g.KQ / 16;
  std::vector<unsigned long long> X((size_t)g.Np * 16);
  std::memcpy(X.data(), x, sizeof(double) * Nz * 16);
  std::vector<int> A((size_t)g.NQ * KT * kD64Digits * 256);
  int E[16];
  for (int li = 0; li < 16; ++li) {
    for (int jj = 0; jj < C; ++jj)
      X[(size_t)(Nz + jj) * 16 + li] = d64_continuation(jj, d, C, Mr, &X[li], &X[(size_t)(Nz - d) * 16 + li], 16);
    E[li] = 1;
    for (int n = 0; n < g.Np; ++n) E[li] = std::max(E[li], (int)(X[(size_t)n * 16 + li] >> 52) & 0x7ff);
    for (int j = 0; j < g.KQ; ++j)
      for (int q = 0; q < g.NQ; ++q) {
        long long u = 0;
        for (int i = 0; i < g.NQ && j < g.No && E[li] < 0x7ff; ++i) {
          const long long v = d64_fixed(X[(size_t)dense_row(g, j, i) * 16 + li], E[li]);
          u += __builtin_popcount(q & i) & 1 ? -v : v;
        }
        const unsigned long long w = d64_bias(u);
        for (int i = 0; i < kD64Digits; ++i)
          A[((size_t)(q * KT + j / 16) * kD64Digits + i) * 256 + d64_a_index(li, j % 16)] = d64_field(w, i) - 128;
      }
  }
  std::vector<int> B(blocks.size());
  for (size_t i = 0; i < blocks.size(); ++i) B[i] = (int)__half2float(blocks[i]);
  for (int li = 0; li < 16; ++li)
    for (int j = 0; j < g.No; ++j) {
      long long row[4] = {};
      for (int q = 0; q < g.NQ; ++q) {
        long long s[kD64Sums] = {};
        for (int ks = 0; ks < KT; ++ks)
          for (int i = 0; i < kD64Digits; ++i)
            for (int b = 0; b < kD64Digits && i + b < kD64Sums; ++b)
              for (int k = 0; k < 16; ++k)
                s[i + b] += (long long)A[((size_t)(q * KT + ks) * kD64Digits + i) * 256 + d64_a_index(li, k)] *
                            B[((((size_t)(j / 16) * g.NQ + q) * KT + ks) * kD64Digits + b) * 256 + d64_b_index(k, j % 16)];
        int si[kD64Sums];
        for (int i = 0; i < kD64Sums; ++i) {
          if (s[i] > (1 << 24) || s[i] < -(1 << 24)) return 3;
          si[i] = (int)s[i];
        }
        const long long v = d64_combine(si, sh);
        for (int i = 0; i < g.NQ; ++i) row[i] += (__builtin_popcount(q & i) + (order == 1 ? i : 0)) & 1 ? -v : v;
      }
      for (int i = 0; i < g.NQ; ++i) {
        const int n = dense_row(g, j, i);
        if (n < Nz) y[(size_t)n * 16 + li] = E[li] == 0x7ff ? NAN : std::ldexp((double)row[i], 56 + sh + E[li] - 1082 - ex);
      }
    }
  return 0;
}
// thread order inside a phase (0 ascending, 1 descending) and shared-memory
// poisoning of the emulation (see phased_emulate)
void fchc_set_emulation(int order, int poison) {
  emu_order() = order;
  emu_poison() = poison;
}
}
