// Launch of the dense z operators (dense_z.cuh).
#include <atomic>
#include <cmath>

#include "dense_build.cuh"
#include "dense_z.cuh"
#include "internal.hpp"

namespace fcns {

static fc_status launch_dense(DenseArgs a, cudaStream_t stream) {
  // as many slabs as fit beside the tile; a block set that fits whole is loaded once per CTA
  const int nord = (a.orders & 1) + (a.orders >> 1);
  const int all = nord * a.g.chunks * a.g.NQ * a.g.slabs;
  a.stages = dense_stages(a.g, a.d, a.Cc);   // (at least two: dense_plan)
  a.resident = all <= a.stages ? 1 : 0;
  // low x low products where the contraction is short and the tile's time is its loads: see the header
  a.low_low = a.g.NQ == 4 && a.g.KQ <= 48 ? 1 : 0;
  const DenseSmem so = dense_smem(a.g, a.d, a.Cc, a.stages);
  // d = 5 (the default continuation) is compiled on its own
  const int form = (a.g.NQ == 4 ? 1 : 0) + (a.d == 5 ? 2 : 0);
  auto kern = form == 0 ? dense_z_kernel<2, 0> : form == 1 ? dense_z_kernel<4, 0> : form == 2 ? dense_z_kernel<2, 5> : dense_z_kernel<4, 5>;
  static std::atomic<unsigned long long> attr_set[4];
  std::atomic<unsigned long long>& attr = attr_set[form];
  static std::atomic<int> sm_count[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64 || !(attr.load() >> dev & 1ull)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDenseSmemMax);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute(dense z)");
    if (dev < 64) attr.fetch_or(1ull << dev);
  }
  int sms = dev < 64 ? sm_count[dev].load() : 0;
  if (!sms) {
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_status(e, "cudaDeviceGetAttribute");
    if (dev < 64) sm_count[dev].store(sms);
  }
  a.tiles = (a.lines + kDenseLines - 1) / kDenseLines;
  const unsigned grid = (unsigned)(a.tiles < sms ? a.tiles : sms);
  kern<<<grid, kDenseThreads, so.total, stream>>>(a, so);
  return cuda_status(cudaGetLastError(), "dense z launch");
}

// The words that kernels set when a wait runs out, one per plan (by its serial number; two of a thousand plans in use
// share one).  Managed: a kernel's store reaches the host without a call, a host's read of a page that no kernel has written
// is an ordinary one, and nothing is allocated (a pinned word of its own cost a plan's first call 107 us).
constexpr int kErrWords = 1024;
static __managed__ unsigned g_dense_err[kErrWords];

static unsigned* err_word(const PlanData& p) {
  unsigned* w = p.gave_up.load();
  if (w) return w;
  // (where the host may not read managed memory while kernels run, there is no word; the outputs are NaN all the same)
  int dev = 0, ok = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&ok, cudaDevAttrConcurrentManagedAccess, dev) != cudaSuccess || !ok) return nullptr;
  w = &g_dense_err[p.serial % kErrWords];
  p.gave_up.store(w);
  return w;
}

fc_status dense_gave_up(const PlanData& p, const char* who) {
  unsigned* w = p.gave_up.load();
  const unsigned id = w ? *static_cast<volatile unsigned*>(w) : 0;
  if (!id) return FC_OK;
  *static_cast<volatile unsigned*>(w) = 0;
  set_error(std::string(who) + ": a kernel of the plan gave up wait " + std::to_string(id));
  return FC_ERR_TIMEOUT;
}

fc_status launch_deriv_dense(const DerivDevTables& t, const PlanData& p, int batch, long long lines, double Lz,
                             const void* f, void* df, void* d2f, cudaStream_t stream) {
  DenseArgs a = {};
  a.g = p.dense;
  a.d = p.d;
  a.Cc = p.C;
  a.orders = (df ? 1 : 0) | (d2f ? 2 : 0);
  a.per = lines;
  a.outer = lines * p.Nz;
  a.lines = lines * batch;
  a.in = static_cast<const float*>(f);
  a.out1 = static_cast<float*>(df);
  a.out2 = static_cast<float*>(d2f);
  a.B = static_cast<const __half*>(t.dense);
  a.order_halves = dense_order_halves(a.g);
  a.Mr2 = t.Mr2;
  const double dz = Lz / (p.Nz - 1), sc[2] = {1.0 / dz, 1.0 / (dz * dz)};
  for (int o = 0; o < 2; ++o) {   // (at least 1 after rounding: frexp's mantissa is in [1/2, 1))
    int e = 0;
    a.f[o] = (float)(2 * std::frexp(sc[o], &e));
    a.fe[o] = e - 1 - p.kern.e[o];
    if (!(sc[o] > 0) || std::isinf(sc[o])) {   // (no exponent: as a product)
      a.f[o] = (float)sc[o];
      a.fe[o] = 1000;
    }
  }
  a.err = err_word(p);
  const fc_status s = launch_dense(a, stream);
  if (!s && a.err && injected_event("dense_z_kernel")) *static_cast<volatile unsigned*>(a.err) = 1;   // (as the kernel would)
  return s;
}

__global__ void dense_build_kernel(const __grid_constant__ DenseGeom g, const double* __restrict__ c, int e1, int e2, __half* out) {
  const long long n = dense_pairs(g), i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * n) return;
  const int o = i >= n;
  dense_pair(g, c + o * g.Np, o ? e2 : e1, i - o * n, out + o * dense_order_halves(g));
}

fc_status launch_dense_build(const PlanData& p, const double* c, void* out, cudaStream_t stream) {
  const long long n = 2 * dense_pairs(p.dense);
  dense_build_kernel<<<(unsigned)((n + 127) / 128), 128, 0, stream>>>(p.dense, c, p.kern.e[0], p.kern.e[1], static_cast<__half*>(out));
  return cuda_status(cudaGetLastError(), "dense z blocks launch");
}

}  // namespace fcns
