// C ABI of libfcns: argument validation, plan objects, dispatch to launchers.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "host_tables.hpp"
#include "slabs.hpp"
#include "internal.hpp"

namespace fcns {

static thread_local std::string g_last_error;

void set_error(const std::string& msg) { g_last_error = msg; }

fc_status cuda_status(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return FC_OK;
  set_error(std::string(what) + ": " + cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? FC_ERR_NOMEM : FC_ERR_CUDA;
}

// Failure injection (tests of callers' error handling; nothing reaches the
// GPU): rules "entry:status:skip:count" from fc_inject_failure or from the
// FCNS_INJECT environment variable (comma-separated rules, read on the first
// check).  A rule lets `skip` calls of its entry point through, then fails
// the next `count` calls (count < 0: every later call); entry "*" matches
// every entry point that checks.
namespace {
struct InjectRule {
  std::string entry;
  fc_status status;
  long long skip, count;
};
std::mutex g_inj_mtx;
std::vector<InjectRule> g_inj;
std::atomic<int> g_inj_state{-1};  // -1: environment not read; 0: no rules; 1: rules armed

bool parse_status(const std::string& t, fc_status* out) {
  static const char* names[] = {"FC_OK", "FC_ERR_ARG", "FC_ERR_UNSUPPORTED", "FC_ERR_CUDA",
                                "FC_ERR_NOMEM", "FC_ERR_TIMEOUT", "FC_ERR_NONFINITE", "FC_ERR_STATE"};
  for (int i = 1; i < 8; ++i)
    if (t == names[i] || t == std::to_string(i)) { *out = (fc_status)i; return true; }
  return false;
}

// caller holds g_inj_mtx
void read_env_rules() {
  const char* env = std::getenv("FCNS_INJECT");
  std::string all = env ? env : "";
  size_t pos = 0;
  while (pos < all.size()) {
    size_t end = all.find(',', pos);
    if (end == std::string::npos) end = all.size();
    std::string rule = all.substr(pos, end - pos), f[4];
    pos = end + 1;
    int k = 0;
    size_t q = 0;
    while (k < 4) {
      size_t c = rule.find(':', q);
      f[k++] = rule.substr(q, c == std::string::npos ? std::string::npos : c - q);
      if (c == std::string::npos) break;
      q = c + 1;
    }
    fc_status st;
    if (f[0].empty() || !parse_status(f[1], &st)) continue;
    g_inj.push_back({f[0], st, f[2].empty() ? 0 : std::atoll(f[2].c_str()), f[3].empty() ? 1 : std::atoll(f[3].c_str())});
  }
  g_inj_state.store(g_inj.empty() ? 0 : 1);
}
}  // namespace

fc_status injected(const char* entry) {
  if (g_inj_state.load(std::memory_order_acquire) == 0) return FC_OK;
  std::lock_guard<std::mutex> lk(g_inj_mtx);
  if (g_inj_state.load() < 0) read_env_rules();
  fc_status out = FC_OK;
  for (auto& r : g_inj) {
    if (r.entry != "*" && r.entry != entry) continue;
    if (r.skip > 0) { --r.skip; continue; }
    if (r.count == 0) continue;
    if (r.count > 0) --r.count;
    out = r.status;
    break;
  }
  std::vector<InjectRule> live;
  for (auto& r : g_inj)
    if (r.count != 0) live.push_back(r);
  g_inj.swap(live);
  g_inj_state.store(g_inj.empty() ? 0 : 1);
  if (out) set_error(std::string(entry) + ": injected failure");
  return out;
}

bool injected_event(const char* name) {
  if (g_inj_state.load(std::memory_order_acquire) <= 0) return false;
  std::lock_guard<std::mutex> lk(g_inj_mtx);
  for (auto& r : g_inj) {
    if (r.entry != name || r.count == 0) continue;
    if (r.skip > 0) { --r.skip; continue; }
    if (r.count > 0) --r.count;
    return true;
  }
  return false;
}

// Which float32 calls take the dense operators instead of the transforms.  A
// tile of 128 lines passes through one SM in 10 us (N' = 115) to 45 us (538), so
// a call needs a wave of tiles (152 x 128 lines) or more, and the gain depends
// on how far the transform length lies above N'.  Measured, dense against
// transform (us, inputs that rotate over more than the L2):
//   padded, N' >= 180   Nz = 155 x 16k lines 29 / 34, 257 x 16k 39 / 48, 400 x 16k 52 /
//                       80, 513 x 16k 58 / 65, 400 x 98k 221 / 395; 8k lines: about
//                       33 / 22 and 46 / 31, so from 16384 lines on
//   padded, N' >= 100   from 131072 lines on (129 x 41k 51 / 42), and where the
//                       transform has 288 points or more (129 x 131k 112 / 132, 150
//                       101 / 208), or 256 and the line two parts, which short lines
//                       prefer to four (N' odd: 104 89 / 97, but 115 105 / 99); below
//                       that the transforms are even or faster (75 x 131k 87 / 81)
//   direct, N' >= 400   (the transform has length N') 487 x 98k 245 / 272, 41k
//                       124 / 121: from 98304 lines on
//   direct, shorter     231 x 132k 167 / 139: transforms
static long long dense_min_lines(const PlanData& p, int L) {
  const long long never = 1LL << 62;
  if (p.dense_direct) return p.Np >= 400 ? 98304 : never;
  if (p.Np >= 180) return 16384;
  return p.Np >= 100 && (L >= 288 || (L == 256 && p.Np % 2)) ? 131072 : never;
}
// Float64 calls take them wherever the plan has them: the transforms sit on the
// float64 pipe.  Measured, dense against transform (us): 11 x 512 lines 29 / 58,
// 65 x 8k 80 / 197, 103 (direct) x 3072 64 / 85, 231 (direct) x 8k 205 / 255, 487
// (direct) x 8k 420 / 462, 513 x 512 60 / 130, x 32k 1467 / 4104.  Only where the
// transform has length N' = 512 and the second wave of 152 tiles of 16 lines is
// half empty are they slower (3072 lines: 217 / 199).
bool deriv_is_dense(const PlanData& p, fc_dtype dtype, long long lines) {
  if (dtype == FC_F64) return p.dense64.NQ && !(p.dense_direct && p.Np >= 400 && lines > 2432 && lines <= 3648);
  return p.dense.NQ && lines >= p.dense_lines;
}

}  // namespace fcns

using namespace fcns;

extern "C" {

const char* fc_status_str(fc_status s) {
  switch (s) {
    case FC_OK: return "FC_OK";
    case FC_ERR_ARG: return "FC_ERR_ARG";
    case FC_ERR_UNSUPPORTED: return "FC_ERR_UNSUPPORTED";
    case FC_ERR_CUDA: return "FC_ERR_CUDA";
    case FC_ERR_NOMEM: return "FC_ERR_NOMEM";
    case FC_ERR_TIMEOUT: return "FC_ERR_TIMEOUT";
    case FC_ERR_NONFINITE: return "FC_ERR_NONFINITE";
    case FC_ERR_STATE: return "FC_ERR_STATE";
  }
  return "FC_ERR_UNKNOWN";
}

const char* fc_last_error(void) { return g_last_error.c_str(); }

fc_status fc_inject_failure(const char* entry, fc_status status, long long skip, long long count) {
  std::lock_guard<std::mutex> lk(g_inj_mtx);
  if (g_inj_state.load() < 0) read_env_rules();
  if (!entry) {
    g_inj.clear();
    g_inj_state.store(0);
    return FC_OK;
  }
  if (status == FC_OK || (int)status < 0 || (int)status > 7 || skip < 0 || count == 0) {
    set_error("fc_inject_failure: status must be an error code, skip >= 0 and count != 0");
    return FC_ERR_ARG;
  }
  g_inj.push_back({entry, status, skip, count});
  g_inj_state.store(1);
  return FC_OK;
}

fc_status fc_setup_ex(int d, int C, int Nz, int M, int n_os, fc_plan_t* out) {
  if (fc_status inj = injected("fc_setup")) return inj;
  if (!out) { set_error("fc_setup: out is NULL"); return FC_ERR_ARG; }
  *out = nullptr;
  if (d < 2 || d > 10 || C < d || C > 64 || Nz < 2 * d || M < 1 || n_os < 1 || 2 * M + 1 > 2 * ((d - 1) * n_os + 1)) {
    set_error("fc_setup: invalid d, C, Nz, M or n_os");
    return FC_ERR_ARG;
  }
  fc_plan* p = new (std::nothrow) fc_plan;
  if (!p) return FC_ERR_NOMEM;
  static std::atomic<unsigned long long> next_serial{1};
  p->data.serial = next_serial.fetch_add(1);
  FcTables T;
  if (!build_fc_tables(d, C, M, n_os, &T)) { delete p; set_error("fc_setup: table construction failed"); return FC_ERR_ARG; }
  p->data.d = d; p->data.C = C; p->data.Nz = Nz; p->data.Np = Nz + C;
  p->data.M = M; p->data.n_os = n_os; p->data.ls_residual = T.ls_residual;
  // per-device tables are handed out by address and used outside the plan's
  // lock: the vector never reallocates (one entry per device, at most 64)
  p->data.dev.reserve(64);
  p->data.Mr = T.Mr;
  // transform length: N' itself when it is one of the compiled (smooth)
  // lengths -- the paper's choice of N' (Sec. 6, Sec. 7 tables) -- else the
  // padded circular-convolution length L >= N' + Nz - 1
  int L = 0;
  for (auto& sh : engine_shapes())
    if (sh.L == p->data.Np) L = sh.L;
  if (!L) L = pick_engine_length(p->data.Np + Nz - 1);
  if (L > 0) {
    for (auto& s : engine_shapes())
      if (s.L == L) { p->deriv.L = L; p->deriv.L1 = s.L1; p->deriv.L2 = s.L2; }
    engine_twiddles(p->deriv.L1, p->deriv.L2, &p->deriv.tw);
    auto& t = p->deriv;
    std::vector<std::complex<double>> H1, H2;
    deriv_conv_spectra(Nz, p->data.Np, L, &H1, &H2);
    t.H1_32.resize(L); t.H2_32.resize(L); t.H1_64.resize(L); t.H2_64.resize(L);
    for (int i = 0; i < L; ++i) {
      t.H1_32[i] = make_float2((float)H1[i].real(), (float)H1[i].imag());
      t.H2_32[i] = make_float2((float)H2[i].real(), (float)H2[i].imag());
      t.H1_64[i] = make_double2(H1[i].real(), H1[i].imag());
      t.H2_64[i] = make_double2(H2[i].real(), H2[i].imag());
    }
    t.tw32.resize(2 * L); t.tw64.resize(2 * L);
    for (int i = 0; i < 2 * L; ++i) {
      t.tw32[i] = make_float2((float)t.tw[i].real(), (float)t.tw[i].imag());
      t.tw64[i] = make_double2(t.tw[i].real(), t.tw[i].imag());
    }
  }
  p->deriv.Mr2.resize(p->data.Mr.size());
  for (size_t i = 0; i < p->data.Mr.size(); ++i) {
    const float hi = (float)p->data.Mr[i];
    p->deriv.Mr2[i] = make_float2(hi, (float)(p->data.Mr[i] - (double)hi));
  }
  PlanData& pd = p->data;
  pd.dense_direct = L == pd.Np;
  pd.dense_lines = dense_min_lines(pd, L);
  const bool f32 = L > 0 && pd.dense_lines < (1LL << 31) && dense_plan(Nz, d, C, &pd.dense);
  const bool f64 = L > 0 && dense64_geom(Nz, pd.Np, &pd.dense64);
  if (!f32) pd.dense = DenseGeom();
  if (!f64) pd.dense64 = DenseGeom();
  if (f32 || f64) dense_kernels(f32 ? pd.dense : pd.dense64, &pd.kern);
  *out = p;
  return FC_OK;
}

fc_status fc_setup(int d, int C, int Nz, fc_plan_t* out) {
  return fc_setup_ex(d, C, Nz, (2 * (d + C)) / 3, 20, out);
}

fc_status fc_plan_matrix(fc_plan_t plan, double* Mr_out) {
  if (!plan || !Mr_out) { set_error("fc_plan_matrix: NULL argument"); return FC_ERR_ARG; }
  std::memcpy(Mr_out, plan->data.Mr.data(), sizeof(double) * plan->data.Mr.size());
  return FC_OK;
}

fc_status fc_plan_info(fc_plan_t plan, int* d, int* C, int* Nz, int* M, int* n_os, double* ls_residual) {
  if (!plan) { set_error("fc_plan_info: NULL plan"); return FC_ERR_ARG; }
  if (d) *d = plan->data.d;
  if (C) *C = plan->data.C;
  if (Nz) *Nz = plan->data.Nz;
  if (M) *M = plan->data.M;
  if (n_os) *n_os = plan->data.n_os;
  if (ls_residual) *ls_residual = plan->data.ls_residual;
  return FC_OK;
}

fc_status fc_destroy(fc_plan_t plan) {
  if (!plan) return FC_ERR_ARG;
  int cur = -1;
  if (!plan->data.dev.empty() && cudaGetDevice(&cur) == cudaSuccess) {
    for (auto& t : plan->data.dev) {
      cudaSetDevice(t.device);
      cudaDeviceSynchronize();
      cudaFree(t.block);
      cudaFree(t.dense); cudaFree(t.dense64);
      for (auto& slot : t.stage)
        for (void* b : slot) cudaFree(b);
      for (int k = 0; k < 3; ++k) {
        if (t.ev_in[k]) cudaEventDestroy(t.ev_in[k]);
        if (t.ev_run[k]) cudaEventDestroy(t.ev_run[k]);
        if (t.ev_out[k]) cudaEventDestroy(t.ev_out[k]);
      }
      if (t.st_in) cudaStreamDestroy(t.st_in);
      if (t.st_run) cudaStreamDestroy(t.st_run);
      if (t.st_out) cudaStreamDestroy(t.st_out);
    }
    cudaSetDevice(cur);
  }
  // (the devices have finished: what no later call has reported)
  const fc_status s = dense_gave_up(plan->data, "fc_destroy");
  delete plan;
  return s;
}

}  // extern "C"

namespace fcns {

static fc_status deriv_tables_locked(fc_plan* plan, DerivDevTables** out) {
  int dev = -1;
  fc_status s = cuda_status(cudaGetDevice(&dev), "cudaGetDevice");
  if (s) return s;
  for (auto& t : plan->data.dev)
    if (t.device == dev) { *out = &t; return FC_OK; }
  if (plan->data.dev.size() >= plan->data.dev.capacity()) {
    set_error("fc_deriv_z: more devices than the plan supports (64)");
    return FC_ERR_UNSUPPORTED;
  }
  // every table in one allocation and one copy (the dense operators' blocks follow when a call takes them)
  const PlanData& pd = plan->data;
  const PlanHostTables& h = plan->deriv;
  std::vector<unsigned char> up;
  auto put = [&up](const void* src, size_t bytes) {
    const size_t at = (up.size() + 255) & ~(size_t)255;
    up.resize(at + bytes);
    std::memcpy(up.data() + at, src, bytes);
    return at;
  };
  const size_t L = h.L;
  const size_t oMr = put(pd.Mr.data(), sizeof(double) * pd.Mr.size()), oMr2 = put(h.Mr2.data(), sizeof(float2) * h.Mr2.size());
  const size_t oH1 = put(h.H1_32.data(), 8 * L), oH2 = put(h.H2_32.data(), 8 * L), oT = put(h.tw32.data(), 16 * L);
  const size_t oG1 = put(h.H1_64.data(), 16 * L), oG2 = put(h.H2_64.data(), 16 * L), oU = put(h.tw64.data(), 32 * L);
  const size_t oC = pd.dense.NQ ? put(pd.kern.c.data(), 8 * pd.kern.c.size()) : 0;
  const size_t oI = pd.dense64.NQ ? put(pd.kern.ci.data(), 8 * pd.kern.ci.size()) : 0;
  DerivDevTables t;
  t.device = dev;
  t.L = h.L;
  s = cuda_status(cudaMalloc(&t.block, up.size()), "cudaMalloc(tables)");
  if (s) return s;
  unsigned char* at = static_cast<unsigned char*>(t.block);
  t.Mr = reinterpret_cast<double*>(at + oMr);
  t.Mr2 = reinterpret_cast<float2*>(at + oMr2);
  t.H1_32 = at + oH1; t.H2_32 = at + oH2; t.tw32 = at + oT;
  t.H1_64 = at + oG1; t.H2_64 = at + oG2; t.tw64 = at + oU;
  s = cuda_status(cudaMemcpy(at, up.data(), up.size(), cudaMemcpyHostToDevice), "cudaMemcpy(tables)");
  if (pd.dense.NQ) t.kern = reinterpret_cast<const double*>(at + oC);
  if (pd.dense64.NQ) t.kern64 = reinterpret_cast<const long long*>(at + oI);
  // in place before any stream reads them, non-blocking ones too
  if (!s) s = cuda_status(cudaStreamSynchronize(nullptr), "cudaStreamSynchronize(tables)");
  if (s) {
    cudaFree(t.block);
    return s;
  }
  plan->data.dev.push_back(t);
  *out = &plan->data.dev.back();
  return FC_OK;
}

// The dense operators' blocks of a precision, at its first call that takes them (an allocation of more than 2 MB is 90 us,
// and most plans are used in one precision).  On a stream of its own and with the thread's capture mode relaxed, so that
// the call may be a captured one: the blocks belong to the plan, not to the graph.
static fc_status dense_blocks_locked(const PlanData& pd, DerivDevTables* t, fc_dtype dtype) {
  void*& slot = dtype == FC_F64 ? t->dense64 : t->dense;
  if (slot) return FC_OK;
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  fc_status s = cuda_status(cudaThreadExchangeStreamCaptureMode(&mode), "cudaThreadExchangeStreamCaptureMode");
  if (s) return s;
  void* b = nullptr;
  cudaStream_t st = nullptr;
  s = cuda_status(cudaMalloc(&b, dtype == FC_F64 ? dense64_bytes(pd) : dense_bytes(pd)), "cudaMalloc(blocks)");
  if (!s) s = cuda_status(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking), "cudaStreamCreate");
  if (!s) s = dtype == FC_F64 ? launch_dense64_build(pd, t->kern64, b, st) : launch_dense_build(pd, t->kern, b, st);
  if (!s) s = cuda_status(cudaStreamSynchronize(st), "cudaStreamSynchronize(blocks)");
  if (st) cudaStreamDestroy(st);
  if (s) cudaFree(b);
  else slot = b;
  cudaThreadExchangeStreamCaptureMode(&mode);
  return s;
}

}  // namespace fcns

fc_status fcns::check_deriv_args(const PlanData& pd, const PlanHostTables& t, fc_dtype dtype, int batch, int Nx,
                                 int Ny, double Lz, const void* f, void* df, void* d2f, const char* who) {
  std::string w(who);
  if (!f || (!df && !d2f)) { set_error(w + ": NULL input or both outputs"); return FC_ERR_ARG; }
  if (dtype != FC_F32 && dtype != FC_F64) { set_error(w + ": bad dtype"); return FC_ERR_ARG; }
  if (batch < 1 || Nx < 1 || Ny < 1 || !(Lz > 0) || !std::isfinite(Lz)) { set_error(w + ": bad sizes"); return FC_ERR_ARG; }
  const long long lines = (long long)Nx * Ny;
  if (lines * batch >= (1LL << 31)) { set_error(w + ": too many lines"); return FC_ERR_UNSUPPORTED; }
  if (t.L == 0) { set_error(w + ": N' + Nz - 1 exceeds the compiled transform lengths"); return FC_ERR_UNSUPPORTED; }
  const size_t es = dtype == FC_F32 ? 4 : 8;
  const size_t bytes = es * (size_t)lines * pd.Nz * batch;
  auto overlap = [&](const void* a, const void* b) {
    if (!a || !b) return false;
    const char* x = (const char*)a;
    const char* y = (const char*)b;
    return x < y + bytes && y < x + bytes;
  };
  if (overlap(f, df) || overlap(f, d2f) || overlap(df, d2f)) { set_error(w + ": overlapping buffers"); return FC_ERR_ARG; }
  return FC_OK;
}

extern "C" fc_status fc_deriv_z(fc_plan_t plan, fc_dtype dtype, int batch, int Nx, int Ny, double Lz,
                                const void* f, void* df, void* d2f, fc_stream_t stream) {
  if (fc_status inj = injected("fc_deriv_z")) return inj;
  if (!plan) { set_error("fc_deriv_z: NULL plan"); return FC_ERR_ARG; }
  fc_status s = check_deriv_args(plan->data, plan->deriv, dtype, batch, Nx, Ny, Lz, f, df, d2f, "fc_deriv_z");
  if (!s) s = dense_gave_up(plan->data, "fc_deriv_z");
  if (s) return s;
  const bool dense = deriv_is_dense(plan->data, dtype, (long long)Nx * Ny * batch);
  DerivDevTables* t = nullptr;
  {
    std::lock_guard<std::mutex> lk(plan->data.mtx);
    s = deriv_tables_locked(plan, &t);
    if (!s && dense) s = dense_blocks_locked(plan->data, t, dtype);
  }
  if (s) return s;
  return launch_deriv_any(dense, *t, plan->data, dtype, batch, (long long)Nx * Ny, Lz, f, df, d2f, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// fc_deriv_z on host arrays: slabs of y rows (all z, all x) are copied in,
// differentiated and copied out on three streams, so that the copies of one
// slab overlap the kernel of another and the two copy directions overlap
// each other.
// ---------------------------------------------------------------------------
static fc_status stage_for(DerivDevTables* t, size_t bytes) {
  fc_status s = FC_OK;
  if (!t->st_in) {
    s = cuda_status(cudaStreamCreateWithFlags(&t->st_in, cudaStreamNonBlocking), "cudaStreamCreate");
    if (!s) s = cuda_status(cudaStreamCreateWithFlags(&t->st_run, cudaStreamNonBlocking), "cudaStreamCreate");
    if (!s) s = cuda_status(cudaStreamCreateWithFlags(&t->st_out, cudaStreamNonBlocking), "cudaStreamCreate");
    for (int k = 0; k < 3 && !s; ++k) {
      s = cuda_status(cudaEventCreateWithFlags(&t->ev_in[k], cudaEventDisableTiming), "cudaEventCreate");
      if (!s) s = cuda_status(cudaEventCreateWithFlags(&t->ev_run[k], cudaEventDisableTiming), "cudaEventCreate");
      if (!s) s = cuda_status(cudaEventCreateWithFlags(&t->ev_out[k], cudaEventDisableTiming), "cudaEventCreate");
    }
    if (s) return s;
  }
  if (t->stage_bytes >= bytes) return FC_OK;
  for (auto& slot : t->stage)
    for (void*& b : slot) {
      cudaFree(b);
      b = nullptr;
    }
  t->stage_bytes = 0;
  for (auto& slot : t->stage)
    for (void*& b : slot) {
      s = cuda_status(cudaMalloc(&b, bytes), "cudaMalloc(fc_deriv_z_host staging)");
      if (s) return s;
    }
  t->stage_bytes = bytes;
  return FC_OK;
}

extern "C" fc_status fc_deriv_z_host_ex(fc_plan_t plan, fc_dtype dtype, int batch, int Nx, int Ny, double Lz,
                                        const void* f, void* df, void* d2f, size_t slab_bytes, fc_stream_t stream) {
  if (fc_status inj = injected("fc_deriv_z_host")) return inj;
  if (!plan) { set_error("fc_deriv_z_host: NULL plan"); return FC_ERR_ARG; }
  fc_status s = check_deriv_args(plan->data, plan->deriv, dtype, batch, Nx, Ny, Lz, f, df, d2f, "fc_deriv_z_host");
  if (!s) s = dense_gave_up(plan->data, "fc_deriv_z_host");
  if (s) return s;
  // the whole call picks the kernel, so that the slabs give what one call on device arrays gives
  const bool dense = deriv_is_dense(plan->data, dtype, (long long)Nx * Ny * batch);
  DerivDevTables* t = nullptr;
  {
    std::lock_guard<std::mutex> lk(plan->data.mtx);
    s = deriv_tables_locked(plan, &t);
    if (!s && dense) s = dense_blocks_locked(plan->data, t, dtype);
  }
  if (s) return s;
  std::lock_guard<std::mutex> hl(plan->data.host_mtx);
  const size_t es = dtype == FC_F32 ? 4 : 8;
  const int Nz = plan->data.Nz;
  const size_t yrow = (size_t)Nz * Nx * es;   // bytes of one y row over all z
  std::vector<Slab> slabs;
  const long long Yc = plan_slabs(batch, Ny, yrow, slab_bytes, &slabs);
  s = stage_for(t, (size_t)Yc * yrow);
  if (s) return s;
  // the slabs start after the work already queued on the caller's stream
  cudaEvent_t e0 = nullptr;
  s = cuda_status(cudaEventCreateWithFlags(&e0, cudaEventDisableTiming), "cudaEventCreate");
  if (!s) s = cuda_status(cudaEventRecord(e0, (cudaStream_t)stream), "cudaEventRecord");
  if (!s) s = cuda_status(cudaStreamWaitEvent(t->st_in, e0, 0), "cudaStreamWaitEvent");
  const char* fh = static_cast<const char*>(f);
  char* oh[2] = {static_cast<char*>(df), static_cast<char*>(d2f)};
  const size_t hp = (size_t)Ny * Nx * es;     // host pitch between z rows
  long long i = 0;
  for (size_t si = 0; si < slabs.size() && !s; ++si, ++i) {
    {  // slab si in staging slot i % 3
      const int b = slabs[si].b;
      const long long y0 = slabs[si].y0, yc = slabs[si].yc;
      const int k = (int)(i % 3);
      const size_t w = (size_t)yc * Nx * es, off = ((size_t)b * Nz * Ny + (size_t)y0) * Nx * es;
      if (i >= 3) s = cuda_status(cudaStreamWaitEvent(t->st_in, t->ev_out[k], 0), "cudaStreamWaitEvent");
      if (!s) s = cuda_status(cudaMemcpy2DAsync(t->stage[k][0], w, fh + off, hp, w, Nz, cudaMemcpyHostToDevice, t->st_in),
                              "cudaMemcpy2DAsync(H2D)");
      if (!s) s = cuda_status(cudaEventRecord(t->ev_in[k], t->st_in), "cudaEventRecord");
      if (!s) s = cuda_status(cudaStreamWaitEvent(t->st_run, t->ev_in[k], 0), "cudaStreamWaitEvent");
      void *o1 = df ? t->stage[k][1] : nullptr, *o2 = d2f ? t->stage[k][2] : nullptr;
      if (!s) s = launch_deriv_any(dense, *t, plan->data, dtype, 1, (long long)Nx * yc, Lz, t->stage[k][0], o1, o2, t->st_run);
      if (!s) s = cuda_status(cudaEventRecord(t->ev_run[k], t->st_run), "cudaEventRecord");
      if (!s) s = cuda_status(cudaStreamWaitEvent(t->st_out, t->ev_run[k], 0), "cudaStreamWaitEvent");
      for (int o = 0; o < 2 && !s; ++o)
        if (oh[o])
          s = cuda_status(cudaMemcpy2DAsync(oh[o] + off, hp, t->stage[k][1 + o], w, w, Nz, cudaMemcpyDeviceToHost,
                                            t->st_out), "cudaMemcpy2DAsync(D2H)");
      if (!s) s = cuda_status(cudaEventRecord(t->ev_out[k], t->st_out), "cudaEventRecord");
    }
  }
  // synchronous: the outputs are in host memory on return (also after an error)
  const fc_status s1 = cuda_status(cudaStreamSynchronize(t->st_in), "cudaStreamSynchronize");
  const fc_status s2 = cuda_status(cudaStreamSynchronize(t->st_run), "cudaStreamSynchronize");
  const fc_status s3 = cuda_status(cudaStreamSynchronize(t->st_out), "cudaStreamSynchronize");
  if (e0) cudaEventDestroy(e0);
  const fc_status s4 = dense_gave_up(plan->data, "fc_deriv_z_host");
  return s ? s : (s1 ? s1 : (s2 ? s2 : (s3 ? s3 : s4)));
}

extern "C" fc_status fc_deriv_z_host(fc_plan_t plan, fc_dtype dtype, int batch, int Nx, int Ny, double Lz,
                                     const void* f, void* df, void* d2f, fc_stream_t stream) {
  // 256 MB slabs: every copy moves Nz rows of ~0.5 MB; with 64 MB slabs (rows
  // of 128 KB at 512^2 x 513) the strided copies ran at half the speed
  return fc_deriv_z_host_ex(plan, dtype, batch, Nx, Ny, Lz, f, df, d2f, (size_t)256 << 20, stream);
}
