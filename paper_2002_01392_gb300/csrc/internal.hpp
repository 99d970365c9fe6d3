// Internal declarations shared by the C ABI and the kernel launchers.
#pragma once
#include <cuda_runtime.h>
#include <complex>
#include <atomic>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/fcns.h"
#include "dense64.hpp"
#include "dense_geom.hpp"
#include "host_tables.hpp"

namespace fcns {

void set_error(const std::string& msg);
fc_status cuda_status(cudaError_t e, const char* what);
// host-side failure injection: the status an armed entry point must return
// now (FC_OK when it is not armed); checked first thing by the entry points
fc_status injected(const char* entry);

// lengths of the two-pass line engine that are compiled: L = L1 * L2
struct EngineShape { int L, L1, L2; };
const std::vector<EngineShape>& engine_shapes();
// smallest compiled L >= need (0 if none)
int pick_engine_length(int need);

// per-device copies of the derivative tables of one plan
struct DerivDevTables {
  int device = -1;
  int L = 0;
  void* block = nullptr;  // one allocation holds all of the following but the blocks
  double* Mr = nullptr;
  float2* Mr2 = nullptr;  // (hi, lo) float split of Mr
  void* tw32 = nullptr;  // float2[L]
  void* tw64 = nullptr;  // double2[L]
  void* H1_32 = nullptr; // spectra of d1 and d2 separately (paired-line kernel)
  void* H1_64 = nullptr;
  void* H2_32 = nullptr;
  void* H2_64 = nullptr;
  const double* kern = nullptr;      // what the blocks are built from (PlanData::kern)
  const long long* kern64 = nullptr;
  void* dense = nullptr;          // blocks of the dense operators (float16 pairs), both orders; null: not used
  void* dense64 = nullptr;        // the same for float64 (digit fragments)
  // staging of fc_deriv_z_host: three rotating slots of (input, d1, d2) slab
  // buffers of stage_bytes each, and the copy-in / compute / copy-out streams
  size_t stage_bytes = 0;
  void* stage[3][3] = {};
  cudaStream_t st_in = nullptr, st_run = nullptr, st_out = nullptr;
  cudaEvent_t ev_in[3] = {}, ev_run[3] = {}, ev_out[3] = {};
};

struct PlanData {
  unsigned long long serial = 0;          // unique per plan in the process (never reused)
  int d, C, Nz, Np, M, n_os;
  double ls_residual;
  std::vector<double> Mr;
  DenseGeom dense;                        // dense operators (NQ = 0: none)
  long long dense_lines = 0;              // float32 calls of this many lines or more take them
  DenseGeom dense64;                      // the same for float64 (dense64.hpp)
  bool dense_direct = false;              // the transform kernel would run at length N' itself
  DenseKernels kern;                      // what the blocks are built from, where either exists
  // word that a float32 dense kernel of the plan sets when a wait runs out (null before the first one)
  mutable std::atomic<unsigned*> gave_up{nullptr};
  std::mutex mtx;
  std::mutex host_mtx;   // serialises fc_deriv_z_host calls on the plan (shared staging)
  std::vector<DerivDevTables> dev;
};


// host copies of the derivative tables of one plan, in both precisions
struct PlanHostTables {
  int L = 0, L1 = 0, L2 = 0;
  std::vector<std::complex<double>> tw;
  std::vector<float2> tw32, Mr2, H1_32, H2_32;
  std::vector<double2> tw64, H1_64, H2_64;
};

// argument checks shared by the fc_deriv_z entry points
fc_status check_deriv_args(const PlanData& p, const PlanHostTables& t, fc_dtype dtype, int batch, int Nx, int Ny,
                           double Lz, const void* f, void* df, void* d2f, const char* who);

}  // namespace fcns

struct fc_plan {
  fcns::PlanData data;
  fcns::PlanHostTables deriv;
};

namespace fcns {

fc_status launch_deriv_z(const DerivDevTables& t, const PlanData& p, fc_dtype dtype, int batch,
                         long long lines, double Lz, const void* f, void* df, void* d2f,
                         cudaStream_t stream);
// the same by the dense operators (float32; plans with a dense geometry)
fc_status launch_deriv_dense(const DerivDevTables& t, const PlanData& p, int batch, long long lines, double Lz,
                             const void* f, void* df, void* d2f, cudaStream_t stream);
fc_status launch_deriv_dense64(const DerivDevTables& t, const PlanData& p, int batch, long long lines, double Lz,
                               const void* f, void* df, void* d2f, cudaStream_t stream);
// the kernel of a whole call by its type and lines: transforms, or the dense operators of its precision
inline fc_status launch_deriv_any(bool dense, const DerivDevTables& t, const PlanData& p, fc_dtype dtype, int batch,
                                  long long lines, double Lz, const void* f, void* df, void* d2f, cudaStream_t stream) {
  if (!dense) return launch_deriv_z(t, p, dtype, batch, lines, Lz, f, df, d2f, stream);
  return dtype == FC_F64 ? launch_deriv_dense64(t, p, batch, lines, Lz, f, df, d2f, stream)
                         : launch_deriv_dense(t, p, batch, lines, Lz, f, df, d2f, stream);
}
// builds the blocks of both orders in `out` (bytes: dense_bytes / dense64_bytes) from the kernels `c` (plan.kern.c or
// plan.kern.ci, both orders, on the device)
fc_status launch_dense_build(const PlanData& p, const double* c, void* out, cudaStream_t stream);
fc_status launch_dense64_build(const PlanData& p, const long long* c, void* out, cudaStream_t stream);
inline size_t dense_bytes(const PlanData& p) { return p.dense.NQ ? 4 * (size_t)dense_order_halves(p.dense) : 0; }
inline size_t dense64_bytes(const PlanData& p) { return p.dense64.NQ ? 4 * (size_t)dense64_order_halves(p.dense64) : 0; }
// FC_ERR_TIMEOUT (once) where a float32 dense kernel of the plan gave up a bounded wait
fc_status dense_gave_up(const PlanData& p, const char* who);
// whether a rule of fc_inject_failure for exactly this name fires; sets no error text
bool injected_event(const char* name);
// whether a whole call (all its lines) takes the dense operators
bool deriv_is_dense(const PlanData& p, fc_dtype dtype, long long lines);

}  // namespace fcns
