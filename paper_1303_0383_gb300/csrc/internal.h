// internal.h -- declarations shared by the translation units of liblagp (not installed).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "lagp.h"
#include "batch.cuh"
#include "sizes.h"

namespace lagp {

// Upper limits checked by the entry points (see the argument rules in lagp.h).
constexpr int kMaxP = 8;
constexpr int kMaxN = 256;       // local design size n
constexpr int kMaxCand = 8192;   // candidate count

extern std::atomic<int64_t> g_launches;

// Device properties of the current device, cached per device ordinal.
struct DevInfo {
  int device;
  int num_sms;
  size_t smem_optin;
  size_t smem_per_sm;
  size_t l2;
};
int dev_info(DevInfo *out);
// Lets a kernel's launches use any dynamic shared memory the device allows.  The limit is state
// of the function, not of a launch: setting each launch's own size would let one thread lower
// it between another thread's setting and launch.
int allow_smem(const void *fn, const DevInfo &di);

// Kernel (a): candidate sets.
int knn_launch(const double *X, int64_t N, int32_t p, const double *XX, int64_t T, int32_t ncand,
               int32_t *cand, void *ws, size_t ws_bytes, cudaStream_t stream);
int knn_launch_list(const double *X, int64_t N, int32_t p, const double *XX, int64_t nloc,
                    int32_t M, int32_t *cand, void *ws, size_t ws_bytes, cudaStream_t stream,
                    const int32_t *list, const LocDesc *locs, int ldxx, int ctas_per_sm);

// Kernels (b)+(c): greedy design and predictive equations.
struct SelectArgs {
  const double *X, *Z;
  int64_t N;
  int32_t p;
  const double *XX;
  int64_t T;
  const int32_t *cand;
  int32_t M, n0, n;
  double theta, g;
  const double *theta_loc;  // per-location lengthscale (device, T), or nullptr: theta
  const int32_t *start;     // saved start designs (device, T x nstart), or nullptr: n0 nearest
  int32_t nstart;
  double r_min;             // > 1: stopping rule of Sec. 6 (ALC), 0: fixed n
  int32_t *n_out;           // adaptive designs' sizes (device, T), with r_min
  int32_t method, precision;
  double *mean, *s2, *var;
  int32_t *idx;
  int8_t *status;
};
size_t select_workspace_bytes(int64_t T, int32_t p, int32_t n, int32_t ncand, int32_t method,
                              int32_t precision, int num_sms);
int select_launch(const SelectArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream);
// The least workspace that select_launch takes (one CTA per SM, or the FP64 recursion).
size_t select_needed_bytes(const SelectArgs &a, int num_sms);
// The same launch on a caller-chosen grid of G CTAs (G >= 1), and the scratch it needs.
int select_default_grid(int64_t T, int num_sms);
size_t select_scratch_bytes_for_grid(int G, int32_t p, int32_t n, int32_t ncand);
int select_launch_on_grid(const SelectArgs &a, void *ws, size_t ws_bytes, int G,
                          cudaStream_t stream);
// The FP64 recursion on the *count locations (queue positions, both device) in `list`, of a uniform
// launch (a) or of a batch (b): what the ALC screen left to it.  queue: a zeroed counter.
struct BatchLaunch;
struct HandedList {
  int *queue;
  const int32_t *list;
  const int *count;
};
int select_listed_launch(const SelectArgs *a, const BatchLaunch *b, const HandedList &h, void *scratch,
                         size_t bytes, cudaStream_t stream);

// Mixed-precision variant of kernels (b)+(c) (ALC): float-float screen, FP64 decisions.
size_t select_mixed_workspace_bytes(int64_t T, int32_t p, int32_t n, int32_t ncand, int32_t precision, int num_sms);
size_t select_mixed_needed_bytes(const SelectArgs &a);  // room for one CTA per SM
int select_mixed_launch(const SelectArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream);

// ALC in the paper's own form (explicit K_j^{-1}, partition inverse updates), FP64:
// kernel (b) then kernel (c) on the selected design (select_dense.cu).
int select_dense_max_n();
size_t select_dense_workspace_bytes(int64_t T, int32_t p, int32_t n, int32_t ncand, int num_sms);
int select_dense_launch(const SelectArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream);

// Kernel (c) on a selected design: FP64 predictive equations for every location from its
// design indices (idx < 0 marks a location whose screen failed).
struct PredictArgs {
  const double *X, *Z;
  int32_t p;
  const double *XX;
  int64_t T;
  int32_t n, nmax;
  double theta, g;
  const int32_t *idx;
  BatchView B;  // per-location tables, or designs == nullptr for a uniform launch
  // the FP64 recursion's own rounding (chol_flat_fp64), and idx set to -1 where it fails
  int32_t recip = 0;
  // NN: the candidate lists (location t's M at its offset); the design, the n nearest, goes to
  // idx where that is given
  const int32_t *nn = nullptr;
  int32_t M = 0;
  int64_t N = INT64_MAX;
  int *queue = nullptr;  // a counter that is zero already, or nullptr: one in the workspace
  double *mean, *s2, *var;
  int8_t *status;
};
size_t predict_fp64_workspace_bytes(int64_t T, int32_t nmax, int num_sms);
int predict_fp64_launch(const PredictArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream);
int predict_fp64_prepare();

// Local maximum-likelihood lengthscale of each location's design (mle.cu).
struct MleArgs {
  const double *X, *Z;
  int32_t p;
  int64_t T;
  const int32_t *idx;
  int32_t n;
  double theta0;
  const double *theta0_loc;
  double g, tmin, tmax, tol;
  int32_t maxit;
  double *theta_out;
  int32_t *iters;
  int8_t *status;
};
size_t mle_workspace_bytes(int64_t T, int32_t n, int num_sms);
int mle_launch(const MleArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream);
int mle_prepare();

// MSPE variant of kernels (b)+(c), FP64.
size_t select_mspe_workspace_bytes(int64_t T, int32_t p, int32_t n, int32_t ncand, int num_sms);
size_t select_mspe_needed_bytes(int64_t T, int32_t p, int32_t n, int32_t ncand, int num_sms);
int select_mspe_launch(const SelectArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream);
// MSPE, mixed precision: float-float screen, FP64 bookkeeping and decisions.
size_t select_mspe_mixed_workspace_bytes(int64_t T, int32_t p, int32_t n, int32_t ncand, int num_sms);
int select_mspe_mixed_launch(const SelectArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream);
#define LAGP_MSPE_MIX_CTAS_PER_SM 2  // resident CTAs per SM of the mixed MSPE kernel
#define LAGP_MSPE_CTAS_PER_SM 2      // resident CTAs per SM of the FP64 MSPE kernel

// Batched launch of kernels (b)+(c): per-location tables in device memory (batch.cuh),
// one persistent launch of G = ctas_per_sm x SMs CTAs over the cost-ordered queue.
struct BatchDesign;
struct BatchLaunch {
  int32_t method, precision;
  int64_t T;
  const BatchDesign *designs;  // device
  const LocDesc *locs;         // device, T entries
  const int32_t *order;        // device, queue position -> location
  const double *XX;
  int32_t ldxx;
  const int32_t *cand;         // device; location t's list at locs[t].cand_off
  int32_t nmax, pmax, Mmax;
  double gmin;                 // smallest nugget of the designs
  double *mean, *s2, *var;
  int32_t *idx;                // location t's indices at locs[t].idx_off
  int64_t idx_total;           // sum of the locations' n (the length of idx)
  int8_t *status;
  int32_t ctas_per_sm;         // 1 .. select_max_ctas()
};
int select_max_ctas(int32_t method, int32_t precision);
// Per-translation-unit set-up that must not happen during stream capture (constant uploads).
int select_prepare();
int select_mixed_prepare();
int select_mspe_prepare();
int select_mspe_mixed_prepare();
size_t select_batch_workspace_bytes(const BatchLaunch &b, int num_sms);
int select_batch_launch(const BatchLaunch &b, void *ws, size_t ws_bytes, cudaStream_t stream);
size_t select_batch_needed_bytes(const BatchLaunch &b, int num_sms);
size_t select_mixed_batch_workspace_bytes(const BatchLaunch &b);
size_t select_mixed_batch_needed_bytes(const BatchLaunch &b);
int select_mixed_batch_launch(const BatchLaunch &b, void *ws, size_t ws_bytes, cudaStream_t stream);
size_t select_mspe_batch_workspace_bytes(const BatchLaunch &b, int G);
int select_mspe_batch_launch(const BatchLaunch &b, void *ws, size_t ws_bytes, int G, cudaStream_t stream);
size_t select_mspe_mixed_batch_workspace_bytes(const BatchLaunch &b, int G);
int select_mspe_mixed_batch_launch(const BatchLaunch &b, void *ws, size_t ws_bytes, int G,
                                   cudaStream_t stream);

// Argument checks shared by the entry points (api.cu).
int check_common(int64_t N, int32_t p, int64_t T, int32_t n0, int32_t n, int32_t ncand,
                 double theta, double g, int32_t method, int32_t precision);
int check_supported(int32_t method, int32_t precision);

// Unique id of the calling thread's current CUDA context, 0 if none (api.cu).
int current_context_id(unsigned long long *id);

// Bounds-check records of the checked build (check.cuh): one per instrumented translation
// unit, read and cleared by these (all zero in normal builds).
struct CheckRec {
  unsigned long long count;  // violations since the last take
  long long site, index, bound;
};
int knn_check_take(CheckRec *out);
int select_check_take(CheckRec *out);
int select_mixed_check_take(CheckRec *out);
int select_dense_check_take(CheckRec *out);
int predict_check_take(CheckRec *out);

// Map the last CUDA error to a library code.
int cuda_status(cudaError_t e);

}  // namespace lagp
