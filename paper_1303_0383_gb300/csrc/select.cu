// select.cu -- kernels (b)+(c): greedy local design and predictive equations, FP64.
//
// Gramacy & Apley, Sec. 3: starting from the n0 nearest neighbours, the local design
// grows one point at a time; each step adds the candidate c that maximises the ALC
// reduction in variance at x (Eq. dxy; SM "partial correlations", Eq. dxy2):
//     score(c) = cov_j(x,c)^2 / v_j(c),
//     cov_j(a,b) = K(a,b) - k_j(a)^T K_j^{-1} k_j(b),  v_j(c) = cov_j(c,c),
// or, for NN, simply the next nearest.  Sec. 3.2 requires every step to cost O(j^2)
// per candidate at most; this kernel costs O(j) per candidate per step by carrying,
// for every candidate, the row u_c = L_j^{-1} k_j(c) of the bordered Cholesky factor
// L_j of K_j together with v_j(c) and cov_j(x,c).  Adding point s appends
//     L_{j+1} = [[L_j, 0], [u_s^T, sqrt(v_j(s))]]
// (the Cholesky counterpart of the partitioned inverse of SM Sec. 1, with the same
// Schur-complement scalar v_j(s)), and every candidate updates in O(j):
//     u_c[j]     = (K(s,c) - u_s . u_c) / sqrt(v_j(s))      (= cov_j(s,c)/sqrt(v_j(s)))
//     v_{j+1}(c) = v_j(c) - u_c[j]^2                         (Eq. dxy applied at c)
//     cov_{j+1}(x,c) = cov_j(x,c) - u_x[j] u_c[j].
// The same recursion gives u_x = L^{-1} k(x) and ytil = L^{-1} Y, hence
//     psi_{j+1} = psi_j + ytil_j^2   with ytil_j = (y_s - mu_j(s)) / sqrt(v_j(s))
// (Eq. psiup in the form the SM derives for E{psi_{j+1}}), and at the end
// mu = u_x . ytil, v_n(x) = K(x,x) - ||u_x||^2, s2 = psi v_n(x)/n, V = psi v_n(x)/(n-2)
// (Eqs. predgp, preds2).  The start design is built by the same recursion with the
// pivot forced to ranks 0..n0-1.
//
// Correlations use the library's table-driven FP64 exponential (fp64_exp.cuh); ALC scores
// are compared as fractions, without a division per candidate.
//
// Layout: one persistent CTA per resident location (a work counter hands out
// locations).  Per CTA, scratch holds U[j][c] (row j of every candidate, coalesced
// over c) and the candidates' coordinates Xc[k][c]; v, cov(x,.) and the used flags
// live in shared memory.
#include <math.h>

#include <algorithm>

#include "batch.cuh"
#include "check.cuh"
#include "fp64_exp.cuh"
#include "internal.h"

namespace lagp {
namespace {

constexpr int SB = 256;  // threads per CTA

struct SelParams {
  const double *X, *Z;
  int64_t N;       // design rows (uniform launches; batched ones take each design's)
  int p;
  const double *XX;
  int64_t T;
  const int32_t *cand;
  int M, Mpad, n0, n, method;
  int nmax, pmax;  // slot dimensions (the largest n and p of the launch)
  double theta, g;
  double *mean, *s2, *var;
  int32_t *idx;
  int8_t *status;
  double *U;      // gridDim.x slots of nmax x Mpad
  double *Xc;     // gridDim.x slots of pmax x Mpad
  int *queue;
  BatchView B;    // per-location tables (B.designs == nullptr: uniform launch)
  const int32_t *start;  // saved start designs (T x nstart design indices), or nullptr
  int nstart;
  double r_min;          // > 1: stopping rule of Sec. 6 (ALC); 0: the design has n points
  int32_t *n_out;        // design sizes (T) when r_min > 1
  const int32_t *list;   // queue positions to take (*count of them), or nullptr: all T
  const int *count;
};

// ALC scores are compared as fractions cov^2 / v without dividing: a/da beats b/db when
// a*db > b*da (both denominators are positive), ties going to the smaller rank.
__device__ __forceinline__ bool score_better(double a, double da, int ra, double b, double db,
                                             int rb) {
  const double l = a * db, r = b * da;
  return l > r || (l == r && ra < rb);
}

__global__ void __launch_bounds__(SB, 2) select_fp64_kernel(SelParams P) {
  extern __shared__ __align__(16) double sm[];
  const int Mpad = P.Mpad, nmax = P.nmax;
  double *v = sm;                       // Mpad
  double *covx = v + Mpad;              // Mpad
  double *srow = covx + Mpad;           // nmax  (u_s, the new row of L)
  double *ux = srow + nmax;             // nmax  (u_x = L^{-1} k(x))
  double *yt = ux + nmax;               // nmax  (ytil = L^{-1} Y)
  unsigned char *used = reinterpret_cast<unsigned char *>(yt + nmax);  // Mpad
  int *sr = reinterpret_cast<int *>(used + Mpad);                     // nmax: start ranks
  __shared__ double xs[kMaxP], xl[kMaxP];
  __shared__ double red_s[SB / 32], red_d[SB / 32];
  __shared__ int red_r[SB / 32];
  __shared__ double etab[64];
  if (threadIdx.x < 64) etab[threadIdx.x] = c_exp.tab[threadIdx.x];
  __shared__ int sh_loc, sh_best, sh_fail, sh_n;
  __shared__ double sh_inv, sh_uxj, sh_vx, sh_psi;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double *U = P.U + (size_t)blockIdx.x * nmax * Mpad;
  double *Xc = P.Xc + (size_t)blockIdx.x * P.pmax * Mpad;
  // checked build: the layout above ends within the launch's dynamic shared memory
  if (!LAGP_CHK(reinterpret_cast<unsigned char *>(sr + nmax) - reinterpret_cast<unsigned char *>(sm),
                dynamic_smem_bytes() + 1u, 25))
    return;

  // the list's launch may start before kernel (c) has ended: wait for it
  if (P.list) asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t T = P.list ? *P.count : P.T;
  for (;;) {
    __syncthreads();
    if (tid == 0) sh_loc = atomicAdd(P.queue, 1);
    __syncthreads();
    if (sh_loc >= T) break;
    const LocParams L = resolve_loc(P.B, P.list ? P.list[sh_loc] : sh_loc, P.X, P.Z, P.XX, P.p, P.n, P.M, P.n0, P.theta,
                                    P.g, P.cand, P.idx, P.N);
    const int64_t loc = L.loc;
    const int n = L.n, p = L.p, M = L.M;
    // checked build: the location fits the slot (rows, candidates, coordinates)
    if (!(LAGP_CHK(n - 1, nmax, 21) && LAGP_CHK(M - 1, Mpad, 22) && LAGP_CHK(p - 1, P.pmax, 23)))
      continue;
    const int32_t *cnd = L.cand;
    if (tid < p) xl[tid] = L.x[tid];
    if (tid == 0) { sh_fail = 0; sh_vx = L.onepg; sh_psi = 0.0; sh_n = n; }
    __syncthreads();
    // the start design: the n0 nearest, or a saved design (augmentation)
    const int n0e = P.start ? P.nstart : L.n0;
    if (P.start) start_ranks(P.start + loc * P.nstart, P.nstart, cnd, M, sr);
    // Stage candidate coordinates; v = K(c,c) = 1+g, cov_0(x,c) = K(x,c).
    // NN, and ALC without greedy steps (n0 == n), never look past rank n-1
    const int limit = ((P.method == LAGP_NN || n0e == n) && !P.start) ? n : M;
    for (int c = tid; c < limit; c += SB) {
      if (!LAGP_CHK(cnd[c], L.N, 24)) {  // never read, never chosen
        v[c] = 0.0;
        covx[c] = 0.0;
        used[c] = 1;
        continue;
      }
      const double *xc = L.X + (int64_t)cnd[c] * p;
      double acc = 0.0;
      for (int k = 0; k < p; k++) {
        double xk = xc[k];
        Xc[k * Mpad + c] = xk;
        double t = xl[k] - xk;
        acc = fma(t, t, acc);
      }
      v[c] = L.onepg;
      covx[c] = exp_nonpos(-acc * L.theta_inv, etab);
      used[c] = 0;
    }
    __syncthreads();

    int s = 0;
    for (int j = 0; j < n; j++) {
      if (j >= n0e && P.method == LAGP_ALC) s = sh_best;
      else s = (P.start && j < n0e) ? sr[j] : j;
      if (s < 0) {  // nothing admissible left
        if (tid == 0) sh_fail = 1;
        __syncthreads();
        break;
      }
      for (int i = tid; i < j; i += SB) srow[i] = U[(size_t)i * Mpad + s];
      if (tid < p) xs[tid] = Xc[tid * Mpad + s];
      __syncthreads();
      if (tid == 0) {
        const double vs = v[s];
        if (!(vs > 0.0)) {
          sh_fail = 1;
        } else {
          const double sq = sqrt(vs);
          const double uxj = covx[s] / sq;                 // u_x[j]
          const double vxn = fma(-uxj, uxj, sh_vx);       // v_{j+1}(x)
          if (P.r_min > 0.0 && j >= n0e && sh_vx / vxn < P.r_min) {
            // Sec. 6 stopping rule: the design stops before a greedy point whose variance
            // reduction ratio v_j(x) / v_{j+1}(x) (psi cancels) is below r_min
            sh_n = j;
          } else {
            double t = L.Z[cnd[s]];
            for (int i = 0; i < j; i++) t = fma(-srow[i], yt[i], t);
            const double ytj = t / sq;                     // ytil[j]
            ux[j] = uxj;
            yt[j] = ytj;
            sh_vx = vxn;
            sh_psi = fma(ytj, ytj, sh_psi);
            sh_inv = 1.0 / sq;
            sh_uxj = uxj;
            used[s] = 1;
            if (L.idx) L.idx[j] = cnd[s];
          }
        }
      }
      __syncthreads();
      if (sh_n == j) break;
      if (sh_fail) break;
      if (j == n - 1) break;
      const double inv = sh_inv, uxj = sh_uxj;
      const bool want_score = (P.method == LAGP_ALC) && (j + 1 >= n0e);
      double bs = -1.0, bd = 1.0;   // best score as a fraction bs/bd (none yet: -1)
      int br = 0x7fffffff;
      for (int c = tid; c < limit; c += SB) {
        if (used[c]) continue;
        double acc = 0.0;
        for (int k = 0; k < p; k++) {
          double t = xs[k] - Xc[k * Mpad + c];
          acc = fma(t, t, acc);
        }
        double t = exp_nonpos(-acc * L.theta_inv, etab);  // K(s, c)
        const double *Uc = U + c;
        for (int i = 0; i < j; i++, Uc += Mpad) t = fma(-srow[i], *Uc, t);
        const double u = t * inv;                          // u_c[j]
        U[(size_t)j * Mpad + c] = u;
        const double vc = fma(-u, u, v[c]);
        const double cx = fma(-uxj, u, covx[c]);
        v[c] = vc;
        covx[c] = cx;
        if (want_score && vc > 0.0) {
          const double num = cx * cx;                      // ALC reduction num/vc, Eq. dxy
          if (score_better(num, vc, c, bs, bd, br)) { bs = num; bd = vc; br = c; }
        }
      }
      if (want_score) {
        for (int o = 16; o > 0; o >>= 1) {
          double os = __shfl_down_sync(0xffffffffu, bs, o);
          double od = __shfl_down_sync(0xffffffffu, bd, o);
          int orr = __shfl_down_sync(0xffffffffu, br, o);
          if (score_better(os, od, orr, bs, bd, br)) { bs = os; bd = od; br = orr; }
        }
        if (lane == 0) { red_s[warp] = bs; red_d[warp] = bd; red_r[warp] = br; }
        __syncthreads();
        if (warp == 0) {
          bs = (lane < SB / 32) ? red_s[lane] : -1.0;
          bd = (lane < SB / 32) ? red_d[lane] : 1.0;
          br = (lane < SB / 32) ? red_r[lane] : 0x7fffffff;
          for (int o = 16; o > 0; o >>= 1) {
            double os = __shfl_down_sync(0xffffffffu, bs, o);
            double od = __shfl_down_sync(0xffffffffu, bd, o);
            int orr = __shfl_down_sync(0xffffffffu, br, o);
            if (score_better(os, od, orr, bs, bd, br)) { bs = os; bd = od; br = orr; }
          }
          if (lane == 0) sh_best = (br == 0x7fffffff) ? -1 : br;
        }
      }
      __syncthreads();
    }
    __syncthreads();
    const int ne = sh_n;  // the design's size (n, or where the stopping rule ended it)
    if (tid == 0) {
      if (P.n_out) P.n_out[loc] = sh_fail ? 0 : ne;
      if (sh_fail) {
        if (P.status) P.status[loc] = (int8_t)LAGP_ERR_NOT_PD;
        P.mean[loc] = NAN;
        P.s2[loc] = NAN;
        if (P.var) P.var[loc] = NAN;
      } else {
        double mu = 0.0;
        for (int i = 0; i < ne; i++) mu = fma(ux[i], yt[i], mu);
        const double pv = sh_psi * sh_vx;
        P.mean[loc] = mu;
        P.s2[loc] = pv / ne;
        if (P.var) P.var[loc] = pv / (ne - 2);
        if (P.status) P.status[loc] = 0;
      }
    }
    if (L.idx) {
      // A failed location reports no design: every index is -1; an adaptive design's
      // unused slots are -1 too.
      for (int i = tid; i < n; i += SB)
        if (sh_fail || i >= ne) L.idx[i] = -1;
    }
  }
}

int sel_grid(int64_t T, int num_sms) { return (int)rec_grid(T, num_sms); }

int mpad_of(int M) { return (int)align_up((size_t)M, 32); }

size_t sel_smem_bytes(int Mpad, int n) {
  return (size_t)(2 * Mpad + 3 * n) * sizeof(double) + align_up((size_t)Mpad, 16) +
         align_up((size_t)n * sizeof(int), 16);
}

}  // namespace

int select_check_take(CheckRec *out) { return check_take_here(out); }

size_t select_workspace_bytes(int64_t T, int32_t p, int32_t n, int32_t ncand, int32_t method,
                              int32_t precision, int num_sms) {
  if (method == LAGP_MSPE)
    return precision == LAGP_MIXED ? select_mspe_mixed_workspace_bytes(T, p, n, ncand, num_sms)
                                   : select_mspe_workspace_bytes(T, p, n, ncand, num_sms);
  const size_t own = select_scratch_bytes_for_grid(sel_grid(T, num_sms), p, n, ncand);
  if (method == LAGP_NN) return std::max(own, predict_fp64_workspace_bytes(T, n, num_sms));
  const size_t scr = select_mixed_workspace_bytes(T, p, n, ncand, precision, num_sms);
  return precision == LAGP_MIXED || scr > own ? scr : own;
}

// FP64 ALC designs by the fixed-point screen (select_mixed.cu), which resolves v_j(c) >= g at
// least as finely as FP64 does as long as g is well above its unit (2^-57 of 1 + g) and decides
// near ties in this file's own arithmetic; smaller nuggets, where a candidate's v may be
// rounding noise, the stopping rule, NN and callers with the smaller workspace stay here, and so
// does every location that the screen lists (select_listed_launch).
// GB300: 4001 2-d locations, n = 50 of 1000, whole call: 23.1 -> 5.95 ms.
static bool screened(int32_t method, double g, double r_min) {
  return method == LAGP_ALC && g >= 9.3132257461547852e-10 && r_min == 0.0;  // 2^-30
}

// NN's design is given, so it is kernel (c) alone, on the n nearest candidates, with the
// recursion's rounding (bit for bit this file's kernel).  GB300: 10000 locations at n = 50,
// ncand = 1000, with the candidate search: 9.36 -> 2.00 ms; 3000 at n = 208: 27.5 -> 18.1 ms.
static PredictArgs nn_args(const double *XX, int64_t T, int n, const int32_t *cand, int M, double *mean,
                           double *s2, double *var, int32_t *idx, int8_t *status) {
  PredictArgs pa;
  pa.XX = XX; pa.T = T; pa.n = pa.nmax = n; pa.idx = idx;
  pa.recip = 1; pa.nn = cand; pa.M = M;
  pa.mean = mean; pa.s2 = s2; pa.var = var; pa.status = status;
  return pa;
}

size_t select_needed_bytes(const SelectArgs &a, int num_sms) {
  if (a.method == LAGP_MSPE)
    return a.precision == LAGP_MIXED ? select_mspe_mixed_workspace_bytes(a.T, a.p, a.n, a.M, num_sms)
                                     : select_mspe_needed_bytes(a.T, a.p, a.n, a.M, num_sms);
  const size_t own = select_scratch_bytes_for_grid(sel_grid(a.T, num_sms), a.p, a.n, a.M);
  if (a.method == LAGP_NN) return std::min(own, predict_fp64_workspace_bytes(a.T, a.n, num_sms));
  const size_t scr = select_mixed_needed_bytes(a);
  return a.precision == LAGP_MIXED ? scr : screened(a.method, a.g, a.r_min) ? std::min(own, scr) : own;
}

int select_launch(const SelectArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream) {
  if (a.T == 0) return LAGP_OK;
  if (a.method == LAGP_MSPE)
    return a.precision == LAGP_MIXED ? select_mspe_mixed_launch(a, ws, ws_bytes, stream)
                                     : select_mspe_launch(a, ws, ws_bytes, stream);
  if (a.precision == LAGP_MIXED && a.method == LAGP_ALC)
    return select_mixed_launch(a, ws, ws_bytes, stream);
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  st = exp_table_upload();
  if (st) return st;
  if (screened(a.method, a.g, a.r_min) && ws_bytes >= select_mixed_needed_bytes(a))
    return select_mixed_launch(a, ws, ws_bytes, stream);
  if (a.method == LAGP_NN && ws_bytes >= predict_fp64_workspace_bytes(a.T, a.n, di.num_sms)) {
    PredictArgs pa = nn_args(a.XX, a.T, a.n, a.cand, a.M, a.mean, a.s2, a.var, a.idx, a.status);
    pa.X = a.X; pa.Z = a.Z; pa.p = a.p; pa.N = a.N; pa.theta = a.theta; pa.g = a.g;
    pa.B = BatchView{nullptr, nullptr, nullptr, 0, a.theta_loc, nullptr};
    return predict_fp64_launch(pa, ws, ws_bytes, stream);
  }
  const int G = sel_grid(a.T, di.num_sms);
  return select_launch_on_grid(a, ws, ws_bytes, G, stream);
}

int select_default_grid(int64_t T, int num_sms) { return sel_grid(T, num_sms); }

size_t select_scratch_bytes_for_grid(int G, int32_t p, int32_t n, int32_t ncand) {
  return 256 + rec_slots_bytes(G, p, n, ncand);
}

// The arguments of a uniform launch, and of a batch.
static SelParams sel_params(const SelectArgs &a) {
  SelParams P = {};
  P.X = a.X; P.Z = a.Z; P.N = a.N; P.p = a.p; P.XX = a.XX; P.T = a.T; P.cand = a.cand;
  P.M = a.M; P.Mpad = mpad_of(a.M); P.n0 = a.n0; P.n = a.n; P.method = a.method;
  P.theta = a.theta;
  P.g = a.g;
  P.nmax = a.n;
  P.pmax = a.p;
  P.B = BatchView{nullptr, nullptr, nullptr, 0, a.theta_loc, nullptr};
  P.start = a.start; P.nstart = a.nstart;
  P.r_min = a.r_min; P.n_out = a.n_out;
  P.mean = a.mean; P.s2 = a.s2; P.var = a.var; P.idx = a.idx; P.status = a.status;
  return P;
}
static SelParams sel_params(const BatchLaunch &b) {
  SelParams P = {};
  P.p = b.pmax; P.XX = b.XX; P.T = b.T; P.cand = b.cand;
  P.M = b.Mmax; P.Mpad = mpad_of(b.Mmax); P.n = b.nmax; P.method = b.method;
  P.theta = 1.0; P.nmax = b.nmax; P.pmax = b.pmax;
  P.B = BatchView{b.designs, b.locs, b.order, b.ldxx, nullptr, nullptr};
  P.mean = b.mean; P.s2 = b.s2; P.var = b.var; P.idx = b.idx; P.status = b.status;
  return P;
}

// The recursion on G CTAs; slots: rec_slots_bytes(G) of scratch, P.queue a zeroed counter.
static int sel_run(SelParams P, int G, void *slots, const DevInfo &di, cudaStream_t stream) {
  P.U = static_cast<double *>(slots);
  P.Xc = reinterpret_cast<double *>(static_cast<char *>(slots) +
                                    align_up((size_t)G * P.nmax * P.Mpad * sizeof(double), 256));
  const size_t smem = sel_smem_bytes(P.Mpad, P.nmax);
  if (smem > di.smem_optin) return LAGP_ERR_INVALID_ARG;
  const int st = allow_smem(reinterpret_cast<const void *>(select_fp64_kernel), di);
  if (st) return st;
  // A list is empty in nearly every call: its launch overlaps the end of kernel (c), which it waits for
  // itself, instead of following it (one location of 60 candidates: 205 us, 208 following, 202 without).
  cudaLaunchAttribute early;
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(SB);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &early;
  cfg.numAttrs = P.list ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, select_fp64_kernel, P);
  if (e != cudaSuccess) return cuda_status(e);
  g_launches.fetch_add(1);
  return cuda_status(cudaGetLastError());
}

int select_launch_on_grid(const SelectArgs &a, void *ws, size_t ws_bytes, int G,
                          cudaStream_t stream) {
  if (a.T == 0) return LAGP_OK;
  if (G < 1) return LAGP_ERR_INVALID_ARG;
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  st = exp_table_upload();
  if (st) return st;
  if (ws_bytes < select_scratch_bytes_for_grid(G, a.p, a.n, a.M)) return LAGP_ERR_INVALID_ARG;
  SelParams P = sel_params(a);
  P.queue = static_cast<int *>(ws);
  const cudaError_t e = cudaMemsetAsync(P.queue, 0, sizeof(int), stream);   // the work counter starts at zero
  if (e != cudaSuccess) return cuda_status(e);
  return sel_run(P, G, static_cast<char *>(ws) + 256, di, stream);
}

int select_listed_launch(const SelectArgs *a, const BatchLaunch *b, const HandedList &h, void *scratch,
                         size_t bytes, cudaStream_t stream) {
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  st = exp_table_upload();
  if (st) return st;
  SelParams P = a ? sel_params(*a) : sel_params(*b);
  const int64_t G = rec_fit(P.T, bytes, P.pmax, P.nmax, P.M, di.num_sms);
  if (G < 1) return LAGP_ERR_INVALID_ARG;
  P.queue = h.queue; P.list = h.list; P.count = h.count;
  return sel_run(P, (int)G, scratch, di, stream);
}

int select_max_ctas(int32_t method, int32_t precision) {
  if (method == LAGP_MSPE) return precision == LAGP_MIXED ? LAGP_MSPE_MIX_CTAS_PER_SM : LAGP_MSPE_CTAS_PER_SM;
  return 2;
}

static int batch_grid(const BatchLaunch &b, int num_sms) {
  int c = b.ctas_per_sm;
  const int cmax = select_max_ctas(b.method, b.precision);
  if (c < 1 || c > cmax) c = cmax;
  const int64_t g = (int64_t)num_sms * c;
  return (int)(b.T < g ? (b.T > 0 ? b.T : 1) : g);
}

size_t select_batch_workspace_bytes(const BatchLaunch &b, int num_sms) {
  const int G = batch_grid(b, num_sms);
  if (b.method == LAGP_MSPE)
    return b.precision == LAGP_MIXED ? select_mspe_mixed_batch_workspace_bytes(b, G)
                                     : select_mspe_batch_workspace_bytes(b, G);
  const size_t own = select_scratch_bytes_for_grid(G, b.pmax, b.nmax, b.Mmax);
  if (b.method == LAGP_NN) return std::max(own, predict_fp64_workspace_bytes(b.T, b.nmax, num_sms));
  const size_t scr = select_mixed_batch_workspace_bytes(b);
  return b.precision == LAGP_MIXED || scr > own ? scr : own;
}

size_t select_batch_needed_bytes(const BatchLaunch &b, int num_sms) {
  const int G = batch_grid(b, num_sms);
  if (b.method == LAGP_MSPE)
    return b.precision == LAGP_MIXED ? select_mspe_mixed_batch_workspace_bytes(b, G)
                                     : select_mspe_batch_workspace_bytes(b, std::min(G, num_sms));
  const size_t own = select_scratch_bytes_for_grid(G, b.pmax, b.nmax, b.Mmax);
  if (b.method == LAGP_NN) return std::min(own, predict_fp64_workspace_bytes(b.T, b.nmax, num_sms));
  const size_t scr = select_mixed_batch_needed_bytes(b);
  return b.precision == LAGP_MIXED ? scr : screened(b.method, b.gmin, 0.0) ? std::min(own, scr) : own;
}

int select_batch_launch(const BatchLaunch &b, void *ws, size_t ws_bytes, cudaStream_t stream) {
  if (b.T == 0) return LAGP_OK;
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  st = exp_table_upload();
  if (st) return st;
  int G = batch_grid(b, di.num_sms);
  if (b.method == LAGP_MSPE) {
    if (b.precision == LAGP_MIXED) return select_mspe_mixed_batch_launch(b, ws, ws_bytes, G, stream);
    if (ws_bytes < select_mspe_batch_workspace_bytes(b, G)) G = std::min(G, di.num_sms);  // one CTA per SM
    return select_mspe_batch_launch(b, ws, ws_bytes, G, stream);
  }
  if ((b.precision == LAGP_MIXED && b.method == LAGP_ALC) ||
      (screened(b.method, b.gmin, 0.0) && ws_bytes >= select_mixed_batch_needed_bytes(b)))
    return select_mixed_batch_launch(b, ws, ws_bytes, stream);
  if (b.method == LAGP_NN && ws_bytes >= predict_fp64_workspace_bytes(b.T, b.nmax, di.num_sms)) {
    PredictArgs pa = nn_args(b.XX, b.T, b.nmax, b.cand, b.Mmax, b.mean, b.s2, b.var, b.idx, b.status);
    pa.X = pa.Z = nullptr; pa.p = b.pmax; pa.theta = 1.0; pa.g = 0.0;
    pa.B = BatchView{b.designs, b.locs, b.order, b.ldxx, nullptr, nullptr};
    return predict_fp64_launch(pa, ws, ws_bytes, stream);
  }
  if (ws_bytes < select_scratch_bytes_for_grid(G, b.pmax, b.nmax, b.Mmax)) return LAGP_ERR_INVALID_ARG;
  SelParams P = sel_params(b);
  P.queue = static_cast<int *>(ws);
  const cudaError_t e = cudaMemsetAsync(P.queue, 0, sizeof(int), stream);
  if (e != cudaSuccess) return cuda_status(e);
  return sel_run(P, G, static_cast<char *>(ws) + 256, di, stream);
}

int select_prepare() {
  const int st = exp_table_upload();
  return st ? st : predict_fp64_prepare();
}

}  // namespace lagp
