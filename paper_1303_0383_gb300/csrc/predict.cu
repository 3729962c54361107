// predict.cu -- kernel (c): the FP64 predictive equations (Sec. 2, Eqs. predgp and preds2) on
// the selected design of every location, or (NN) on its n nearest candidates, with the
// per-location arithmetic of predict_loc.cuh.
//
// FP64 issues two lanes per clock and SM here, so a warp instruction costs the same 16 clocks
// for one lane as for 32: a pivot's square root and reciprocal, taken by one thread, were half
// of the FP64 work of a 50-point factorisation.  The group kernel factors several locations in
// step, one team of threads each, and one further warp takes all their pivots in its lanes,
// while the teams update the rest of their matrices: a step is two barriers.  Every entry's
// operations and their order are those of chol_flat_fp64, so the results are bit for bit the
// one-location kernel's, which stays for matrices too large for shared memory (n > 208, the
// line: packed triangles of one location and of the index table fill the 227 KB).
// GB300, NN's 3000 locations, one-location kernel or the recursion before -> groups: n = 50
// 2.65 -> 0.45 ms, n = 100 7.74 -> 1.95, n = 180 20.8 -> 12.7, n = 208 27.5 -> 18.1 (one-location
// kernel at n = 209, 128 threads: 24.8); one location: n = 50 267 -> 69 us, n = 208 2.40 -> 0.91 ms.
#include <math.h>

#include "check.cuh"
#include "predict_loc.cuh"

namespace lagp {
namespace {

constexpr int PB = 512;              // threads per CTA of the one-location kernel
constexpr int kMaxGroup = 8;         // locations of a group
constexpr int kGroupMaxN = 208;      // largest n of the group kernel
constexpr size_t kGroupSmem = 112 * 1024;  // two CTAs per SM where a group of two or more fits

struct PredParams {
  const double *X, *Z;
  int p;
  const double *XX;
  int64_t T;
  int n, nmax;
  double theta, g;
  const int32_t *idx;     // selected design indices (location t's n at its offset)
  BatchView B;
  int recip;              // chol_flat_fp64's; and a failed location's design is set to -1
  const int32_t *nn;      // NN: the candidate lists (location t's M at its offset), else nullptr
  int M;
  int64_t N;
  double *mean, *s2, *var;
  int8_t *status;
  double *Ag;             // per-CTA matrix slots when the matrix is not in shared memory
  int group;              // locations per CTA (group kernel)
  int *queue;
};

__device__ __forceinline__ LocParams pred_loc(const PredParams &P, int64_t q) {
  LocParams L = resolve_loc(P.B, q, P.X, P.Z, P.XX, P.p, P.n, P.M, 0, P.theta, P.g,
                            P.nn, const_cast<int32_t *>(P.idx), P.N);
  return L;
}

// The location's design: its own indices, or its n nearest candidates.
__device__ __forceinline__ const int32_t *pred_design(const PredParams &P, const LocParams &L) {
  return P.nn ? L.cand : L.idx;
}

// NN's design to the caller, or -1 where a factorisation failed.
__device__ __forceinline__ void pred_idx_out(const PredParams &P, const LocParams &L, bool fail, int i0,
                                             int step) {
  if (!L.idx || !(P.nn || (P.recip && fail))) return;
  for (int i = i0; i < L.n; i += step) L.idx[i] = fail ? -1 : L.cand[i];
}

// checked build: a design index past N fails the location
__device__ __forceinline__ bool pred_index_ok(const PredParams &P, const LocParams &L, const int32_t *d,
                                              int i) {
  return LAGP_CHK(d[i], L.N, P.nn ? 24 : 41);
}

// One location in 512 threads: each column's update is n^2 / 2 entries behind two block barriers, and
// 128 threads took 110 rounds of loads from L2 for it at n = 256.  GB300, 128 -> 512 threads: n = 220
// one location 5.12 -> 1.51 ms, 600 9.71 -> 4.59, 3000 29.7 -> 22.0; n = 256 8.67 -> 2.46, 16.3 -> 7.26,
// 46.1 -> 34.4.
__global__ void __launch_bounds__(PB, 2) predict_fp64_kernel(PredParams P) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nmax = P.nmax;
  double *rl = reinterpret_cast<double *>(smraw);     // nmax: 1 / l_kk
  double *A = P.Ag + (size_t)blockIdx.x * nmax * (nmax + 2);
  __shared__ double etab[64];
  __shared__ double xl[kMaxP];
  __shared__ int sh_loc, sh_fail;
  const int tid = threadIdx.x;
  if (tid < 64) etab[tid] = c_exp.tab[tid];

  for (;;) {
    __syncthreads();
    if (tid == 0) sh_loc = atomicAdd(P.queue, 1);
    __syncthreads();
    if (sh_loc >= P.T) break;
    const LocParams L = pred_loc(P, sh_loc);
    const int32_t *d = pred_design(P, L);
    if (tid < L.p) xl[tid] = L.x[tid];
    bool ok = d[0] >= 0;  // (a failed location has no design: nothing to check)
    if (ok)
      for (int i = tid; i < L.n; i += PB) ok = ok && pred_index_ok(P, L, d, i);
    if (!__syncthreads_and(ok)) {
      if (tid == 0) predict_failed(L.loc, P.mean, P.s2, P.var, P.status);
      pred_idx_out(P, L, true, tid, PB);
      continue;
    }
    predict_location(L, d, L.n, xl, A, rl, etab, &sh_fail, L.loc, P.mean, P.s2, P.var,
                     P.status, P.recip != 0);
    pred_idx_out(P, L, sh_fail != 0, tid, PB);
  }
}

// A location of the group: the matrix's lower triangle, packed, then k(x), Y and 1 / l_kk.
__host__ __device__ constexpr size_t group_loc_words(int nmax) {
  return (size_t)nmax * (nmax + 1) / 2 + 3 * (size_t)nmax;
}
size_t group_smem_bytes(int nmax, int G) {
  return G * group_loc_words(nmax) * sizeof(double) +
         align_up((size_t)nmax * (nmax + 1) / 2 * sizeof(uint16_t), 16);
}

// P.group teams of TT threads, one location each, and one warp for their pivots.
template <int TT>
__global__ void __launch_bounds__(TT == 64 ? 64 * kMaxGroup + 32 : 2 * TT + 32)
predict_group_kernel(PredParams P) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nmax = P.nmax, G = P.group;
  const size_t words = group_loc_words(nmax);
  double *As = reinterpret_cast<double *>(smraw);              // G locations
  uint16_t *tri = reinterpret_cast<uint16_t *>(As + G * words);  // entry e of a triangle: row << 8 | column
  __shared__ double etab[64];
  __shared__ LocParams Ls[kMaxGroup];
  __shared__ double xls[kMaxGroup][kMaxP];
  __shared__ int sh_loc, sh_fail[kMaxGroup];
  const int tid = threadIdx.x, lane = tid & 31;
  const int g = tid / TT, t = tid % TT;  // team and thread in it; g == G: the pivot warp
  const bool pivots = g == G;
  for (int i = tid; i < 64; i += blockDim.x) etab[i] = c_exp.tab[i];
  for (int a = tid; a < nmax; a += blockDim.x)
    for (int b = 0; b <= a; b++) tri[a * (a + 1) / 2 + b] = (uint16_t)(a << 8 | b);

  for (;;) {
    __syncthreads();
    if (tid == 0) sh_loc = atomicAdd(P.queue, G);
    __syncthreads();
    const int64_t base = sh_loc;
    if (base >= P.T) break;
    const int live = (int)(P.T - base < G ? P.T - base : G);
    if (pivots && lane < live) {
      Ls[lane] = pred_loc(P, base + lane);
      const LocParams &L = Ls[lane];
      for (int k = 0; k < L.p; k++) xls[lane][k] = L.x[k];
      sh_fail[lane] = pred_design(P, L)[0] < 0;
    }
    __syncthreads();
    int steps = 0;  // the group's largest n
    for (int h = 0; h < live; h++) steps = max(steps, Ls[h].n);
    const bool mine = !pivots && g < live;
    double *A = As + (size_t)(pivots ? (lane < G ? lane : 0) : g) * words;
    const int own = pivots ? lane : g;
    const int n = own < live ? Ls[own].n : 0, ntri = n * (n + 1) / 2;
    double *B = A + ntri, *rl = B + 2 * n;  // k(x) and Y interleaved; 1 / l_kk
    if (mine && !sh_fail[g]) {
      const int32_t *d = pred_design(P, Ls[g]);
      for (int i = t; i < n; i += TT)
        if (!pred_index_ok(P, Ls[g], d, i)) sh_fail[g] = 1;
    }
    __syncthreads();
    if (mine && !sh_fail[g]) {
      // K_n + g I (lower triangle), k(x) and Y
      const LocParams &L = Ls[g];
      const int32_t *d = pred_design(P, L);
      const int p = L.p;
      for (int e = t; e < ntri + 2 * n; e += TT) {
        if (e < ntri) {
          const int a = tri[e] >> 8, b = tri[e] & 255;
          A[e] = (a == b) ? L.onepg
                          : pl_corr(L.X + (int64_t)d[a] * p, L.X + (int64_t)d[b] * p, p, L.theta_inv, etab);
        } else {
          const int a = (e - ntri) >> 1, col = (e - ntri) & 1;
          B[e - ntri] = col == 0 ? pl_corr(L.X + (int64_t)d[a] * p, xls[g], p, L.theta_inv, etab) : L.Z[d[a]];
        }
      }
    }
    __syncthreads();
    // right-looking Cholesky of the group's matrices in step (chol_flat_fp64's operations)
    for (int k = -1; k < steps; k++) {
      const int kk = k * (k + 1) / 2 + k;  // the pivot's entry (k >= 0)
      if (mine && k >= 0 && k < n && !sh_fail[g]) {
        const double lkk = A[kk], r = rl[k];
        for (int i = k + 1 + t; i < n + 2; i += TT) {
          double *ap = i < n ? &A[i * (i + 1) / 2 + k] : &B[2 * k + i - n];
          const double a = *ap, q = a * r;
          *ap = (P.recip && i < n) ? q : div_by_pivot(a, q, lkk, r, false);
        }
      }
      __syncthreads();
      if (pivots) {
        const int i = k + 1, row = i * (i + 1) / 2;
        if (i < n && !sh_fail[lane]) {
          double v = A[row + i];
          if (k >= 0) v = fma(-A[row + k], A[row + k], v);
          if (!(v > 0.0)) sh_fail[lane] = 1;
          const double lv = sqrt(v);
          A[row + i] = lv;
          rl[i] = 1.0 / lv;
        }
      } else if (mine && k >= 0 && k < n) {
        const int rows = n - k - 1, ntr = rows * (rows + 1) / 2;
        for (int e = 1 + t; e < ntr + 2 * rows; e += TT) {
          if (e < ntr) {
            const int i = k + 1 + (tri[e] >> 8), l = k + 1 + (tri[e] & 255), row = i * (i + 1) / 2;
            A[row + l] = fma(-A[row + k], A[l * (l + 1) / 2 + k], A[row + l]);
          } else {
            const int i = k + 1 + ((e - ntr) >> 1), col = (e - ntr) & 1;
            B[2 * i + col] = fma(-A[i * (i + 1) / 2 + k], B[2 * k + col], B[2 * i + col]);
          }
        }
      }
      __syncthreads();
    }
    // Where a quotient of k(x) or Y may not be the division's (div_sure): their forward substitutions
    // once more, divided.  A zero is sure if it leads its column and was zero there.  A check at each
    // division instead cost every pivot (NN, n = 50, 100 locations: 69.9 us; unchecked 68.0, so 68.1).
    bool redo = false;
    if (P.recip && mine && !sh_fail[g])
      for (int e = t; e < 2 * n; e += TT)
        if (!div_sure(B[e]))
          redo = redo || B[e] != 0.0 || !(e & 1) || (e > 1 && B[e - 2] != 0.0) ||
                 Ls[g].Z[pred_design(P, Ls[g])[e >> 1]] != 0.0;
    if (__syncthreads_or(redo)) {
      const bool again = mine && !sh_fail[g];
      if (again) {
        const LocParams &L = Ls[g];
        const int32_t *d = pred_design(P, L);
        for (int e = t; e < 2 * n; e += TT) {
          const int a = e >> 1;
          B[e] = (e & 1) == 0 ? pl_corr(L.X + (int64_t)d[a] * L.p, xls[g], L.p, L.theta_inv, etab) : L.Z[d[a]];
        }
      }
      __syncthreads();
      for (int k = 0; k < steps; k++) {
        if (again && k < n && t < 2) B[2 * k + t] = B[2 * k + t] / A[k * (k + 1) / 2 + k];
        __syncthreads();
        if (again)
          for (int e = 2 * (k + 1) + t; e < 2 * n; e += TT)
            B[e] = fma(-A[(e >> 1) * ((e >> 1) + 1) / 2 + k], B[2 * k + (e & 1)], B[e]);
        __syncthreads();
      }
    }
    if (pivots && lane < live) {
      const LocParams &L = Ls[lane];
      if (sh_fail[lane]) predict_failed(L.loc, P.mean, P.s2, P.var, P.status);
      else predict_sums(B, 2, n, L.onepg, L.loc, P.mean, P.s2, P.var, P.status);
    }
    if (mine) pred_idx_out(P, Ls[g], sh_fail[g] != 0, t, TT);
  }
}

// Locations per CTA and threads per location: as many as two CTAs per SM leave room for, but
// no more than spread the locations over the SMs; 64 threads each, or 256 for one or two.
struct GroupShape {
  int G, TT;
};
GroupShape group_shape(int64_t T, int nmax, const DevInfo &di) {
  int G = (int)(kGroupSmem / (group_loc_words(nmax) * sizeof(double) + 1024));
  if (G < 1) G = 1;
  if (G > kMaxGroup) G = kMaxGroup;
  const int64_t even = ceil_div(T, 2 * (int64_t)di.num_sms);  // spreads the locations evenly
  if (even < G) G = (int)even;
  return GroupShape{G, G <= 2 ? 256 : 64};
}

bool use_group(int nmax) { return nmax <= kGroupMaxN; }

size_t pred_smem_bytes(int nmax) { return (size_t)nmax * sizeof(double); }

int pred_grid(int64_t T, int nmax, const DevInfo &di) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, predict_fp64_kernel, PB,
                                                    pred_smem_bytes(nmax)) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  const int64_t g = (int64_t)di.num_sms * per_sm;
  return (int)(T < g ? (T > 0 ? T : 1) : g);
}

// Worst-case grid for sizing the workspace before the occupancy is known: at most this many
// CTAs of 512 threads per SM (2048 threads per SM).
int pred_grid_bound(int64_t T, int num_sms) {
  const int64_t g = (int64_t)num_sms * (2048 / PB);
  return (int)(T < g ? (T > 0 ? T : 1) : g);
}

}  // namespace

size_t predict_fp64_workspace_bytes(int64_t T, int32_t nmax, int num_sms) {
  size_t b = 256;
  if (!use_group(nmax))
    b += align_up((size_t)pred_grid_bound(T, num_sms) * nmax * (nmax + 2) * sizeof(double), 256);
  return b;
}

int predict_fp64_launch(const PredictArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream) {
  if (a.T == 0) return LAGP_OK;
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  st = exp_table_upload();  // this translation unit's copy of the exp constants
  if (st) return st;
  if (ws_bytes < predict_fp64_workspace_bytes(a.T, a.nmax, di.num_sms)) return LAGP_ERR_INVALID_ARG;
  char *w = static_cast<char *>(ws);
  PredParams P;
  P.X = a.X; P.Z = a.Z; P.p = a.p; P.XX = a.XX; P.T = a.T; P.n = a.n; P.nmax = a.nmax;
  P.theta = a.theta; P.g = a.g; P.idx = a.idx;
  P.B = a.B;
  P.recip = a.recip; P.nn = a.nn; P.M = a.M; P.N = a.N;
  P.mean = a.mean; P.s2 = a.s2; P.var = a.var; P.status = a.status;
  P.queue = a.queue ? a.queue : reinterpret_cast<int *>(w);
  P.Ag = nullptr;
  P.group = 0;
  cudaError_t e = a.queue ? cudaSuccess : cudaMemsetAsync(P.queue, 0, sizeof(int), stream);
  if (e != cudaSuccess) return cuda_status(e);
  if (use_group(a.nmax)) {
    const GroupShape s = group_shape(a.T, a.nmax, di);
    P.group = s.G;
    const size_t smem = group_smem_bytes(a.nmax, s.G);
    const void *fn = s.TT == 64 ? reinterpret_cast<const void *>(predict_group_kernel<64>)
                                : reinterpret_cast<const void *>(predict_group_kernel<256>);
    const int threads = s.G * s.TT + 32;
    st = allow_smem(fn, di);
    if (st) return st;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
    if (e != cudaSuccess) return cuda_status(e);
    if (per_sm < 1) return LAGP_ERR_CUDA;
    const int64_t groups = ceil_div(a.T, s.G), most = (int64_t)di.num_sms * per_sm;
    void *args[] = {&P};
    e = cudaLaunchKernel(fn, dim3((unsigned)(groups < most ? groups : most)), dim3(threads), args, smem, stream);
    if (e != cudaSuccess) return cuda_status(e);
  } else {
    int G = pred_grid(a.T, a.nmax, di);
    const int Gb = pred_grid_bound(a.T, di.num_sms);
    if (G > Gb) G = Gb;
    P.Ag = reinterpret_cast<double *>(w + 256);
    predict_fp64_kernel<<<G, PB, pred_smem_bytes(a.nmax), stream>>>(P);
  }
  g_launches.fetch_add(1);
  return cuda_status(cudaGetLastError());
}

int predict_check_take(CheckRec *out) { return check_take_here(out); }

int predict_fp64_prepare() { return exp_table_upload(); }

}  // namespace lagp
