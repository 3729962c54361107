// select_mixed.cu -- kernels (b)+(c) for ALC: a candidate screen, FP64 decisions where it is
// close, and FP64 predictive equations.
//
// Gramacy & Apley, Sec. 3: the greedy local design adds, at each step, the candidate that
// maximises the ALC reduction cov_j(x,c)^2 / v_j(c) (Eq. dxy; SM Eq. dxy2).  The screen
// carries, for every candidate, its row of the bordered Cholesky factor, v_j(c) and
// cov_j(x,c) as the FP64 recursion does (select.cu).  FP64 runs at 1/64 of the FP32 rate on
// this GPU, and plain FP32 cannot be used because v_j(c) ~ g = 1e-6 is the difference of O(1)
// quantities, so there are two arithmetics (alc_screen.cuh): LAGP_MIXED screens in compensated
// float-float on the FP32 pipe (46 bits), LAGP_FP64 in 64-bit fixed point on the integer pipe,
// whose scores are as close to the exact ones as those of the FP64 recursion.
//
// Decisions stay FP64-exact where they are close: when the screen's second-best score is
// within DELTA (relative) of its best, the design's FP64 Cholesky factor is rebuilt from
// scratch and every candidate within DELTA is re-scored in FP64 (forward substitution,
// one warp per candidate), the FP64 best winning with ties to the nearer candidate.
// Otherwise the screen's best is taken.  DELTA = 1e-5 is about five times the largest
// discrepancy between the FP64 scores and those of a screen of 46 bits, by emulation (2e-6
// of the best score); with the fixed-point screen the factor and the re-score round exactly as
// the FP64 recursion does, so that every decision is that recursion's.  A location that the fixed
// point does not resolve as FP64 does is listed, and the recursion itself takes it afterwards.
//
// Each thread screens a pair of candidates, and a step needs one block barrier: every thread
// merges the per-warp best/second-best results and derives the step's pivot scalars itself.
// The pivot's coordinates, state and factor row are read from a record that the warp holding
// the step's best wrote before that barrier: no read of the row after it.
//
// The predictive equations (Eqs. predgp, preds2) are evaluated in FP64 on the selected
// designs by kernel (c) in predict.cu afterwards, so mu, s2 and V carry FP64 accuracy
// whatever screened the candidates.
#include <cooperative_groups.h>
#include <math.h>
#include <stdlib.h>

#include <algorithm>

#include "alc_screen.cuh"
#include "batch.cuh"
#include "check.cuh"

namespace lagp {
namespace {

namespace cg = cooperative_groups;


// A location's formats (fx.cuh), and what they are found from.
struct FxFormat {
  int fmt[2];           // sh2b, e
  unsigned dmax, kmax;  // high words of the largest |x_c - x| and K(x, c)
  int near;             // candidates with a K(x, c) within 2^-100 of the largest
  int odd;              // a coordinate is not finite
};

struct MixParams {
  const double *X, *Z;
  int64_t N;       // design rows (uniform launches; batched ones take each design's)
  int p;
  const double *XX;
  int64_t T;
  const int32_t *cand;
  int M, Mpad, Qpad, n0, n;  // Mpad = 2 Qpad: candidates (pairs) per CTA slot, padded
  int nmax, pmax;  // slot dimensions (the largest n and p of the launch)
  double theta, theta_inv, g, onepg;
  BatchView B;     // per-location tables (B.designs == nullptr: uniform launch)
  int32_t *idx;   // selected design indices (required: the caller's or the workspace's)
  void *U;       // slots of n x Qpad candidate pairs: row j of every candidate's factor row
  int smem;      // bytes of dynamic shared memory
  void *Xr;      // slots of p x Qpad pairs: candidate coordinates minus x
  double *A;     // slots of n x (n + 2): FP64 factorisation
  int32_t *list; // FxArith: queue positions left to the FP64 recursion, *nlist of them
  int *nlist;
  int *queue;
  int *rescores; // count of FP64 re-score passes (diagnostics)
  const int32_t *start;  // saved start designs (T x nstart design indices), or nullptr
  int nstart;
  double r_min;          // > 1: stopping rule of Sec. 6; 0: the design has n points
  int32_t *n_out;        // design sizes (T) when r_min > 1
  double *mean, *s2, *var;
  int8_t *status;
  int CL;                // CTAs per cluster (cluster form): they share one location
  int nrec;              // pivot records of a CTA
  int tmem;              // 1: rows in tensor memory
};

// FxArith: a location's state (one CTA): v = 1+g, cov_0(x, c) = K(x, c) in FP64, the coordinates
// relative to x, in formats set by the largest coordinate difference and K(x, c) (compared by
// the high words of their doubles, which are ordered like the values).  Returns whether the
// location is the FP64 recursion's: coordinates that are not finite, or spread so far that the
// format's resolution, 2^(b-58), falls short of FP64's (beyond b = 14 distances lose whole bits, and
// the correlations are no covariance any more); and, where the design is to grow (greedy), x so far
// from every candidate that cov^2 leaves FP64's normal range: there the recursion's scores lose bits
// or tie at 0, and the screen's, scaled by the largest K(x, c) = 2^-w or more, do not.  cov shrinks
// from 2^-w by 2^-53 at most before it is rounding error, and is compared as cov^2 v' with v' of
// 2^-30 or more: 2 (w + 53) + 30 < 1022 for w <= 400.  And fewer than 4 n / 5 candidates with a K(x, c)
// within 2^-100 of the largest (small lengthscales): the later steps would be among candidates whose
// scores are rounding error, a re-score of them all each.  (Emulated, 2000 points on a square of
// side 4, n = 50 of 200, theta = 1e-3: 20 such steps at 20 candidates, 7 at 28, 0.7 at 36; none at 40 and theta
// = 1.3e-3.)
template <int MBT>
__device__ __noinline__ bool fx_location(const LocParams &L, const double *xl, const double *etab, int4 *vp,
                                         int4 *cp, int4 *Xr, unsigned char *used, int Qpad, bool greedy, FxFormat &F) {
  const int tid = threadIdx.x, p = L.p, M = L.M, n = L.n;
  long long *v = reinterpret_cast<long long *>(vp), *cov = reinterpret_cast<long long *>(cp);
  // e even with 1 + g < 2^(e+1)
  const int e = (ilogb(L.onepg) + 1) & ~1;
  const long long onepg = __double2ll_rn(scalbn(L.onepg, 60 - e));
  const double csc = sqrt(L.theta_inv * 1.4426950408889634);  // K = 2^-(squared distance) in these units
  if (tid == 0) {
    F.dmax = F.kmax = 0u;
    F.near = 0;
    F.odd = !(csc >= 0.0 && csc < INFINITY);
  }
  __syncthreads();
  unsigned dmax = 0u, kmax = 0u;
  for (int c = tid; c < 2 * Qpad; c += MBT) {
    // (checked build: a design index past N gets v = 0, so that a start design holding it fails
    // instead of reading its index)
    const bool inside = c < M, live = inside && LAGP_CHK(L.cand[c], L.N, 24);
    double kx = -1.0;  // no coordinates
    if (live) {
      const double *xc = L.X + (int64_t)L.cand[c] * p;
      double acc = 0.0;
      unsigned dm = 0u;
      for (int k = 0; k < p; k++) {
        const double dk = xc[k] - xl[k];
        acc = fma(dk, dk, acc);
        dm = max(dm, (unsigned)__double2hiint(dk) & 0x7fffffffu);
      }
      if (dm < 0x7ff00000u) {
        kx = exp_nonpos(-acc * L.theta_inv, etab);
        dmax = max(dmax, dm);
        kmax = max(kmax, (unsigned)__double2hiint(kx) & 0x7fffffffu);
      } else {
        F.odd = 1;
      }
    }
    used[c] = live ? 0 : 1;
    v[c] = inside && !live ? 0 : onepg;
    reinterpret_cast<double *>(cov)[c] = kx;
  }
  dmax = __reduce_max_sync(0xffffffffu, dmax);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if ((tid & 31) == 0) {
    atomicMax(&F.dmax, dmax);
    atomicMax(&F.kmax, kmax);
  }
  __syncthreads();
  // coordinates at most 2^b in size; K(x, c) scaled by 2^(59 - e + w), the largest in
  // [2^(59-e), 2^(60-e))
  const int b = max(0, (int)(F.dmax >> 20) - 1023 + ilogb(csc) + 2);
  const double fsc = scalbn(csc, 28 - b);
  const int w = min(max(1023 - (int)(F.kmax >> 20), 0), 1022);
  const double kw = scalbn(1.0, w), ke = scalbn(1.0, 59 - e);
  int near = 0;
  for (int c = tid; c < 2 * Qpad; c += MBT) {
    const double kx = reinterpret_cast<double *>(cov)[c];
    const bool live = kx >= 0.0;
    cov[c] = live ? __double2ll_rn(kx * kw * ke) : 0;
    near += kx * kw >= 0x1p-100;
    const double *xc = L.X + (live ? (int64_t)L.cand[c] * p : 0);
    for (int k = 0; k < p; k++) {
      const double f = live ? (xc[k] - xl[k]) * fsc : 0.0;
      const int xh = __double2int_rn(f);
      int *slot = reinterpret_cast<int *>(Xr + k * Qpad + (c >> 1)) + (c & 1);
      slot[0] = xh;
      slot[2] = __double2int_rn((f - (double)xh) * 1073741824.0);  // 2^30
    }
  }
  near = __reduce_add_sync(0xffffffffu, near);
  if ((tid & 31) == 0) atomicAdd(&F.near, near);
  if (tid == 0) {
    F.fmt[0] = min(2 * b, 62);
    F.fmt[1] = e;
  }
  __syncthreads();
  return b > 8 || F.odd || (greedy && (w > 400 || 5 * F.near < 4 * n));
}

// FxArith: whether a location is better left to the FP64 recursion after re-scores of weight m / 8 (8 and
// one per candidate each) in `steps` greedy steps, at a design of j + 1 points: if they go on at that
// pace, they take more than half as long as the recursion.  A pass rebuilds the design's factor, a
// chain of about 3.2 us per column; the recursion takes 8 us a step and 0.25 ns more per candidate
// and (n + 60) (GB300, 300 locations, n = 50 and 100, M = 200 to 2000).  Designs without such structure
// re-score 0 to 2 times in 44 steps.  Whole calls, the recursion alone, every re-score made, this
// rule: near-duplicate points, n = 50 of 200 0.65, 4.28, 0.80 ms, n = 100 of 400 2.49, 27.9, 2.76; theta =
// 1e-3, n = 50 of 1000 1.77, 261, 1.85.
__device__ __forceinline__ bool rescore_pace(int m, int steps, int j, int n, int M) {
  const float rest = 0.2f * (float)(n * n - j * j) * (float)m / (float)steps;
  const float all = (float)n * (8.0f + (float)M * (float)(n + 60) * 2.5e-4f);
  return m >= 24 && 2.0f * rest > all;
}

// MBT threads per CTA, one location per CTA, one or two candidate pairs per thread up to 1024
// candidates (more in turn beyond).  An SM always holds kScrThreads threads of 128 registers: a
// spilled operand comes back from L2, since shared memory leaves no L1, and the row loops are
// free of spills at 128 only.  A location of more candidates gets a larger share of an SM's
// shared and tensor memory and fewer locations are in flight: the factor rows -- read again at
// every later step -- then stay on the chip or in L2.  GB300, whole calls in float-float,
// against three or four CTAs of 256 threads at 80 or 64 registers for every size, records of
// the pivot gathered after the barrier and a ring of prefetched rows: 10000 2-d locations, n =
// 50 of 1000, 14.05 -> 13.32 ms; 10000 8-d ones, n = 100 of 2000, 131.4 -> 118.2 ms; one location,
// n = 50 of 1000, 524 -> 442 us.
// TM: rows R .. R + RT - 1 of each candidate are also kept in the CTA's tensor memory (its
// share of the 512 columns: 128 words per thread, RT = 32, 16 or 8 rows for 1, 2 or up to 4
// pairs per thread) and the screen reads them from there instead of L2 (four 16-byte loads per
// thread: about 200 cycles from tensor memory against about 580 for L2 hits).  One CTA per location only (not the cluster form).
// CLU: the cluster form.  The P.CL CTAs of a thread-block cluster share one location, CTA
// `crank` holding the candidate pairs crank*Qc .. crank*Qc + Qc - 1 (its own v, cov, flags,
// factor rows and coordinates); a step's pivot state -- v_j(s), cov_j(x,s), u_s and x_s -- is
// read from the CTA that holds s (its shared memory through the cluster, its global rows),
// and the per-warp best scores are merged over the cluster after one cluster barrier.  With
// 1/CL of the locations in flight, the live factor rows shrink by CL and more of each
// CTA's rows fit in shared memory.  Every candidate's arithmetic is the same in both forms.
template <class A, int MBT, int NP, bool CLU>
__global__ void __launch_bounds__(MBT, kScrThreads / MBT) select_mixed_kernel(const __grid_constant__ MixParams P) {
  constexpr bool TM = !CLU;
  using Word = typename A::Word;
  constexpr int NWARP = MBT / 32;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nmax = P.nmax;
  __shared__ __align__(8) uint32_t ytab[A::kFixed ? 2 * kFxTab : 128];
  __shared__ double etab[64];
  __shared__ double xl[kMaxP];
  constexpr int NRED = NWARP * (CLU ? kMaxCL : 1);  // per-warp results (of the cluster)
  __shared__ unsigned red_k1[2][NRED], red_k2[2][NRED];  // score keys, double-buffered by step
  __shared__ int red_r1[2][NRED], red_buf[2][NWARP];
  __shared__ double xr_n[CLU ? kMaxCL : 1], xr_d[CLU ? kMaxCL : 1];  // per-CTA FP64 re-score bests
  __shared__ int xr_r[CLU ? kMaxCL : 1];
  __shared__ double red_n[NWARP], red_d[NWARP];
  __shared__ int red_rr[NWARP];
  __shared__ int sh_loc, sh_fail, sh_nlist, sh_per, sh_passes;
  __shared__ LocParams L;  // the location's parameters: read where they are used
  __shared__ FxFormat fx;                // the location's formats (FxArith)
  __shared__ unsigned sh_top[3], sh_nwr[3];  // by step: best score key of the warps that are done,
                                             // records begun
  __shared__ uint32_t sh_tmem;
  if constexpr (TM) {
    // this CTA's share of the SM's tensor memory (the host checks that the resident CTAs'
    // shares fit, so the allocation never waits), released at the end of the kernel
    if (threadIdx.x < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(&sh_tmem)),
                   "n"(tmem_cols(MBT))
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  if (threadIdx.x < 64) etab[threadIdx.x] = c_exp.tab[threadIdx.x];
  if constexpr (A::kFixed) {
    for (int i = threadIdx.x; i < kFxTab; i += MBT)
      reinterpret_cast<uint64_t *>(ytab)[i] = c_exp.fx.tab[i];
  } else if (threadIdx.x < 64) {
    ytab[threadIdx.x] = __float_as_uint(c_exp.tabf_h[threadIdx.x]);
    ytab[64 + threadIdx.x] = __float_as_uint(c_exp.tabf_l[threadIdx.x]);
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int CL = CLU ? P.CL : 1;
  int crank = 0;
  if constexpr (CLU) crank = (int)cg::this_cluster().block_rank();
  Word *U = static_cast<Word *>(P.U) + (size_t)blockIdx.x * nmax * P.Qpad;
  Word *Xr = static_cast<Word *>(P.Xr) + (size_t)blockIdx.x * P.pmax * P.Qpad;
  const int lda = nmax + 1;
  double *Af = P.A + (size_t)blockIdx.x * nmax * (nmax + 2);
  // this thread's tensor-memory words: its warp's lane quarter, its part of the columns
  const uint32_t tb = TM ? sh_tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(kTmemWords * (warp >> 2))
                         : 0u;

  for (;;) {
    int qloc;  // the location's queue position (one per cluster in the cluster form)
    if constexpr (CLU) {
      cg::this_cluster().sync();
      if (crank == 0 && tid == 0) sh_loc = atomicAdd(P.queue, 1);
      cg::this_cluster().sync();
      qloc = *cg::this_cluster().map_shared_rank(&sh_loc, 0);
    } else {
      __syncthreads();
      if (tid == 0) sh_loc = atomicAdd(P.queue, 1);
      __syncthreads();
      qloc = sh_loc;
    }
    if (qloc >= P.T) break;
    if (tid == 0)
      L = resolve_loc(P.B, qloc, P.X, P.Z, P.XX, P.p, P.n, P.M, P.n0, P.theta, P.g, P.cand, P.idx, P.N);
    __syncthreads();
    const int n = L.n, p = L.p, M = L.M;
    // checked build: the location fits the slot (rows, candidates, coordinates)
    if (!(LAGP_CHK(n - 1, nmax, 13) && LAGP_CHK(M - 1, CL * P.Mpad, 14) && LAGP_CHK(p - 1, P.pmax, 15)))
      continue;
    // the start design: the n0 nearest, or a saved design (augmentation)
    const int n0e = P.start ? P.nstart : L.n0;
    // Without greedy steps (n0 == n) only the start design's own rows are ever read.
    const int Q = ((n0e == n && !P.start ? n : M) + 1) >> 1;
    // this CTA's candidate pairs: q0 .. q0 + Ql - 1 of the location's (M + 1) / 2 (all of
    // them outside the cluster form), of which the first Qs are screened
    const int Qm = (M + 1) >> 1;
    const int Qc = CLU ? (Qm + CL - 1) / CL : Qm;
    const int q0 = CLU ? crank * Qc : 0;
    const int Ql = CLU ? max(0, min(Qc, Qm - q0)) : Qm;
    const int Qs = CLU ? max(0, min(Ql, Q - q0)) : Q;
    // Shared memory is laid out for the location: its pairs' v and cov, the pivot records, the
    // design, the used flags, and as many of its factor rows as the rest holds.
    const int Qpad = (Qc + 31) & ~31, nrow = (n + 1) & ~1, recw = A::rec_words(n);
    Word *vp = reinterpret_cast<Word *>(smraw);                // Qpad: v_j(c) pairs
    Word *cp = vp + Qpad;                                      // Qpad: cov_j(x, c) pairs
    int2 *recs = reinterpret_cast<int2 *>(cp + Qpad);          // P.nrec x recw
    int *dr = reinterpret_cast<int *>(recs + P.nrec * recw);   // n (padded to 4)
    int *rlist = dr + ((n + 3) & ~3);                          // RESCORE_CAP
    unsigned char *used = reinterpret_cast<unsigned char *>(rlist + RESCORE_CAP);  // 2 Qpad
    Word *Us = reinterpret_cast<Word *>(used + 2 * Qpad);      // R x Qpad: first factor rows
    int R = (P.smem - (int)(reinterpret_cast<unsigned char *>(Us) - smraw)) / (Qpad * (int)sizeof(Word));
    R = R < n ? R & ~1 : n;  // even: every stretch of the row loops starts at an even entry
    // rows R .. R + RT - 1 in tensor memory: 16, 8 or 4 rows per pair for up to 2, 4 or 8 pairs
    // per thread (one: 32), so that they fit the thread's words in whole loads of four rows
    const int slots = NP * ((Qpad + NP * MBT - 1) / (NP * MBT));
    const int RT = TM && P.tmem ? 4 * (kTmemWords / 16 / slots) : 0;
    // checked build: the layout above ends within the launch's dynamic shared memory
    if (!LAGP_CHK(reinterpret_cast<unsigned char *>(Us + (size_t)R * Qpad) - smraw,
                  dynamic_smem_bytes() + 1u, 20))
      continue;
    if (tid < p) xl[tid] = L.x[tid];
    if (tid == 0) {
      sh_fail = sh_passes = 0;
      // a last round of up to 64 pairs would leave nearly all threads idle for its row loops' latency:
      // rounds of like size then (600 8-d locations, n = 100 of 2100: 11.3 -> 10.3 ms; a larger rest is
      // better on its own)
      const int full = NP * MBT, q32 = (Qs + 31) & ~31, rest = q32 % full, rounds = (q32 + full - 1) / full;
      sh_per = MBT == 512 && q32 > full && rest > 0 && rest <= 64 ? ((q32 + rounds - 1) / rounds + 31) & ~31 : full;
    }
    __syncthreads();
    bool hand = false;  // (FxArith) the location is left to the FP64 recursion
    if constexpr (A::kFixed) {
      hand = fx_location<MBT>(L, xl, etab, vp, cp, Xr, used, Qpad, n0e < n, fx);
      if (hand && tid == 0) sh_fail = 1;
    } else {
      // coordinates relative to x over sqrt(theta), v = 1+g, cov_0(x,c) = K(x,c) in FP64, all as
      // float-float pairs
      const ff onepg = ff_from_double(L.onepg);
      const double sc = sqrt(L.theta_inv);
      for (int q = tid; q < Qpad; q += MBT) {
        ff cv[2];
        bool flagged[2] = {false, false};  // checked build: a design index past N
        for (int h = 0; h < 2; h++) {
          const int c = 2 * q + h;             // this CTA's index
          const int cgl = 2 * (q0 + q) + h;    // the location's candidate rank
          bool live = CLU ? (q < Ql && cgl < M) : (c < M);
          if (live && !LAGP_CHK(L.cand[cgl], L.N, 11)) {
            live = false;
            flagged[h] = true;
          }
          cv[h] = ff{0.0f, 0.0f};
          const double *xc = L.X + (live ? (int64_t)L.cand[cgl] * p : 0);
          double acc = 0.0;
          for (int k = 0; k < p; k++) {
            const double dk = live ? xc[k] - xl[k] : 0.0;
            const ff fk = ff_from_double(dk * sc);
            float *slot = reinterpret_cast<float *>(Xr + k * Qpad + q);
            slot[h] = fk.h;
            slot[2 + h] = fk.l;
            acc = fma(dk, dk, acc);
          }
          if (live) cv[h] = ff_from_double(exp_nonpos(-acc * L.theta_inv, etab));
          used[c] = live ? 0 : 1;
        }
        // (a flagged candidate gets v = 0, so that a start design holding it fails instead of
        // reading its index)
        vp[q] = Word{(decltype(Word::x))(flagged[0] ? 0.0f : onepg.h), (decltype(Word::x))(flagged[1] ? 0.0f : onepg.h),
                     (decltype(Word::x))(flagged[0] ? 0.0f : onepg.l), (decltype(Word::x))(flagged[1] ? 0.0f : onepg.l)};
        cp[q] = Word{(decltype(Word::x))cv[0].h, (decltype(Word::x))cv[1].h, (decltype(Word::x))cv[0].l,
                     (decltype(Word::x))cv[1].l};
      }
    }
    if (tid == 0) sh_top[0] = sh_nwr[0] = 0u;
    // Cluster form: the first steps read the start pivots' v, cov and coordinates from
    // the CTA holding them, so every CTA's state must be in place before any step begins
    // (a stale value read there would let the CTAs' decisions, and barriers, diverge).
    if constexpr (CLU) cg::this_cluster().sync();
    else __syncthreads();
    if (P.start) start_ranks(P.start + L.loc * P.nstart, P.nstart, L.cand, M, dr);

    int best = 0;
    int ne = n;       // the design's size (n, or where the stopping rule ends it)
    ff vx = ff_from_double(L.onepg);  // v_j(x), carried by every thread for the stopping rule
    // the pivot record in use, and whether it holds the step's pivot already
    int active = 0;
    bool have = false;
    for (int j = hand ? n : 0; j < n; j++) {
      const int s = (j < n0e) ? (P.start ? dr[j] : j) : best;
      if (s < 0) {  // nothing admissible left (the same for every thread)
        if (tid == 0) sh_fail = 1;
        break;
      }
      // the pivot's CTA in the cluster (so) and its index there (sl)
      int so = 0, sl = s;
      if constexpr (CLU) {
        so = (s >> 1) / Qc;
        sl = s - 2 * so * Qc;
      }
      if (CLU || !have) {
        // a pivot whose record is not in place (forced, re-scored, or held by another CTA):
        // every thread derives the scalars, the CTA gathers the row
        const Word *vps = vp, *cps = cp, *Uss = Us, *Ugs = U, *Xrs = Xr;
        if constexpr (CLU) {
          cg::cluster_group cl = cg::this_cluster();
          vps = cl.map_shared_rank(vp, so);
          cps = cl.map_shared_rank(cp, so);
          Uss = cl.map_shared_rank(Us, so);
          const size_t other = (size_t)((int)blockIdx.x - crank + so);
          Ugs = static_cast<const Word *>(P.U) + other * nmax * P.Qpad;
          Xrs = static_cast<const Word *>(P.Xr) + other * P.pmax * P.Qpad;
        }
        if (!A::positive(vps, sl)) {
          if (tid == 0) sh_fail = 1;
          break;
        }
        const typename A::Scalars ps = A::scalars(vps, cps, sl);
        active = 0;
        int2 *rec = recs + active * recw;
        for (int i = tid; i < j; i += MBT)
          A::rec_entry(rec, i, nrow, (i < R ? Uss : Ugs) + (size_t)i * Qpad, sl);
        if (tid < p) A::rec_coord(rec, tid, Xrs + tid * Qpad, sl);
        if (tid == 0) A::scalars_store(rec, ps);
        __syncthreads();
      }
      const int2 *rec = recs + active * recw;
      if (!A::kFixed && P.r_min > 0.0) {
        // Sec. 6 stopping rule: stop before a greedy point whose variance reduction ratio
        // v_j(x) / v_{j+1}(x) (psi cancels) is below r_min; every thread decides alike
        const ff ux = A::scalars_ux(rec);
        const ff vxn = ff_sub(vx, ff_mul(ux, ux));
        if (j >= n0e && ff_to_double(vx) / ff_to_double(vxn) < P.r_min) {
          ne = j;
          break;
        }
        vx = vxn;
      }
      if (tid == 0) dr[j] = s;
      if (crank == so && tid == 0) used[sl] = 1;  // (the screen tests for the pivot itself)
      if (j == n - 1) break;
      const bool want = j + 1 >= n0e;
      float b1 = -1.0f, b2 = -1.0f;
      int r1 = 0x7fffffff;
      const StepCtx<A> C{U, Us, R, Xr, vp, cp, used, rec, ytab, fx.fmt, Qpad, nrow, p, j,
                         CLU && crank != so ? -1 : sl, 2 * q0, want, tb, RT};
      // whole warps (tensor-memory accesses are warp-collective): pairs up to the next
      // multiple of 32 (all within Qpad; those past Qs only update state nobody reads), each
      // round's in two halves of whole warps
      const int Q32 = (Qs + 31) & ~31;
      // (two forms: the first alone spills in fixed point, the second alone runs the 256-thread
      // float-float instance 4 % slower, n = 100 of 1000)
      if constexpr (MBT == 512 || !A::kFixed) {
        const int per = sh_per;  // pairs of a round
        for (int base = 0, k = 0; base < Q32; base += per, k += NP) {
          const int left = min(per, Q32 - base), dq = NP == 1 ? MBT : min(MBT, ((left >> 1) + 31) & ~31);
          if (tid < min(dq, left)) screen_pairs<A, MBT, NP, TM>(C, base + tid, b1, r1, b2, k, tid + dq < left ? dq : 0);
        }
      } else {
        for (int q = tid, k = 0; q - tid < Q32; q += NP * MBT, k += NP) {
          const int left = Q32 - (q - tid), dq = NP == 1 ? MBT : min(MBT, ((left >> 1) + 31) & ~31);
          if (tid < min(dq, left)) screen_pairs<A, MBT, NP, TM>(C, q, b1, r1, b2, k, q + dq < Q32 ? dq : 0);
        }
      }
      // best and second-best screen scores of the warp; the warp writes the record of its own
      // best candidate as the next step's pivot before the barrier, so that the gather of the
      // row (L2) and the scalars are off the path between the barrier and the next screen.
      // Only a warp ahead of all that are done writes one (the winner always is; of eight warps
      // in any order, 2.7 on average), in the records other than the one in use in turn; where
      // they run out, the CTA gathers the pivot after the barrier.
      const int par = j & 1;
      if (tid == 0) sh_top[(j + 1) % 3] = sh_nwr[(j + 1) % 3] = 0u;  // (last used two steps ago)
      if (want) {
        unsigned k1 = score_key(b1), k2 = score_key(b2);
        warp_best2(k1, r1, k2);
        unsigned top = 0u;
        if (!CLU && lane == 0) top = atomicMax(&sh_top[j % 3], k1);
        int buf = -1;
        if (!CLU && k1 && k1 >= __shfl_sync(0xffffffffu, top, 0)) {
          if (lane == 0) buf = (int)atomicAdd(&sh_nwr[j % 3], 1u);
          buf = __shfl_sync(0xffffffffu, buf, 0);
          buf = buf < P.nrec - 1 ? buf + (buf >= active ? 1 : 0) : -1;
        }
        if (buf >= 0) {
          const int sl2 = r1;
          int2 *nrec_ = recs + buf * recw;
          __syncwarp();  // this step's rows, v and cov of the warp's candidates are in place
          if (j + 2 < n)
            for (int i = lane; i <= j; i += 32)
              A::rec_entry(nrec_, i, nrow, (i < R ? Us : U) + (size_t)i * Qpad, sl2);
          if (lane < p) A::rec_coord(nrec_, lane, Xr + lane * Qpad, sl2);
          const typename A::Scalars np = A::scalars(vp, cp, sl2);
          if (lane == 0) A::scalars_store(nrec_, np);
        }
        if (lane == 0) {
          if constexpr (CLU) {  // into every CTA of the cluster
            cg::cluster_group cl = cg::this_cluster();
            const int en = crank * NWARP + warp;
            for (int r = 0; r < CL; r++) {
              cl.map_shared_rank(&red_k1[par][0], r)[en] = k1;
              cl.map_shared_rank(&red_k2[par][0], r)[en] = k2;
              cl.map_shared_rank(&red_r1[par][0], r)[en] = r1;
            }
          } else {
            red_k1[par][warp] = k1;
            red_k2[par][warp] = k2;
            red_r1[par][warp] = r1;
            red_buf[par][warp] = buf;
          }
        }
      }
      if constexpr (CLU) cg::this_cluster().sync();
      else __syncthreads();
      have = false;
      if (!want) continue;
      // every warp merges the CTA's (the cluster's) entries: lane l takes entries l, l + 32
      unsigned K1 = 0u, K2 = 0u;
      int R1 = 0x7fffffff;
      const int nred = CL * NWARP;
      if (lane < nred) {
        K1 = red_k1[par][lane];
        K2 = red_k2[par][lane];
        R1 = red_r1[par][lane];
      }
      if (CLU && lane + 32 < nred) merge_keys(red_k1[par][lane + 32], red_r1[par][lane + 32],
                                              red_k2[par][lane + 32], K1, R1, K2);
      const int ew = warp_best2(K1, R1, K2);
      best = K1 ? R1 : -1;
      if (!CLU && K1) {
        const int buf = red_buf[par][ew];
        have = buf >= 0;
        if (have) active = buf;
      }
      // Candidates closer than DELTA are decided in FP64.  For the FP64 precision the margin
      // also covers the FP64 recursion's own rounding of cov_j(x, c) where that is small: 2^13
      // units, 2^-46 of the largest K(x, c), or where cov has outgrown that and has been shifted
      // (Scalars::csh), of the largest u_x u_c, which fills the same 2^59 units.
      float delta = DELTA;
      if constexpr (A::kFixed) {
        if (K1) delta += 8192.0f / fmaxf(fabsf(fx_to_float(A::get64(cp, best))), 1.0f);
      }
      const float B1 = __uint_as_float(K1 - 1u), B2 = __uint_as_float(K2 - 1u);
      const bool near = K1 && K2 && B2 >= B1 * (1.0f - delta);
      if (!near) continue;
      // ---- FP64 re-score of the near-tied candidates (rare) ----
      if (tid == 0 && crank == 0 && P.rescores) atomicAdd(P.rescores, 1);
      // each CTA re-scores its own near-tied candidates (the FP64 factor of the design, the
      // same in every CTA, is formed by each)
      const RescoreCtx R{L.X, L.cand, xl, etab, used, vp, cp, dr, Af, Af + nmax * lda, rlist, &sh_nlist, &sh_fail,
                         red_n, red_d, red_rr, p, 2 * q0, CLU ? min(2 * Ql, M - 2 * q0) : M, j + 1, lda,
                         L.theta_inv, L.onepg, delta, A::kFixed};
      double bn, bd;
      int br;
      rescore_fp64<A>(R, B1, &bn, &bd, &br);
      if (sh_fail) break;  // the same in every CTA of a cluster
      if constexpr (A::kFixed) {
        __syncthreads();  // (every thread has read sh_fail)
        if (tid == 0 && rescore_pace(sh_passes += 8 + sh_nlist, j + 2 - n0e, j, L.n, L.M)) sh_fail = 1;
        __syncthreads();
        if (sh_fail) break;
      }
      if constexpr (CLU) {  // the cluster's FP64 best, ties to the nearer candidate
        cg::cluster_group cl = cg::this_cluster();
        if (tid == 0)
          for (int r = 0; r < CL; r++) {
            cl.map_shared_rank(xr_n, r)[crank] = bn;
            cl.map_shared_rank(xr_d, r)[crank] = bd;
            cl.map_shared_rank(xr_r, r)[crank] = br;
          }
        cl.sync();
        bn = xr_n[0];
        bd = xr_d[0];
        br = xr_r[0];
        for (int r = 1; r < CL; r++)
          if (frac_better(xr_n[r], xr_d[r], xr_r[r], bn, bd, br)) {
            bn = xr_n[r];
            bd = xr_d[r];
            br = xr_r[r];
          }
      }
      const int rb = br != 0x7fffffff ? br : A::kFixed ? -1 : best;
      if (rb != best) have = false;
      best = rb;
    }
    // (cluster form: the last step's pivot reads of the other CTAs' state are done before
    // any CTA moves on and reuses or discards it)
    if constexpr (CLU) cg::this_cluster().sync();
    else __syncthreads();
    // the design (design indices), or -1 when a step failed; kernel (c) (predict.cu)
    // evaluates the predictive equations on it in FP64.  (FxArith: whatever stopped the screen, the
    // recursion decides whether the location fails.)
    if constexpr (A::kFixed)
      if (sh_fail && tid == 0) P.list[atomicAdd(P.nlist, 1)] = sh_loc;  // (its queue position)
    if (crank == 0) {
      for (int i = tid; i < n; i += MBT)
        L.idx[i] = (sh_fail || i >= ne || !LAGP_CHK(dr[i], M, 16)) ? -1 : L.cand[dr[i]];
      if (P.n_out && tid == 0) P.n_out[L.loc] = sh_fail ? 0 : ne;
    }
    // The factor rows in global memory are dead now (the next location rewrites each row
    // before reading it): drop their L2 lines without writing them back to DRAM.
    {
      char *u0 = reinterpret_cast<char *>(U + (size_t)R * Qpad);
      const int nlines = (int)(((size_t)(n > R ? n - R : 0) * Qpad * sizeof(int4)) / 128);
      for (int l = tid; l < nlines; l += MBT)
        asm volatile("discard.global.L2 [%0], 128;" ::"l"(u0 + (size_t)l * 128) : "memory");
    }
  }
  // no CTA of a cluster exits while another may still read its shared memory
  if constexpr (CLU) cg::this_cluster().sync();
  if constexpr (TM) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (threadIdx.x < 32)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sh_tmem),
                   "n"(tmem_cols(MBT))
                   : "memory");
  }
}

// The kernel instance of a launch: threads per CTA and CTAs per location (CL > 1: the cluster
// form, 256 threads).
struct MixVariant {
  int MBT;
  int NP;      // pairs a thread takes at a time
  int CL;
  bool fixed;  // FxArith (LAGP_FP64) instead of FfArith (LAGP_MIXED)
};

// Pivot records of a CTA: the one in use and up to six begun in a step; fewer where the rest of
// the state would leave the SM fewer CTAs.
constexpr int kRecords = 7;

// Dynamic shared memory without the factor rows.
size_t mix_state_bytes(int Qpad, int n, int nrec, MixVariant v) {
  const size_t recw = v.fixed ? FxArith::rec_words(n) : FfArith::rec_words(n);
  return (size_t)Qpad * 2 * sizeof(int4) + nrec * recw * sizeof(int2) +
         (size_t)((n + 3) & ~3) * sizeof(int) + RESCORE_CAP * sizeof(int) + (size_t)2 * Qpad;
}

template <class A>
const void *mix_kernel_of(int MBT, int NP) {
  return NP == 1      ? reinterpret_cast<const void *>(select_mixed_kernel<A, 128, 1, false>)
         : MBT == 128 ? reinterpret_cast<const void *>(select_mixed_kernel<A, 128, 2, false>)
         : MBT == 256 ? reinterpret_cast<const void *>(select_mixed_kernel<A, 256, 2, false>)
                      : reinterpret_cast<const void *>(select_mixed_kernel<A, 512, 2, false>);
}
const void *mix_kernel(MixVariant v) {
  if (v.CL > 1) return reinterpret_cast<const void *>(select_mixed_kernel<FfArith, 256, 2, true>);
  return v.fixed ? mix_kernel_of<FxArith>(v.MBT, v.NP) : mix_kernel_of<FfArith>(v.MBT, v.NP);
}

size_t mix_static_smem(MixVariant v) {
  cudaFuncAttributes fa;
  return cudaFuncGetAttributes(&fa, mix_kernel(v)) == cudaSuccess ? fa.sharedSizeBytes : 4096;
}

// Resident CTAs per SM the instance is compiled for.
int mix_minb(MixVariant v) { return kScrThreads / v.MBT; }

// Launch-shape overrides for measurements (they change no result): LAGP_MIX_CLUSTER = CTAs
// per location (1, 2, 4 or 8), LAGP_MIX_TMEM = 0 (no rows in tensor memory).  -1: not set.
int mix_env(const char *name) {
  const char *e = getenv(name);
  return e && *e ? atoi(e) : -1;
}

// One CTA per location: the cluster form (several) measured slower on every workload.
int mix_cluster_size() {
  const int e = mix_env("LAGP_MIX_CLUSTER");
  return e == 1 || e == 2 || e == 4 || e == 8 ? e : 1;
}

MixVariant mix_variant(int64_t T, int M, int n, int p, int CL, bool fixed, const DevInfo &di) {
  if (CL > 1) return MixVariant{256, 2, CL, false};
  const int threads = mix_threads(T, M, n, p, ScreenChip{di.num_sms, di.l2, di.smem_per_sm + kTmemBytes});
  return MixVariant{threads, mix_qpad(M, 1) <= 128 ? 1 : 2, 1, fixed};
}

// A CTA's share of an SM's shared memory, without what it takes besides (static, 1 KB reserved).
size_t mix_share(MixVariant v, const DevInfo &di) {
  return std::min(di.smem_per_sm / mix_minb(v), di.smem_optin + 1024) - (mix_static_smem(v) + 1024);
}

// Records and dynamic shared memory of a launch whose largest location has Qpad pairs and n
// points: a CTA takes its whole share of the SM, the factor rows filling what the state leaves
// (row i is read at every step after step i, so the first rows carry the most traffic; the
// rest stream from tensor memory and L2); a state larger than the share takes what it needs.
void mix_smem(int Qpad, int n, MixVariant v, const DevInfo &di, int *nrec, size_t *smem) {
  const size_t share = mix_share(v, di);
  *nrec = v.CL > 1 ? 1 : kRecords;
  while (*nrec > 1 && mix_state_bytes(Qpad, n, *nrec, v) > share) --*nrec;
  const size_t need = mix_state_bytes(Qpad, n, *nrec, v);
  *smem = need > share ? need : share;
  const size_t all = need + (size_t)n * Qpad * sizeof(int4);  // every row
  if (*smem > all) *smem = all;
}

// CTAs of a uniform launch: the instance's resident CTAs per SM (one location each), or in
// the cluster form as many clusters of CL as can be resident at once (at most one per
// location).
int mix_grid(int64_t T, int num_sms, MixVariant v) {
  int64_t g = (int64_t)num_sms * mix_minb(v);
  return (int)(T < g ? (T > 0 ? T : 1) : g);
}

cudaLaunchConfig_t mix_config(MixVariant v, int G, size_t smem, cudaStream_t stream,
                              cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G, 1, 1);
  cfg.blockDim = dim3(v.MBT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  if (v.CL > 1) {
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = v.CL;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  return cfg;
}

int mix_cluster_grid(int64_t T, MixVariant v, size_t smem, const DevInfo &di, int *G) {
  const int st = allow_smem(mix_kernel(v), di);
  if (st) return st;
  const int num_sms = di.num_sms;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = mix_config(v, v.CL, smem, nullptr, attr);
  int nc = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&nc, mix_kernel(v), &cfg);
  if (e != cudaSuccess) return cuda_status(e);
  if (nc < 1) return LAGP_ERR_INVALID_ARG;
  int64_t c = nc;
  c = c < (int64_t)num_sms * mix_minb(v) / v.CL ? c : (int64_t)num_sms * mix_minb(v) / v.CL;
  c = c < (T > 0 ? T : 1) ? c : (T > 0 ? T : 1);
  *G = (int)(c * v.CL);
  return LAGP_OK;
}

// The screen, then kernel (c) on the designs it selected, then (FP64) the recursion on the listed
// locations, whose designs are -1 until then.
int mix_run(MixParams P, MixVariant v, const MixLayout &L, int G, char *w, size_t ws_bytes, int32_t *user_idx,
            const SelectArgs *sa, const BatchLaunch *sb, const DevInfo &di, cudaStream_t stream) {
  P.queue = reinterpret_cast<int *>(w);
  P.nlist = reinterpret_cast<int *>(w + 64);
  P.rescores = reinterpret_cast<int *>(w + 256);
  P.list = reinterpret_cast<int32_t *>(w + 512);
  char *o = w + 512 + L.list;
  P.U = o;
  o += L.u;
  P.Xr = o;
  o += L.xr;
  P.A = reinterpret_cast<double *>(o);
  o += L.a;
  // the design goes to the caller's idx, or to the workspace when the caller wants none
  P.idx = user_idx ? user_idx : reinterpret_cast<int32_t *>(o);
  o += L.idx;
  P.CL = v.CL;
  // LAGP_MIX_TMEM=0 turns the rows in tensor memory off (for measurements; no result changes)
  P.tmem = mix_env("LAGP_MIX_TMEM") != 0;
  size_t smem;
  mix_smem(P.Qpad, P.nmax, v, di, &P.nrec, &smem);
  P.smem = (int)smem;
  if (smem > di.smem_optin) return LAGP_ERR_INVALID_ARG;
  const int st = allow_smem(mix_kernel(v), di);
  if (st) return st;
  cudaError_t e;
  if (v.CL == 1) {
    // every resident CTA holds its share of the SM's 512 tensor-memory columns, and an allocation
    // must never wait: no more than mix_minb CTAs may be resident.  Their registers see to it
    // unless the compiler needs fewer than the 128 it may take; then the CTA's whole share of
    // shared memory, of which one more would not find any left, does
    int k = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, mix_kernel(v), v.MBT, smem);
    if (e != cudaSuccess) return cuda_status(e);
    if (k > mix_minb(v)) {
      smem = std::max(smem, mix_share(v, di));
      P.smem = (int)smem;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, mix_kernel(v), v.MBT, smem);
      if (e != cudaSuccess) return cuda_status(e);
    }
    if (k * tmem_cols(v.MBT) > 512) return LAGP_ERR_CUDA;
  }
  e = cudaMemsetAsync(w, 0, 512, stream);  // the counters
  if (e != cudaSuccess) return cuda_status(e);
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = mix_config(v, G, smem, stream, attr);
  void *args[] = {&P};
  e = cudaLaunchKernelExC(&cfg, mix_kernel(v), args);
  if (e != cudaSuccess) return cuda_status(e);
  g_launches.fetch_add(1);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e);
  PredictArgs pa;
  pa.X = P.X; pa.Z = P.Z; pa.p = P.pmax; pa.XX = P.XX; pa.T = P.T; pa.n = P.n; pa.nmax = P.nmax;
  pa.theta = P.theta; pa.g = P.g; pa.idx = P.idx; pa.B = P.B;
  pa.B.n_loc = P.n_out;  // adaptive designs: kernel (c) on each location's own size
  pa.recip = v.fixed;    // FP64: the recursion's own rounding, and no design where it fails
  pa.mean = P.mean; pa.s2 = P.s2; pa.var = P.var; pa.status = P.status;
  pa.queue = reinterpret_cast<int *>(w + 192);  // (one of the counters: no launch between the two kernels)
  const int sp = predict_fp64_launch(pa, o, L.pred, stream);
  if (sp || !v.fixed) return sp;
  const size_t used = 512 + L.list;
  return select_listed_launch(sa, sb, HandedList{reinterpret_cast<int *>(w + 128), P.list, P.nlist}, w + used,
                              ws_bytes - used, stream);
}

// A batch's instance suits its largest candidate count; the grid is the batch's share of
// select_max_ctas() CTAs per SM, of that instance's residents.
MixVariant mix_batch_variant(const BatchLaunch &b, const DevInfo &di) {
  return mix_variant(b.T, b.Mmax, b.nmax, b.pmax, 1, b.precision == LAGP_FP64, di);
}
int mix_batch_grid(const BatchLaunch &b, const DevInfo &di) {
  const int most = select_max_ctas(b.method, b.precision);
  const int ctas = b.ctas_per_sm < 1 || b.ctas_per_sm > most ? most : b.ctas_per_sm;
  const int64_t g = (int64_t)di.num_sms * mix_minb(mix_batch_variant(b, di)) * ctas / most;
  return (int)(g < 1 ? 1 : g < b.T ? g : b.T);
}

}  // namespace

int select_mixed_check_take(CheckRec *out) { return check_take_here(out); }

size_t select_mixed_workspace_bytes(int64_t T, int32_t p, int32_t n, int32_t ncand, int32_t precision, int num_sms) {
  const bool fixed = precision == LAGP_FP64;
  return mix_asked_bytes(T, p, n, ncand, T * n, predict_fp64_workspace_bytes(T, n, num_sms), num_sms, !fixed,
                         fixed ? T : 0);
}

// The grid of a uniform launch (not the cluster form) in ws_bytes, 0: no room.
static int mix_uniform_fit(const SelectArgs &a, MixVariant v, size_t ws_bytes, const DevInfo &di) {
  return mix_fit(mix_grid(a.T, di.num_sms, v), ws_bytes, a.p, a.n, mix_qpad(a.M, 1), a.T * a.n,
                 predict_fp64_workspace_bytes(a.T, a.n, di.num_sms), di.num_sms, v.fixed ? a.T : 0);
}

size_t select_mixed_needed_bytes(const SelectArgs &a) {
  DevInfo di;
  if (dev_info(&di)) return SIZE_MAX;
  const bool fixed = a.precision == LAGP_FP64;
  const MixVariant v = mix_variant(a.T, a.M, a.n, a.p, fixed ? 1 : mix_cluster_size(), fixed, di);
  if (v.CL > 1) return select_mixed_workspace_bytes(a.T, a.p, a.n, a.M, a.precision, di.num_sms);
  const int64_t G = std::min<int64_t>(mix_grid(a.T, di.num_sms, v), di.num_sms);
  return mix_layout(G, a.p, a.n, mix_qpad(a.M, 1), a.T * a.n, predict_fp64_workspace_bytes(a.T, a.n, di.num_sms),
                    fixed ? a.T : 0).total;
}

int select_mixed_launch(const SelectArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream) {
  if (a.T == 0) return LAGP_OK;
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  st = exp_table_upload();
  if (st) return st;
  const bool fixed = a.precision == LAGP_FP64;
  const MixVariant v = mix_variant(a.T, a.M, a.n, a.p, fixed ? 1 : mix_cluster_size(), fixed, di);
  const int Qpad = mix_qpad(a.M, v.CL);
  int G = mix_grid(a.T, di.num_sms, v);
  if (v.CL > 1) {
    int nrec;
    size_t smem;
    mix_smem(Qpad, a.n, v, di, &nrec, &smem);
    st = mix_cluster_grid(a.T, v, smem, di, &G);
    if (st) return st;
  }
  const size_t pred = predict_fp64_workspace_bytes(a.T, a.n, di.num_sms);
  if (v.CL == 1) G = mix_uniform_fit(a, v, ws_bytes, di);
  if (G < 1) return LAGP_ERR_INVALID_ARG;
  const MixLayout L = mix_layout(G, a.p, a.n, Qpad, a.T * a.n, pred, v.fixed ? a.T : 0);
  if (ws_bytes < L.total) return LAGP_ERR_INVALID_ARG;
  MixParams P;
  P.X = a.X; P.Z = a.Z; P.N = a.N; P.p = a.p; P.XX = a.XX; P.T = a.T; P.cand = a.cand;
  P.M = a.M; P.Qpad = Qpad; P.Mpad = 2 * Qpad; P.n0 = a.n0; P.n = a.n;
  P.theta = a.theta; P.theta_inv = 1.0 / a.theta; P.g = a.g; P.onepg = 1.0 + a.g;
  P.nmax = a.n; P.pmax = a.p;
  P.B = BatchView{nullptr, nullptr, nullptr, 0, a.theta_loc, nullptr};
  P.start = a.start; P.nstart = a.nstart;
  P.r_min = a.r_min; P.n_out = a.n_out;
  P.mean = a.mean; P.s2 = a.s2; P.var = a.var; P.status = a.status;
  return mix_run(P, v, L, G, static_cast<char *>(ws), ws_bytes, a.idx, &a, nullptr, di, stream);
}

size_t select_mixed_batch_workspace_bytes(const BatchLaunch &b) {
  DevInfo di;
  const int sms = dev_info(&di) == LAGP_OK ? di.num_sms : 152;
  return mix_asked_bytes(b.T, b.pmax, b.nmax, b.Mmax, b.idx_total, predict_fp64_workspace_bytes(b.T, b.nmax, sms), sms,
                         false, b.precision == LAGP_FP64 ? b.T : 0);
}

// A batch's grid in ws_bytes, 0: no room.
static int mix_batch_fit(const BatchLaunch &b, size_t ws_bytes, const DevInfo &di) {
  return mix_fit(mix_batch_grid(b, di), ws_bytes, b.pmax, b.nmax, mix_qpad(b.Mmax, 1), b.idx_total,
                 predict_fp64_workspace_bytes(b.T, b.nmax, di.num_sms), di.num_sms,
                 b.precision == LAGP_FP64 ? b.T : 0);
}

size_t select_mixed_batch_needed_bytes(const BatchLaunch &b) {
  DevInfo di;
  if (dev_info(&di)) return SIZE_MAX;
  const int64_t G = std::min<int64_t>(mix_batch_grid(b, di), di.num_sms);
  return mix_layout(G, b.pmax, b.nmax, mix_qpad(b.Mmax, 1), b.idx_total,
                    predict_fp64_workspace_bytes(b.T, b.nmax, di.num_sms), b.precision == LAGP_FP64 ? b.T : 0).total;
}

// (Locations grouped by candidate count, one launch of a fitting instance each, measured slower:
// 3000 locations of up to 4000 candidates 90.6 -> 97.1 ms, the launches' tails.)
int select_mixed_batch_launch(const BatchLaunch &b, void *ws, size_t ws_bytes, cudaStream_t stream) {
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  st = exp_table_upload();  // this translation unit's copy of the exp constants
  if (st) return st;
  const int Qpad = mix_qpad(b.Mmax, 1), G = mix_batch_fit(b, ws_bytes, di);
  if (G < 1) return LAGP_ERR_INVALID_ARG;
  const MixLayout L = mix_layout(G, b.pmax, b.nmax, Qpad, b.idx_total,
                                 predict_fp64_workspace_bytes(b.T, b.nmax, di.num_sms),
                                 b.precision == LAGP_FP64 ? b.T : 0);
  MixParams P;
  P.X = nullptr; P.Z = nullptr; P.N = 0; P.p = b.pmax; P.XX = b.XX; P.T = b.T; P.cand = b.cand;
  P.M = b.Mmax; P.Qpad = Qpad; P.Mpad = 2 * Qpad; P.n0 = 0; P.n = b.nmax;
  P.theta = 1.0; P.theta_inv = 1.0; P.g = 0.0; P.onepg = 1.0;
  P.nmax = b.nmax; P.pmax = b.pmax;
  P.B = BatchView{b.designs, b.locs, b.order, b.ldxx, nullptr, nullptr};
  P.start = nullptr; P.nstart = 0;
  P.r_min = 0.0; P.n_out = nullptr;
  P.mean = b.mean; P.s2 = b.s2; P.var = b.var; P.status = b.status;
  return mix_run(P, mix_batch_variant(b, di), L, G, static_cast<char *>(ws), ws_bytes, b.idx, nullptr, &b, di, stream);
}

int select_mixed_prepare() {
  const int st = exp_table_upload();
  return st ? st : predict_fp64_prepare();
}

}  // namespace lagp
