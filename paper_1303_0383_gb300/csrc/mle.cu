// mle.cu -- the local maximum-likelihood lengthscale of each location's design.
//
// Gramacy & Apley, Sec. 4.2 (step 3 of the stagewise scheme): given the local design
// D_n(x), the lengthscale theta maximising the log likelihood Eq. gpk of its responses,
// found by Newton's method with the analytic derivatives Eqs. dl, d2l (Sec. 3.2):
//   l'  = -tr(K^-1 Kd)/2 + (n/2) w^T Kd w / psi,
//   l'' = -tr(K^-1 [Kdd - Kd K^-1 Kd])/2 + n/(2 psi) w^T [Kdd - 2 Kd K^-1 Kd] w
//         + n/(2 psi^2) (w^T Kd w)^2,
// with K = K(X_n, X_n) + g I, w = K^-1 Y, psi = Y^T w, Kd = dK/dtheta = K o R2 / theta^2 and
// Kdd = Kd o (R2 / theta^2 - 2 / theta) off the diagonal (R2 the squared distances; the
// diagonal does not depend on theta).
//
// The iteration is safeguarded: a bracket [lo, hi] of the maximum is narrowed by the sign
// of l'; the Newton step is taken when l'' < 0 and it stays strictly inside the bracket,
// otherwise the iterate goes to the end of [tmin, tmax] uphill of theta if that end has
// not been evaluated, else to the bracket's midpoint; it stops when a step is at most
// tol * theta (the new point is returned), when l' = 0, or at an end of [tmin, tmax]
// where l' points outward.
//
// One CTA per location.  Per iteration, in FP64: K and Kd (one exp per pair), the
// Cholesky factor (fp64_chol.cuh), L^-1 by forward substitution (right-looking, one barrier
// per column), K^-1 = L^-T L^-1 and the O(n^2) vector terms; the n^3 product K^-1 Kd behind
// tr((K^-1 Kd)^2) runs in float-float on the FP32 pipes (K^-1 has large entries of both
// signs, so plain FP32 would leave l'' without a correct digit; float-float keeps about
// 48 bits per product).  The matrices live in shared memory
// when they fit, else in a per-CTA slot of the workspace.
#include <math.h>

#include <algorithm>

#include "ff.cuh"
#include "fp64_chol.cuh"
#include "fp64_exp.cuh"
#include "internal.h"

namespace lagp {
namespace {

constexpr int LB = 256;                      // threads per CTA
constexpr size_t kSmemMle = 110 * 1024;      // largest per-CTA set kept in shared memory
constexpr int kSums = 7;                     // block sums per Newton iteration

struct MleParams {
  const double *X, *Z;
  int p;
  int64_t T;
  const int32_t *idx;  // T x n design indices
  int n;
  double theta0;
  const double *theta0_loc;  // may be null
  double g, tmin, tmax, tol;
  int maxit;
  double *theta_out;
  int32_t *iters;
  int8_t *status;
  unsigned char *slots;  // per-CTA buffers when not in shared memory
  size_t slot_bytes;
  int *queue;
};

// Per-CTA buffers in shared memory: two squares of rows of lda doubles (odd: a column's entries
// lie in different banks), each a symmetric or triangular matrix in its lower triangle, diagonal
// included, and another in its upper one, a packed triangle, and four vectors.
//   S1  lower K, its Cholesky factor L, then K^-1;  upper the squared distances
//   S2  lower Kd;  upper X = L^-1, transposed (x_ii = 1 / l_ii is in rl), then A_ab
//   S3  the design's coordinates, then Kdd, then A_ba
// so that four CTAs share an SM at n = 50 (three with full matrices: 500 locations were a wave
// and a tenth): the factorisation's pivot chain is sequential, and more locations in flight
// hide it.  Squared distances are formed once per location, Kdd once per iteration.  GB300, two
// stages over 500 8-d locations, n = 50, the MLE of the first among them: 11.99 -> 8.22 ms.
__host__ __device__ constexpr int mle_lda(int n) { return n | 1; }
__host__ __device__ constexpr size_t mle_s3_words(int n) {
  return (size_t)n * (n + 1) / 2 > (size_t)n * kMaxP ? (size_t)n * (n + 1) / 2 : (size_t)n * kMaxP;
}
size_t mle_set_bytes(int n) {
  return (2 * (size_t)n * mle_lda(n) + mle_s3_words(n) + 4 * (size_t)n) * sizeof(double);
}
// Larger designs (n > 73), in a slot of the workspace: three full squares (K, L, then K^-1; Kd;
// L^-1, then A), four vectors and the coordinates.  There a walk down a column costs a sector of
// L2 per entry, so symmetric matrices are kept whole and read along rows, or with neighbouring
// threads on neighbouring entries of a row, and distances are formed again from the coordinates.
// GB300, 500 8-d locations, n = 100, packed squares -> these: 50.6 -> 22.6 ms; 100 locations, n =
// 256, 361 -> 211 (in shared memory, n = 73, the packed ones are a fifth faster).
size_t mle_slot_bytes(int n) { return align_up(((size_t)n * n * 3 + (size_t)n * (4 + kMaxP)) * sizeof(double), 256); }

// Lane 0's shuffle-tree sum of v over its warp.
__device__ __forceinline__ double warp_tree_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// What a Newton iteration sums over the design, this thread's share: psi, w^T Kd w, w^T Kdd w,
// kdw^T K^-1 kdw, tr(K^-1 Kd), tr(K^-1 Kdd), tr((K^-1 Kd)^2).
struct MleTerms {
  double psi, q3, q1, q2, t1, t3, t2p;
};

// At lengthscale 1 / tinv, in the packed squares (see above); false (for every thread) where K
// has no factor.
__device__ __forceinline__ bool mle_terms_packed(double *S1, double *S2, double *S3, const double *Y, double *w,
                                                 double *kdw, double *rl, int n, double tinv, double g,
                                                 const double *etab, int *fail, int turn, MleTerms *out) {
  const int tid = threadIdx.x, lda = mle_lda(n), ntri = n * (n + 1) / 2;
  const double tinv2 = tinv * tinv;
  // K, Kd and Kdd: one exp per pair a > b
  for (int e = tid; e < ntri; e += LB) {
    const int a = tri_row(e), b = e - a * (a + 1) / 2;
    double r2 = 0.0, kd = 0.0;
    if (a == b) {
      S1[a * lda + a] = 1.0 + g;
    } else {
      r2 = S1[b * lda + a];
      const double k = exp_nonpos(-r2 * tinv, etab);
      S1[a * lda + b] = k;
      kd = k * r2 * tinv2;
    }
    S2[a * lda + b] = kd;
    S3[e] = kd * fma(r2, tinv2, -2.0 * tinv);
  }
  chol_flat_fp64(S1, n, lda, 0, rl, fail, false, turn);
  if (*fail) return false;
  // X = L^-1: x_ic = -(sum_{c<=m<i} l_im x_mc) / l_ii, x_ii = 1 / l_ii.  Right-looking: at
  // step m every entry (i > m, c <= m) takes its term l_im x_mc -- the same terms in the
  // same order as the row-by-row sums -- and the thread that adds the last term of row
  // m + 1 finishes that entry, so a step is one barrier and all threads share its FP64
  // work.  Row m + 1 runs in a loop of its own: in the shared loop its multiply by 1 / l_ii
  // would be a predicated FP64 instruction issued by every warp.
  for (int m = 0; m < n - 1; m++) {
    const int w1 = m + 1, cnt = (n - 1 - m) * w1;
    {  // row m + 1: its last term, then the division by its pivot
      const int i = m + 1;
      for (int c = tid; c < w1; c += LB) {
        const double x = c == m ? rl[m] : S2[c * lda + m], s = c == m ? 0.0 : S2[c * lda + i];
        S2[c * lda + i] = -fma(S1[i * lda + m], x, s) * rl[i];
      }
    }
    for (int e = w1 + tid; e < cnt; e += LB) {
      const int i = m + 1 + e / w1, c = e % w1;
      const double x = c == m ? rl[m] : S2[c * lda + m], s = c == m ? 0.0 : S2[c * lda + i];
      S2[c * lda + i] = fma(S1[i * lda + m], x, s);
    }
    __syncthreads();
  }
  // K^-1 = X^T X into L's storage, which is no longer needed
  for (int e = tid; e < ntri; e += LB) {
    const int a = tri_row(e), b = e - a * (a + 1) / 2;
    double s = fma(rl[a], a == b ? rl[a] : S2[b * lda + a], 0.0);
    for (int m = a + 1; m < n; m++) s = fma(S2[a * lda + m], S2[b * lda + m], s);
    S1[a * lda + b] = s;
  }
  __syncthreads();
  // w = K^-1 Y, then Kd w (entry (a, b) of a symmetric matrix: along row a up to the
  // diagonal, then down column a)
  for (int a = tid; a < n; a += LB) {
    double s = 0.0;
    for (int b = 0, q = a * lda; b < n; q += b < a ? 1 : lda, b++) s = fma(S1[q], Y[b], s);
    w[a] = s;
  }
  __syncthreads();
  for (int a = tid; a < n; a += LB) {
    double s = 0.0;
    for (int b = 0, q = a * lda; b < n; q += b < a ? 1 : lda, b++) s = fma(S2[q], w[b], s);
    kdw[a] = s;
  }
  __syncthreads();
  // per-row pieces of psi, w^T Kd w, w^T Kdd w, kdw^T K^-1 kdw, tr(K^-1 Kd), tr(K^-1 Kdd)
  double psi = 0.0, q3 = 0.0, q1 = 0.0, q2 = 0.0, t1 = 0.0, t3 = 0.0;
  for (int a = tid; a < n; a += LB) {
    psi = fma(Y[a], w[a], psi);
    q3 = fma(w[a], kdw[a], q3);
    double sdd = 0.0, sq2 = 0.0, st1 = 0.0, st3 = 0.0;
    for (int b = 0, q = a * lda, t = a * (a + 1) / 2; b < n; q += b < a ? 1 : lda, b++, t += b > a ? b : 1) {
      const double kd = S2[q], kdd = S3[t], ki = S1[q];
      sdd = fma(kdd, w[b], sdd);
      sq2 = fma(ki, kdw[b], sq2);
      st1 = fma(ki, kd, st1);
      st3 = fma(ki, kdd, st3);
    }
    q1 = fma(w[a], sdd, q1);
    q2 = fma(kdw[a], sq2, q2);
    t1 += st1;
    t3 += st3;
  }
  __syncthreads();
  // tr((K^-1 Kd)^2) = sum_ab A_ab A_ba with A = K^-1 Kd, the n^3 term: formed in
  // float-float on the FP32 pipes (compensated dots, about 2^-48 per product).  It
  // enters l'' only, which sets the Newton step, not the root l' = 0 the iteration
  // converges to.  K^-1 and Kd are converted in place (their FP64 uses are done), one
  // float-float pair per FP64 slot.
  float2 *Kif = reinterpret_cast<float2 *>(S1), *Kdf = reinterpret_cast<float2 *>(S2);
  for (int e = tid; e < ntri; e += LB) {
    const int a = tri_row(e), q = a * lda + e - a * (a + 1) / 2;
    const ff ki = ff_from_double(S1[q]), kd = ff_from_double(S2[q]);
    Kif[q] = make_float2(ki.h, ki.l);
    Kdf[q] = make_float2(kd.h, kd.l);
  }
  __syncthreads();
  // The pairs a <= b, all lanes busy: (a == b ? 1 : 2) A_ab and A_ba (for a == b both are
  // A_aa)
  for (int e = tid; e < ntri; e += LB) {
    const int b = tri_row(e), a = e - b * (b + 1) / 2;
    ffacc sab{0.0f, 0.0f}, sba{0.0f, 0.0f};
    for (int m = 0, qa = a * lda, qb = b * lda; m < n; qa += m < a ? 1 : lda, qb += m < b ? 1 : lda, m++) {
      const float2 x1 = Kif[qa], y1 = Kdf[qb], x2 = Kif[qb], y2 = Kdf[qa];
      ffacc_add_prod(sab, ff{x1.x, x1.y}, ff{y1.x, y1.y});
      ffacc_add_prod(sba, ff{x2.x, x2.y}, ff{y2.x, y2.y});
    }
    const double vab = (double)sab.h + (double)sab.l, vba = (double)sba.h + (double)sba.l;
    if (a != b) S2[a * lda + b] = 2.0 * vab;
    S3[e] = vba;
  }
  __syncthreads();
  // each thread adds its pairs in the order of the row-major (a, b) scan
  double t2p = 0.0;
  for (int e = tid; e < n * n; e += LB) {
    const int a = e / n, b = e % n;
    if (b < a) continue;
    const double v = S3[b * (b + 1) / 2 + a];
    t2p = fma(a == b ? v : S2[a * lda + b], v, t2p);
  }
  *out = MleTerms{psi, q3, q1, q2, t1, t3, t2p};
  return true;
}

// The same operations on full squares, from the coordinates xd (p per point).
__device__ __forceinline__ bool mle_terms_full(double *Lm, double *Kd, double *Ki, const double *xd, const double *Y,
                                               double *w, double *kdw, double *rl, int n, int p, double tinv, double g,
                                               const double *etab, int *fail, int turn, MleTerms *out) {
  const int tid = threadIdx.x, ntri = n * (n + 1) / 2;
  const double tinv2 = tinv * tinv;
  // squared distance of design points a and b
  auto r2of = [&](int a, int b) {
    double r2 = 0.0;
    for (int k = 0; k < p; k++) {
      const double t = xd[a * p + k] - xd[b * p + k];
      r2 = fma(t, t, r2);
    }
    return r2;
  };
  // K (lower triangle) and Kd (full): one exp per pair a > b, mirrored
  for (int e = tid; e < ntri; e += LB) {
    const int a = tri_row(e), b = e - a * (a + 1) / 2;
    if (a == b) {
      Lm[a * n + a] = 1.0 + g;
      Kd[a * n + a] = 0.0;
    } else {
      const double r2 = r2of(a, b);
      const double k = exp_nonpos(-r2 * tinv, etab);
      Lm[a * n + b] = k;
      const double kd = k * r2 * tinv2;
      Kd[a * n + b] = kd;
      Kd[b * n + a] = kd;
    }
  }
  chol_flat_fp64(Lm, n, n, 0, rl, fail, false, turn);
  if (*fail) return false;
  // X = L^-1 (lower triangle, in Ki's storage): x_ic = -(sum_{c<=m<i} l_im x_mc) / l_ii,
  // x_ii = 1 / l_ii.  Right-looking: at step m every entry (i > m, c <= m) takes its
  // term l_im x_mc -- the same terms in the same order as the row-by-row sums -- and
  // the thread that adds the last term of row m + 1 finishes that entry, so a step is
  // one barrier and all threads share its FP64 work.  Row m + 1 runs in a loop of its
  // own: in the shared loop its multiply by 1 / l_ii would be a predicated FP64
  // instruction issued by every warp.
  double *Xb = Ki;
  for (int e = tid; e < ntri; e += LB) {
    const int a = tri_row(e), b = e - a * (a + 1) / 2;
    Xb[a * n + b] = (a == b) ? rl[a] : 0.0;
  }
  __syncthreads();
  for (int m = 0; m < n - 1; m++) {
    const int w1 = m + 1, cnt = (n - 1 - m) * w1;
    {  // row m + 1: its last term, then the division by its pivot
      const int i = m + 1;
      for (int c = tid; c < w1; c += LB)
        Xb[i * n + c] = -fma(Lm[i * n + m], Xb[m * n + c], Xb[i * n + c]) * rl[i];
    }
    for (int e = w1 + tid; e < cnt; e += LB) {
      const int i = m + 1 + e / w1, c = e % w1;
      Xb[i * n + c] = fma(Lm[i * n + m], Xb[m * n + c], Xb[i * n + c]);
    }
    __syncthreads();
  }
  // K^-1 = X^T X (both triangles) into L's storage, which is no longer needed
  double *KiM = Lm;
  for (int e = tid; e < ntri; e += LB) {
    const int a = tri_row(e), b = e - a * (a + 1) / 2;
    double s = 0.0;
    for (int m = a; m < n; m++) s = fma(Xb[m * n + a], Xb[m * n + b], s);
    KiM[a * n + b] = s;
    KiM[b * n + a] = s;
  }
  __syncthreads();
  // w = K^-1 Y, then Kd w
  for (int a = tid; a < n; a += LB) {
    double s = 0.0;
    for (int b = 0; b < n; b++) s = fma(KiM[a * n + b], Y[b], s);
    w[a] = s;
  }
  __syncthreads();
  for (int a = tid; a < n; a += LB) {
    double s = 0.0;
    for (int b = 0; b < n; b++) s = fma(Kd[a * n + b], w[b], s);
    kdw[a] = s;
  }
  __syncthreads();
  // per-row pieces of psi, w^T Kd w, w^T Kdd w, kdw^T K^-1 kdw, tr(K^-1 Kd), tr(K^-1 Kdd)
  double psi = 0.0, q3 = 0.0, q1 = 0.0, q2 = 0.0, t1 = 0.0, t3 = 0.0;
  for (int a = tid; a < n; a += LB) {
    psi = fma(Y[a], w[a], psi);
    q3 = fma(w[a], kdw[a], q3);
    double sdd = 0.0, sq2 = 0.0, st1 = 0.0, st3 = 0.0;
    for (int b = 0; b < n; b++) {
      const double kd = Kd[a * n + b], kdd = kd * (r2of(a, b) * tinv2 - 2.0 * tinv);
      const double ki = KiM[a * n + b];
      sdd = fma(kdd, w[b], sdd);
      sq2 = fma(ki, kdw[b], sq2);
      st1 = fma(ki, kd, st1);
      st3 = fma(ki, kdd, st3);
    }
    q1 = fma(w[a], sdd, q1);
    q2 = fma(kdw[a], sq2, q2);
    t1 += st1;
    t3 += st3;
  }
  __syncthreads();
  // tr((K^-1 Kd)^2) = sum_ab A_ab A_ba with A = K^-1 Kd, the n^3 term: formed in
  // float-float on the FP32 pipes (compensated dots, about 2^-48 per product).  It
  // enters l'' only, which sets the Newton step, not the root l' = 0 the iteration
  // converges to.  K^-1 and Kd are converted in place (their FP64 uses are done), one
  // float-float pair per FP64 slot.
  float2 *Kif = reinterpret_cast<float2 *>(KiM), *Kdf = reinterpret_cast<float2 *>(Kd);
  for (int e = tid; e < n * n; e += LB) {
    const ff ki = ff_from_double(KiM[e]), kd = ff_from_double(Kd[e]);
    Kif[e] = make_float2(ki.h, ki.l);
    Kdf[e] = make_float2(kd.h, kd.l);
  }
  __syncthreads();
  // The pairs a <= b, all lanes busy: (a == b ? 1 : 2) A_ab into slot (a, b) and A_ba into
  // slot (b, a) of the dead L^-1 storage (for a == b both are A_aa, in one slot).
  for (int e = tid; e < ntri; e += LB) {
    const int b = tri_row(e), a = e - b * (b + 1) / 2;
    ffacc sab{0.0f, 0.0f}, sba{0.0f, 0.0f};
    for (int m = 0; m < n; m++) {
      const float2 x1 = Kif[a * n + m], y1 = Kdf[m * n + b];
      const float2 x2 = Kif[b * n + m], y2 = Kdf[m * n + a];
      ffacc_add_prod(sab, ff{x1.x, x1.y}, ff{y1.x, y1.y});
      ffacc_add_prod(sba, ff{x2.x, x2.y}, ff{y2.x, y2.y});
    }
    const double vab = (double)sab.h + (double)sab.l, vba = (double)sba.h + (double)sba.l;
    Xb[a * n + b] = (a == b ? 1.0 : 2.0) * vab;
    if (a != b) Xb[b * n + a] = vba;
  }
  __syncthreads();
  // each thread adds its pairs in the order of the row-major (a, b) scan
  double t2p = 0.0;
  for (int e = tid; e < n * n; e += LB) {
    const int a = e / n, b = e % n;
    if (b < a) continue;
    t2p = fma(Xb[a * n + b], Xb[b * n + a], t2p);
  }
  *out = MleTerms{psi, q3, q1, q2, t1, t3, t2p};
  return true;
}

// Packed: the set is in shared memory; otherwise it is a slot of the workspace.
template <bool Packed>
__global__ void __launch_bounds__(LB, 4) mle_fp64_kernel(MleParams P) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int n = P.n, p = P.p, ntri = n * (n + 1) / 2;
  const size_t sq = (size_t)n * (Packed ? mle_lda(n) : n);
  double *S1 = reinterpret_cast<double *>(Packed ? smraw : P.slots + (size_t)blockIdx.x * P.slot_bytes);
  double *S2 = S1 + sq, *S3 = S2 + sq;
  double *Y = S3 + (Packed ? mle_s3_words(n) : sq), *w = Y + n, *kdw = w + n, *rl = kdw + n;
  double *xd = Packed ? S3 : rl + n;  // n x p coordinates of the design
  __shared__ double etab[64];
  __shared__ double red[kSums][LB / 32];
  __shared__ double sh_th, sh_lo, sh_hi;
  __shared__ int sh_loc, sh_fail, sh_done, sh_lo_open, sh_hi_open, sh_it, sh_st;
  const int tid = threadIdx.x;
  if (tid < 64) etab[tid] = c_exp.tab[tid];
  // one pivot warp per sub-partition for the CTAs of an SM (dealt to the SMs in turn)
  unsigned nsm;
  asm("mov.u32 %0, %%nsmid;" : "=r"(nsm));
  const int turn = (int)(blockIdx.x / nsm) & 3;

  for (;;) {
    __syncthreads();
    if (tid == 0) sh_loc = atomicAdd(P.queue, 1);
    __syncthreads();
    if (sh_loc >= P.T) break;
    const int64_t loc = sh_loc;
    const int32_t *d = P.idx + loc * n;
    if (tid == 0) {
      sh_fail = d[0] < 0;  // no design (its screen failed)
      const double t0 = P.theta0_loc ? P.theta0_loc[loc] : P.theta0;
      sh_th = fmin(fmax(t0, P.tmin), P.tmax);
      sh_lo = P.tmin;
      sh_hi = P.tmax;
      sh_lo_open = sh_hi_open = 1;
      sh_done = 0;
      sh_it = 0;
      sh_st = LAGP_ERR_NO_CONVERGENCE;
    }
    __syncthreads();
    if (!sh_fail) {
      for (int i = tid; i < n; i += LB) Y[i] = P.Z[d[i]];
      for (int e = tid; e < n * p; e += LB) xd[e] = P.X[(int64_t)d[e / p] * p + e % p];
    }
    __syncthreads();  // the coordinates are read by other threads below
    if (Packed && !sh_fail)
      for (int e = tid; e < ntri; e += LB) {
        const int a = tri_row(e), b = e - a * (a + 1) / 2;
        if (a == b) continue;
        double r2 = 0.0;
        for (int k = 0; k < p; k++) {
          const double t = xd[a * p + k] - xd[b * p + k];
          r2 = fma(t, t, r2);
        }
        S1[b * mle_lda(n) + a] = r2;
      }
    __syncthreads();
    while (!sh_fail && !sh_done) {
      const double th = sh_th;
      MleTerms mt;
      const bool ok = Packed ? mle_terms_packed(S1, S2, S3, Y, w, kdw, rl, n, 1.0 / th, P.g, etab, &sh_fail, turn, &mt)
                             : mle_terms_full(S1, S2, S3, xd, Y, w, kdw, rl, n, p, 1.0 / th, P.g, etab, &sh_fail,
                                              turn, &mt);
      if (!ok) break;
      // The seven block sums: a shuffle tree per warp, then thread 0 adds the warp totals in
      // warp order.  The six row sums are exactly +0.0 in a warp none of whose threads holds
      // a row (warp * 32 >= n), whose tree would give +0.0, so such warps skip it.
      {
        const int lane = tid & 31, warp = tid >> 5;
        double v[kSums] = {mt.psi, mt.q3, mt.q1, mt.q2, mt.t1, mt.t3, mt.t2p};
        if (warp * 32 < n) {
#pragma unroll
          for (int j = 0; j < kSums - 1; j++) v[j] = warp_tree_sum(v[j]);
        }
        v[kSums - 1] = warp_tree_sum(v[kSums - 1]);
        if (lane == 0) {
#pragma unroll
          for (int j = 0; j < kSums; j++) red[j][warp] = v[j];
        }
      }
      __syncthreads();
      if (tid == 0) {
        double v[kSums];
#pragma unroll
        for (int j = 0; j < kSums; j++) {
          double s = 0.0;
          for (int w = 0; w < LB / 32; w++) s += red[j][w];
          v[j] = s;
        }
        const double psi = v[0], q3 = v[1], q1 = v[2], q2 = v[3], t1 = v[4], t3 = v[5], t2 = v[6];
        const double dn = n;
        const double d1 = -0.5 * t1 + dn / 2.0 * q3 / psi;
        const double d2 = -0.5 * (t3 - t2) + dn / (2.0 * psi) * (q1 - 2.0 * q2) +
                          dn / (2.0 * psi * psi) * q3 * q3;
        sh_it++;
        bool stop = false;
        if (d1 == 0.0) {
          stop = true;
        } else if (d1 > 0.0) {
          sh_lo = th;
          sh_lo_open = 0;
          stop = th >= P.tmax;
        } else {
          sh_hi = th;
          sh_hi_open = 0;
          stop = th <= P.tmin;
        }
        if (stop) {
          sh_st = 0;
          sh_done = 1;
        } else {
          double tn = (d2 < 0.0) ? th - d1 / d2 : NAN;
          if (!(tn > sh_lo && tn < sh_hi)) {
            if (d1 > 0.0 && sh_hi_open) tn = sh_hi;  // uphill to an end not yet evaluated
            else if (d1 < 0.0 && sh_lo_open) tn = sh_lo;
            else tn = 0.5 * (sh_lo + sh_hi);
          }
          const bool small = fabs(tn - th) <= P.tol * th;
          sh_th = tn;
          if (small) {
            sh_st = 0;
            sh_done = 1;
          } else if (sh_it >= P.maxit) {
            sh_done = 1;  // sh_st stays LAGP_ERR_NO_CONVERGENCE
          }
        }
      }
      __syncthreads();
    }
    __syncthreads();
    if (tid == 0) {
      P.theta_out[loc] = sh_fail ? NAN : sh_th;
      if (P.iters) P.iters[loc] = sh_it;
      if (P.status) P.status[loc] = sh_fail ? (int8_t)LAGP_ERR_NOT_PD : (int8_t)sh_st;
    }
  }
}

bool mle_in_smem(int n) { return mle_set_bytes(n) <= kSmemMle; }

int mle_grid(int64_t T, int n, const DevInfo &di) {
  int per_sm = 1;
  const cudaError_t e =
      mle_in_smem(n) ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mle_fp64_kernel<true>, LB, mle_set_bytes(n))
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mle_fp64_kernel<false>, LB, 0);
  if (e != cudaSuccess || per_sm < 1) per_sm = 1;
  const int64_t g = (int64_t)di.num_sms * per_sm;
  return (int)(T < g ? (T > 0 ? T : 1) : g);
}

// At most 2048 / LB CTAs per SM: the bound used to size the per-CTA slots.
int mle_grid_bound(int64_t T, int num_sms) {
  const int64_t g = (int64_t)num_sms * (2048 / LB);
  return (int)(T < g ? (T > 0 ? T : 1) : g);
}

}  // namespace

size_t mle_workspace_bytes(int64_t T, int32_t n, int num_sms) {
  return 256 + (mle_in_smem(n) ? 0 : (size_t)mle_grid_bound(T, num_sms) * mle_slot_bytes(n));
}

int mle_launch(const MleArgs &a, void *ws, size_t ws_bytes, cudaStream_t stream) {
  if (a.T == 0) return LAGP_OK;
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  st = exp_table_upload();  // this translation unit's copy of the exp constants
  if (st) return st;
  if (ws_bytes < 256) return LAGP_ERR_INVALID_ARG;
  const bool sm = mle_in_smem(a.n);
  const size_t smem = sm ? mle_set_bytes(a.n) : 0;
  if (sm) {
    st = allow_smem(reinterpret_cast<const void *>(mle_fp64_kernel<true>), di);
    if (st) return st;
  }
  cudaError_t e;
  int G = mle_grid(a.T, a.n, di);
  if (!sm) {  // as many slots as there are, one per SM at least
    const int64_t slots = (int64_t)((ws_bytes - 256) / mle_slot_bytes(a.n));
    if (slots < std::min<int64_t>(a.T, di.num_sms)) return LAGP_ERR_INVALID_ARG;
    G = (int)std::min<int64_t>(G, slots);
  }
  char *w = static_cast<char *>(ws);
  MleParams P;
  P.X = a.X; P.Z = a.Z; P.p = a.p; P.T = a.T; P.idx = a.idx; P.n = a.n;
  P.theta0 = a.theta0; P.theta0_loc = a.theta0_loc; P.g = a.g; P.tmin = a.tmin; P.tmax = a.tmax;
  P.tol = a.tol; P.maxit = a.maxit;
  P.theta_out = a.theta_out; P.iters = a.iters; P.status = a.status;
  P.queue = reinterpret_cast<int *>(w);
  P.slot_bytes = mle_slot_bytes(a.n);
  P.slots = sm ? nullptr : reinterpret_cast<unsigned char *>(w + 256);
  e = cudaMemsetAsync(P.queue, 0, sizeof(int), stream);
  if (e != cudaSuccess) return cuda_status(e);
  if (sm) mle_fp64_kernel<true><<<G, LB, smem, stream>>>(P);
  else mle_fp64_kernel<false><<<G, LB, 0, stream>>>(P);
  g_launches.fetch_add(1);
  return cuda_status(cudaGetLastError());
}

int mle_prepare() { return exp_table_upload(); }

}  // namespace lagp
