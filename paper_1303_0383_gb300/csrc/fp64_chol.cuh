// fp64_chol.cuh -- block-cooperative FP64 Cholesky for one small matrix per CTA.
//
// FP64 runs at 1/64 of the FP32 rate on this GPU, so the factorisation keeps every FP64
// instruction busy on all lanes: each step's column scaling and trailing update are
// flattened over the CTA's threads.  A division by the pivot is a product with its
// reciprocal plus one correction (Markstein: with the correctly rounded reciprocal y of b
// and q = rn(a y), q + (a - b q) y is the correctly rounded a / b), and the pivot's square
// root and reciprocal are taken by the thread that finishes the pivot in the previous
// step's update, so a step costs two block barriers.  The right-looking order makes for
// every entry the same subtractions, in the same order, as the row-by-row factorisation.
#pragma once

#include <math.h>

namespace lagp {
namespace {

// Row of the lower triangle {(a, b): 0 <= b <= a} that holds flat entry e.
__device__ __forceinline__ int tri_row(int e) {
  int a = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while (a * (a + 1) / 2 > e) a--;
  while ((a + 1) * (a + 2) / 2 <= e) a++;
  return a;
}

// a / l from q = rn(a r), r = rn(1 / l).  exact: also where the correction would leave the normal
// range or meet an infinity (there it turns an infinite quotient into NaN), as a division.
__device__ __forceinline__ double div_by_pivot(double a, double q, double l, double r, bool exact) {
  if (exact) {
    const unsigned ha = (unsigned)__double2hiint(a) & 0x7fffffffu, hq = (unsigned)__double2hiint(q) & 0x7fffffffu;
    // both within 2^-960 .. 2^1023, or a = 0
    if ((ha < (64u << 20) || hq < (64u << 20) || hq >= 0x7ff00000u) && (ha | (unsigned)__double2loint(a))) return a / l;
  }
  return fma(fma(-q, l, a), r, q);
}

// Whether c, not zero, from div_by_pivot(a, q, l, r, false) is a / l: c within 2^-399 .. 2^399, so q
// within 2^-400 .. 2^400.  With l = sqrt(v) within 2^-537 .. 2^512, a is then normal and the
// residual a - q l, a multiple of 2^-1041, exact; a q beyond gives a c beyond (or NaN).
__device__ __forceinline__ bool div_sure(double c) {
  return (((unsigned)__double2hiint(c) >> 20 & 0x7ffu) - 624u) < 799u;
}

// In-place Cholesky A = L L^T of the n x n lower triangle of A (row-major, leading
// dimension lda), carrying naug extra columns n .. n+naug-1 along so that they end as
// L^{-1} b (forward substitution).  rl[k] receives 1 / l_kk.  Sets *fail (shared) on a
// pivot <= 0; every thread returns after the same barriers.
// recip: the matrix entries (not the extra columns) are multiplied by 1 / l_kk instead of
// divided by l_kk, and the extra columns divided whatever their values: the rounding of the FP64
// recursion (select.cu), so a design's rows come out bit for bit as that recursion forms them.
// turn: the warp that takes the pivots.  Warp w of every CTA runs on sub-partition w mod 4, so
// CTAs that share an SM should have them taken by different ones.
__device__ void chol_flat_fp64(double *A, int n, int lda, int naug, double *rl, int *fail,
                               bool recip = false, int turn = 0) {
  const int nt = blockDim.x, first = (int)threadIdx.x - 32 * turn, tid = first < 0 ? first + nt : first;
  __syncthreads();
  if (tid == 0) {
    const double d0 = A[0];
    if (!(d0 > 0.0)) *fail = 1;
    const double l0 = sqrt(d0);
    A[0] = l0;
    rl[0] = 1.0 / l0;
  }
  __syncthreads();
  for (int k = 0; k < n && !*fail; k++) {
    const double lkk = A[k * lda + k], r = rl[k];
    // column k and the extra columns of row k divided by the pivot
    for (int i = k + 1 + tid; i < n + naug; i += nt) {
      double *ap = (i < n) ? &A[i * lda + k] : &A[k * lda + i];
      const double a = *ap, q = a * r;
      *ap = (recip && i < n) ? q : div_by_pivot(a, q, lkk, r, recip);
    }
    __syncthreads();
    // a_il -= l_ik l_lk for k < l <= i, and the extra columns: b_i -= l_ik b_k
    const int rows = n - k - 1, ntr = rows * (rows + 1) / 2;
    for (int e = tid; e < ntr + naug * rows; e += nt) {
      if (e < ntr) {
        const int t = tri_row(e), c = e - t * (t + 1) / 2;
        const int i = k + 1 + t, l = k + 1 + c;
        const double v = fma(-A[i * lda + k], A[l * lda + k], A[i * lda + l]);
        if (e == 0) {  // the next pivot is final: its square root and reciprocal
          if (!(v > 0.0)) *fail = 1;
          const double lv = sqrt(v);
          A[i * lda + l] = lv;
          rl[k + 1] = 1.0 / lv;
        } else {
          A[i * lda + l] = v;
        }
      } else {
        const int i = k + 1 + (e - ntr) / naug, col = (e - ntr) % naug;
        A[i * lda + n + col] = fma(-A[i * lda + k], A[k * lda + n + col], A[i * lda + n + col]);
      }
    }
    __syncthreads();
  }
}

}  // namespace
}  // namespace lagp
