// fx.cuh -- 64-bit fixed-point arithmetic of the ALC candidate screen, on the integer pipe.
//
// Every quantity of the bordered Cholesky recursion is bounded: correlations, conditional
// covariances and variances by 1 + g, factor entries by sqrt(1 + g) (Cauchy-Schwarz).  So
// the screen of the FP64 designs carries them in fixed point, and the row dot u_s . u_c -- its
// inner loop -- becomes three 32 x 32 + 64-bit multiply-adds per term (IMAD.WIDE), exact but
// for the products' bits below 2^-116.  GB300, per warp instruction and SM sub-partition:
// IMAD.WIDE 4 cycles (12 a term and candidate), a compensated float-float term six packed
// FFMA2 of 2 for two candidates (6), an FP64 DFMA 64.  Scores by emulation, largest relative
// error over a uniform 2-d design: FP64 9e-9, fixed point 1.1e-8, float-float 6e-7.
//
// Formats, with e even and 1 + g < 2^(e+1):
//   variance units (v, K, cov, dots)   int64, value 2^(60-e)
//   factor entries u                   u64 = value 2^(58-e/2) = h 2^28 + l: int32 h,
//                                      l in [-2^27, 2^27]
//   u_s.u_c = sum h h' + (sum (h l' + l h')) 2^-28: the first sum is at most (1+g) 2^(60-e)
//   in size, the second at most 2^30.5 16 2^27 2 < 2^63 for 256 terms; the products l l'
//   are below 2^-4 units each and left out.
//   coordinates relative to x          value 2^(28-b) = h + l 2^-30, all |value| < 2^b
//                                      (value in units where K = 2^-(squared distance))
// Plain integer code, so the host can run it too (the unit test compares it with long
// double there).
#pragma once

#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define LAGP_HD __host__ __device__ __forceinline__
#else
#define LAGP_HD inline
#endif

namespace lagp {

// Constants of 2^-y: 2^(-i/256), i = 0..255, times 2^63, and c_m = (ln2 / 256)^m / m! times 2^60.
constexpr int kFxTab = 256;
struct FxConsts {
  uint64_t tab[kFxTab];
  uint64_t c1, c2;
  uint32_t c3, c4, c5, pad;
};

// High word of a b, rounded: the addend makes it one IMAD.WIDE (4 cycles per warp; a truncated
// high product would be an IMAD.HI, 8).
LAGP_HD uint32_t fx_mulhi(uint32_t a, uint32_t b) {
  return (uint32_t)(((uint64_t)a * b + 0x80000000u) >> 32);
}

// 64-bit shifts by 0 .. 31 as funnel shifts.
LAGP_HD uint64_t fx_make(uint32_t hi, uint32_t lo) { return ((uint64_t)hi << 32) | lo; }
LAGP_HD uint64_t fx_shl31(uint64_t x, int n) {
#ifdef __CUDA_ARCH__
  const uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
  return fx_make(__funnelshift_l(lo, hi, n), lo << n);
#else
  return x << n;
#endif
}

// Float of a 64-bit integer to two ulp and 2^7, from its words (a 64-bit conversion
// instruction runs at the FP64 rate).
LAGP_HD float fx_to_float(int64_t x) {
  return fmaf((float)(int32_t)(x >> 32), 4294967296.0f, (float)(uint32_t)x);
}

// 2^-y for y = Y 2^-56 in [0, 64), times 2^60 (Tang's table-driven method, ACM TOMS 15(2),
// 1989, with N = 256): y = k + i/256 + rho/256, and 2^(-rho/256) by its Taylor series through
// rho^5 (the next term is below 2^-60).  The inner coefficients need 32 bits at the scale
// 2^60, so they cost one multiplication each; 12 in all.
LAGP_HD int64_t fx_exp2(uint64_t Y, const uint64_t *tab, uint64_t c1, uint64_t c2, uint32_t c3,
                        uint32_t c4, uint32_t c5, int shift) {
  const int k = (int)(Y >> 56) + shift;
  const uint32_t i = (uint32_t)(Y >> 48) & 255u;
  const uint32_t rh = (uint32_t)(Y >> 16), rl = (uint32_t)Y << 16;  // rho 2^32, then its low bits
  const uint32_t q = c3 - fx_mulhi(rh, c4 - fx_mulhi(rh, c5));
  const uint64_t q2 = c2 - fx_mulhi(rh, q);
  const uint32_t q2h = (uint32_t)(q2 >> 32), q2l = (uint32_t)q2;
  const uint64_t q1 = c1 - ((uint64_t)rh * q2h + fx_mulhi(rh, q2l) + fx_mulhi(rl, q2h));
  const uint32_t q1h = (uint32_t)(q1 >> 32), q1l = (uint32_t)q1;
  const uint64_t E = (uint64_t)rh * q1h + fx_mulhi(rh, q1l) + fx_mulhi(rl, q1h);  // 1 - 2^(-rho/256)
  const uint64_t T = tab[i];
  const uint32_t Th = (uint32_t)(T >> 32), Tl = (uint32_t)T;
  const uint32_t Eh = (uint32_t)(E >> 32), El = (uint32_t)E;
  const uint64_t P = (uint64_t)Th * Eh + fx_mulhi(Th, El) + fx_mulhi(Tl, Eh);  // T E 2^-64
  const uint64_t K = (T >> 3) - (P << 1);
  return k > 63 ? 0 : (int64_t)(K >> k);
}

// K = 2^-y in variance units, y the squared distance from the sums of the coordinate
// differences dh + dl 2^-30: hh = sum dh^2 (scale 2^(56-2b)), hl = sum dh dl, ll = sum dl^2
// (used where sh2b = min(2b, 62) is not 0; below one unit otherwise).  A distance of 64 or more
// is a correlation below 2^-64, 0 here.
LAGP_HD int64_t fx_corr(int64_t hh, int64_t hl, int64_t ll, int sh2b, const uint64_t *tab, uint64_t c1,
                        uint64_t c2, uint32_t c3, uint32_t c4, uint32_t c5, int e) {
  int64_t y = hh + (hl >> 29);
  bool zero = false;
  if (sh2b) {  // the same for the whole location
    // hh 2^sh2b + (2 hl + ll 2^-30) 2^(sh2b-30): the low part keeps the bits that hh's scale lacks
    zero = ((uint64_t)(y > 0 ? y : 0) >> (62 - sh2b)) != 0;
    const int64_t low = hl + (ll >> 31);
    y = sh2b <= 29 ? (int64_t)((uint64_t)hh << sh2b) + (low >> (29 - sh2b)) : (int64_t)((uint64_t)y << sh2b);
  }
  const int64_t K = fx_exp2((uint64_t)(y > 0 ? y : 0), tab, c1, c2, c3, c4, c5, e);
  return zero ? 0 : K;
}

// 1 / sqrt(nu) for nu = V 2^-60, V in (0, 2^62): u64 = hi64((t << q) R), with
// R = 2^62 rho, rho = 1 / sqrt(nu 4^q) in (1/2, 1].  FP32 estimate and one step of third order
// in integers (relative error about 2^-58).
struct FxRsqrt {
  int32_t Rh, Rl;  // R = Rh 2^32 + Rl, Rl signed
  int q;
};

LAGP_HD int fx_clz(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}
LAGP_HD uint64_t fx_umulhi64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

LAGP_HD FxRsqrt fx_rsqrt(int64_t V) {
  FxRsqrt r;
  r.q = (fx_clz((uint64_t)V) - 2) >> 1;
  const uint64_t N = (uint64_t)V << (2 * r.q);  // nu 4^q 2^60, in [2^60, 2^62)
  const float nf = (float)(uint32_t)(N >> 32) * 3.7252903e-09f;  // 2^-28
#ifdef __CUDA_ARCH__
  const float y0 = rsqrtf(nf);
#else
  const float y0 = 1.0f / sqrtf(nf);
#endif
  const uint32_t Y0 = (uint32_t)(y0 * 2147483648.0f);          // rho 2^31
  const uint64_t S = (uint64_t)Y0 * Y0;                         // rho^2 2^62
  const int64_t e = (int64_t)(1ull << 60) - (int64_t)fx_umulhi64(N << 1, S << 1);  // 1 - nu rho^2
  const int64_t et = e >> 20;
  const int64_t c = (e >> 1) + ((3 * et * et) >> 23);           // (1 - e)^(-1/2) - 1 at 2^60
  const int64_t ch = c >> 20, cl = c & 0xfffff;
  const int64_t R = ((int64_t)Y0 << 31) + (((int64_t)Y0 * ch) >> 9) + (((int64_t)Y0 * cl) >> 29);
  r.Rl = (int32_t)R;
  r.Rh = (int32_t)((R - r.Rl) >> 32);
  return r;
}

// t / sqrt(nu) in the format of factor entries, t in variance units with |t| <= sqrt(nu (1+g)).
LAGP_HD int64_t fx_mul_rsqrt(int64_t t, FxRsqrt r) {
  const int64_t ts = (int64_t)fx_shl31((uint64_t)t, r.q);  // q <= 30
  const int32_t th = (int32_t)(ts >> 32);
  const uint32_t tl = (uint32_t)ts;
  return (int64_t)th * r.Rh + (int64_t)(((uint64_t)tl * (uint32_t)r.Rh) >> 32) +
         (((int64_t)th * r.Rl) >> 32);
}

struct FxU {  // a factor entry: h 2^28 + l
  int32_t h, l;
};
LAGP_HD FxU fx_split(int64_t u) {
  FxU r;
  r.h = (int32_t)((u + (1 << 27)) >> 28);
  r.l = (int32_t)((uint32_t)u - ((uint32_t)r.h << 28));
  return r;
}

// a b in variance units
LAGP_HD int64_t fx_mul_uu(FxU a, FxU b) {
  return (int64_t)a.h * b.h + (((int64_t)a.h * b.l + (int64_t)a.l * b.h) >> 28);
}

}  // namespace lagp
