// mixed_screen.cuh -- device code shared by the candidate screens (select_mixed.cu through
// alc_screen.cuh, select_mspe_mixed.cu): the float-float exp, the FP64 correlation, the
// asynchronous row copies and L2 policies.
// Included by one translation unit each: c_exp is that unit's copy of the exp constants.
#pragma once

#include <math.h>

#include "check.cuh"
#include "ff.cuh"
#include "ff2.cuh"
#include "fp64_exp.cuh"
#include "internal.h"

namespace lagp {
namespace {

constexpr float DELTA = 1e-5f;     // near-tie margin for the FP64 re-score
constexpr int RESCORE_CAP = 64;    // candidates re-scored per pass

// exp(a) for a <= 0 on a pair, in float-float (Tang's table-driven method with N = 64, see
// fp64_exp.cuh): a = k ln2/64 + r, exp(r) - 1 = r + r^2/2 + r^3/6 + r^4/24 + r^5/120 with
// the first two terms in float-float and the rest in FP32 (they are below 3e-8).
// Arguments below -87 give 0.
__device__ __forceinline__ ff2 exp_ff2(ff2 a, const float *tabh, const float *tabl) {
  const float2 ah = make_float2(fmaxf(a.h.x, -87.0f), fmaxf(a.h.y, -87.0f));
  const float2 magic = f2s(12582912.0f);  // 1.5 * 2^23
  const float2 t = fma2(ah, f2s(c_exp.inv_ln2_64f), magic);
  const float2 kf = sub2(t, magic);
  const int kx = __float_as_int(t.x) - 0x4B400000, ky = __float_as_int(t.y) - 0x4B400000;
  const float2 r1 = fma2(neg2(kf), f2s(c_exp.c1), ah);  // exact
  const float2 p2h = mul2(kf, f2s(c_exp.c2));
  const float2 p2l = fma2(kf, f2s(c_exp.c2), neg2(p2h));
  const ff2 s = two_sum2(r1, neg2(p2h));
  const float2 rl = add2(sub2(sub2(s.l, p2l), mul2(kf, f2s(c_exp.c3))), a.l);
  const ff2 r = fast_two_sum2(s.h, rl);
  const float2 sqh = mul2(r.h, r.h);
  const float2 sql = fma2(add2(r.h, r.h), r.l, fma2(r.h, r.h, neg2(sqh)));
  const float2 P = mul2(mul2(r.h, sqh),
                        fma2(r.h, fma2(r.h, f2s(1.0f / 120.0f), f2s(1.0f / 24.0f)), f2s(1.0f / 6.0f)));
  const ff2 e = two_sum2(r.h, mul2(f2s(0.5f), sqh));
  const ff2 E = fast_two_sum2(e.h, add2(add2(e.l, r.l), fma2(f2s(0.5f), sql, P)));
  const float2 Th = f2(tabh[kx & 63], tabh[ky & 63]), Tl = f2(tabl[kx & 63], tabl[ky & 63]);
  const float2 ph = mul2(Th, E.h);
  const float2 pl = fma2(Th, E.h, neg2(ph));
  const ff2 s2 = two_sum2(Th, ph);
  const float2 low = add2(add2(s2.l, pl), fma2(Th, E.l, fma2(Tl, E.h, Tl)));
  const ff2 res = fast_two_sum2(s2.h, low);
  const float2 sc = f2(__int_as_float(((kx >> 6) + 127) << 23), __int_as_float(((ky >> 6) + 127) << 23));
  ff2 out{mul2(res.h, sc), mul2(res.l, sc)};
  if (a.h.x < -87.0f) out.h.x = out.l.x = 0.0f;
  if (a.h.y < -87.0f) out.h.y = out.l.y = 0.0f;
  return out;
}

__device__ __forceinline__ double corr64(const double *a, const double *b, int p, double theta_inv,
                                         const double *etab) {
  double acc = 0.0;
  for (int k = 0; k < p; k++) {
    const double t = a[k] - b[k];
    acc = fma(t, t, acc);
  }
  return exp_nonpos(-acc * theta_inv, etab);
}

// Asynchronous 16-byte copies global -> shared (cp.async, L2 only) and their groups: a
// thread's factor rows in global memory reach its own slots of a ring in shared memory a
// few rows ahead of their use, so that the loads of the next rows are in flight while a
// row is consumed.  Each thread waits only for its own copies (no barrier).

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Factor-row loads with an L2 evict-last policy: a row is read again at every later step of
// the location, so on the workloads whose live rows fit in L2 they are kept there ahead of
// data read once (candidate lists, coordinates).  paper-2d: 14.85 -> 14.38 ms.
__device__ __forceinline__ unsigned long long l2_evict_last_policy() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ unsigned long long l2_evict_first_policy() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ double ld_l2_hint(const double *a, unsigned long long pol) {
  double v;
  asm volatile("ld.global.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(a), "l"(pol));
  return v;
}
// (V16: float4 or int4)
template <class V16>
__device__ __forceinline__ void cp_async16_l2_hint(V16 *smem_dst, const V16 *gmem_src,
                                                   unsigned long long pol) {
  static_assert(sizeof(V16) == 16, "16-byte copies");
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(s),
               "l"(gmem_src), "l"(pol)
               : "memory");
}
__device__ __forceinline__ float4 ld_l2_hint(const float4 *a, unsigned long long pol) {
  float4 v;
  asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(a), "l"(pol));
  return v;
}
__device__ __forceinline__ int4 ld_l2_hint(const int4 *a, unsigned long long pol) {
  int4 v;
  asm volatile("ld.global.L2::cache_hint.v4.s32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(a), "l"(pol));
  return v;
}

}  // namespace
}  // namespace lagp
