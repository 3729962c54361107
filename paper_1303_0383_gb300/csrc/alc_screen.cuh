// alc_screen.cuh -- device code of the ALC candidate screen (select_mixed.cu): its two
// arithmetics, rows in tensor memory, the per-pair step, score tracking, and the FP64 re-score
// of candidates the screen cannot separate.
//
// Gramacy & Apley, Sec. 3: the greedy local design adds the candidate that maximises the
// ALC reduction cov_j(x,c)^2 / v_j(c) (Eq. dxy; SM Eq. dxy2); Sec. 3.2 gives the O(j)
// update of every candidate's quantities when the design grows by one point.
#pragma once

#include "fp64_chol.cuh"
#include "fx.cuh"
#include "mixed_screen.cuh"

namespace lagp {
namespace {

__device__ __forceinline__ bool frac_better(double a, double da, int ra, double b, double db,
                                            int rb) {
  const double l = a * db, r = b * da;
  return l > r || (l == r && ra < rb);
}

// Screen score comparison: larger score, ties to the smaller rank (a thread meets its
// candidates in rank order); -1: no score.
__device__ __forceinline__ void track2(float sc, int c, float &b1, int &r1, float &b2) {
  b2 = fmaxf(b2, fminf(sc, b1));
  r1 = sc > b1 ? c : r1;
  b1 = fmaxf(b1, sc);
}

// Score keys: 0 for none, else the bits of the (non-negative) score plus one, which order like
// the scores, so that a warp's best is one integer reduction.
__device__ __forceinline__ unsigned score_key(float sc) {
  return sc >= 0.0f ? __float_as_uint(sc) + 1u : 0u;
}
// (k1, r1, k2): best key, its rank, second-best key.  Ties go to the smaller rank; ranks differ.
__device__ __forceinline__ void merge_keys(unsigned o1, int orr, unsigned o2, unsigned &k1, int &r1,
                                           unsigned &k2) {
  if (o1 > k1 || (o1 == k1 && orr < r1)) {
    k2 = max(k1, o2);
    k1 = o1;
    r1 = orr;
  } else {
    k2 = max(k2, o1);
  }
}
// The warp's, in every lane; returns the lane that holds the best (-1: none).
__device__ __forceinline__ int warp_best2(unsigned &k1, int &r1, unsigned &k2) {
  const unsigned K = __reduce_max_sync(0xffffffffu, k1);
  const int r = (int)__reduce_min_sync(0xffffffffu, K && k1 == K ? (unsigned)r1 : 0x7fffffffu);
  const bool win = K && k1 == K && r1 == r;
  k2 = __reduce_max_sync(0xffffffffu, win ? k2 : k1);
  k1 = K;
  r1 = r;
  return __ffs(__ballot_sync(0xffffffffu, win)) - 1;
}

// Tensor memory as a second on-chip store for factor rows (no tensor-core work): a CTA
// allocates its share of its SM's 512 columns; warp w may address only the 32 lanes of
// its sub-partition, 32 (w & 3) .. 32 (w & 3) + 31, and takes columns 128 (w >> 2) .. + 127 of
// them, so every thread owns 128 32-bit words of its own lane.  Loads and stores are
// warp-collective (every lane of the warp executes them with the same address).  The load's
// wait is tied to the registers it delivers, so no use of them can be scheduled before it.
__device__ __forceinline__ void tmem_ld16_issue(uint32_t ta, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(ta));
}
__device__ __forceinline__ void tmem_wait16(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),
                 "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]),
                 "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
               :
               : "memory");
}
__device__ __forceinline__ uint32_t as_word(float x) { return __float_as_uint(x); }
__device__ __forceinline__ uint32_t as_word(int x) { return (uint32_t)x; }
template <class Word>
__device__ __forceinline__ Word tmem_word(const uint32_t *w);
template <>
__device__ __forceinline__ float4 tmem_word<float4>(const uint32_t *w) {
  return make_float4(__uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]), __uint_as_float(w[3]));
}
template <>
__device__ __forceinline__ int4 tmem_word<int4>(const uint32_t *w) {
  return make_int4((int)w[0], (int)w[1], (int)w[2], (int)w[3]);
}
template <class Word>
__device__ __forceinline__ void tmem_st4(uint32_t ta, Word v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ta),
               "r"(as_word(v.x)), "r"(as_word(v.y)), "r"(as_word(v.z)), "r"(as_word(v.w))
               : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
constexpr int kTmemWords = 128;  // words of one thread
constexpr size_t kTmemBytes = 256 * 1024;  // of an SM
// columns of a CTA of nt threads
__host__ __device__ constexpr int tmem_cols(int nt) { return nt * kTmemWords / 128; }

// ---- the screen's arithmetics
// Two candidates (2q, 2q + 1) per pair; every 16-byte word holds a pair's {a, b} high and low
// parts.  Kept per pair: v_j(c), cov_j(x, c), the coordinates (relative to x) and the factor
// rows; per step a record of the pivot s: its coordinates, scalars and factor row.
// An arithmetic gives: Acc and row() (one term of K(s, c) - u_s . u_c for a pair), corr() (K(s, c)
// from the coordinates), finish() (u_c[j], v and cov of the pair), score().

// The screen's ALC score cov^2 / v in FP32, with the approximate quotient (a reciprocal and a
// product, within 2 ulp): the screen only ranks, and any pair of scores whose order that
// error could swap lies well inside the near-tie band DELTA, whose candidates are re-scored
// in FP64.  The same expression forms every screen score, so the tracked best and the
// near-tie list agree.
__device__ __forceinline__ float score32(float cov, float v) { return __fdividef(cov * cov, v); }

constexpr int kRecHead = kMaxP + 4;  // 8-byte words of a record before its row: coordinates, scalars

// LAGP_MIXED: float-float on the FP32 pipes (ff.cuh, ff2.cuh).
struct FfArith {
  using Word = float4;
  static constexpr bool kFixed = false;
  // record row: {h, h, -h, -h} per entry, then {l, l}: no term needs a move or a sign flip
  static __host__ __device__ constexpr int rec_words(int n) { return 3 * ((n + 1) & ~1) + kRecHead; }
  struct Scalars {
    ff inv, ux;  // 1 / sqrt(v_j(s)), u_x[j]
  };
  static __device__ __forceinline__ bool positive(const Word *v, int c) { return ff2_get(v, c).h > 0.0f; }
  static __device__ __forceinline__ float score(const Word *cov, const Word *v, int c) {
    return score32(ff2_get(cov, c).h, ff2_get(v, c).h);
  }
  static __device__ __forceinline__ Scalars scalars(const Word *v, const Word *cov, int c) {
    Scalars s;
    s.inv = ff_rcp(ff_sqrt(ff2_get(v, c)));
    s.ux = ff_mul(ff2_get(cov, c), s.inv);
    return s;
  }
  static __device__ __forceinline__ void scalars_store(int2 *rec, const Scalars &s) {
    reinterpret_cast<float4 *>(rec + kMaxP)[0] = make_float4(s.inv.h, s.inv.l, s.ux.h, s.ux.l);
  }
  static __device__ __forceinline__ Scalars scalars_load(const int2 *rec) {
    const float4 a = reinterpret_cast<const float4 *>(rec + kMaxP)[0];
    return Scalars{ff{a.x, a.y}, ff{a.z, a.w}};
  }
  static __device__ __forceinline__ ff scalars_ux(const int2 *rec) { return scalars_load(rec).ux; }
  static __device__ __forceinline__ void rec_coord(int2 *rec, int k, const Word *row, int c) {
    const ff x = ff2_get(row, c);
    reinterpret_cast<float2 *>(rec)[k] = make_float2(x.h, x.l);
  }
  static __device__ __forceinline__ void rec_entry(int2 *rec, int i, int nrow, const Word *row, int c) {
    const ff u = ff2_get(row, c);
    reinterpret_cast<float4 *>(rec + kRecHead)[i] = make_float4(u.h, u.h, -u.h, -u.h);
    reinterpret_cast<float2 *>(rec + kRecHead + 2 * nrow)[i] = f2s(u.l);
  }
  using Acc = ff2acc;
  struct Dist {
    float2 h, l;
  };
  static __device__ __forceinline__ void dist_clear(Dist &d) { d.h = d.l = f2s(0.0f); }
  static __device__ __forceinline__ void dist_add(Dist &d, const int2 *rec, int k, Word w, int) {
    const ff2 b{make_float2(w.x, w.y), make_float2(w.z, w.w)};
    const float2 a = reinterpret_cast<const float2 *>(rec)[k];
    const ff2 df = two_sum2(f2s(a.x), neg2(b.h));
    const float2 dfl = add2(df.l, sub2(f2s(a.y), b.l));
    const float2 ph = mul2(df.h, df.h);
    const float2 pl = fma2(add2(df.h, df.h), dfl, fma2(df.h, df.h, neg2(ph)));
    const ff2 sacc = two_sum2(d.h, ph);
    d.h = sacc.h;
    d.l = add2(add2(sacc.l, d.l), pl);
  }
  // the coordinates are in units of sqrt(theta), so K = exp(-d^2)
  static __device__ __forceinline__ Acc corr(const Dist &d, const void *tab, const int *) {
    const ff2 d2 = fast_two_sum2(d.h, d.l);
    const float *th = static_cast<const float *>(tab);
    const ff2 kc = exp_ff2(ff2{neg2(d2.h), neg2(d2.l)}, th, th + 64);
    return Acc{kc.h, kc.l};
  }
  // entries i .. i + R - 1 of the record's row (nrow words of high parts), R rows of a pair
  template <int R, int NP>
  static __device__ __forceinline__ void rows(Acc (&acc)[NP], const int2 *rec, int i, int nrow,
                                              const Word (&b)[R][NP]) {
    const float4 *s4 = reinterpret_cast<const float4 *>(rec + kRecHead) + i;
    const float2 *s2 = reinterpret_cast<const float2 *>(rec + kRecHead + 2 * nrow) + i;
#pragma unroll
    for (int r = 0; r < R; r++) {
      const float4 h = s4[r];
      const float2 l = s2[r];
#pragma unroll
      for (int m = 0; m < NP; m++) ff2acc_sub_prod(acc[m], h, l, b[r][m]);
    }
  }
  static __device__ __forceinline__ Word finish(const Acc &acc, const Scalars &s, Word v0, Word c0,
                                                Word *v, Word *cov) {
    const ff2 u = ff2_mul(ff2acc_result(acc), ff2_bcast(s.inv));
    const ff2 vn = ff2_sub(ff2{make_float2(v0.x, v0.y), make_float2(v0.z, v0.w)}, ff2_mul(u, u));
    const ff2 cn = ff2_sub(ff2{make_float2(c0.x, c0.y), make_float2(c0.z, c0.w)},
                           ff2_mul(ff2_bcast(s.ux), u));
    *v = make_float4(vn.h.x, vn.h.y, vn.l.x, vn.l.y);
    *cov = make_float4(cn.h.x, cn.h.y, cn.l.x, cn.l.y);
    return make_float4(u.h.x, u.h.y, u.l.x, u.l.y);
  }
  static __device__ __forceinline__ void keep_a(Word &w, Word o) { w.x = o.x; w.z = o.z; }
  static __device__ __forceinline__ void keep_b(Word &w, Word o) { w.y = o.y; w.w = o.w; }
  static __device__ __forceinline__ float score_a(Word c, Word v) { return v.x > 0.0f ? score32(c.x, v.x) : -1.0f; }
  static __device__ __forceinline__ float score_b(Word c, Word v) { return v.y > 0.0f ? score32(c.y, v.y) : -1.0f; }
};

// LAGP_FP64: 64-bit fixed point on the integer pipe (fx.cuh), at FP64's resolution or below it.
// v and cov are an int64 per candidate; rows hold {h_a, h_b, l_a, l_b}.
struct FxArith {
  using Word = int4;
  static constexpr bool kFixed = true;
  static __host__ __device__ constexpr int rec_words(int n) { return ((n + 1) & ~1) + kRecHead; }
  struct Scalars {
    FxRsqrt rs;  // 1 / sqrt(v_j(s))
    FxU nux;     // -u_x[j]
    int csh;     // cov_j(x, .) is shifted right by this much in this step
  };
  static __device__ __forceinline__ long long get64(const Word *w, int c) {
    return reinterpret_cast<const long long *>(w)[c];
  }
  static __device__ __forceinline__ FxU get(const Word *row, int c) {
    const int4 v = row[c >> 1];
    return (c & 1) ? FxU{v.y, v.w} : FxU{v.x, v.z};
  }
  static __device__ __forceinline__ bool positive(const Word *v, int c) { return get64(v, c) > 0; }
  static __device__ __forceinline__ float score(const Word *cov, const Word *v, int c) {
    return score32(fx_to_float(get64(cov, c)), fx_to_float(get64(v, c)));
  }
  // u_x[j] = cov_j(x, s) / sqrt(v_j(s)); where it would leave its format (x far from candidates
  // that are close to one another) cov is shifted right first, here and by every candidate.
  static __device__ __forceinline__ Scalars scalars(const Word *v, const Word *cov, int c) {
    Scalars r;
    const long long cs = get64(cov, c);
    r.rs = fx_rsqrt(get64(v, c));
    r.csh = max(0, 64 - fx_clz((uint64_t)(cs < 0 ? -cs : cs)) + r.rs.q - 60);
    r.nux = fx_split(-fx_mul_rsqrt(cs >> r.csh, r.rs));
    return r;
  }
  static __device__ __forceinline__ void scalars_store(int2 *rec, const Scalars &s) {
    int4 *o = reinterpret_cast<int4 *>(rec + kMaxP);
    o[0] = make_int4(s.rs.Rh, s.rs.Rl, s.rs.q, s.csh);
    o[1] = make_int4(s.nux.h, s.nux.l, 0, 0);
  }
  static __device__ __forceinline__ Scalars scalars_load(const int2 *rec) {
    const int4 *o = reinterpret_cast<const int4 *>(rec + kMaxP);
    const int4 a = o[0], b = o[1];
    return Scalars{FxRsqrt{a.x, a.y, a.z}, FxU{b.x, b.y}, a.w};
  }
  static __device__ __forceinline__ ff scalars_ux(const int2 *) { return ff{0.0f, 0.0f}; }  // (not kept)
  static __device__ __forceinline__ void rec_coord(int2 *rec, int k, const Word *row, int c) {
    const FxU x = get(row, c);
    rec[k] = make_int2(x.h, x.l);
  }
  static __device__ __forceinline__ void rec_entry(int2 *rec, int i, int, const Word *row, int c) {
    const FxU u = get(row, c);
    rec[kRecHead + i] = make_int2(-u.h, -u.l);
  }
  // h collects the products of the high parts (variance units), x the cross products (2^-28)
  struct Acc {
    long long h0, h1, x0, x1;
  };
  struct Dist {
    long long hh[2], hl[2], ll[2];
  };
  static __device__ __forceinline__ void dist_clear(Dist &d) {
    d.hh[0] = d.hh[1] = d.hl[0] = d.hl[1] = d.ll[0] = d.ll[1] = 0;
  }
  static __device__ __forceinline__ void dist_add(Dist &d, const int2 *rec, int k, Word b, int sh2b) {
    const int2 a = rec[k];
    const int h0 = a.x - b.x, h1 = a.x - b.y, l0 = a.y - b.z, l1 = a.y - b.w;
    d.hh[0] += (long long)h0 * h0;
    d.hh[1] += (long long)h1 * h1;
    d.hl[0] += (long long)h0 * l0;
    d.hl[1] += (long long)h1 * l1;
    if (sh2b) {
      d.ll[0] += (long long)l0 * l0;
      d.ll[1] += (long long)l1 * l1;
    }
  }
  static __device__ __forceinline__ Acc corr(const Dist &d, const void *tab, const int *fmt) {
    const uint64_t *t = static_cast<const uint64_t *>(tab);
    const int sh2b = fmt[0], e = fmt[1];
    Acc a;
    a.h0 = fx_corr(d.hh[0], d.hl[0], d.ll[0], sh2b, t, c_exp.fx.c1, c_exp.fx.c2, c_exp.fx.c3,
                   c_exp.fx.c4, c_exp.fx.c5, e);
    a.h1 = fx_corr(d.hh[1], d.hl[1], d.ll[1], sh2b, t, c_exp.fx.c1, c_exp.fx.c2, c_exp.fx.c3,
                   c_exp.fx.c4, c_exp.fx.c5, e);
    a.x0 = a.x1 = 0;
    return a;
  }
  static __device__ __forceinline__ void add(Acc &a, int ush, int usl, Word b) {
    a.h0 += (long long)ush * b.x;
    a.h1 += (long long)ush * b.y;
    a.x0 += (long long)ush * b.z;
    a.x1 += (long long)ush * b.w;
    a.x0 += (long long)usl * b.x;
    a.x1 += (long long)usl * b.y;
  }
  template <int R, int NP>
  static __device__ __forceinline__ void rows(Acc (&acc)[NP], const int2 *rec, int i, int,
                                              const Word (&b)[R][NP]) {
    const int2 *s = rec + kRecHead + i;
#pragma unroll
    for (int r = 0; r + 1 < R; r += 2) {  // two entries per load: i is even where R > 1
      const int4 w = *reinterpret_cast<const int4 *>(s + r);
#pragma unroll
      for (int m = 0; m < NP; m++) {
        add(acc[m], w.x, w.y, b[r][m]);
        add(acc[m], w.z, w.w, b[r + 1][m]);
      }
    }
    if constexpr (R & 1) {
      const int2 w = s[R - 1];
#pragma unroll
      for (int m = 0; m < NP; m++) add(acc[m], w.x, w.y, b[R - 1][m]);
    }
  }
  static __device__ __forceinline__ Word finish(const Acc &acc, const Scalars &s, Word v0, Word c0,
                                                Word *v, Word *cov) {
    const FxU ua = fx_split(fx_mul_rsqrt(acc.h0 + (acc.x0 >> 28), s.rs));
    const FxU ub = fx_split(fx_mul_rsqrt(acc.h1 + (acc.x1 >> 28), s.rs));
    long long ca = a64(c0), cb = b64(c0);
    if (s.csh) {  // the same for the whole CTA
      ca >>= s.csh;
      cb >>= s.csh;
    }
    *v = word(a64(v0) - fx_mul_uu(ua, ua), b64(v0) - fx_mul_uu(ub, ub));
    *cov = word(ca + fx_mul_uu(s.nux, ua), cb + fx_mul_uu(s.nux, ub));
    return make_int4(ua.h, ub.h, ua.l, ub.l);
  }
  static __device__ __forceinline__ long long a64(Word w) { return (long long)fx_make(w.y, w.x); }
  static __device__ __forceinline__ long long b64(Word w) { return (long long)fx_make(w.w, w.z); }
  static __device__ __forceinline__ Word word(long long a, long long b) {
    return make_int4((int)a, (int)(a >> 32), (int)b, (int)(b >> 32));
  }
  static __device__ __forceinline__ void keep_a(Word &w, Word o) { w.x = o.x; w.y = o.y; }
  static __device__ __forceinline__ void keep_b(Word &w, Word o) { w.z = o.z; w.w = o.w; }
  static __device__ __forceinline__ float score_a(Word c, Word v) {
    return v.y >= 0 && (v.x | v.y) ? score32(fx_to_float(a64(c)), fx_to_float(a64(v))) : -1.0f;
  }
  static __device__ __forceinline__ float score_b(Word c, Word v) {
    return v.w >= 0 && (v.z | v.w) ? score32(fx_to_float(b64(c)), fx_to_float(b64(v))) : -1.0f;
  }
};

// One step of the screen for NP candidate pairs of this thread (Sec. 3.2 update): K(s, c) from
// the squared distance, the new factor entry u_c[j] = (K(s, c) - u_s . u_c) / L_jj, then
// v_{j+1}(c) = v_j(c) - u_c[j]^2, cov_{j+1}(x, c) = cov_j(x, c) - u_x[j] u_c[j], and the ALC
// screen score cov^2 / v.  The step's scalars and the location's formats are read from shared
// memory where they are used, so that the row loops keep their registers.
template <class A>
struct StepCtx {
  typename A::Word *U;      // factor rows in global memory (rows R .. n-1 are used)
  typename A::Word *Us;     // the first R rows, in shared memory
  int R;                    // even, or all n rows
  const typename A::Word *Xr;
  typename A::Word *vp, *cp;  // v_j(c) and cov_j(x, c) pairs
  const unsigned char *used;
  const int2 *rec;         // the pivot's record
  const void *tab;         // the exponential's table
  const int *fmt;          // formats of the location (FxArith): sh2b, e
  int Qpad, nrow, p, j;
  int s;         // the pivot, if it is held here (its flag may not be in place yet)
  int c0;        // global rank of the first candidate held here
  bool want;
  uint32_t tb;   // tensor-memory instance: this thread's first column (lane and column fields)
  int RT;        // rows R .. R + RT - 1 also held there (a read copy), RT words x 4 per pair
};

// The pairs are q and, NP = 2, q + dq: two per thread share every load of u_s and keep eight
// row loads in flight.  dq is the same for a warp; 0: there is no second pair, the first is
// computed in its place and not stored (a second instantiation for one pair would spill
// registers in both).
// TM: rows R .. R + RT - 1 are read from this thread's tensor-memory words instead of L2
// (they are still written to global memory, where the step's pivot row is
// gathered from); the caller keeps every warp convergent.
// slot: the first pair's place among this thread's pairs.
template <class A, int MBT, int NP, bool TM>
__device__ __forceinline__ void screen_pairs(const StepCtx<A> &C, int q, float &b1, int &r1, float &b2,
                                             int slot, int dq) {
  using Word = typename A::Word;
  const int Q = C.Qpad;
  const int jr = C.j < C.R ? C.j : C.R;  // rows R .. j-1 come from global memory
  // with tensor memory: rows R .. jt-1 from there, jt .. j-1 from global memory
  const int jt = TM ? max(jr, min(C.j, C.R + C.RT)) : jr;
  const uint32_t ta = TM ? C.tb + (uint32_t)(slot * C.RT * 4) : 0u;
  const uint32_t dt = dq ? (uint32_t)(C.RT * 4) : 0u;
  // checked build: the pairs' tensor-memory words end within the thread's 128 (the test is
  // the same for a whole warp, whose pairs share the slot)
  if constexpr (TM)
    if (!LAGP_CHK((slot + (dq ? 2 : 1)) * C.RT * 4 - 1, kTmemWords, 18)) return;
  typename A::Acc acc[NP];
  {
    typename A::Dist d[NP];
#pragma unroll
    for (int m = 0; m < NP; m++) A::dist_clear(d[m]);
    const int sh2b = A::kFixed ? C.fmt[0] : 0;
    for (int k = 0; k < C.p; k += 4) {  // four coordinates' loads in flight
      Word b[4][NP];
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (k + u < C.p)
#pragma unroll
          for (int m = 0; m < NP; m++) b[u][m] = C.Xr[(k + u) * Q + q + m * dq];
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (k + u < C.p)
#pragma unroll
          for (int m = 0; m < NP; m++) A::dist_add(d[m], C.rec, k + u, b[u][m], sh2b);
    }
#pragma unroll
    for (int m = 0; m < NP; m++) acc[m] = A::corr(d[m], C.tab, C.fmt);
  }
  // K(s, c) - sum_i u_s[i] u_c[i] over the rows held in shared memory, then tensor memory,
  // then global memory, four rows per iteration: their loads are issued before their terms are
  // accumulated.
  {
    const Word *us = C.Us + q;
    int i = 0;
    for (; i + 4 <= jr; i += 4, us += 4 * Q) {
      Word b[4][NP];
#pragma unroll
      for (int r = 0; r < 4; r++)
#pragma unroll
        for (int m = 0; m < NP; m++) b[r][m] = us[r * Q + m * dq];
      A::template rows<4>(acc, C.rec, i, C.nrow, b);
    }
    for (; i < jr; i++, us += Q) {
      Word b[1][NP];
#pragma unroll
      for (int m = 0; m < NP; m++) b[0][m] = us[m * dq];
      A::template rows<1>(acc, C.rec, i, C.nrow, b);
    }
  }
  if constexpr (TM) {
    for (int i = jr; i < jt; i += 4) {  // rows past jt are loaded but not used
      uint32_t tw[NP][16];
#pragma unroll
      for (int m = 0; m < NP; m++) tmem_ld16_issue(ta + m * dt + (uint32_t)(4 * (i - C.R)), tw[m]);
#pragma unroll
      for (int m = 0; m < NP; m++) tmem_wait16(tw[m]);
      if (i + 4 <= jt) {  // a whole group (the usual case): no per-row tests
        Word b[4][NP];
#pragma unroll
        for (int r = 0; r < 4; r++)
#pragma unroll
          for (int m = 0; m < NP; m++) b[r][m] = tmem_word<Word>(tw[m] + 4 * r);
        A::template rows<4>(acc, C.rec, i, C.nrow, b);
      } else {
#pragma unroll
        for (int r = 0; r < 3; r++)
          if (i + r < jt) {
            Word b[1][NP];
#pragma unroll
            for (int m = 0; m < NP; m++) b[0][m] = tmem_word<Word>(tw[m] + 4 * r);
            A::template rows<1>(acc, C.rec, i + r, C.nrow, b);
          }
      }
    }
  }
  {
    const unsigned long long pol = l2_evict_last_policy();
    const Word *ug = C.U + (size_t)jt * Q + q;
    int i = jt;
    for (; i + 4 <= C.j; i += 4, ug += 4 * (size_t)Q) {
      Word b[4][NP];
#pragma unroll
      for (int r = 0; r < 4; r++)
#pragma unroll
        for (int m = 0; m < NP; m++) b[r][m] = ld_l2_hint(ug + r * Q + m * dq, pol);
      A::template rows<4>(acc, C.rec, i, C.nrow, b);
    }
    for (; i < C.j; i++, ug += Q) {
      Word b[1][NP];
#pragma unroll
      for (int m = 0; m < NP; m++) b[0][m] = ld_l2_hint(ug + m * dq, pol);
      A::template rows<1>(acc, C.rec, i, C.nrow, b);
    }
  }
  const typename A::Scalars ps = A::scalars_load(C.rec);
#pragma unroll
  for (int m = 0; m < NP; m++) {
    if (m == 1 && !dq) break;
    const int qm = q + m * dq;
    const Word v0 = C.vp[qm], c0 = C.cp[qm];
    Word v, cx;
    const Word u = A::finish(acc[m], ps, v0, c0, &v, &cx);  // u_c[j]
    // the same for the whole CTA: a shared or a global store instead of a generic one
    if (!LAGP_CHK(qm, Q, 12)) continue;
    if (C.j < C.R) {
      C.Us[C.j * Q + qm] = u;
    } else {
      C.U[(size_t)C.j * Q + qm] = u;
      if constexpr (TM)
        if (C.j < C.R + C.RT) tmem_st4(ta + m * dt + (uint32_t)(4 * (C.j - C.R)), u);
    }
    // A used lane keeps its values: the step's pivot may be the partner of a live
    // candidate, and other threads read the pivot's v and cov at the start of the step
    // without a barrier after it.
    const bool u0 = C.used[2 * qm] || 2 * qm == C.s, u1 = C.used[2 * qm + 1] || 2 * qm + 1 == C.s;
    if (u0) { A::keep_a(v, v0); A::keep_a(cx, c0); }
    if (u1) { A::keep_b(v, v0); A::keep_b(cx, c0); }
    C.vp[qm] = v;
    C.cp[qm] = cx;
    if (C.want) {
      track2(u0 ? -1.0f : A::score_a(cx, v), C.c0 + 2 * qm, b1, r1, b2);
      track2(u1 ? -1.0f : A::score_b(cx, v), C.c0 + 2 * qm + 1, b1, r1, b2);
    }
  }
}

// ---- FP64 re-score of near-tied candidates (Sec. 3.3 decisions in FP64) ----
// Scratch and inputs of one CTA's re-score pass.  The CTA holds candidates with global
// ranks c0 .. c0 + Mloc - 1 (local index c = rank - c0); the current design is dr[0..jd)
// (global ranks), its FP64 factor is formed in A (global memory, jd x (jd + 1), the
// reciprocals of its diagonal in rl).
struct RescoreCtx {
  const double *X;
  const int32_t *cnd;          // the location's candidate list (global ranks -> design rows)
  const double *xl;            // x (shared memory)
  const double *etab;
  const unsigned char *used;   // local flags
  const void *vp, *cp;         // local screen state
  const int *dr;
  double *A, *rl;
  int *rlist, *nlist, *fail;
  double *red_n, *red_d;
  int *red_rr;
  int p, c0, Mloc, jd, lda;
  double theta_inv, onepg;
  float delta;                 // the near-tie margin of this step
  bool recip;                  // the FP64 recursion's own rounding (select.cu): entries u = t (1 / l)
};

// Every candidate of this CTA whose screen score is within 2 delta of B1 is re-scored in
// FP64: the design's FP64 Cholesky factor (with k(x) as an extra column) is formed from
// scratch, and each listed candidate's u = L^{-1} k_c is obtained by forward substitution
// (one warp per candidate), giving v_j(c) = 1 + g - |u|^2 and cov_j(x, c) = k(x, c) - u.u_x.
// On return (all threads, after a barrier): *bn / *bd is the CTA's best FP64 score as a
// fraction, *br its global rank (0x7fffffff if none), or *R.fail set (factor not PD; FxArith also:
// more candidates than the list holds).
template <class A>
__device__ __noinline__ void rescore_fp64(const RescoreCtx &R, float B1, double *bn_out, double *bd_out,
                             int *br_out) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int jd = R.jd, lda = R.lda, p = R.p;
  if (tid == 0) *R.nlist = 0;
  __syncthreads();
  for (int c = tid; c < R.Mloc; c += nt) {
    if (R.used[c]) continue;
    const typename A::Word *vp = static_cast<const typename A::Word *>(R.vp);
    if (!A::positive(vp, c)) continue;
    const float sc = A::score(static_cast<const typename A::Word *>(R.cp), vp, c);
    if (sc >= B1 * (1.0f - 2.0f * R.delta)) {
      const int pos = atomicAdd(R.nlist, 1);
      if (pos < RESCORE_CAP) R.rlist[pos] = c;
    }
  }
  if constexpr (A::kFixed) {  // more near-ties than the list holds: the recursion's work
    __syncthreads();
    if (*R.nlist > RESCORE_CAP) {
      if (tid == 0) *R.fail = 1;
      __syncthreads();
      return;
    }
  }
  // FP64 factor of the current design with k(x) as an extra column (lower triangle)
  for (int qq = tid; qq < jd * (jd + 1); qq += nt) {
    const int a = qq / (jd + 1), b = qq % (jd + 1);
    if (b < jd && b > a) continue;
    const double *xa = R.X + (int64_t)R.cnd[R.dr[a]] * p;
    double val;
    if (b < jd) val = (a == b) ? R.onepg : corr64(xa, R.X + (int64_t)R.cnd[R.dr[b]] * p, p, R.theta_inv, R.etab);
    else val = corr64(xa, R.xl, p, R.theta_inv, R.etab);
    R.A[a * lda + b] = val;
  }
  chol_flat_fp64(R.A, jd, lda, 1, R.rl, R.fail, R.recip);
  if (*R.fail) return;
  const double *L = R.A;
  // more near-ties than the list holds: re-score every remaining candidate
  const bool all = *R.nlist > RESCORE_CAP;
  const int nl = all ? R.Mloc : *R.nlist;
  double bn = -1.0, bd = 1.0;
  int br = 0x7fffffff;
  for (int item = warp; item < nl; item += nt / 32) {
    const int c = all ? item : R.rlist[item];
    if (R.used[c]) continue;
    const int rank = R.c0 + c;
    const double *xc = R.X + (int64_t)R.cnd[rank] * p;
    double tv[kMaxN / 32];
#pragma unroll
    for (int r = 0; r < kMaxN / 32; r++) {
      const int i = 32 * r + lane;
      tv[r] = (i < jd) ? corr64(R.X + (int64_t)R.cnd[R.dr[i]] * p, xc, p, R.theta_inv, R.etab) : 0.0;
    }
    double vsum = R.onepg;
    double cov = corr64(R.xl, xc, p, R.theta_inv, R.etab);
    for (int m = 0; m < jd; m++) {
      double own = 0.0;
#pragma unroll
      for (int r = 0; r < kMaxN / 32; r++)
        if (32 * r + lane == m) own = tv[r];
      const double r = R.rl[m], uq = own * r;  // divided by l_mm as chol_flat_fp64 does
      const double um_l = R.recip ? uq : fma(fma(-uq, L[m * lda + m], own), r, uq);
      const double um = __shfl_sync(0xffffffffu, um_l, m & 31);
      vsum = fma(-um, um, vsum);
      cov = fma(-L[m * lda + jd], um, cov);
#pragma unroll
      for (int r = 0; r < kMaxN / 32; r++) {
        const int i = 32 * r + lane;
        if (i > m && i < jd) tv[r] = fma(-L[i * lda + m], um, tv[r]);
      }
    }
    if (vsum > 0.0) {
      const double num = cov * cov;
      if (frac_better(num, vsum, rank, bn, bd, br)) {
        bn = num;
        bd = vsum;
        br = rank;
      }
    }
  }
  if (lane == 0) {
    R.red_n[warp] = bn;
    R.red_d[warp] = bd;
    R.red_rr[warp] = br;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < nt / 32; w++)
      if (frac_better(R.red_n[w], R.red_d[w], R.red_rr[w], bn, bd, br)) {
        bn = R.red_n[w];
        bd = R.red_d[w];
        br = R.red_rr[w];
      }
    R.red_n[0] = bn;
    R.red_d[0] = bd;
    R.red_rr[0] = br;
  }
  __syncthreads();
  *bn_out = R.red_n[0];
  *bd_out = R.red_d[0];
  *br_out = R.red_rr[0];
}

}  // namespace
}  // namespace lagp
