// knn.cu -- kernel (a): candidate sets of the ncand nearest design points.
//
// Gramacy & Apley, Sec. 3 (the nearest-neighbour sub-design, also the start design
// D_{n0}) and Sec. 6 (every search is restricted to the N' nearest candidates).  For
// each predictive location x the kernel returns the ncand design indices with the
// smallest exact FP64 squared distance, ordered by (d2, index).
//
// FP64 is 1/64 of FP32 throughput on this GPU, so exact distances are computed only for
// the few points that can be members.  One CTA owns one location at a time:
//   prep    (once per call) an FP32 copy of X, rows padded to a vector load, and
//           B = max |coordinate|;
//   pass 0  FP32 squared distances d2f of a sample of the design, and a 4096-bin histogram of
//           the top 12 bits of d2f (non-negative floats order like their bit patterns), bound
//           the ncand-th smallest from above;
//   pass 1  the points with d2f <= bound are listed, with a histogram of their d2f.  Large
//           designs: the scan below lists them for 64 locations at a time on the tensor cores
//           (and pass 0 is a kernel before it); the location's CTA starts from its list;
//   select  a block scan finds the bin b* holding the ncand-th smallest d2f; tau is the
//           upper edge of b*.  Every listed point with d2f <= tau + 2E survives, where
//           E bounds |d2f - d2| (FP32 rounding of the coordinates, the differences and the
//           fused sum; see fp32_err_bound) -- all true members survive; the survivors get
//           their exact FP64 d2 from a list, so the FP64 work runs on full warps.  Where the
//           sample is too small or its bound missed, two passes over all points do the same;
//   sort    the survivors in (d2, index) order: a bucket sort on d2 with insertion in the
//           buckets, or a bitonic sort on (d2 bits, index) where buckets overflow; the
//           first ncand indices are written out.
// If the survivors do not fit in shared memory (many points tied at the boundary), the
// CTA redoes that location exactly in FP64: a 4096-bin histogram of float(d2) over exact
// d2 (recomputed in every pass: no scratch), and radix refinement on the 96-bit key (d2 bits, index) for an
// oversized boundary bin.  Either way the result is bit-identical to a full sort.
#include <cuda_fp16.h>
#include <float.h>
#include <math.h>

#include <algorithm>

#include "batch.cuh"
#include "check.cuh"
#include "internal.h"

namespace lagp {
namespace {

constexpr int KB = 256;               // threads per CTA (the location kernel: this or twice it)
constexpr int HBITS = 12;
constexpr int KS = 16;                // the sample that bounds the M-th distance: one block of
                                      // 32 consecutive design points in every KS blocks
constexpr int HBINS = 1 << HBITS;     // 4096 histogram bins
// The bucket sort's permutation gets cap entries of its own where they fit in shared
// memory next to the keys (cap <= 8192); otherwise it uses the histogram's second half
// (HBINS / 2 entries) and larger survivor sets take the bitonic sort.
__host__ __device__ constexpr bool knn_own_perm(int cap) { return cap > HBINS / 2 && cap <= 8192; }


__device__ __forceinline__ double sqdist_exact(const double *x, const double *xi, int p) {
  double acc = 0.0;
  for (int k = 0; k < p; k++) {
    double t = __dsub_rn(x[k], xi[k]);
    acc = __dadd_rn(acc, __dmul_rn(t, t));
  }
  return acc;
}

__device__ __forceinline__ uint32_t coarse_bin(double d2) {
  return __float_as_uint(__double2float_rn(d2)) >> (31 - HBITS);
}

// Keys are (d2 bits, index) compared as three 32-bit words (hi, lo, index): non-negative
// doubles order like their bit patterns.
__device__ __forceinline__ bool key_less3(uint32_t ah, uint32_t al, int32_t ai, uint32_t bh,
                                          uint32_t bl, int32_t bi) {
  return ah < bh || (ah == bh && (al < bl || (al == bl && ai < bi)));
}

// Digit d (0..11, most significant first) of the 96-bit key (bits:64 | index:32).
__device__ __forceinline__ uint32_t key_digit(uint64_t bits, uint32_t idx, int d) {
  return d < 8 ? (uint32_t)(bits >> (56 - 8 * d)) & 0xFFu : (idx >> (24 - 8 * (d - 8))) & 0xFFu;
}

// True if the top 8*nd bits of the key equal the recorded prefix digits.
__device__ __forceinline__ bool key_prefix_eq(uint64_t bits, uint32_t idx, int nd,
                                              const uint32_t *pref) {
  for (int d = 0; d < nd; d++)
    if (key_digit(bits, idx, d) != pref[d]) return false;
  return true;
}

// Exclusive block scan of one value per thread; returns the prefix, *total gets the sum.
template <int NT>
__device__ uint32_t block_excl_scan(uint32_t v, uint32_t *warp_tmp, uint32_t *total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) warp_tmp[w] = inc;
  __syncthreads();
  if (w == 0) {
    uint32_t s = (lane < NT / 32) ? warp_tmp[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    if (lane < NT / 32) warp_tmp[lane] = s;  // inclusive warp totals
  }
  __syncthreads();
  uint32_t base = (w > 0) ? warp_tmp[w - 1] : 0;
  *total = warp_tmp[NT / 32 - 1];
  __syncthreads();
  return base + inc - v;
}

// Find, over hist[0..nbins), the bin where the cumulative count first reaches `rank`
// (1-based); returns the bin and the count strictly below it.  nbins == HBINS or 256.
template <int NT>
__device__ void find_rank_bin(const uint32_t *hist, int nbins, uint32_t rank, uint32_t *warp_tmp,
                              int *bin_out, uint32_t *below_out) {
  const int per = nbins / NT > 0 ? nbins / NT : 1;  // a power of two
  const int first = threadIdx.x * per;
  uint32_t part = 0;
  // each thread's range starts at its own rotation: the lanes of a warp read different
  // banks instead of all `per` apart (a per-way bank conflict)
  if (first < nbins)
    for (int b = 0; b < per; b++) part += hist[first + ((b + threadIdx.x) & (per - 1))];
  uint32_t total;
  uint32_t pre = block_excl_scan<NT>(part, warp_tmp, &total);
  if (first < nbins && pre < rank && rank <= pre + part) {
    uint32_t cum = pre;
    for (int b = 0; b < per; b++) {
      uint32_t h = hist[first + b];
      if (cum + h >= rank) {
        *bin_out = first + b;
        *below_out = cum;
        break;
      }
      cum += h;
    }
  }
  __syncthreads();
}

// Bitonic sort of n2 (a power of two) keys held as (hi, lo, index) words in shared memory;
// each stage visits exactly its n2/2 compare-exchange pairs.
template <int NT>
__device__ void bitonic_sort(uint32_t *kh, uint32_t *kl, int32_t *idx, int n2) {
  for (int k = 2; k <= n2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      const int lj = __ffs(j) - 1;
      for (int pp = threadIdx.x; pp < (n2 >> 1); pp += NT) {
        const int i = ((pp >> lj) << (lj + 1)) | (pp & (j - 1));
        const int ixj = i + j;
        const uint32_t ah = kh[i], al = kl[i], bh = kh[ixj], bl = kl[ixj];
        const int32_t ai = idx[i], bi = idx[ixj];
        const bool up = (i & k) == 0;
        const bool sw = up ? key_less3(bh, bl, bi, ah, al, ai) : key_less3(ah, al, ai, bh, bl, bi);
        if (sw) {
          kh[i] = bh; kl[i] = bl; idx[i] = bi;
          kh[ixj] = ah; kl[ixj] = al; idx[ixj] = ai;
        }
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ void put_key(uint32_t *kh, uint32_t *kl, int32_t *sidx, uint32_t pos,
                                        double d2, int32_t i) {
  const uint64_t b = (uint64_t)__double_as_longlong(d2);
  kh[pos] = (uint32_t)(b >> 32);
  kl[pos] = (uint32_t)b;
  sidx[pos] = i;
}

// Bound on |d2f - d2| for a squared distance d2 <= d computed in FP32 from coordinates
// of magnitude <= B (u = 2^-24): rounding the coordinates and each difference gives
// |diff_f - diff| <= 2uB + u|diff|, squaring and the p fused additions add (2+p)u d2;
// summed over k with sum |diff_k| <= sqrt(p d2).  Constants doubled for safety.
__device__ __forceinline__ double fp32_err_bound(double d, double B, int p) {
  const double u = 5.9604644775390625e-08;  // 2^-24
  return 8.0 * u * B * sqrt((double)p * d) + (4.0 + 2.0 * p) * u * d + 16.0 * p * u * u * B * B;
}

// Exact path for one location (the fallback when many points tie at the boundary):
// exact FP64 d2 of every point (recomputed in each pass, no scratch), coarse histogram of
// float(d2), boundary resolution by radix refinement; keys into shared memory; returns
// the count.
template <int NT>
__device__ int knn_exact_location(const double *__restrict__ X, int N, int p, int M,
                                  const double *xs, uint32_t *kh, uint32_t *kl, int32_t *sidx,
                                  uint32_t *hist, int cap, uint32_t *warp_tmp, int *sh_bin,
                                  uint32_t *sh_below, uint32_t *sh_count, uint32_t *pref) {
  for (int b = threadIdx.x; b < HBINS; b += NT) hist[b] = 0;
  if (threadIdx.x == 0) *sh_count = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < N; i += NT)
    atomicAdd(&hist[coarse_bin(sqdist_exact(xs, X + (size_t)i * p, p))], 1u);
  __syncthreads();
  find_rank_bin<NT>(hist, HBINS, (uint32_t)M, warp_tmp, sh_bin, sh_below);
  const uint32_t bstar = (uint32_t)*sh_bin;
  const uint32_t below = *sh_below;
  const uint32_t nb = hist[bstar];
  const bool fits = below + nb <= (uint32_t)cap;
  for (int i = threadIdx.x; i < N; i += NT) {
    const double d2 = sqdist_exact(xs, X + (size_t)i * p, p);
    const uint32_t b = coarse_bin(d2);
    if (b < bstar || (fits && b == bstar)) put_key(kh, kl, sidx, atomicAdd(sh_count, 1u), d2, i);
  }
  __syncthreads();
  if (!fits) {
    uint32_t need = (uint32_t)M - below;
    uint32_t *h256 = hist;
    for (int d = 0; d < 12; d++) {
      for (int b = threadIdx.x; b < 256; b += NT) h256[b] = 0;
      __syncthreads();
      for (int i = threadIdx.x; i < N; i += NT) {
        const double d2 = sqdist_exact(xs, X + (size_t)i * p, p);
        if (coarse_bin(d2) != bstar) continue;
        const uint64_t bits = (uint64_t)__double_as_longlong(d2);
        if (!key_prefix_eq(bits, (uint32_t)i, d, pref)) continue;
        atomicAdd(&h256[key_digit(bits, (uint32_t)i, d)], 1u);
      }
      __syncthreads();
      const uint32_t cnt0 = *sh_count;  // stable here: no thread appends until after the scan
      find_rank_bin<NT>(h256, 256, need, warp_tmp, sh_bin, sh_below);
      const uint32_t dd = (uint32_t)*sh_bin, dbelow = *sh_below, deq = h256[dd];
      const bool last = cnt0 + dbelow + deq <= (uint32_t)cap;
      for (int i = threadIdx.x; i < N; i += NT) {
        const double d2 = sqdist_exact(xs, X + (size_t)i * p, p);
        if (coarse_bin(d2) != bstar) continue;
        const uint64_t bits = (uint64_t)__double_as_longlong(d2);
        if (!key_prefix_eq(bits, (uint32_t)i, d, pref)) continue;
        const uint32_t dg = key_digit(bits, (uint32_t)i, d);
        if (dg < dd || (last && dg == dd)) put_key(kh, kl, sidx, atomicAdd(sh_count, 1u), d2, i);
      }
      __syncthreads();
      if (last) break;
      need -= dbelow;
      if (threadIdx.x == 0) pref[d] = dd;
      __syncthreads();
    }
  }
  const int cnt = (int)*sh_count;
  __syncthreads();  // the caller reuses the counter
  return cnt;
}

// Floats per row of the FP32 copy of X: the dimension, padded with zeros to 1, 2, 4 or 8, so
// that a row is one or two vector loads.
__host__ __device__ constexpr int knn_row(int p) { return p > 4 ? 8 : p > 2 ? 4 : p; }

// The FP32 copy of X (N x p, row-major), and B = max |coordinate|.
__global__ void knn_prep_kernel(const double *__restrict__ X, int64_t N, int p,
                                float *__restrict__ Xf, unsigned int *__restrict__ bmax) {
  __shared__ unsigned int wmax[KB / 32];
  unsigned int m = 0;
  const int S = knn_row(p);
  const int64_t n = N * S;
  for (int64_t i = blockIdx.x * (int64_t)KB + threadIdx.x; i < n; i += (int64_t)gridDim.x * KB) {
    const int64_t r = i / S;
    const int k = (int)(i - r * S);
    const double x = k < p ? X[r * p + k] : 0.0;
    Xf[i] = __double2float_rn(x);
    const float a = __double2float_ru(fabs(x));
    m = max(m, __float_as_uint(a));
  }
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < KB / 32; w++) m = max(m, wmax[w]);
    atomicMax(bmax, m);
  }
}

// FP32 d2 of point i from its row of Xf (the padding adds exact zeros).
template <int S>
__device__ __forceinline__ float sqdist_f32(const float *xf, const float *__restrict__ Xf, int i) {
  const float *row = Xf + (size_t)i * S;
  float y[S];
  if constexpr (S >= 4) {
#pragma unroll
    for (int k = 0; k < S; k += 4) {
      const float4 v = *reinterpret_cast<const float4 *>(row + k);
      y[k] = v.x, y[k + 1] = v.y, y[k + 2] = v.z, y[k + 3] = v.w;
    }
  } else if constexpr (S == 2) {
    const float2 v = *reinterpret_cast<const float2 *>(row);
    y[0] = v.x, y[1] = v.y;
  } else {
    y[0] = row[0];
  }
  float acc = 0.0f;
#pragma unroll
  for (int k = 0; k < S; k++) {
    const float dk = __fsub_rn(xf[k], y[k]);
    acc = __fmaf_rn(dk, dk, acc);
  }
  return acc;
}

// Visits the points i = first, first + stride, ... < N: the FP32 distances of KU points are
// formed -- their loads in flight together -- before f(d2f, i) uses any of them (one point
// at a time, each pass was bound by the L2 latency of its dependent loads).  first is the
// thread's lane past a multiple of 32, stride a multiple of 32: a warp visits 32 neighbours.
// Rows of 8: a lane that loaded its own point's row would touch every line of 32 rows twice; the
// warp loads them as they lie instead, lane l the half row l & 1 of point l / 2, the even lanes start
// the sum and the odd ones end it (the same operations in the same order), and the even lanes
// take over half of the points.  GB300, 3000 8-d locations over 100000 points far from the origin
// (not scanned), ncand = 1000: 1.00 ms a row per lane -> 0.87 (a dimension-major copy: 0.83; the
// lists of the scan want rows); 20000 points: 0.36 -> 0.35.
constexpr int KU = 4;
template <int S, typename F>
__device__ __forceinline__ void each_point(const float *xf, const float *__restrict__ Xf, int N,
                                           int first, int stride, F f) {
  int i = first;
  if constexpr (S == 8) {
    const int lane = threadIdx.x & 31, odd = lane & 1;
    const float x0 = xf[4 * odd], x1 = xf[4 * odd + 1], x2 = xf[4 * odd + 2], x3 = xf[4 * odd + 3];
    // the half row's sum, on top of a
    auto half = [&](float a, const float4 &v) {
      const float d0 = __fsub_rn(x0, v.x), d1 = __fsub_rn(x1, v.y), d2 = __fsub_rn(x2, v.z), d3 = __fsub_rn(x3, v.w);
      return __fmaf_rn(d3, d3, __fmaf_rn(d2, d2, __fmaf_rn(d1, d1, __fmaf_rn(d0, d0, a))));
    };
    const int mine = odd ? lane >> 1 : 16 + (lane >> 1);
    for (; i - lane + (KU - 1) * stride + 31 < N; i += KU * stride) {
      float4 v[KU][2];
      float d[KU];
#pragma unroll
      for (int u = 0; u < KU; u++) {
        const float4 *r = reinterpret_cast<const float4 *>(Xf + (size_t)(i - lane + u * stride) * S) + lane;
        v[u][0] = r[0];
        v[u][1] = r[32];
      }
#pragma unroll
      for (int u = 0; u < KU; u++) {
        const float a = half(__shfl_up_sync(0xffffffffu, half(0.0f, v[u][0]), 1), v[u][0]);  // points 0 .. 15
        const float b = half(__shfl_up_sync(0xffffffffu, half(0.0f, v[u][1]), 1), v[u][1]);  // 16 .. 31
        const float o = __shfl_down_sync(0xffffffffu, b, 1);
        d[u] = odd ? a : o;
      }
#pragma unroll
      for (int u = 0; u < KU; u++) f(d[u], i - lane + u * stride + mine);
    }
  } else {
    for (; i + (KU - 1) * stride < N; i += KU * stride) {
      float d[KU];
#pragma unroll
      for (int u = 0; u < KU; u++) d[u] = sqdist_f32<S>(xf, Xf, i + u * stride);
#pragma unroll
      for (int u = 0; u < KU; u++) f(d[u], i + u * stride);
    }
  }
  for (; i < N; i += stride) f(sqdist_f32<S>(xf, Xf, i), i);
}

// Pass 0: a sample of the design -- 32 consecutive points (whole lines) out of every 32 KS,
// spread over any ordering of X -- bounds the M-th smallest d2f from above: the bound is the
// upper edge of the bin holding the sample's ceil(1.5 M ns / N)-th smallest, about 1.5 M points
// of the whole design.  sample_rank: that rank, 0 where the sample is too small for it.
__device__ __forceinline__ int sample_rank(int N, int M) {
  const int ns = (N / (32 * KS)) * 32 + min(32, N % (32 * KS));
  const int ks = (int)(((int64_t)3 * M * ns + 2 * (int64_t)N - 1) / (2 * (int64_t)N));
  return ks < ns ? ks : 0;
}
// hist: zeroed, HBINS bins.  Every thread returns after the same barriers.
template <int S, int NT>
__device__ float sample_bound(const float *xf, const float *__restrict__ Xf, int N, int ks, uint32_t *hist,
                              uint32_t *warp_tmp, int *sh_bin, uint32_t *sh_below) {
  each_point<S>(xf, Xf, N, (threadIdx.x >> 5) * 32 * KS + (threadIdx.x & 31), (NT / 32) * 32 * KS,
                [&](float d2f, int) { atomicAdd(&hist[__float_as_uint(d2f) >> (31 - HBITS)], 1u); });
  __syncthreads();
  find_rank_bin<NT>(hist, HBINS, (uint32_t)ks, warp_tmp, sh_bin, sh_below);
  return __uint_as_float(((uint32_t)*sh_bin + 1u) << (31 - HBITS));
}

// ---- The scan: pass 1 of many locations at once, on the tensor cores
// d2 = |y|^2 - 2 x.y + |x|^2 for 16 points by 8 locations is one m16n8k16 MMA in FP16 with FP32
// sums: a point's 16 values against a location's.  Coordinates are scaled by a power of two so
// that |y| <= 1; |y|^2 takes three slots (11 bits each) against 1, and with p <= 4 the
// coordinates are split in two halves, y_h x_h + y_l x_h + y_h x_l, so that the products keep
// 22 bits.  The result only decides which points can have an FP32 distance within the sample's
// bound: the threshold adds an upper bound of every rounding (scan_bound), and a location for
// which that is not small (x far outside the design, values out of range) is not scanned.
// GB300: one location at a time, pass 1 reads the FP32 copy from L2 and spends 2 p FP32
// instructions per point; here 64 locations share every read, and an MMA (2 cycles of an SM),
// four comparisons and four votes serve 128 distances.  100000 8-d points, 10000 locations, ncand =
// 2000, the whole search: 4.15 -> 2.27 ms (per-location passes at this kernel's 512 threads: 3.46);
// 40000 2-d points, ncand = 1000: 0.78 -> 0.61; one 2-d location: 57 -> 51 us.
struct Scan {
  int64_t first;      // launch position of the first location of this wave
  uint32_t *cnt;      // points listed for each location of the wave; nullptr: no scan
  float *bound;       // the sample's bound
  int32_t *list;      // cap indices per location
  int cap;
  uint4 *frag;        // the design: ceil(N / 16) tiles of 32 lanes' A operands; row r of tile k
                      // is point r tiles + k, so that neighbours in X lie in different tiles
  uint32_t *xfrag;    // the locations: 8 words (16 halves) each
  float *thr;         // threshold - |x|^2; -inf: not scanned
};
constexpr int kScanTiles = 128;  // row tiles (16 points) between two extractions

// The 16 values of a point (y = its scaled coordinates) or, x = true, of a location.
__device__ __forceinline__ void scan_values(const float *y, int p, bool x, __half (&v)[16], float *norm) {
  const bool split = p <= 4;
  for (int k = 0; k < 16; k++) v[k] = __float2half_rn(0.0f);
  float nn = 0.0f;
#pragma unroll
  for (int k = 0; k < kMaxP; k++) {
    if (k >= p) break;
    const __half h = __float2half_rn(y[k]);
    const float hf = __half2float(h);
    const __half l = split ? __float2half_rn(y[k] - hf) : __float2half_rn(0.0f);
    const float r = hf + __half2float(l);
    nn = fmaf(r, r, nn);
    const __half m2 = __float2half_rn(-2.0f);
    v[k] = x ? __hmul(m2, h) : h;  // exact
    if (split) {
      v[p + k] = x ? __hmul(m2, h) : l;
      v[2 * p + k] = x ? __hmul(m2, l) : h;
    }
  }
  *norm = nn;
  for (int k = 0; k < 3; k++) {
    const __half h = __float2half_rn(nn);
    v[13 + k] = x ? __float2half_rn(1.0f) : h;
    nn -= __half2float(h);
  }
}

// The scale 2^-e with |coordinate| 2^-e <= 1 for every |coordinate| <= B; false where there is none.
__device__ __forceinline__ bool scan_scale(float B, float *s) {
  if (!(B > 8.6736174e-19f && B < 1.1529215e18f)) return false;  // 2^-60 .. 2^60
  int e;
  frexpf(B, &e);  // B = f 2^e, f < 1
  *s = ldexpf(1.0f, -e);
  return true;
}

// Threshold for the scaled squared distances as the scan forms them: every point with d2f <=
// bound passes.  -inf: the location is not to be scanned.
//   d2 <= bound + the FP32 bound of fp32_err_bound;
//   coordinates rounded to d each (11 bits, or 22 split: 2^-12 or 2^-22 of 1 and of X, a power
//   of two >= |x|): 2 sqrt(p d2) d + p d^2;
//   the products left out when split, 2 p 2^-24 X, and the parts of the norms, 2^-24;
//   FP32 sums: 17 terms of at most p X^2 each to 2^-23 of the largest, |x|^2, |y|^2 and their
//   difference from the threshold to a few 2^-24: 2^-17 p X^2 in all.
__device__ __forceinline__ float scan_bound(float bound, float s, const float *xf, int p) {
  float X = 1.0f;
  bool ok = true;
  for (int k = 0; k < p; k++) {
    const float a = fabsf(xf[k] * s);
    ok = ok && a <= 16.0f;
    while (ok && X < a) X *= 2.0f;
  }
  const float bn = bound * s * s, fp = (float)p;
  if (!ok || !(bn >= 0.0f && bn < 1e4f)) return -INFINITY;
  const float rt = sqrtf(fp * bn);
  const float e32 = 4.7683716e-7f * X * rt + 1.5e-6f * bn + 1e-12f * fp * X * X;
  const float d = (p <= 4 ? 2.3841858e-7f : 2.4414062e-4f) * (1.0f + X);
  const float e16 = 2.01f * sqrtf(fp * (bn + e32)) * d + fp * d * d + fp * 2.3841858e-7f * X +
                    7.6293945e-6f * fp * X * X;
  const float e = 1.01f * (e32 + e16);
  return e <= 0.125f * bn ? bn + e : -INFINITY;
}

// The sample's bound, threshold and operand of every location of a wave (one CTA each, up to
// npad, a multiple of kScanLocs), and, convert, the design's operands (the CTAs beyond).
template <int P>
__global__ void __launch_bounds__(KB) knn_bound_kernel(const Scan S_, int N, int p, const double *__restrict__ XX,
                                                       int nloc, int npad, int M, const float *__restrict__ Xf,
                                                       const unsigned int *__restrict__ bmax,
                                                       const int32_t *__restrict__ list,
                                                       const LocDesc *__restrict__ locs, int ldxx) {
  constexpr int S = P ? knn_row(P) : kMaxP, NT = KB;
  if (P > 0) p = P;
  const float B = __uint_as_float(*bmax);
  float s = 1.0f;
  const bool scaled = scan_scale(B, &s);
  if ((int)blockIdx.x >= npad) {
    const int tiles = (N + 15) / 16, step = (gridDim.x - npad) * KB;
    uint32_t *words = reinterpret_cast<uint32_t *>(S_.frag);
    for (int i = (blockIdx.x - npad) * KB + threadIdx.x; i < 16 * tiles; i += step) {
      float y[kMaxP], nn;
      __half v[16];
      for (int k = 0; k < kMaxP; k++) y[k] = i < N && k < p && scaled ? Xf[(size_t)i * S + k] * s : 0.0f;
      scan_values(y, p, false, v, &nn);
      if (i >= N) v[13] = __float2half_rn(60000.0f);  // past every threshold
      const int row = i / tiles, g = row & 7, hi = row >> 3;
      uint32_t *w = words + (size_t)(i - row * tiles) * 128 + g * 16 + hi;
#pragma unroll
      for (int kk = 0; kk < 8; kk++)
        w[(kk & 3) * 4 + 2 * (kk >> 2)] =
            (uint32_t)__half_as_ushort(v[2 * kk]) | (uint32_t)__half_as_ushort(v[2 * kk + 1]) << 16;
    }
    return;
  }
  __shared__ uint32_t hist[HBINS];
  __shared__ float xf[kMaxP];
  __shared__ uint32_t warp_tmp[32];
  __shared__ int sh_bin;
  __shared__ uint32_t sh_below;
  const int tt = blockIdx.x;
  float bound = INFINITY, thr = -INFINITY;
  int ks = 0;
  if (tt < nloc) {
    const int64_t t = list ? list[S_.first + tt] : S_.first + tt;
    if (locs) M = locs[t].M;
    if (threadIdx.x < kMaxP)
      xf[threadIdx.x] = threadIdx.x < p ? __double2float_rn(XX[t * (locs ? ldxx : p) + threadIdx.x]) : 0.0f;
    for (int b = threadIdx.x; b < HBINS; b += KB) hist[b] = 0;
    __syncthreads();
    ks = scaled ? sample_rank(N, M) : 0;
    if (ks > 0) bound = sample_bound<S, NT>(xf, Xf, N, ks, hist, warp_tmp, &sh_bin, &sh_below);
  }
  if (threadIdx.x == 0) {
    float y[kMaxP], nn;
    __half v[16];
    if (ks > 0) thr = scan_bound(bound, s, xf, p);
    for (int k = 0; k < kMaxP; k++) y[k] = k < p && thr > -INFINITY ? xf[k] * s : 0.0f;
    scan_values(y, p, true, v, &nn);
    for (int kk = 0; kk < 8; kk++)
      S_.xfrag[(size_t)tt * 8 + kk] =
          (uint32_t)__half_as_ushort(v[2 * kk]) | (uint32_t)__half_as_ushort(v[2 * kk + 1]) << 16;
    S_.thr[tt] = thr - nn;
    S_.bound[tt] = bound;
    S_.cnt[tt] = 0u;
  }
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint4 &a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "f"(0.0f));
}

// Lists, for 64 locations, the points of a range of tiles whose distance passes.  A warp holds
// the 64 locations' operands and thresholds and takes every eighth tile; the four votes of a
// tile and column tile are its result, 128 bits.  After kScanTiles tiles each warp takes one
// column tile's bits to its eight lists.  blockIdx: 64 locations, part of the design.
__global__ void __launch_bounds__(KB) knn_scan_kernel(const Scan S_, int tiles, int part) {
  __shared__ uint4 votes[kScanLocs / 8][kScanTiles];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
  const int loc0 = blockIdx.x * kScanLocs;
  uint32_t b0[kScanLocs / 8], b1[kScanLocs / 8];
  float2 th[kScanLocs / 8];
#pragma unroll
  for (int c = 0; c < kScanLocs / 8; c++) {
    const uint32_t *x = S_.xfrag + (size_t)(loc0 + 8 * c + g) * 8;
    b0[c] = x[q];
    b1[c] = x[q + 4];
    th[c] = *reinterpret_cast<const float2 *>(S_.thr + loc0 + 8 * c + 2 * q);
  }
  // nothing to do where none of the 64 is to be scanned (each warp holds all their thresholds)
  bool any = false;
#pragma unroll
  for (int c = 0; c < kScanLocs / 8; c++) any = any || th[c].x > -INFINITY || th[c].y > -INFINITY;
  if (!__any_sync(0xffffffffu, any)) return;
  const int first = blockIdx.y * part, last = min(first + part, tiles);
  for (int base = first; base < last; base += kScanTiles) {
    const int end = min(kScanTiles, last - base);
    uint4 a = make_uint4(0u, 0u, 0u, 0u);
    if (warp < end) a = __ldg(S_.frag + (size_t)(base + warp) * 32 + lane);
    for (int k = warp; k < end; k += KB / 32) {
      const uint4 cur = a;
      if (k + KB / 32 < end) a = __ldg(S_.frag + (size_t)(base + k + KB / 32) * 32 + lane);
#pragma unroll
      for (int c = 0; c < kScanLocs / 8; c++) {
        float d[4];
        mma_f16(d, cur, b0[c], b1[c]);
        uint4 v;
        v.x = __ballot_sync(0xffffffffu, d[0] <= th[c].x);
        v.y = __ballot_sync(0xffffffffu, d[1] <= th[c].y);
        v.z = __ballot_sync(0xffffffffu, d[2] <= th[c].x);
        v.w = __ballot_sync(0xffffffffu, d[3] <= th[c].y);
        if (lane == 0) votes[c][k] = v;
      }
    }
    __syncthreads();
    uint4 v[kScanTiles / 32];
#pragma unroll
    for (int u = 0; u < kScanTiles / 32; u++)
      v[u] = 32 * u + lane < end ? votes[warp][32 * u + lane] : make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
#pragma unroll 1
    for (int c = 0; c < 8; c++) {  // column c: votes of lanes 4 g + c / 2; d[c & 1] and d[2 + (c & 1)]
      uint32_t m[kScanTiles / 32];
      int n = 0;
#pragma unroll
      for (int u = 0; u < kScanTiles / 32; u++) {
        const uint32_t lo = (c & 1) ? v[u].y : v[u].x, hi = (c & 1) ? v[u].w : v[u].z;
        m[u] = ((lo >> (c >> 1)) & 0x11111111u) | ((hi >> (c >> 1)) & 0x11111111u) << 1;  // bit 4 g + half
        n += __popc(m[u]);
      }
      int inc = n;
      for (int o = 1; o < 32; o <<= 1) {
        const int w = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += w;
      }
      const int total = __shfl_sync(0xffffffffu, inc, 31);
      if (!total) continue;
      const int loc = loc0 + 8 * warp + c;
      uint32_t at = 0;
      if (lane == 0) at = atomicAdd(S_.cnt + loc, (uint32_t)total);
      at = __shfl_sync(0xffffffffu, at, 0) + (uint32_t)(inc - n);
      int32_t *out = S_.list + (size_t)loc * S_.cap;
#pragma unroll
      for (int u = 0; u < kScanTiles / 32; u++) {
        uint32_t w = m[u];
        const int tile = base + 32 * u + lane;
        while (w) {
          const int b = __ffs(w) - 1;
          w &= w - 1;
          if (at < (uint32_t)S_.cap) out[at] = ((b >> 2) + 8 * (b & 1)) * tiles + tile;
          at++;
        }
      }
    }
  }
}

constexpr int BUCKET_CAP = 32; // largest bucket sorted in place; beyond, the bitonic sort

// Rank order of the cnt survivors (keys (d2 hi, d2 lo, index) in kh/kl/sidx) by a bucket
// sort: floor(d2 (nb - 1) / max d2) is monotone in d2, so buckets in index order hold
// increasing distances; each bucket is then put in exact key order by insertion (buckets
// hold a few survivors on average).  Writes the first M indices to out and returns true;
// returns false (nothing written) when a bucket holds more than BUCKET_CAP survivors
// (many equal distances), leaving the keys for the bitonic sort.  The bucket bounds use
// hist[0, nb); the permutation goes to perm (cnt entries), which may be hist + nb.
// Every thread returns after the same barriers.
template <int NT>
__device__ bool bucket_order(const uint32_t *kh, const uint32_t *kl, const int32_t *sidx, int cnt,
                             int M, uint32_t *hist, int nb, uint32_t *perm, uint32_t *warp_tmp,
                             uint32_t *sh_flag, unsigned long long *sh_dmax, int32_t *out) {
  uint32_t *bound = hist;
  if (threadIdx.x == 0) {
    *sh_dmax = 0ull;
    *sh_flag = 0u;
  }
  for (int b = threadIdx.x; b < nb; b += NT) bound[b] = 0;
  // the largest key (non-negative doubles order like their bits): a warp maximum, then one
  // shared atomic per warp
  unsigned long long wmax = 0ull;
  for (int r = threadIdx.x; r < cnt; r += NT) {
    const unsigned long long k = ((unsigned long long)kh[r] << 32) | kl[r];
    wmax = k > wmax ? k : wmax;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, wmax, o);
    wmax = w > wmax ? w : wmax;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0 && wmax) atomicMax(sh_dmax, wmax);
  __syncthreads();
  // buckets from FP32: float(d2) is non-decreasing in d2 and so is its product with a
  // positive scale and the truncation, so bucket order is distance order (equal floats
  // share a bucket, which the insertion below orders by the exact key)
  const float dmax = __double2float_ru(__longlong_as_double((long long)*sh_dmax));
  if (!(dmax > 0.0f)) return false;
  const float scale = (float)(nb - 1) / dmax;
  auto bucket_of = [&](int r) {
    const float d2 = __double2float_rn(
        __longlong_as_double((long long)(((unsigned long long)kh[r] << 32) | kl[r])));
    const int b = (int)(d2 * scale);
    return b < nb - 1 ? b : nb - 1;
  };
  for (int r = threadIdx.x; r < cnt; r += NT) atomicAdd(&bound[bucket_of(r)], 1u);
  __syncthreads();
  // exclusive scan of the counts (nb / NT buckets per thread), flagging an oversized bucket
  const int per = nb / NT;  // a power of two
  uint32_t part = 0;
  for (int k = 0; k < per; k++) {  // rotated start per thread: no bank conflicts
    const uint32_t c = bound[threadIdx.x * per + ((k + threadIdx.x) & (per - 1))];
    part += c;
    if (c > BUCKET_CAP) *sh_flag = 1u;
  }
  uint32_t total;
  uint32_t run = block_excl_scan<NT>(part, warp_tmp, &total);
  for (int k = 0; k < per; k++) {
    const uint32_t c = bound[threadIdx.x * per + k];
    bound[threadIdx.x * per + k] = run;
    run += c;
  }
  __syncthreads();
  if (*sh_flag) return false;
  // scatter: afterwards bound[b] is the end of bucket b (= the start of bucket b + 1)
  for (int r = threadIdx.x; r < cnt; r += NT) {
    const uint32_t at = atomicAdd(&bound[bucket_of(r)], 1u);
    if (LAGP_CHK(at, cnt, 3)) perm[at] = r;
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nb; b += NT) {
    const uint32_t lo = b ? bound[b - 1] : 0u, hi = bound[b];
    for (uint32_t i = lo + 1; i < hi; i++) {  // insertion by the exact key
      const uint32_t v = perm[i];
      uint32_t k = i;
      while (k > lo) {
        const uint32_t u = perm[k - 1];
        if (!key_less3(kh[v], kl[v], sidx[v], kh[u], kl[u], sidx[u])) break;
        perm[k] = u;
        k--;
      }
      perm[k] = v;
    }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < M; r += NT) {
    const uint32_t pr = perm[r];
    out[r] = LAGP_CHK(pr, cnt, 4) ? sidx[pr] : -1;
  }
  return true;
}

// P > 0: the dimension is a compile-time constant; P == 0: runtime p.
// Batched launches pass `list` (launch position -> location), `locs` (each location's
// candidate count and output offset) and the row stride of XX; uniform launches pass
// nullptr and use M, t*M and t*p.
template <int P, int NT>
__global__ void __launch_bounds__(NT, 4 * KB / NT) knn_kernel(const Scan S_, const double *__restrict__ X, int N, int p,
                                                 const double *__restrict__ XX, int64_t T, int M,
                                                 int32_t *__restrict__ cand,
                                                 const float *__restrict__ Xf,
                                                 const unsigned int *__restrict__ bmax, int cap,
                                                 const int32_t *__restrict__ list,
                                                 const LocDesc *__restrict__ locs, int ldxx) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t *kh = reinterpret_cast<uint32_t *>(smem);   // cap
  uint32_t *kl = kh + cap;                              // cap
  int32_t *sidx = reinterpret_cast<int32_t *>(kl + cap);  // cap
  uint32_t *hist = reinterpret_cast<uint32_t *>(sidx + cap);  // HBINS
  // the bucket sort's permutation: the histogram's second half, or its own cap entries
  const bool own_perm = knn_own_perm(cap);
  uint32_t *perm = own_perm ? hist + HBINS : hist + HBINS / 2;
  const int nb = own_perm ? HBINS : HBINS / 2;
  const int perm_cap = own_perm ? cap : HBINS / 2;
  __shared__ double xs[kMaxP];
  __shared__ float xf[kMaxP];
  __shared__ uint32_t warp_tmp[32];
  __shared__ int sh_bin;
  __shared__ uint32_t sh_below, sh_count;
  __shared__ uint32_t pref[12];
  __shared__ float sh_thr;
  __shared__ unsigned long long sh_dmax;
  if (P > 0) p = P;
  constexpr int S = P ? knn_row(P) : kMaxP;

  const double Bx = (double)__uint_as_float(*bmax);
  const int Mu = M;
  for (int64_t tt = blockIdx.x; tt < T; tt += gridDim.x) {
    const int64_t t = list ? list[S_.first + tt] : S_.first + tt;
    int32_t *out = cand + (locs ? locs[t].cand_off : t * Mu);
    M = locs ? locs[t].M : Mu;
    if (threadIdx.x < S) {
      const double x = threadIdx.x < p ? XX[t * (locs ? ldxx : p) + threadIdx.x] : 0.0;
      xs[threadIdx.x] = x;
      xf[threadIdx.x] = __double2float_rn(x);
    }
    for (int b = threadIdx.x; b < HBINS; b += NT) hist[b] = 0;
    if (threadIdx.x == 0) sh_count = 0;
    __syncthreads();
    // The screen's threshold thr = tau + 2E: tau the upper edge of the bin holding the M-th
    // smallest d2f in `hist` (complete up to that bin), E the FP32 error bound.
    auto set_threshold = [&]() {
      find_rank_bin<NT>(hist, HBINS, (uint32_t)M, warp_tmp, &sh_bin, &sh_below);
      if (threadIdx.x == 0) {
        double B = Bx;
        for (int k = 0; k < p; k++) B = fmax(B, fabs(xs[k]));
        const double tau = (double)__uint_as_float(((uint32_t)sh_bin + 1u) << (31 - HBITS));
        const double E0 = fp32_err_bound(tau, B, p);
        const double E = fp32_err_bound(tau + 2.0 * E0, B, p);
        sh_thr = __double2float_ru(tau + 2.0 * E);
      }
      __syncthreads();
    };
    int cnt = 0;
    bool listed = false;
    float bound = 0.0f;
    bool some = false;  // (d2f, index) of the points with d2f <= bound are listed
    const bool scanned = S_.cnt && S_.thr[tt] > -INFINITY;
    const uint32_t pre = scanned ? S_.cnt[tt] : 0u;
    if (pre >= (uint32_t)M && pre <= (uint32_t)S_.cap) {
      // the scan listed every point that can have d2f <= bound (and a few more)
      some = true;
      bound = S_.bound[tt];
      const int32_t *pl = S_.list + (size_t)tt * S_.cap;
      for (int r0 = threadIdx.x & ~31; r0 < (int)pre; r0 += KU * NT) {
        float d[KU];
        int id[KU];
#pragma unroll
        for (int u = 0; u < KU; u++) {
          const int r = r0 + u * NT + (threadIdx.x & 31);
          id[u] = r < (int)pre ? pl[r] : -1;
          if (id[u] >= 0 && !LAGP_CHK(id[u], N, 2)) id[u] = -1;
        }
#pragma unroll
        for (int u = 0; u < KU; u++) d[u] = id[u] >= 0 ? sqdist_f32<S>(xf, Xf, id[u]) : INFINITY;
#pragma unroll
        for (int u = 0; u < KU; u++) {  // warp-aggregated appends
          const bool keep = id[u] >= 0 && d[u] <= bound;
          const unsigned ball = __ballot_sync(0xffffffffu, keep);
          uint32_t base = 0;
          if ((threadIdx.x & 31) == 0 && ball) base = atomicAdd(&sh_count, (uint32_t)__popc(ball));
          base = __shfl_sync(0xffffffffu, base, 0);
          const uint32_t pos = base + __popc(ball & ((1u << (threadIdx.x & 31)) - 1u));
          if (keep) {
            if (pos < (uint32_t)cap) {
              kh[pos] = __float_as_uint(d[u]);
              kl[pos] = (uint32_t)id[u];
            }
            atomicAdd(&hist[__float_as_uint(d[u]) >> (31 - HBITS)], 1u);
          }
        }
      }
    }
    // (a scan that listed fewer than M has shown that the sample's bound missed: two full passes)
    const int ks = scanned && pre < (uint32_t)M ? 0 : sample_rank(N, M);
    if (!some && ks > 0) {
      some = true;
      bound = S_.cnt ? S_.bound[tt] : INFINITY;  // the kernel before the scan has it
      if (!(bound < INFINITY)) {
        bound = sample_bound<S, NT>(xf, Xf, N, ks, hist, warp_tmp, &sh_bin, &sh_below);
        for (int b = threadIdx.x; b < HBINS; b += NT) hist[b] = 0;
        __syncthreads();
      }
      // pass 1: the points with d2f <= bound are listed (d2f bits, index) and histogrammed;
      // the list's histogram is the whole design's in every bin up to the M-th's
      each_point<S>(xf, Xf, N, threadIdx.x, NT, [&](float d2f, int i) {
        if (d2f <= bound) {
          const uint32_t pos = atomicAdd(&sh_count, 1u);
          if (pos < (uint32_t)cap) {
            kh[pos] = __float_as_uint(d2f);
            kl[pos] = (uint32_t)i;
          }
          atomicAdd(&hist[__float_as_uint(d2f) >> (31 - HBITS)], 1u);
        }
      });
    }
    if (some) {
      __syncthreads();
      const uint32_t nl = sh_count;
      if (nl >= (uint32_t)M && nl <= (uint32_t)cap) {
        set_threshold();
        const float thr = sh_thr;
        if (thr <= bound) {  // every point with d2f <= thr is in the list: keep those
          listed = true;
          __syncthreads();
          if (threadIdx.x == 0) sh_count = 0;
          __syncthreads();
          // warp-aggregated appends: one shared atomic per warp and pass
          for (int r0 = threadIdx.x & ~31; r0 < (int)nl; r0 += NT) {
            const int r = r0 + (threadIdx.x & 31);
            const bool keep = r < (int)nl && __uint_as_float(kh[r]) <= thr;
            const unsigned ball = __ballot_sync(0xffffffffu, keep);
            uint32_t base = 0;
            if ((threadIdx.x & 31) == 0 && ball) base = atomicAdd(&sh_count, (uint32_t)__popc(ball));
            base = __shfl_sync(0xffffffffu, base, 0);
            const uint32_t at = base + __popc(ball & ((1u << (threadIdx.x & 31)) - 1u));
            if (keep && LAGP_CHK(at, cap, 1)) sidx[at] = (int32_t)kl[r];
          }
          __syncthreads();
          cnt = (int)sh_count;
        }
      }
      if (!listed) {  // the sample's bound missed (rare): the two full passes below
        __syncthreads();
        for (int b = threadIdx.x; b < HBINS; b += NT) hist[b] = 0;
        if (threadIdx.x == 0) sh_count = 0;
        __syncthreads();
      }
    }
    if (!listed) {
      // pass 1: histogram of the FP32 distances of every point
      each_point<S>(xf, Xf, N, threadIdx.x, NT, [&](float d2f, int) {
        atomicAdd(&hist[__float_as_uint(d2f) >> (31 - HBITS)], 1u);
      });
      __syncthreads();
      set_threshold();
      const float thr = sh_thr;
      // pass 2: the same FP32 distances again (bit for bit); survivors are listed first
      each_point<S>(xf, Xf, N, threadIdx.x, NT, [&](float d2f, int i) {
        if (d2f <= thr) {
          const uint32_t pos = atomicAdd(&sh_count, 1u);
          if (pos < (uint32_t)cap) sidx[pos] = i;
        }
      });
      __syncthreads();
      cnt = (int)sh_count;
    }
    // then get their exact FP64 distances from the compacted list: a warp instruction of
    // the FP64 pipe serves 32 survivors instead of the few a strided pass would hold
    if (cnt <= cap)
      for (int r = threadIdx.x; r < cnt; r += NT) {
        const int32_t i = sidx[r];
        if (LAGP_CHK(i, N, 2)) put_key(kh, kl, sidx, (uint32_t)r, sqdist_exact(xs, X + (size_t)i * p, p), i);
      }
    __syncthreads();
    if (cnt > cap || cnt < M)  // too many ties at the boundary (or, defensively, too few)
      cnt = knn_exact_location<NT>(X, N, p, M, xs, kh, kl, sidx, hist, cap, warp_tmp, &sh_bin,
                               &sh_below, &sh_count, pref);
    if (cnt > cap || cnt > perm_cap ||
        !bucket_order<NT>(kh, kl, sidx, cnt, M, hist, nb, perm, warp_tmp, &sh_count,
                                   &sh_dmax, out)) {
      int n2 = 1;
      while (n2 < cnt) n2 <<= 1;
      for (int i = cnt + threadIdx.x; i < n2; i += NT) {
        kh[i] = 0xffffffffu;
        kl[i] = 0xffffffffu;
        sidx[i] = 0x7fffffff;
      }
      __syncthreads();
      bitonic_sort<NT>(kh, kl, sidx, n2);
      for (int r = threadIdx.x; r < M; r += NT) {
        const int32_t v = sidx[r];
        out[r] = LAGP_CHK(v, N, 5) ? v : -1;
      }
    }
    __syncthreads();
  }
}

size_t knn_smem_bytes(int cap) {
  return (size_t)cap * (4 + 4 + 4) + HBINS * 4 + (knn_own_perm(cap) ? (size_t)cap * 4 : 0);
}

int knn_per_sm(size_t smem) {
  const int per_sm = (int)(200000 / (smem + 1024));  // leave room, at most 8 CTAs
  return per_sm < 1 ? 1 : per_sm > 8 ? 8 : per_sm;
}
int knn_grid(int64_t T, int num_sms, size_t smem) {
  const int64_t g = (int64_t)num_sms * knn_per_sm(smem);
  return (int)(T < g ? (T > 0 ? T : 1) : g);
}

}  // namespace

int knn_check_take(CheckRec *out) { return check_take_here(out); }

// The scan is three launches (bounds, scan, lists to candidates) instead of one, for designs
// large enough that pass 1 is most of a location's work.  GB300, whole search, per-location
// passes -> scan: N = 40000 as above, 100 locations of 500 among 100000 70 -> 58 us; N = 16384, 2-d,
// ncand = 1000: one location 35 -> 41 us, 100 44 -> 54, 3000 183 -> 194.
// The last condition: distances that the scan's precision separates, if the points fill a box.
static bool scan_pays(int64_t N, int32_t M, int p) {
  return N >= kScanMinN && N >= 8 * (int64_t)M && pow(1.5 * M / N, 2.0 / p) >= (p <= 4 ? 4e-4 : 3e-2);
}

// Launch kernel (a) over nloc locations of one design.  Uniform launches: list == nullptr,
// locs == nullptr, candidate count M.  Batched: the design's locations in list, their
// counts and offsets in locs (M is then the largest count, which sizes shared memory).
// A workspace without room for the scan takes the per-location passes.
int knn_launch_list(const double *X, int64_t N, int32_t p, const double *XX, int64_t nloc,
                    int32_t M, int32_t *cand, void *ws, size_t ws_bytes, cudaStream_t stream,
                    const int32_t *list, const LocDesc *locs, int ldxx, int ctas_per_sm) {
  if (nloc == 0) return LAGP_OK;
  DevInfo di;
  int st = dev_info(&di);
  if (st) return st;
  if (ws_bytes < knn_base_bytes(N)) return LAGP_ERR_INVALID_ARG;
  const int cap = knn_cap(M);
  const size_t smem = knn_smem_bytes(cap);
  if (smem > di.smem_optin) return LAGP_ERR_INVALID_ARG;
  // 512 threads where shared memory holds three CTAs per SM or fewer (10000 8-d locations, ncand =
  // 2000, two CTAs: 4.15 -> 3.46 ms without the scan, 2.49 -> 2.27 with it)
  const bool wide = knn_per_sm(smem) <= 3;
  const int threads = wide ? 2 * KB : KB;
  const void *fn, *bfn;
  switch (p) {
#define LAGP_KNN_CASE(P) \
  case P: fn = wide ? (const void *)knn_kernel<P, 2 * KB> : (const void *)knn_kernel<P, KB>; \
    bfn = (const void *)knn_bound_kernel<P>; break;
    LAGP_KNN_CASE(1)
    LAGP_KNN_CASE(2)
    LAGP_KNN_CASE(3)
    LAGP_KNN_CASE(4)
    LAGP_KNN_CASE(8)
#undef LAGP_KNN_CASE
    default: fn = wide ? (const void *)knn_kernel<0, 2 * KB> : (const void *)knn_kernel<0, KB>;
      bfn = (const void *)knn_bound_kernel<0>; break;
  }
  st = allow_smem(fn, di);
  if (st) return st;
  char *w = static_cast<char *>(ws);
  unsigned int *bmax = reinterpret_cast<unsigned int *>(w);
  float *Xf = reinterpret_cast<float *>(w + 256);
  cudaError_t e = cudaMemsetAsync(bmax, 0, sizeof(unsigned int), stream);
  if (e != cudaSuccess) return cuda_status(e);
  const int64_t n = N * knn_row(p);
  int pblocks = (int)((n + KB - 1) / KB);
  if (pblocks > 4 * di.num_sms) pblocks = 4 * di.num_sms;
  knn_prep_kernel<<<pblocks, KB, 0, stream>>>(X, N, p, Xf, bmax);
  g_launches.fetch_add(1);
  const int Ni = (int)N;
  // the scan's part of the workspace: its operands, then as many locations as there is room for
  // (a batch's is sized for its largest N, M and T)
  const size_t frag_off = knn_base_bytes(N), loc_off = frag_off + scan_frag_bytes(N);
  const int lcap = scan_cap(M);
  const int64_t wave = ws_bytes < loc_off + 256 ? 0 : scan_wave(ws_bytes - loc_off - 256, nloc, M);
  const bool scan = scan_pays(N, M, p) && wave > 0;
  const int64_t waves = scan ? ceil_div(nloc, wave) : 1;
  const int64_t share = ceil_div(ceil_div(nloc, waves), kScanLocs) * kScanLocs;  // <= wave
  for (int64_t first = 0; first < nloc; first += share) {
    int64_t cnt = waves == 1 || nloc - first < share ? nloc - first : share;
    Scan S;
    S.first = first;
    S.cnt = nullptr;
    if (scan) {
      S.cnt = reinterpret_cast<uint32_t *>(w + loc_off);
      S.bound = reinterpret_cast<float *>(S.cnt + wave);
      S.thr = S.bound + wave;
      S.xfrag = reinterpret_cast<uint32_t *>(S.thr + wave);
      S.list = reinterpret_cast<int32_t *>(w + loc_off + align_up((size_t)wave * 44, 256));
      S.frag = reinterpret_cast<uint4 *>(w + frag_off);
      S.cap = lcap;
      int c = (int)cnt, npad = (int)(ceil_div(cnt, kScanLocs) * kScanLocs);
      const int tiles = (int)ceil_div(N, 16);
      const int conv = first ? 0 : (int)std::min<int64_t>(ceil_div(16 * (int64_t)tiles, KB), 4 * di.num_sms);
      void *bargs[] = {(void *)&S, (void *)&Ni, (void *)&p, (void *)&XX, (void *)&c, (void *)&npad, (void *)&M,
                       (void *)&Xf, (void *)&bmax, (void *)&list, (void *)&locs, (void *)&ldxx};
      e = cudaLaunchKernel(bfn, dim3(npad + conv), dim3(KB), bargs, 0, stream);
      if (e != cudaSuccess) return cuda_status(e);
      // about 16 CTAs per SM, each over whole rounds of kScanTiles tiles, or a quarter of one
      // where that leaves SMs idle
      const int groups = npad / kScanLocs;
      const int round = groups * ceil_div(tiles, kScanTiles) < 4 * di.num_sms ? kScanTiles / 4 : kScanTiles;
      const int64_t parts = ceil_div((int64_t)16 * di.num_sms, groups);
      const int part = (int)(ceil_div(ceil_div(tiles, parts), round) * round);
      knn_scan_kernel<<<dim3(groups, (unsigned)ceil_div(tiles, part)), KB, 0, stream>>>(S, tiles, part);
      g_launches.fetch_add(2);
    }
    int grid = knn_grid(cnt, di.num_sms, smem);
    if (ctas_per_sm > 0) {
      const int64_t g2 = (int64_t)di.num_sms * ctas_per_sm;
      grid = (int)(cnt < g2 ? cnt : g2);
    }
    void *args[] = {(void *)&S, (void *)&X, (void *)&Ni, (void *)&p, (void *)&XX, (void *)&cnt, (void *)&M,
                    (void *)&cand, (void *)&Xf, (void *)&bmax, (void *)&cap, (void *)&list,
                    (void *)&locs, (void *)&ldxx};
    e = cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, smem, stream);
    if (e != cudaSuccess) return cuda_status(e);
    g_launches.fetch_add(1);
    if (waves == 1) break;
  }
  return cuda_status(cudaGetLastError());
}

int knn_launch(const double *X, int64_t N, int32_t p, const double *XX, int64_t T, int32_t ncand,
               int32_t *cand, void *ws, size_t ws_bytes, cudaStream_t stream) {
  return knn_launch_list(X, N, p, XX, T, ncand, cand, ws, ws_bytes, stream, nullptr, nullptr, p, 0);
}

}  // namespace lagp
