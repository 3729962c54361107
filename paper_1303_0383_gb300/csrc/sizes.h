// sizes.h -- launch shapes and workspace layouts of the ALC candidate screen (select_mixed.cu)
// and of the candidate search's scan (knn.cu): plain host arithmetic, which the tests compile
// alone.
//
// A workspace query has to grow with every size that it is asked for: a program that takes one
// workspace for its largest problem (the server's slots) also runs smaller ones in it.  The
// shapes do not grow by themselves -- a location of more candidates gets a larger share of an
// SM, so fewer are in flight -- so the queries take the largest over all shapes of sizes up to
// the one asked for.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace lagp {

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// ---- the ALC candidate screen

constexpr int kScrThreads = 512;  // threads per SM: CTAs of 128, 256 or 512 threads, 128 registers each
constexpr int kMaxCL = 8;         // CTAs per cluster in the cluster form

// Candidate pairs of one CTA slot: M candidates over CL CTAs, padded to 32 pairs (so the
// shared-memory rows after the Mpad = 2 Qpad flag bytes start 16-byte aligned).
inline int mix_qpad(int M, int CL) { return (int)align_up((size_t)ceil_div(ceil_div(M, 2), CL), 32); }

struct ScreenChip {
  int num_sms;
  size_t l2, on_chip;  // bytes of L2, and of shared and tensor memory per SM
};

// Threads per CTA for T locations of M candidates and n points: one or two candidate pairs per
// thread, 512 threads per SM in all.  Small CTAs leave fewer threads idle and hide each other's
// barriers; large ones have a location to themselves sooner and keep fewer factor rows live.  So
// CTAs of 128 and 256 threads are taken for up to 512 and 1024 candidates, and for half as many again
// where more than two locations per SM are asked for and the rows and coordinates of those in
// flight stay within nine tenths of L2 and the chip; with two per SM or fewer, 256 threads from 257
// candidates on.  GB300, mixed, 2000 2-d
// locations, n = 50, in ms for 128 / 256 / 512 threads: M = 400 1.50 / 1.79 / 2.51, 600 2.21 / 2.26 /
// 3.17, 700 2.25 / 2.53 / 3.22, 1024 3.04 / 2.73 / 3.44, 1100 4.36 / 3.64 / 4.19, 1300 5.07 / 4.06 / 4.39,
// 1500 5.72 / 4.72 / 4.42; 300 locations, M = 400 0.44 / 0.40 / 0.44; one, 0.27 / 0.24 / 0.24, M = 1100
// 0.63 / 0.46 / 0.36; 600 8-d ones, n = 100: M = 300 1.67 / 2.08 / 2.48, 500 2.86 / 2.13 / 2.72, 1030 6.54 /
// 5.67 / 4.23 (rows beyond L2); n = 60, M = 700 1.52 / 1.31 (just beyond the line).  kMixTop: the largest M of the first two.
constexpr int kMixTop[2] = {768, 1344};
inline int mix_threads(int64_t T, int M, int n, int p, const ScreenChip &c) {
  const int Qpad = mix_qpad(M, 1);
  const bool many = T > 2 * (int64_t)c.num_sms;
  const double room = 0.9 * ((double)c.l2 + (double)c.num_sms * c.on_chip);
  auto fits = [&](int k) { return 16.0 * k * c.num_sms * (n + p) * Qpad <= room; };  // k locations per SM
  if (Qpad <= 128 || (many && 2 * Qpad <= kMixTop[0] && fits(4))) return 128;
  if (2 * Qpad <= 1024 || (many && 2 * Qpad <= kMixTop[1] && fits(2))) return 256;
  return 512;
}

struct MixLayout {
  size_t list, u, xr, a, idx, pred, total;
};

// [counters, 512 bytes | list | U | Xr | A | design indices | kernel (c) workspace] of G CTAs, each
// with a slot of n x Qpad factor rows and p x Qpad coordinates (16 bytes per pair) and of the
// n x (n + 2) FP64 factorisation; pred: kernel (c)'s bytes.  listed: the locations that the list
// of those left to the FP64 recursion has room for (FP64: all of them; mixed: 0).  The recursion
// runs last, in all that follows the list.
inline MixLayout mix_layout(int64_t G, int p, int n, int Qpad, int64_t idx_total, size_t pred, int64_t listed) {
  MixLayout L;
  // (512: a warp reads 512 bytes of a row; rows that lie across such blocks stream 3 % slower)
  L.list = align_up((size_t)listed * sizeof(int32_t), 512);
  L.u = align_up((size_t)G * n * Qpad * 16, 256);
  L.xr = align_up((size_t)G * p * Qpad * 16, 256);
  L.a = align_up((size_t)G * n * (n + 2) * sizeof(double), 256);
  L.idx = align_up((size_t)idx_total * sizeof(int32_t), 256);
  L.pred = pred;
  L.total = 512 + L.list + L.u + L.xr + L.a + L.idx + L.pred;
  return L;
}

// Scratch of the FP64 recursion's slots (select.cu): n x Mpad factor rows and p x Mpad coordinates.
inline size_t rec_slots_bytes(int64_t G, int p, int n, int M) {
  const size_t Mpad = align_up((size_t)M, 32);
  return align_up((size_t)G * (size_t)n * Mpad * sizeof(double), 256) +
         align_up((size_t)G * (size_t)p * Mpad * sizeof(double), 256);
}
// CTAs of the recursion for T locations: two per SM.
inline int64_t rec_grid(int64_t T, int num_sms) { return std::min<int64_t>(2 * (int64_t)num_sms, T > 0 ? T : 1); }
// Of those, as many as fit in `bytes`.
inline int64_t rec_fit(int64_t T, size_t bytes, int p, int n, int M, int num_sms) {
  return std::min<int64_t>(rec_grid(T, num_sms), (int64_t)(bytes / rec_slots_bytes(1, p, n, M)));
}

// What a workspace query returns: enough for the full grid of every shape, for T locations of at
// most M candidates and n points.
inline size_t mix_asked_bytes(int64_t T, int p, int n, int M, int64_t idx_total, size_t pred, int num_sms,
                              bool clusters, int64_t listed) {
  const int64_t T1 = T > 0 ? T : 1;
  size_t most = 0;
  for (int k = 0; k < 3; k++) {  // 128, 256 and 512 threads
    const int Mk = k < 2 ? std::min(M, kMixTop[k]) : M;
    const int64_t G = std::min<int64_t>((int64_t)num_sms * (4 >> k), T1);
    most = std::max(most, mix_layout(G, p, n, mix_qpad(Mk, 1), idx_total, pred, listed).total);
  }
  for (int CL = 2; clusters && CL <= kMaxCL; CL *= 2) {
    const int64_t G = std::min<int64_t>((int64_t)num_sms * (kScrThreads / 256), CL * T1);
    most = std::max(most, mix_layout(G, p, n, mix_qpad(M, CL), idx_total, pred, listed).total);
  }
  if (listed)
    most = std::max(most, 512 + mix_layout(0, p, n, 0, 0, 0, listed).list + rec_slots_bytes(rec_grid(T, num_sms), p, n, M));
  return most;
}

// The largest grid of at most G CTAs that fits in `bytes`; 0 where not even one CTA per SM (or
// G, if that is fewer) does.
inline int mix_fit(int64_t G, size_t bytes, int p, int n, int Qpad, int64_t idx_total, size_t pred, int num_sms,
                   int64_t listed) {
  const int64_t least = std::min<int64_t>(G, num_sms);
  if (mix_layout(least, p, n, Qpad, idx_total, pred, listed).total > bytes) return 0;
  while (mix_layout(G, p, n, Qpad, idx_total, pred, listed).total > bytes) {
    const MixLayout L = mix_layout(G, p, n, Qpad, idx_total, pred, listed);
    const size_t slot = (L.u + L.xr + L.a) / (size_t)G;  // at most 768 / G above a slot's own bytes
    const int64_t over = (int64_t)((L.total - bytes) / (slot + 1)) + 1;
    G = std::max(least, G - over);
  }
  return (int)G;
}

// ---- the candidate search

// Entries of a location's lists in shared memory (knn.cu).
inline int knn_cap(int M) {
  int cap = 2048;
  while (cap < 2 * M && cap < 16384) cap <<= 1;
  return cap;
}

// Scratch layout: [bmax (256 B)] [Xf: N rows of up to 8 floats], then, for the scan, the design's
// operands and a wave of locations: [counts, bounds, thresholds, operands, lists].
constexpr size_t kScanListBytes = 128u << 20;
constexpr int kScanLocs = 64;      // locations of a CTA of the scan
constexpr int kScanMinN = 32768;   // smallest design that is scanned

inline size_t knn_base_bytes(int64_t N) { return 256 + align_up((size_t)N * 8 * sizeof(float), 256); }
inline int scan_cap(int M) { return knn_cap(M) + knn_cap(M) / 2; }  // list entries per location
inline size_t scan_loc_bytes(int cap) { return 44 + (size_t)cap * sizeof(int32_t); }
inline size_t scan_frag_bytes(int64_t N) { return align_up((size_t)ceil_div(N, 16) * 512, 256); }

// Bytes of the locations of a wave at most: all T, or what kScanListBytes (lists beyond L2 are
// read back from DRAM) or 512 locations hold.
inline size_t scan_wave_bytes(int64_t T, int M) {
  const size_t per = scan_loc_bytes(scan_cap(M));
  return std::min((size_t)(ceil_div(T, kScanLocs) * kScanLocs) * per, std::max(kScanListBytes, 512 * per));
}
// Locations of a wave in `bytes`, a multiple of kScanLocs.
inline int64_t scan_wave(size_t bytes, int64_t T, int M) {
  return (int64_t)(std::min(bytes, scan_wave_bytes(T, M)) / scan_loc_bytes(scan_cap(M))) / kScanLocs * kScanLocs;
}

inline size_t knn_asked_bytes(int64_t N, int64_t T, int M) {
  const size_t base = knn_base_bytes(N);
  return N >= kScanMinN && T > 0 ? base + scan_frag_bytes(N) + 256 + scan_wave_bytes(T, M) : base;
}

}  // namespace lagp
