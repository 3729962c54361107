"""Workspace queries (csrc/sizes.h, compiled on the host) grow with every size, so that one
taken for the largest problem holds every smaller one, and a launch that is given a workspace
asked for at larger sizes fits its whole grid in it.  On the GPU: a server takes its largest
batches at candidate counts below the one its slots are sized for."""
from __future__ import annotations

import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "sizes.h"
#include <cstdio>
using namespace lagp;
static int bad(const char *what, long a, long b, long c) { printf("%s %ld %ld %ld\n", what, a, b, c); return 1; }
int main() {
  const int sms = 152;
  const ScreenChip chip{sms, 132120576, 495616};
  const int Ms[] = {3, 64, 200, 256, 257, 500, 511, 512, 513, 600, 767, 768, 769, 800, 1000, 1023, 1024, 1025, 1100, 1343, 1344, 1345,
                    1500, 2000, 2047, 2048, 2049, 3000, 4096, 4097, 6000, 8192};
  const int ns[] = {3, 20, 50, 73, 100, 208, 209, 256};
  const long Ts[] = {1, 2, 63, 64, 65, 151, 152, 153, 304, 305, 608, 609, 3000, 4096, 10000, 100000};
  for (int n : ns)
    for (long T : Ts)
      for (int c = 0; c < 2; c++) {
        size_t prev = 0;
        for (int M : Ms) {
          if (M < n) continue;
          const size_t a = mix_asked_bytes(T, 8, n, M, T * n, 256, sms, c, 0);
          if (a < prev) return bad("mix M", T, n, M);
          prev = a;
          // the grid of the shape that runs, whole, in what was asked for at this or any larger size
          const int64_t G = std::min<int64_t>((int64_t)sms * (kScrThreads / mix_threads(T, M, n, 8, chip)), T);
          if (mix_fit(G, a, 8, n, mix_qpad(M, 1), T * n, 256, sms, 0) != G) return bad("mix fit", T, n, M);
          if (mix_asked_bytes(T + 1, 8, n, M, (T + 1) * n, 256, sms, c, 0) < a) return bad("mix T", T, n, M);
          if (n < 256 && M > n && mix_asked_bytes(T, 8, n + 1, M, T * (n + 1), 256, sms, c, 0) < a) return bad("mix n", T, n, M);
          // and less of it in less, down to one CTA per SM
          const int64_t least = std::min<int64_t>(G, sms);
          const size_t small = mix_layout(least, 8, n, mix_qpad(M, 1), T * n, 256, 0).total;
          if (mix_fit(G, small, 8, n, mix_qpad(M, 1), T * n, 256, sms, 0) != least) return bad("mix least", T, n, M);
          if (mix_fit(G, small - 1, 8, n, mix_qpad(M, 1), T * n, 256, sms, 0)) return bad("mix refused", T, n, M);
          if (G > least) {
            const size_t mid = mix_layout(G - 1, 8, n, mix_qpad(M, 1), T * n, 256, 0).total;
            const int g = mix_fit(G, mid, 8, n, mix_qpad(M, 1), T * n, 256, sms, 0);
            if (g < G - 3 || mix_layout(g, 8, n, mix_qpad(M, 1), T * n, 256, 0).total > mid) return bad("mix mid", T, n, M);
          }
        }
      }
  for (long N : {1L, 32767L, 32768L, 40001L, 2000000L})
    for (long T : Ts) {
      size_t prev = 0;
      for (int M : Ms) {
        const size_t a = knn_asked_bytes(N, T, M);
        if (a < prev) return bad("knn M", N, T, M);
        prev = a;
        if (knn_asked_bytes(N, T + 1, M) < a || knn_asked_bytes(N + 1, T, M) < a) return bad("knn N T", N, T, M);
        if (N >= kScanMinN) {
          const size_t room = a - knn_base_bytes(N) - scan_frag_bytes(N) - 256;
          const long w = scan_wave(room, T, M);
          if (w < std::min(T, 448L) || w * (long)scan_loc_bytes(scan_cap(M)) > (long)room) return bad("wave", N, T, M);
        }
      }
    }
  return 0;
}
"""


def test_queries_grow_with_every_size(tmp_path):
    src = tmp_path / "sizes.cpp"
    src.write_text(SRC)
    exe = tmp_path / "sizes"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1303_0383_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("nmax,ncand_max,below", [(128, 1100, (1024, 512)), (64, 800, (512,)), (64, 1500, (1000,))])
def test_server_takes_full_batches_below_its_largest_count(precision, nmax, ncand_max, below):
    import torch

    from paper_1303_0383_gb300 import lagp
    rng = np.random.default_rng(nmax + ncand_max)
    X = rng.random((30000, 2))
    Z = np.sin(3 * X[:, 0]) + X[:, 1]
    Xd, Zd = torch.as_tensor(X).cuda(), torch.as_tensor(Z).cuda()
    srv = lagp.Server([dict(X=Xd, Z=Zd, n0=6, theta=0.3, g=1e-5)], "alc", precision, nmax=nmax,
                      ncand_max=ncand_max, max_batch=4096, memory_budget=4 << 30, max_slots=1)
    try:
        x = rng.random((4096, 2))
        for M in below:
            rid = srv.submit(0, x, nmax, M)
            assert srv.wait(rid, 60000)
            r = srv.results(rid)
            assert (r["status"] == 0).all()
            u = lagp.predict_torch(Xd, Zd, torch.as_tensor(x[:50]).cuda(), 6, nmax, M, 0.3, 1e-5, "alc", precision)
            assert np.array_equal(u["idx"].cpu().numpy(), r["idx"][:50])
        assert srv.stats()["last_error"] == 0
    finally:
        srv.close()
