"""When two batched calls may share a captured graph (csrc/batch_plan.h, compiled on the host):
every value that a launch is made from changes the key, and values that the kernels read from
the tables copied in before a replay do not.  On the GPU: calls with the same T and buffers but
other splits and sizes equal the same calls without a graph."""
from __future__ import annotations

import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "batch_plan.h"
#include <cstdio>
#include <functional>
using namespace lagp;
struct All { BatchPlan P; BatchLayout L; BatchCall C; };
static All base() {
  All a;
  a.P.designs = {BatchDesign{(double *)8, (double *)16, 100, 2, 4, 0.5, 1e-6},
                 BatchDesign{(double *)24, (double *)32, 200, 3, 5, 0.7, 1e-5}};
  a.P.locs = {LocDesc{0, 10, 20, 0, 0, 0}, LocDesc{1, 30, 40, 0, 20, 10}};
  a.P.order = {1, 0}, a.P.lists = {0, 1}, a.P.list_off = {0, 1, 2}, a.P.list_cnt = {1, 1};
  a.P.nmax = 30, a.P.pmax = 3, a.P.Mmax = 40, a.P.Mmax_d = {20, 40};
  a.P.cand_total = 60, a.P.idx_total = 40, a.P.Nmax = 200;
  a.L = BatchLayout{0, 256, 512, 768, 1024, 1280, 4096, 100, 200};
  memset(&a.C, 0, sizeof a.C);
  a.C.workspace = (void *)64, a.C.workspace_bytes = 4096, a.C.XX = (double *)72, a.C.ldxx = 8, a.C.T = 2;
  a.C.precision = 1, a.C.mean = (void *)80, a.C.s2 = (void *)88, a.C.var = (void *)96, a.C.idx = (void *)104;
  a.C.status = (void *)112, a.C.knn_ctas = 2, a.C.sel_ctas = 3, a.C.context = 7;
  return a;
}
static std::string key(const All &a) { return batch_graph_key(a.P, a.L, a.C); }
int main() {
  const std::string k0 = key(base());
  std::function<void(All &)> other[] = {
    [](All &a) { a.P.nmax = 31; }, [](All &a) { a.P.pmax = 4; }, [](All &a) { a.P.Mmax = 41; },
    [](All &a) { a.P.Nmax++; }, [](All &a) { a.P.cand_total++; }, [](All &a) { a.P.idx_total++; },
    [](All &a) { a.P.designs[0].g = 1e-12; }, [](All &a) { a.P.designs[1].X += 8; },
    [](All &a) { a.P.designs[1].Z += 8; }, [](All &a) { a.P.designs[0].N++; }, [](All &a) { a.P.designs[0].p = 1; },
    [](All &a) { a.P.list_cnt = {2, 0}; }, [](All &a) { a.P.list_off[1] = 2; }, [](All &a) { a.P.Mmax_d[0]++; },
    [](All &a) { a.P.designs.pop_back(); },
    [](All &a) { a.L.scratch += 256; }, [](All &a) { a.L.cand += 256; }, [](All &a) { a.L.total++; },
    [](All &a) { a.L.knn_ws++; }, [](All &a) { a.L.sel_ws++; }, [](All &a) { a.L.locs++; },
    [](All &a) { a.L.order++; }, [](All &a) { a.L.lists++; },
    [](All &a) { a.C.workspace = (void *)65; }, [](All &a) { a.C.workspace_bytes++; }, [](All &a) { a.C.XX += 8; },
    [](All &a) { a.C.ldxx++; }, [](All &a) { a.C.T++; }, [](All &a) { a.C.method++; }, [](All &a) { a.C.precision = 0; },
    [](All &a) { a.C.mean = 0; }, [](All &a) { a.C.s2 = 0; }, [](All &a) { a.C.var = 0; }, [](All &a) { a.C.idx = 0; },
    [](All &a) { a.C.status = 0; }, [](All &a) { a.C.knn_ctas++; }, [](All &a) { a.C.sel_ctas--; },
    [](All &a) { a.C.context++; }};
  int i = 0;
  for (auto &f : other) {
    All a = base();
    f(a);
    if (key(a) == k0) { printf("change %d is not in the key\n", i); return 1; }
    i++;
  }
  All a = base();  // tables: the same launches
  a.P.locs[0].n = 12, a.P.locs[1].n = 28, a.P.order = {0, 1}, a.P.designs[0].theta = 0.6, a.P.designs[0].n0 = 5;
  return key(a) == k0 ? 0 : 2;
}
"""


def test_key_holds_what_the_launches_are_made_from(tmp_path):
    src = tmp_path / "key.cpp"
    src.write_text(SRC)
    exe = tmp_path / "key"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1303_0383_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("method,precision", [("alc", "mixed"), ("alc", "fp64"), ("nn", "fp64")])
def test_same_buffers_other_sizes(method, precision):
    import torch

    from paper_1303_0383_gb300 import lagp
    from tests.test_batch_gpu import make_batch, run_batch
    ws, design_of, n, M, XX = make_batch(seed=50, T=40)
    _, designs, out, XXd, wsbuf = run_batch(ws, design_of, n, M, XX, method, precision, lagp.LAGP_BATCH_GRAPH)
    rng = np.random.default_rng(1)
    for step in range(4):
        # within the first call's sizes: other splits over the designs, sums and largest sizes
        d2 = rng.integers(0, 3, size=40).astype(np.int32) if step % 2 else rng.permutation(design_of)
        n2 = np.maximum(rng.permutation(n) - step, 5).astype(np.int32)
        M2 = np.maximum(rng.permutation(M) - step, n2).astype(np.int32)
        n2[n2 > n.max()], M2[M2 > M.max()] = n.max(), M.max()
        if n2.sum() > n.sum() or M2.sum() > M.sum():
            n2, M2 = n.copy(), M.copy()
        got = {k: torch.full_like(v, 7) for k, v in out.items()}
        for k in out:
            out[k].copy_(got[k])
        lagp.lagp_predict_batch_dev(designs, XXd, d2, n2, M2, method, precision, out["mean"], out["s2"], out["var"],
                                    out["idx"], out["status"], lagp.LAGP_BATCH_GRAPH, wsbuf)
        lagp.lagp_predict_batch_dev(designs, XXd, d2, n2, M2, method, precision, got["mean"], got["s2"], got["var"],
                                    got["idx"], got["status"], 0, torch.empty_like(wsbuf))
        torch.cuda.synchronize()
        for k in out:
            assert torch.equal(out[k], got[k]), (step, k)
        assert bool((out["status"] == 0).all())
