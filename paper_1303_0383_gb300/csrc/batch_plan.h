// batch_plan.h -- the host's plan of one batched call: its per-location tables, what they are
// sized from, and the identity of a graph captured from it.  Plain C++ (the tests compile it
// alone).
#pragma once

#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

namespace lagp {

struct BatchDesign {
  const double *X;  // N x p, device
  const double *Z;  // N, device
  int64_t N;
  int32_t p, n0;
  double theta, g;
};

struct LocDesc {
  int32_t design, n, M, pad;
  int64_t cand_off;  // offset of this location's candidate list
  int64_t idx_off;   // offset of this location's selected indices (in the idx output)
};

struct BatchLayout {
  size_t designs, locs, order, lists, cand, scratch, total;
  size_t knn_ws, sel_ws, sel_needed;
};

struct BatchPlan {
  std::vector<BatchDesign> designs;
  std::vector<LocDesc> locs;
  std::vector<int32_t> order, lists, list_off, list_cnt;
  int32_t nmax = 0, pmax = 0, Mmax = 0;
  std::vector<int32_t> Mmax_d;
  int64_t cand_total = 0, idx_total = 0, Nmax = 0;

  double gmin() const {  // the smallest nugget
    double g = designs.empty() ? 0.0 : designs[0].g;
    for (const auto &d : designs) g = std::min(g, d.g);
    return g;
  }
};

// One call's buffers and launch shape.
struct BatchCall {
  const void *workspace;
  size_t workspace_bytes;
  const double *XX;
  int32_t ldxx;
  int64_t T;
  int32_t method, precision;
  const void *mean, *s2, *var, *idx, *status;
  int knn_ctas, sel_ctas;
  unsigned long long context;  // the CUDA context's unique id
};

// Two calls may share a captured graph only if every launch would be made with the same
// arguments: the key holds each value that the launches of a batch are made from (pointers,
// counts, sizes that lay out the workspace and shared memory or choose a kernel).  What the
// kernels read from the tables, which are copied in before each replay, is not in it: n, the
// candidate count and the design of each location within the largest ones, theta, n0.
inline std::string batch_graph_key(const BatchPlan &P, const BatchLayout &L, const BatchCall &C) {
  std::string k;
  auto put = [&k](const auto &v) { k.append(reinterpret_cast<const char *>(&v), sizeof v); };
  put(C.workspace), put(C.workspace_bytes), put(C.XX), put(C.ldxx), put(C.T), put(C.method), put(C.precision);
  put(C.mean), put(C.s2), put(C.var), put(C.idx), put(C.status);
  put(C.knn_ctas), put(C.sel_ctas), put(C.context);
  put(P.nmax), put(P.pmax), put(P.Mmax), put(P.Nmax), put(P.cand_total), put(P.idx_total);
  put(P.gmin());  // chooses the FP64 form
  put(L.designs), put(L.locs), put(L.order), put(L.lists), put(L.cand), put(L.scratch), put(L.total);
  put(L.knn_ws), put(L.sel_ws), put(L.sel_needed);
  for (size_t d = 0; d < P.designs.size(); d++) {
    const BatchDesign &D = P.designs[d];
    put(D.X), put(D.Z), put(D.N), put(D.p);
    put(P.list_off[d]), put(P.list_cnt[d]), put(P.Mmax_d[d]);
  }
  return k;
}

}  // namespace lagp
