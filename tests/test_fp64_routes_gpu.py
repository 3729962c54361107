"""The FP64 ALC designs by the fixed-point screen, and NN by the predictive kernel alone,
against the FP64 recursion (which the no-allocation entry point runs on the same inputs): every
decision of the screen that is not clear by its margin is taken in the recursion's own
arithmetic, and the predictive kernel makes the recursion's operations in its order, so
designs, statuses and values must be the same bit for bit.  Sizes at the edges of the screen's
instances (64, 128, 256 candidate pairs), of the predictive kernel's group form (n = 208) and
its teams (64 threads), odd candidate counts, no greedy step at all, and the options that
change the number format (wide spread, large and tiny nuggets).  And FP64 MSPE in a workspace
of fewer CTAs, whose results are the same."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1303_0383_gb300 import lagp

pytestmark = pytest.mark.gpu


def _both(N, p, T, n0, n, M, theta, g, method, seed, poison=None, spread=1.0):
    import torch
    rng = np.random.default_rng(seed)
    X = rng.random((N, p)) * spread
    Z = np.sin(3 * X[:, 0]) + X.sum(1)
    XX = rng.random((T, p)) * spread
    near = np.argsort(((XX[:, None] - X[None]) ** 2).sum(-1), axis=1, kind="stable")[:, :M]
    if poison is not None:
        X[near[0, M // 2], 0] = poison
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    X, Z, XX, cand = d(X), d(Z), d(XX), d(near.astype(np.int32))
    res = []
    for call in ("workspace", "noalloc"):
        o = dict(mean=torch.full((T,), 7.0, dtype=torch.float64, device="cuda"))
        o["s2"], o["var"] = torch.full_like(o["mean"], 7.0), torch.full_like(o["mean"], 7.0)
        o["idx"] = torch.full((T, n), -7, dtype=torch.int32, device="cuda")
        o["status"] = torch.full((T,), 9, dtype=torch.int8, device="cuda")
        a = (X, Z, XX, cand, n0, n, theta, g, method, "fp64", o["mean"], o["s2"], o["var"], o["idx"], o["status"])
        if call == "workspace":
            lagp.lagp_select_dev(*a, lagp.workspace(lagp.lagp_select_workspace_bytes(T, p, n, M, method)))
        else:
            code = lagp.lagp_select_dev_noalloc(*a)
            assert code == lagp.LAGP_OK, lagp.strerror(code)
        torch.cuda.synchronize()
        res.append({k: v.cpu().numpy() for k, v in o.items()})
    for k in res[0]:
        assert np.array_equal(res[0][k], res[1][k], equal_nan=k not in ("idx", "status")), k
    return res[0]


@pytest.mark.parametrize("N,p,T,n0,n,M", [
    (40, 1, 3, 3, 12, 16), (600, 2, 5, 6, 6, 255), (300, 2, 4, 6, 40, 256), (300, 2, 4, 6, 41, 257),
    (700, 3, 9, 5, 30, 511), (700, 3, 9, 5, 30, 512), (700, 8, 3, 7, 33, 513), (1200, 2, 2, 3, 20, 1025),
    (64, 2, 3, 4, 64, 64), (400, 2, 3, 6, 209, 301), (4200, 2, 1, 6, 12, 4097)])
def test_fp64_alc_sizes(N, p, T, n0, n, M):
    r = _both(N, p, T, n0, n, M, 0.3, 1e-5, "alc", 11 * M + n)
    assert (r["status"] == 0).all()


@pytest.mark.parametrize("theta,g,spread", [
    (0.5, 0.9, 1.0), (0.5, 3.0, 1.0), (0.5, 2.0 ** -30, 1.0), (0.5, 2.0 ** -31, 1.0), (1e-3, 1e-6, 1.0),
    (0.5, 1e-5, 40.0), (0.5, 1e-5, 3e3), (1e3, 1e-6, 1.0), (0.2, 1e-5, 1e-4)])
def test_fp64_alc_formats(theta, g, spread):
    _both(500, 2, 6, 5, 30, 300, theta, g, "alc", 5, spread=spread)


@pytest.mark.parametrize("poison", [np.inf, np.nan, 1e200])
def test_fp64_alc_values_out_of_range(poison):
    _both(500, 2, 4, 5, 20, 200, 0.3, 1e-5, "alc", 6, poison=poison)


@pytest.mark.parametrize("T,n,M", [(1, 3, 3), (700, 50, 60), (7, 64, 64), (310, 65, 70), (5, 208, 210),
                                   (5, 209, 210), (2, 256, 256)])
def test_nn_sizes(T, n, M):
    r = _both(max(300, M), 2, T, 3, n, M, 0.1, 1e-4, "nn", T + n)
    assert (r["status"] == 0).all()


def test_nn_failed_factorisation():
    r = _both(300, 2, 9, 3, 60, 60, 1e4, 0.0, "nn", 3)  # correlations of 1: no factor
    assert (r["status"] != 0).any()


def test_mspe_in_a_smaller_workspace():
    import torch
    T, n, M = 400, 20, 200
    rng = np.random.default_rng(8)
    X, XX = torch.as_tensor(rng.random((900, 2))).cuda(), torch.as_tensor(rng.random((T, 2))).cuda()
    Z = torch.sin(3 * X[:, 0]) + X.sum(1)
    cand = torch.argsort(((XX[:, None] - X[None]) ** 2).sum(-1), dim=1, stable=True)[:, :M].to(torch.int32).contiguous()
    full = lagp.lagp_select_workspace_bytes(T, 2, n, M, "mspe")
    res = []
    for nbytes in (full, full * 6 // 10):
        mean, s2 = (torch.full((T,), 7.0, dtype=torch.float64, device="cuda") for _ in range(2))
        idx = torch.full((T, n), -7, dtype=torch.int32, device="cuda")
        lagp.lagp_select_dev(X, Z, XX, cand, 6, n, 0.3, 1e-4, "mspe", "fp64", mean, s2, None, idx, None,
                             lagp.workspace(nbytes))
        res.append((mean, s2, idx))
    assert all(torch.equal(a, b) for a, b in zip(*res)) and bool(torch.isfinite(res[0][0]).all())
