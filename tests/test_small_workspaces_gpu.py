"""Workspaces between what a call needs and what its query asks for (no room for the candidate
search's scan, or one CTA per SM): the whole path and the batch take them and give the same
results; what is too small for that is refused before anything is launched."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1303_0383_gb300 import lagp

pytestmark = pytest.mark.gpu

N, T, n, M = 100000, 300, 8, 300


def _problem():
    import torch
    rng = np.random.default_rng(1)
    X = torch.as_tensor(rng.random((N, 2))).cuda()
    return X, torch.sin(3 * X[:, 0]) + X[:, 1], torch.as_tensor(rng.random((T, 2))).cuda()


def _outs():
    import torch
    o = {k: torch.full((T,), 7.0, dtype=torch.float64, device="cuda") for k in ("mean", "s2", "var")}
    o["idx"] = torch.full((T, n), -7, dtype=torch.int32, device="cuda")
    o["status"] = torch.full((T,), 9, dtype=torch.int8, device="cuda")
    return o


@pytest.mark.parametrize("method,precision", [("alc", "mixed"), ("alc", "fp64"), ("mspe", "fp64"), ("mspe", "mixed"),
                                              ("nn", "fp64")])
def test_predict_without_room_for_the_scan(method, precision):
    import torch
    X, Z, XX = _problem()
    ask = lagp.lagp_predict_workspace_bytes(N, T, 2, n, M, method, precision)
    cand = -(-T * M * 4 // 256) * 256
    base = 256 + N * 32
    small = cand + max(base, lagp.lagp_select_workspace_bytes(T, 2, n, M, method, precision))
    assert small < ask or method == "mspe"
    res = []
    for nbytes in (ask, small):
        o = _outs()
        lagp.lagp_predict_dev(X, Z, XX, 4, n, M, 0.1, 1e-5, method, precision, *o.values(), lagp.workspace(nbytes))
        res.append(o)
    for k in res[0]:
        assert torch.equal(res[0][k], res[1][k]), k
    with pytest.raises(lagp.LagpError):
        lagp.lagp_predict_dev(X, Z, XX, 4, n, M, 0.1, 1e-5, method, precision, *_outs().values(),
                              lagp.workspace(cand + base - 256))


@pytest.mark.parametrize("method,precision", [("alc", "mixed"), ("alc", "fp64"), ("mspe", "fp64"), ("nn", "fp64")])
def test_batch_in_less_than_asked(method, precision):
    import torch
    X, Z, XX = _problem()
    D = [dict(X=X, Z=Z, n0=4, theta=0.1, g=1e-5), dict(X=X[:50000], Z=Z[:50000], n0=3, theta=0.2, g=1e-6)]
    do, nn, mm = (np.arange(T) % 2).astype(np.int32), np.full(T, n, np.int32), np.full(T, M, np.int32)
    mm[::3] = 120
    ask = lagp.lagp_predict_batch_workspace_bytes(D, do, nn, mm, method, precision)
    tables = -(-2 * 56 // 256) * 256 + T * 64 + int(mm.sum()) * 4  # designs, per-location tables, lists: at most
    res = []
    for nbytes in (ask, tables + 4096 + max(256 + N * 32, (ask - tables) * 7 // 10)):
        o = _outs()
        lagp.lagp_predict_batch_dev(D, XX, do, nn, mm, method, precision, o["mean"], o["s2"], o["var"],
                                    o["idx"].view(-1), o["status"], 0, lagp.workspace(nbytes))
        res.append(o)
    for k in res[0]:
        assert torch.equal(res[0][k], res[1][k]), k
    with pytest.raises(lagp.LagpError):
        lagp.lagp_predict_batch_dev(D, XX, do, nn, mm, method, precision, o["mean"], o["s2"], o["var"],
                                    o["idx"].view(-1), o["status"], 0, lagp.workspace(N * 32))
