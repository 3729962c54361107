"""FP64 ALC where the fixed-point screen does not resolve a location as FP64 does and leaves it to
the FP64 recursion: designs, statuses and values must be that recursion's bit for bit (the
no-allocation entry point runs it on the same inputs), in every entry point that screens --
uniform, one lengthscale per location, augmented, batched, with and without idx, in a workspace
of one CTA per SM."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1303_0383_gb300 import lagp

pytestmark = pytest.mark.gpu


def _square(N=2000, T=20, seed=1):
    rng = np.random.default_rng(seed)
    X, XX = rng.uniform(-2, 2, (N, 2)), rng.uniform(-1.9, 1.9, (T, 2))
    return X, XX, rng


def _cuda(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def _outs(T, n):
    import torch
    o = {k: torch.full((T,), 7.0, dtype=torch.float64, device="cuda") for k in ("mean", "s2", "var")}
    o["idx"] = torch.full((T, n), -7, dtype=torch.int32, device="cuda")
    o["status"] = torch.full((T,), 9, dtype=torch.int8, device="cuda")
    return o


def _same(a, b):
    for k in a:
        x, y = a[k].cpu().numpy(), b[k].cpu().numpy()
        assert np.array_equal(x, y, equal_nan=x.dtype.kind == "f"), k


def _both(X, XX, n0, n, M, theta, g, Z=None):
    cand = np.argsort(((XX[:, None] - X[None]) ** 2).sum(-1), axis=1, kind="stable")[:, :M].astype(np.int32)
    Z = np.sin(3 * X[:, 0]) + np.cos(X).sum(1) if Z is None else Z
    T, p = XX.shape
    a, b = _outs(T, n), _outs(T, n)
    args = (*(_cuda(v) for v in (X, Z, XX, cand)), n0, n, theta, g, "alc", "fp64")
    lagp.lagp_select_dev(*args, *a.values(), lagp.workspace(lagp.lagp_select_workspace_bytes(T, p, n, M, "alc")))
    code = lagp.lagp_select_dev_noalloc(*args, *b.values())
    assert code == lagp.LAGP_OK, lagp.strerror(code)
    _same(a, b)
    return a, args


@pytest.mark.parametrize("g,out", [(1e-9, 3e3), (1e-9, 3e4), (1e-6, 3e5), (1e-6, 1e6), (1e-6, 1e8), (1e-6, 1e9)])
def test_one_point_far_out(g, out):
    X, XX, _ = _square(200)
    X[7] = (out, 0.0)
    a, _ = _both(X, XX, 6, 50, 200, 0.5, g)
    assert bool((a["status"] == 0).all())


def test_other_entry_points():
    import torch
    X, XX, rng = _square(200)
    X[7] = (1e6, 0.0)
    a, args = _both(X, XX, 6, 50, 200, 0.5, 1e-6)
    Xd, Zd, XXd, cd = args[:4]
    T, full = 20, lagp.workspace(lagp.lagp_select_workspace_bytes(20, 2, 50, 200, "alc"))
    # no idx; a workspace of one CTA per SM at most
    o = _outs(T, 50)
    lagp.lagp_select_dev(*args, o["mean"], o["s2"], None, None, None, full)
    _same({k: o[k] for k in ("mean", "s2")}, {k: a[k] for k in ("mean", "s2")})
    # many locations, in workspaces of two CTAs per SM and less (the recursion's share shrinks too)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    many = 2 * sms + 90
    b, margs = _both(X, rng.uniform(-1.9, 1.9, (many, 2)), 6, 20, 200, 0.5, 1e-6)
    ask = lagp.lagp_select_workspace_bytes(many, 2, 20, 200, "alc")
    for share in (0.6, 0.45):
        o = _outs(many, 20)
        lagp.lagp_select_dev(*margs, *o.values(), lagp.workspace(int(ask * share)))
        _same(o, b)
    # one lengthscale per location
    th = torch.as_tensor(np.geomspace(1e-5, 10.0, T)).cuda()
    o = _outs(T, 50)
    lagp.lagp_select_theta_dev(*args[:6], th, 1e-6, "alc", "fp64", *o.values(), full)
    for t in range(T):
        u = _outs(1, 50)
        code = lagp.lagp_select_dev_noalloc(Xd, Zd, XXd[t:t + 1].contiguous(), cd[t:t + 1].contiguous(), 6, 50,
                                            float(th[t]), 1e-6, "alc", "fp64", *u.values())
        assert code == lagp.LAGP_OK
        _same({k: v[t:t + 1] for k, v in o.items()}, u)
    # augmented: from the first 10 points of the design
    o = _outs(T, 50)
    lagp.lagp_select_augment_dev(*args[:4], a["idx"][:, :10].contiguous(), 50, 0.5, 1e-6, "alc", "fp64",
                                 *o.values(), full)
    _same(o, a)
    # a batch of this design and a plain one
    X2, XX2, _ = _square(3000, 1, 5)
    D = [dict(X=Xd, Z=Zd, n0=6, theta=0.5, g=1e-6),
         dict(X=_cuda(X2), Z=_cuda(np.sin(X2).sum(1)), n0=5, theta=0.4, g=1e-5)]
    do = (np.arange(T) % 2).astype(np.int32)
    n, M = np.full(T, 50, np.int32), np.full(T, 200, np.int32)
    n[1::4] = 30
    bo = _outs(T, 50)
    bo["idx"] = torch.full((int(n.sum()),), -7, dtype=torch.int32, device="cuda")
    ws = lagp.workspace(lagp.lagp_predict_batch_workspace_bytes(D, do, n, M, "alc", "fp64"))
    lagp.lagp_predict_batch_dev(D, XXd, do, n, M, "alc", "fp64", bo["mean"], bo["s2"], bo["var"], bo["idx"],
                                bo["status"], 0, ws)
    for k in ("mean", "s2", "var", "status"):
        assert torch.equal(bo[k][0::2], a[k][0::2]), k
    off = np.concatenate([[0], np.cumsum(n)])
    for t in range(0, T, 2):
        assert torch.equal(bo["idx"][off[t]:off[t + 1]], a["idx"][t])
    assert bool((bo["status"] == 0).all())
