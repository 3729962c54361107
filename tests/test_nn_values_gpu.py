"""Kernel (c) where it stands in for the FP64 recursion (NN, FP64 ALC) takes every value as that
recursion's division does: infinite, huge and subnormal responses, correlations with x below the
normal range, and sizes on both sides of the line to the recursion (n = 208)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1303_0383_gb300 import lagp
from tests.test_fp64_handed_gpu import _cuda, _outs, _same

pytestmark = pytest.mark.gpu


def _check(X, Z, XX, n, M, theta, g, method):
    cand = np.argsort(((XX[:, None] - X[None]) ** 2).sum(-1), axis=1, kind="stable")[:, :M].astype(np.int32)
    T, p = XX.shape
    a, b = _outs(T, n), _outs(T, n)
    args = (*(_cuda(v) for v in (X, Z, XX, cand)), 6, n, theta, g, method, "fp64")
    lagp.lagp_select_dev(*args, *a.values(), lagp.workspace(lagp.lagp_select_workspace_bytes(T, p, n, M, method)))
    code = lagp.lagp_select_dev_noalloc(*args, *b.values())
    assert code == lagp.LAGP_OK, lagp.strerror(code)
    _same(a, b)


@pytest.mark.parametrize("method", ["nn", "alc"])
@pytest.mark.parametrize("z", [np.inf, -np.inf, np.nan, 1.7e308, -1.7e308, 1e300, 5e-324, 3e-310, 1e-290, 0.0])
def test_responses(method, z):
    rng = np.random.default_rng(3)
    X, XX = rng.uniform(-2, 2, (300, 2)), rng.uniform(-1.9, 1.9, (8, 2))
    Z = np.sin(3 * X[:, 0])
    Z[::40] = z
    _check(X, Z, XX, 30, 60, 0.5, 1e-6, method)
    _check(X, np.full(300, z), XX, 30, 60, 0.5, 1e-6, method)


@pytest.mark.parametrize("away", [15.0, 18.0, 18.7, 18.8, 18.9, 25.0])
@pytest.mark.parametrize("g", [1e-6, 1e6, 1e300])
def test_correlations_below_the_normal_range(away, g):
    rng = np.random.default_rng(4)
    X, XX = rng.uniform(-0.5, 0.5, (200, 2)), rng.uniform(-0.5, 0.5, (9, 2))
    _check(X, np.cos(X).sum(1), XX + [away, 0.0], 40, 60, 0.5, g, "nn")


@pytest.mark.parametrize("n", [207, 208, 209, 256])
def test_sizes_at_the_line(n):
    rng = np.random.default_rng(n)
    X, XX = rng.uniform(-2, 2, (400, 2)), rng.uniform(-1.9, 1.9, (5, 2))
    _check(X, np.cos(X).sum(1), XX, n, 300, 0.5, 1e-5, "nn")
