"""FP64 ALC where many candidates' scores lie closer than the fixed-point screen's margin: small
lengthscales, near-duplicate points, points symmetric about x, large nuggets.  Whatever the screen
re-scores and whatever it leaves to the FP64 recursion, the results are that recursion's bit for
bit."""
from __future__ import annotations

import numpy as np
import pytest

from tests.test_fp64_handed_gpu import _both, _square

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta", [3e-2, 1e-2, 6e-3, 3e-3, 1e-3, 1e-4, 1e-5])
@pytest.mark.parametrize("n,M", [(50, 200), (30, 300)])
def test_small_lengthscales(theta, n, M):
    X, XX, _ = _square(T=16)
    _both(X, XX, 6, n, M, theta, 1e-6)


@pytest.mark.parametrize("g", [1e-9, 1e-6, 1e-3])
@pytest.mark.parametrize("apart", [0.0, 1e-12, 1e-9, 1e-6, 1e-4])
def test_near_duplicates(g, apart):
    X, XX, rng = _square(T=16)
    X[1000:] = X[:1000] + apart * rng.standard_normal((1000, 2))
    _both(X, XX, 6, 50, 201, 0.5, g)


@pytest.mark.parametrize("half", [0.0, 0.5])
@pytest.mark.parametrize("M", [81, 200, 600])
def test_symmetric_about_x(half, M):
    a = np.arange(45) / 16.0
    X = np.stack(np.meshgrid(a, a), -1).reshape(-1, 2)
    XX = X[np.random.default_rng(M).integers(0, len(X), 24)] + half / 16.0
    _both(X, XX, 5, 40, M, 0.5, 1e-5)


@pytest.mark.parametrize("g", [1.0, 1e3, 1e9, 1e12, 1e15, 1e18, 1e40, 1e300])
def test_large_nuggets(g):
    X, XX, _ = _square(T=8)
    _both(X, XX, 6, 40, 200, 0.5, g)


@pytest.mark.parametrize("spread", [1e2, 1e3, 1e5, 1e100, 1e160])
def test_wide_designs(spread):
    X, XX, _ = _square(T=8)
    _both(X * spread, XX * spread, 6, 40, 200, 0.5, 1e-6)
    _both(X * spread, XX * spread, 6, 40, 200, 0.5 * spread, 1e-6)
