"""FP64 ALC at locations far from their candidates (cov^2 leaves FP64's normal range, and the FP64
recursion's scores tie at 0), and with covariances that outgrow the fixed-point format (x outside
the design): the recursion's results bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from tests.test_fp64_handed_gpu import _both, _square

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("away", [2, 5, 8, 10, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 22, 30])
@pytest.mark.parametrize("g", [1e-9, 1e-6])
def test_far_from_the_design(away, g):
    X, XX, _ = _square(T=12)
    XX[0::2, 0] += away
    XX[1::2] -= away / np.sqrt(2)
    _both(X, XX, 6, 50, 200, 0.5, g)


@pytest.mark.parametrize("n0", [6, 40])
def test_far_without_greedy_steps(n0):
    X, XX, _ = _square(T=5)
    _both(X, XX + [19.0, 0.0], n0, 40, 100, 0.5, 1e-6)
