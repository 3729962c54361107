"""The MLE kernel's storage at its edges: the packed triangle shorter than the coordinates (n <
15), even and odd n, the line between shared memory and the workspace's slots (n = 74), the
largest n.  Well-conditioned designs, the protocol of test_mle_gpu.py (needs a GPU)."""
from __future__ import annotations

from types import SimpleNamespace

import numpy as np
import pytest

import oracle
from tests.test_mle_gpu import THETA_RTOL, gpu_mle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(3, 1), (7, 8), (14, 8), (15, 8), (16, 3), (33, 2), (74, 4), (75, 4), (129, 4), (256, 8)])
def test_mle_sizes(n, p):
    rng = np.random.default_rng(100 * n + p)
    X = rng.random((600, p))
    w = SimpleNamespace(X=X, Z=np.sin(4 * X[:, 0]) + X.sum(1) + 0.1 * rng.standard_normal(600), g=1e-2)
    idx = np.stack([rng.permutation(600)[:n] for _ in range(5)]).astype(np.int32)
    th, it, st = gpu_mle(w, idx, 0.5, 0.005, 50.0)
    ref = oracle.mle_batch(w.X, w.Z, idx, 0.5, w.g, 0.005, 50.0)
    assert np.array_equal(st, ref["status"])
    ok = st == 0
    assert (np.abs(th - ref["theta"])[ok] <= THETA_RTOL * ref["theta"][ok]).all()
    assert np.abs(it.astype(int) - ref["iters"])[ok].max(initial=0) <= 1
