"""Kernel (a) where the scan is launched but some or all locations are not scanned: coordinates
with an offset (distances below the operands' resolution), a column of another unit, clusters
narrower than the sample's bin, and a sample whose bound misses (neighbours that the sampled
blocks do not hold).  Rows of 8 floats also at every remainder of their passes' blocks.  The
lists must equal a brute-force search's."""
from __future__ import annotations

import numpy as np
import pytest

from tests.test_knn_scan_gpu import _check

pytestmark = pytest.mark.gpu


def _check_small(X, XX, M):
    import torch

    from paper_1303_0383_gb300 import lagp
    d2 = np.zeros((len(XX), len(X)))
    for k in range(X.shape[1]):
        t = XX[:, k, None] - X[None, :, k]
        d2 = d2 + t * t
    ref = np.argsort(d2, axis=1, kind="stable")[:, :M]
    cand = torch.full((len(XX), M), -5, dtype=torch.int32, device="cuda")
    lagp.lagp_knn_dev(*(torch.as_tensor(np.ascontiguousarray(a)).cuda() for a in (X, XX)), M, cand,
                      lagp.workspace(lagp.lagp_knn_workspace_bytes(len(X), len(XX), M)))
    assert np.array_equal(cand.cpu().numpy(), ref)


@pytest.mark.parametrize("p", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("offset", [3.0, 10.0, 1e3])
def test_offset_designs(p, offset):
    rng = np.random.default_rng(p + int(offset))
    _check(offset + rng.random((40000, p)), offset + rng.random((70, p)) * np.linspace(1, 3, 70)[:, None], 700)


def test_one_column_of_another_unit():
    rng = np.random.default_rng(2)
    s = np.array([0.1, 5e3, 5e4, 50, 100, 100, 500, 2e3])
    _check(s * rng.random((33000, 8)), s * rng.random((65, 8)), 500)


def test_clusters():
    rng = np.random.default_rng(3)
    X = rng.random((40, 2))[rng.integers(0, 40, 40000)] + 1e-3 * rng.standard_normal((40000, 2))
    _check(X, np.concatenate([X[:60] + 1e-4, rng.random((10, 2))]), 900)


def test_sample_misses():
    # the sample takes 32 points of every 512: here only those lie far away, so its bound is above
    # everything, and then only those lie near, so it is below the M-th
    rng = np.random.default_rng(4)
    near = (np.arange(40960) % 512) < 32
    for inside in (near, ~near):
        X = rng.random((40960, 2))
        X[inside] = 0.5 + 0.05 * (rng.random((inside.sum(), 2)) - 0.5)
        _check(X, 0.5 + 0.04 * (rng.random((66, 2)) - 0.5), 800)


@pytest.mark.parametrize("N", [1024, 1025, 1055, 1056, 3071, 3072, 4095, 8191, 8225])
@pytest.mark.parametrize("p", [5, 8])
def test_rows_of_eight(N, p):
    rng = np.random.default_rng(N + p)
    _check_small(rng.random((N, p)), rng.random((20, p)), 301)
