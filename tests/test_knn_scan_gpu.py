"""Kernel (a)'s tensor-core scan at its edges: the candidate lists are whole numbers in (exact
distance, index) order, so they must equal a brute-force search's, with the scan and without it
(a workspace of the per-location passes' size).  Each dimension's operand form (split up to 4,
padded rows), partial tiles of points and of locations, a location far outside the design (not
scanned), coordinates at extreme scales, and a design of equal distances."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1303_0383_gb300 import lagp

pytestmark = pytest.mark.gpu


def _check(X, XX, M):
    import torch
    d2 = np.zeros((len(XX), len(X)))
    for k in range(X.shape[1]):
        t = XX[:, k, None] - X[None, :, k]
        d2 = d2 + t * t
    ref = np.argsort(d2, axis=1, kind="stable")[:, :M]
    Xd, XXd = (torch.as_tensor(np.ascontiguousarray(a)).cuda() for a in (X, XX))
    base = 256 + -(-len(X) * 32 // 256) * 256
    full = lagp.lagp_knn_workspace_bytes(len(X), len(XX), M)
    assert full > base
    for nbytes in (full, base):
        cand = torch.full((len(XX), M), -5, dtype=torch.int32, device="cuda")
        lagp.lagp_knn_dev(Xd, XXd, M, cand, lagp.workspace(nbytes))
        assert np.array_equal(cand.cpu().numpy(), ref), nbytes


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("N,T,M,scale", [(32768, 1, 100, 1.0), (32769, 64, 900, 1e-5), (40015, 65, 2000, 1e7)])
def test_scan_equals_brute_force(p, N, T, M, scale):
    rng = np.random.default_rng(N + p)
    X, XX = rng.uniform(-1, 1, (N, p)) * scale, rng.uniform(-1, 1, (T, p)) * scale
    if T > 1:
        XX[0] = 50 * scale  # far outside
        XX[1] = X[7]
    _check(X, XX, M)


def test_scan_equal_distances():
    g = np.stack(np.meshgrid(np.arange(200.0), np.arange(200.0), indexing="ij"), -1).reshape(-1, 2)
    _check(g, np.array([[100.0, 100.0], [0.0, 0.0], [99.5, 3.5]]), 1200)
