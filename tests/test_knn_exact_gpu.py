"""Kernel (a)'s exact path (FP32 distances that separate nothing: coordinates far from the
origin), with more locations than the launch has CTAs, so that every CTA takes several: the
candidate lists must equal a brute-force search's.  Sizes on both sides of the bucket sort's
own permutation (ncand = 1000, 1100) and of the scan (N = 32768)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1303_0383_gb300 import lagp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T,M", [(6000, 1500, 300), (6000, 1500, 1000), (9000, 700, 1100), (33000, 1300, 500)])
def test_exact_path_over_many_locations(N, T, M):
    import torch
    rng = np.random.default_rng(N + M)
    X, XX = (torch.as_tensor(5e5 + rng.random((k, 2))).cuda() for k in (N, T))
    cand = torch.full((T, M), -5, dtype=torch.int32, device="cuda")
    lagp.lagp_knn_dev(X, XX, M, cand, lagp.workspace(lagp.lagp_knn_workspace_bytes(N, T, M)))
    for a in range(0, T, 100):
        d2 = torch.zeros((len(XX[a:a + 100]), N), dtype=torch.float64, device="cuda")
        for k in range(2):
            t = XX[a:a + 100, k, None] - X[None, :, k]
            d2 = d2 + t * t
        ref = torch.sort(d2, dim=1, stable=True).indices[:, :M]
        assert torch.equal(cand[a:a + 100].long(), ref)
