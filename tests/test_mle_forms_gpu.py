"""The MLE kernel's slots in the workspace (designs of 74 points and more): a workspace of one slot
per SM gives the same results, a smaller one is refused.  (Values against the oracle at these
sizes: test_mle_sizes_gpu.py.)"""
from __future__ import annotations

import numpy as np
import pytest

from paper_1303_0383_gb300 import lagp

pytestmark = pytest.mark.gpu


def _mle(X, Z, idx, nbytes=None):
    import torch
    T, n = idx.shape
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a)).cuda()
    th = torch.full((T,), 7.0, dtype=torch.float64, device="cuda")
    it, st = torch.full((T,), -1, dtype=torch.int32, device="cuda"), torch.full((T,), 9, dtype=torch.int8, device="cuda")
    ws = lagp.workspace(lagp.lagp_mle_workspace_bytes(T, n) if nbytes is None else nbytes)
    lagp.lagp_mle_dev(d(X), d(Z), d(idx), 0.5, 1e-2, 0.005, 50.0, th, it, st, ws=ws)
    return th.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()


@pytest.mark.parametrize("n", [74, 130])
def test_slots_in_a_smaller_workspace(n):
    import torch
    rng = np.random.default_rng(n)
    X = rng.random((600, 3))
    Z = np.sin(4 * X[:, 0]) + X.sum(1) + 0.1 * rng.standard_normal(600)
    T, sms = 1300, torch.cuda.get_device_properties(0).multi_processor_count
    idx = np.stack([rng.permutation(600)[:n] for _ in range(T)]).astype(np.int32)
    full = _mle(X, Z, idx)
    slot = -(-(3 * n * n + 12 * n) * 8 // 256) * 256
    small = _mle(X, Z, idx, 256 + sms * slot)
    for a, b in zip(full, small):
        assert np.array_equal(a, b)
    assert (full[2] == 0).all()
    with pytest.raises(lagp.LagpError):
        _mle(X, Z, idx, 256 + (sms - 1) * slot)
