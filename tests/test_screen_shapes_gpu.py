"""The ALC screen's launch shapes on both sides of every line between them (64, 384, 512, 672, 1024
candidate pairs; more and fewer than two locations per SM; rows within L2 and beyond; a last round
of up to 64 pairs): a location's results do not depend on its launch, so each call's equal those of
the same locations one by one, whose shape differs."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1303_0383_gb300 import lagp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("M,n", [(256, 20), (257, 20), (512, 20), (700, 20), (768, 20), (769, 20), (1024, 20), (1025, 20),
                                 (1344, 20), (1345, 20), (512, 110), (1030, 110), (2048, 20), (2049, 20), (2113, 30),
                                 (2200, 20)])
def test_shapes(M, n, precision):
    import torch
    rng = np.random.default_rng(M + n)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    X = torch.as_tensor(rng.uniform(-2, 2, (5000, 2))).cuda()
    Z = torch.sin(3 * X[:, 0]) + X[:, 1]
    T = 2 * sms + 40
    XX = torch.as_tensor(rng.uniform(-1.9, 1.9, (T, 2))).cuda()
    a = lagp.predict_torch(X, Z, XX, 6, n, M, 0.5, 1e-5, "alc", precision)
    for lo, hi in ((0, 1), (1, 2 * sms + 1), (T - 3, T)):
        b = lagp.predict_torch(X, Z, XX[lo:hi].contiguous(), 6, n, M, 0.5, 1e-5, "alc", precision)
        for k in a:
            assert torch.equal(a[k][lo:hi], b[k]), (lo, k)
    assert bool((a["status"] == 0).all())
