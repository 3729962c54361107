"""The checked build records nothing for a location that has no design (its screen failed: idx is
-1), on both sides of the predictive kernel's line between its forms (n = 208)."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import numpy as np, torch
from paper_1303_0383_gb300 import lagp
rng = np.random.default_rng(1)
X = torch.as_tensor(rng.random((400, 2))).cuda()
Z = X.sum(1)
XX = torch.as_tensor(rng.random((3, 2))).cuda()
for n in (40, 208, 209, 256):
    idx = torch.as_tensor(np.stack([rng.permutation(400)[:n] for _ in range(3)]).astype(np.int32)).cuda()
    idx[1] = -1
    o = [torch.full((3,), 7.0, dtype=torch.float64, device="cuda") for _ in range(3)]
    st = torch.full((3,), 9, dtype=torch.int8, device="cuda")
    lagp.lagp_design_predict_dev(X, Z, XX, idx, 0.5, 1e-3, *o, st,
                                 ws=lagp.workspace(lagp.lagp_design_predict_workspace_bytes(3, n)))
    assert st.tolist() == [0, lagp.LAGP_ERR_NOT_PD, 0], st
    assert bool(torch.isnan(o[0][1])) and bool(torch.isfinite(o[0][[0, 2]]).all())
r = lagp.lagp_check_take()
assert r["checked"] and r["count"] == 0, r
"""


def test_failed_locations_are_no_violations():
    from paper_1303_0383_gb300 import build
    build.build(checked=True)
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, env=dict(os.environ, LAGP_CHECKED="1"),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
