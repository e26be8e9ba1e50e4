"""Channel-major 1x1 kernel with as many stages as its weight blocks leave room for: shapes on both sides of the rule.

Tolerance: |gpu - ref| <= 1e-5 * S per output, S = |b| + sum |w*x|: an fp32 sum of n <= 130 kept terms is off by at most
n * 2^-24 = 7.8e-6 of S.
"""
import numpy as np
import pytest
import torch

import paper_2310_19509_b200 as sbnn
from oracle import reference as R
from sbnn_inputs import workloads as WL

pytestmark = pytest.mark.gpu


# One step, as many as stages, one more, and many rounds of the ring; pixels and groups that leave a ragged last tile;
# short lists (three stages) and full ones (two).
@pytest.mark.parametrize("out_cm", [True, False])
@pytest.mark.parametrize("g,tile", [(8, (8, 1, 8, 64)), (8, (8, 1, 12, 64)), (4, (8, 2, 8, 64)), (4, (8, 2, 11, 64)), (4, (8, 2, 12, 64)), (4, (8, 1, 16, 64))])
@pytest.mark.parametrize("n,h,w,cin,cout,pct", [(1, 9, 9, 64, 64, 90), (3, 17, 19, 192, 104, 90), (11, 28, 28, 200, 1016, 90), (5, 14, 14, 1024, 120, 90),
                                                 (2, 40, 40, 128, 200, 0), (7, 14, 14, 130, 264, 50)])
def test_stages(n, h, w, cin, cout, pct, g, tile, out_cm):
    d = WL.single_conv_inputs(n, h, w, cin, cout, 1, g, pct, 3, 0.05, 0.05)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
    m = n * h * w
    ld = (m + 3) // 4 * 4 + 8
    x = torch.full((cin, ld), float("nan"), device="cuda")
    x[:, :m] = torch.from_numpy(d["x"].reshape(m, cin).T.copy()).cuda()
    y = torch.full((cout, ld) if out_cm else (m, cout), float("nan"), device="cuda")
    sbnn.conv1x1_gs_cm(p, x, ld, y, ld if out_cm else cout, m, sbnn.SBNN_RELU | (sbnn.SBNN_OUT_CM if out_cm else 0), tile=tile)
    ref, s = R.conv2d(d["x"], d["w"], d["mask"], d["bias"], relu=True)
    out = (y[:, :m].T if out_cm else y).cpu().numpy().astype(np.float64).reshape(ref.shape)
    assert np.all(np.abs(out - ref) <= 1e-5 * s)
    if out_cm:
        assert bool(torch.isnan(y[:, m:]).all())
    sbnn.get_async_status()
