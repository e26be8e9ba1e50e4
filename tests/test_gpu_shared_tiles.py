"""Tiles of the tensor-core kernel whose steps are dealt to three, five, six or seven CTAs of a cluster."""
import numpy as np
import pytest
import torch

import paper_2310_19509_b200 as sbnn
from oracle import reference as R
from sbnn_inputs import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, sbnn.SBNN_BF16_TC])
@pytest.mark.parametrize("split", [3, 5, 6, 7])
def test_tiles_shared_by_any_number_of_ctas(split, flags):
    """Steps (9) and outputs (8 chunks of a thread) are dealt unevenly.  1e-5 * S: the tolerance of every kernel (S = |b| + sum |w*x|)."""
    n, h, w, cin, cout = 2, 11, 13, 516, 132
    d = WL.single_conv_inputs(n, h, w, cin, cout, 1, 4, 50, 11, 0.05, 0.05)
    ref, s = R.conv2d(d["x"], d["w"], d["mask"], d["bias"], relu=False, bf16=bool(flags))
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], d["g"])
    y = torch.full((n, h, w, cout), float("nan"), device="cuda")
    sbnn.debug_conv_gs(p, torch.from_numpy(d["x"]).cuda(), 0, y, 0, n, h, w, flags, 64, split)
    sbnn.get_async_status()
    err = np.abs(y.cpu().numpy().astype(np.float64) - ref.reshape(n, h, w, cout))
    assert np.all(err <= 1e-5 * s.reshape(err.shape))
    p.free()


# 9 rows of kernels of which the last three are half as long: shared by 4 11.0, 10.4 and 10.8 us, by 5 11.6, 10.9 and 11.2; 6 equal rows:
# 8.3 by 6, 10.2 by 4
@pytest.mark.parametrize("n,hw,cin,cout,split", [(1, 56, 144, 32, 4), (10, 14, 148, 48, 4), (8, 13, 148, 80, 4), (5, 14, 128, 64, 6)])
def test_the_last_steps_may_be_short(n, hw, cin, cout, split):
    d = WL.single_conv_inputs(1, 1, 1, cin, cout, 3, 4, 30, 3, 0.05, 0.05)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], 4)
    m = n * hw * hw
    ld = (m + 3) // 4 * 4
    sbnn.conv3x3_gs_cm(p, torch.zeros((cin, ld), device="cuda"), ld, torch.empty((cout, ld), device="cuda"), ld, n, hw, hw, sbnn.SBNN_OUT_CM)
    assert sbnn.debug_last_route() == (64, split)
    p.free()
