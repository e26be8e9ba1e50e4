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
