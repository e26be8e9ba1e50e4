"""The NHWC depthwise kernel that gives a thread one output row: both instances, by the number of CTAs of a launch."""
import numpy as np
import pytest
import torch

import paper_2310_19509_b200 as sbnn
from oracle import reference as R

pytestmark = pytest.mark.gpu


# 1 and 112 CTAs (an instance with more registers); 441 and 350, on 148 SMs more than two an SM, and too few for the sliding kernel
@pytest.mark.parametrize("n,h,w,c,stride", [(1, 5, 9, 12, 1), (2, 28, 28, 256, 2), (9, 28, 28, 256, 1), (25, 28, 28, 256, 2)])
def test_both_instances(n, h, w, c, stride):
    """1e-5 * S: the tolerance of every kernel (S = |b| + sum |w*x|)."""
    rng = np.random.default_rng(n)
    x, wt, b = (rng.standard_normal(s, dtype=np.float32) for s in ((n, h, w, c), (3, 3, c), (c,)))
    ref, s = R.dwconv3x3(x, wt, b, stride=stride, relu=True)
    y = torch.full((ref.size + 128,), float("nan"), device="cuda")
    t = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    sbnn.dwconv3x3(t(wt), t(b), t(x), y[64:], n, h, w, c, stride, sbnn.SBNN_RELU)
    assert bool(torch.isnan(y[:64]).all()) and bool(torch.isnan(y[-64:]).all())
    got = y[64:-64].cpu().numpy().reshape(ref.shape)
    assert np.all(np.abs(got.astype(np.float64) - ref) <= 1e-5 * s)
