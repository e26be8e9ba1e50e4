"""Depthwise kernels that have two instances, one with more registers for launches of few CTAs: the NHWC kernel that gives a thread one
output row, and the channel-major one for 14 x 14 maps."""
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


# 128 and 180 CTAs (an instance with more registers), 455 and 1024, on 148 SMs more than three an SM
@pytest.mark.parametrize("n,c", [(4, 512), (15, 180), (70, 97), (32, 512)])
def test_both_channel_major_14x14_instances(n, c):
    """1e-5 * S, as above."""
    rng = np.random.default_rng(n)
    x, wt, b = (rng.standard_normal(s, dtype=np.float32) for s in ((n, 14, 14, c), (3, 3, c), (c,)))
    ref, s = R.dwconv3x3(x, wt, b, stride=1, relu=True)
    m = n * 196
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    y = torch.full((c, m + 4), float("nan"), device="cuda")
    sbnn.dwconv3x3_cm(t(wt), t(b), t(x.reshape(m, c).T), m, y, m + 4, n, 14, 14, c, 1, sbnn.SBNN_RELU)
    assert bool(torch.isnan(y[:, m:]).all())
    got = y[:, :m].T.cpu().numpy().reshape(ref.shape)
    assert np.all(np.abs(got.astype(np.float64) - ref) <= 1e-5 * s)
