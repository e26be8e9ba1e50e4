"""Depthwise 3x3 on NHWC tensors large enough for the kernel that slides down the rows: ragged strips, rows and channels.

Tolerance: |gpu - ref| <= 1e-5 * S per output, S = |b| + sum |w*x| (nine products and a bias in fp32: 10 * 2^-24 * S)."""
import numpy as np
import pytest
import torch

import paper_2310_19509_b200 as sbnn
from oracle import reference as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,w,c,stride", [
    (40, 13, 13, 516, 1), (24, 15, 31, 256, 1), (150, 4, 3, 1024, 1), (2, 112, 112, 96, 1), (300, 1, 1, 1024, 1),
    (40, 13, 13, 516, 2), (24, 15, 31, 256, 2), (150, 8, 2, 1024, 2), (4, 112, 112, 96, 2),
])
@pytest.mark.parametrize("relu", [True, False])
def test_matches_the_oracle(n, h, w, c, stride, relu):
    rng = np.random.default_rng(n * c + stride)
    x = rng.random((n, h, w, c), dtype=np.float32)
    wt = rng.standard_normal((3, 3, c), dtype=np.float32)
    b = rng.standard_normal(c, dtype=np.float32)
    ho, wo = (h - 1) // stride + 1, (w - 1) // stride + 1
    full = torch.full((n * ho * wo * c + 512,), float("nan"), device="cuda")
    y = full[256:-256].view(n, ho, wo, c)
    dev = [torch.from_numpy(a).cuda() for a in (wt, b, x)]
    sbnn.dwconv3x3(*dev, y, n, h, w, c, stride, sbnn.SBNN_RELU if relu else 0)
    ref, s = R.dwconv3x3(x, wt, b, stride=stride, relu=relu)
    got = y.cpu().numpy()
    assert np.all(np.abs(got.astype(np.float64) - ref) <= 1e-5 * s)
    assert bool(torch.isnan(full[:256]).all()) and bool(torch.isnan(full[-256:]).all())
