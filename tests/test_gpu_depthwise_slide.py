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


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("tap", [0, 1, 2])
def test_taps_outside_the_image_are_not_multiplied(stride, tap):
    """An infinite weight in the first or last kernel row: the outputs whose row lies outside the image stay finite, whichever
    kernel the size selects (one image is too little for the kernel that slides)."""
    n, h, w, c = 40, 13, 13, 516
    rng = np.random.default_rng(stride)
    x = torch.from_numpy(rng.random((n, h, w, c), dtype=np.float32) + np.float32(0.5)).cuda()
    wt = rng.standard_normal((3, 3, c), dtype=np.float32)
    wt[tap, 1, ::7] = np.inf
    wt[tap, 1, 3::7] = np.nan
    wt, b = torch.from_numpy(wt).cuda(), torch.zeros(c, device="cuda")
    ho = (h - 1) // stride + 1
    y, one = torch.empty((n, ho, ho, c), device="cuda"), torch.empty((n, ho, ho, c), device="cuda")
    sbnn.dwconv3x3(wt, b, x, y, n, h, w, c, stride, 0)
    for i in range(n):
        sbnn.dwconv3x3(wt, b, x[i], one[i], 1, h, w, c, stride, 0)
    assert bool(torch.isfinite(one).any()) and not bool(torch.isfinite(one).all())
    torch.testing.assert_close(y, one, rtol=1e-5, atol=1e-5, equal_nan=True)
