"""fp32 layers on the tensor cores (three-way bf16 split): edges of tiles, stages and layouts against the CPU oracle.

Tolerance: |gpu - ref| <= 1e-5 * S per output, S = |b| + sum |w*x|, as for the other fp32 kernels.  The split is exact, the
omitted products are below 2^-25 |w*x| each, a 64-channel step loses at most 24 units in the last place of its sum
(24 * 2^-23 = 2.9e-6 of sum |w*x|) to the accumulator's truncations, and the steps' sums are added in fp32.
"""
import numpy as np
import pytest
import torch

import paper_2310_19509_b200 as sbnn
from oracle import reference as R
from sbnn_inputs import workloads as WL

pytestmark = pytest.mark.gpu
TOL = 1e-5


def layer(n, h, w, cin, cout, k, g, pct, seed=0):
    d = WL.single_conv_inputs(n, h, w, cin, cout, k, g, pct, seed, 0.05, 0.05)
    return d, sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)


def reference(d, relu=True):
    return R.conv2d(d["x"], d["w"], d["mask"], d["bias"], relu=relu)


def check(y, ref, s):
    assert np.all(np.isfinite(y))
    assert np.all(np.abs(y.astype(np.float64) - ref) <= TOL * s)


# (n, h, w, cin, cout, g, pct): pixels and channels at, below and above tiles of 128 pixels and 64 / 128 / 256 output
# channels; one, a half, and several 64-channel steps; one tile per SM and many.
SHAPES = [
    (1, 128, 128, 4, 60, 4, 0),
    (6, 56, 56, 32, 64, 4, 50),
    (3, 57, 59, 36, 68, 4, 30),
    (5, 50, 41, 64, 128, 8, 50),
    (7, 31, 29, 100, 132, 4, 50),
    (9, 28, 28, 160, 260, 4, 30),
    (13, 14, 14, 516, 512, 8, 50),
    (64, 9, 9, 192, 256, 16, 50),
    (11, 23, 23, 128, 252, 2, 50),
    # few tiles: the steps of a tile shared by the 2, 4 or 8 CTAs of a cluster
    (1, 14, 14, 512, 512, 4, 0),
    (4, 7, 7, 1024, 1000, 4, 0),
    (2, 13, 11, 1000, 60, 4, 30),
    (3, 14, 14, 200, 128, 8, 0),
]


@pytest.mark.parametrize("n,h,w,cin,cout,g,pct", SHAPES)
def test_1x1_nhwc(n, h, w, cin, cout, g, pct):
    d, p = layer(n, h, w, cin, cout, 1, g, pct)
    x = torch.from_numpy(d["x"]).cuda()
    y = torch.full((n * h * w * cout + 512,), float("nan"), device="cuda")
    sbnn.conv1x1_gs(p, x, y[256:], n, h, w)
    ref, s = reference(d)
    check(y[256:-256].cpu().numpy().reshape(ref.shape), ref, s)
    assert bool(torch.isnan(y[:256]).all()) and bool(torch.isnan(y[-256:]).all())
    sbnn.get_async_status()


@pytest.mark.parametrize("out_cm", [True, False])
@pytest.mark.parametrize("n,h,w,cin,cout,g,pct", SHAPES)
def test_1x1_channel_major(n, h, w, cin, cout, g, pct, out_cm):
    d, p = layer(n, h, w, cin, cout, 1, g, pct, seed=1)
    m = n * h * w
    ld = (m + 3) // 4 * 4 + 8                                   # padding: unset on input, to be left alone on output
    x = torch.full((cin, ld), float("nan"), device="cuda")
    x[:, :m] = torch.from_numpy(d["x"].reshape(m, cin).T.copy()).cuda()
    y = torch.full((cout, ld) if out_cm else (m, cout), float("nan"), device="cuda")
    sbnn.conv1x1_gs_cm(p, x, ld, y, ld if out_cm else cout, m, sbnn.SBNN_RELU | (sbnn.SBNN_OUT_CM if out_cm else 0))
    ref, s = reference(d)
    got = y.cpu().numpy()
    if out_cm:
        assert np.all(np.isnan(got[:, m:]))
        got = got[:, :m].T
    check(got.reshape(ref.shape), ref, s)
    sbnn.get_async_status()


@pytest.mark.parametrize("n,h,w,cin,cout,g,pct", [
    (1, 56, 56, 4, 256, 4, 0),
    (5, 28, 31, 36, 256, 4, 50),
    (40, 14, 14, 64, 136, 8, 50),
    (120, 7, 7, 100, 128, 4, 30),
    (1, 3, 250, 68, 900, 4, 50),
    (700, 1, 1, 64, 1000, 8, 50),
    (5, 7, 7, 512, 512, 8, 70),
    (1, 14, 14, 64, 64, 4, 50),
    (2, 5, 28, 96, 72, 8, 0),
    (1, 3, 4, 260, 12, 4, 50),
])
def test_3x3(n, h, w, cin, cout, g, pct):
    d, p = layer(n, h, w, cin, cout, 3, g, pct, seed=2)
    x = torch.from_numpy(d["x"]).cuda()
    y = torch.full((n, h, w, cout), float("nan"), device="cuda")
    sbnn.conv3x3_gs(p, x, y, n, h, w)
    ref, s = reference(d)
    check(y.cpu().numpy(), ref, s)
    m = n * h * w
    ld = (m + 3) // 4 * 4 + 4
    xt = torch.full((cin, ld), float("nan"), device="cuda")
    xt[:, :m] = x.reshape(m, cin).T
    for out_cm in (True, False) if w <= 224 else ():
        y = torch.full((cout, ld) if out_cm else (m, cout), float("nan"), device="cuda")
        sbnn.conv3x3_gs_cm(p, xt, ld, y, ld if out_cm else cout, n, h, w, sbnn.SBNN_RELU | (sbnn.SBNN_OUT_CM if out_cm else 0))
        got = y.cpu().numpy()
        if out_cm:
            assert np.all(np.isnan(got[:, m:]))
            got = got[:, :m].T
        check(got.reshape(ref.shape), ref, s)
    sbnn.get_async_status()


def test_values_of_every_size():
    """Products from 1e-16 to 1e14 in one sum: the split must not lose the bits of small or large operands."""
    d, _ = layer(5, 50, 41, 64, 128, 1, 4, 50, seed=3)
    scale = np.float32(2.0) ** np.random.default_rng(0).integers(-50, 50, 64).astype(np.float32)
    d["x"] = np.ascontiguousarray(d["x"] * scale).astype(np.float32)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], 4)
    y = torch.empty((5, 50, 41, 128), device="cuda")
    sbnn.conv1x1_gs(p, torch.from_numpy(d["x"]).cuda(), y, 5, 50, 41, 0)
    ref, s = reference(d, relu=False)
    check(y.cpu().numpy(), ref, s)


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("h,w,cin", [(50, 41, 64), (18, 41, 520)])   # whole tiles; tiles shared by clusters
def test_non_finite_activations_stay_where_they_belong(k, h, w, cin):
    """An infinity or a NaN reaches the outputs whose kept channels read it and no others."""
    n, cout, g = 5 if cin == 64 else 1, 128, 4
    d, p = layer(n, h, w, cin, cout, k, g, 50, seed=4)
    d["x"][0, 0, 0, 3] = np.inf
    d["x"][n // 2, 17, 40, 9] = np.nan
    d["x"][n - 1, h - 1, 39, 63] = -np.inf
    y = torch.empty((n, h, w, cout), device="cuda")
    (sbnn.conv1x1_gs if k == 1 else sbnn.conv3x3_gs)(p, torch.from_numpy(d["x"]).cuda(), y, n, h, w, 0)
    got = y.cpu().numpy()
    clean = dict(d, x=np.where(np.isfinite(d["x"]), d["x"], 0).astype(np.float32))
    ref, s = reference(clean, relu=False)
    touched = np.zeros(ref.shape, bool)
    for b, r, c, ch in np.argwhere(~np.isfinite(d["x"])):
        rr, cc = slice(max(r - k // 2, 0), r + k // 2 + 1), slice(max(c - k // 2, 0), c + k // 2 + 1)
        touched[b, rr, cc] |= d["mask"][:, 0, 0, ch].astype(bool)
    assert not np.isfinite(got[touched]).any()
    assert np.all(np.abs(got[~touched].astype(np.float64) - ref[~touched]) <= TOL * s[~touched])
