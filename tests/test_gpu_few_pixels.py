"""The few-pixel 1x1 kernel with eight warps: both instances, by the number of CTAs of a launch, for every group size."""
import numpy as np
import pytest
import torch

import paper_2310_19509_b200 as sbnn
from oracle import reference as R
from sbnn_inputs import workloads as WL

gpu = pytest.mark.gpu


# Groups x blocks of 32 or 64 pixels just below and above the line between the instances on 148 SMs, with one and with two pixels a
# lane; 516 channels half pruned are more than 256 a group.
@gpu
@pytest.mark.parametrize("g,cout,m", [(1, 592, 32), (1, 593, 32), (1, 148, 65), (1, 149, 65), (2, 296, 17), (2, 298, 17), (2, 592, 64), (2, 594, 64),
                                      (4, 1184, 32), (4, 1188, 1), (4, 592, 197), (4, 596, 225), (8, 2368, 33), (8, 1192, 325), (16, 1200, 33), (16, 64, 1)])
def test_both_instances(g, cout, m):
    """1e-5 * S: the tolerance of every kernel (S = |b| + sum |w*x|)."""
    d = WL.single_conv_inputs(1, 1, m, 516, cout, 1, g, 50, 7, 0.05, 0.05)
    ref, s = R.conv2d(d["x"], d["w"], d["mask"], d["bias"], relu=True)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
    ld = (m + 3) // 4 * 4
    x = torch.zeros((516, ld), device="cuda")
    x[:, :m] = torch.from_numpy(d["x"].reshape(m, 516).T.copy())
    y = torch.full((cout, ld + 4), float("nan"), device="cuda")
    sbnn.debug_conv_gs(p, x, ld, y, ld + 4, 1, 1, m, sbnn.SBNN_RELU | sbnn.SBNN_OUT_CM, 0, 1)
    assert bool(torch.isnan(y[:, m:]).all())
    err = np.abs(y[:, :m].T.cpu().numpy().astype(np.float64) - ref.reshape(m, cout))
    assert np.all(err <= 1e-5 * s.reshape(m, cout))
    p.free()


# Pixels, channels, group, pruned: which side is the faster one, tensor cores or FMA kernel (us: tensor cores and FMA)
@gpu
@pytest.mark.parametrize("m,cin,cout,g,pct,tensor", [
    (49, 1024, 1024, 8, 30, False),      # 8.2, 7.4
    (49, 512, 1024, 4, 0, False),        # 6.9, 6.0
    (49, 1024, 1024, 4, 50, False),      # 8.2, 5.9
    (1, 1024, 1000, 4, 0, False),        # 8.1, 6.6
    (17, 64, 128, 4, 50, False),         # 4.2, 1.7
    (183, 768, 256, 1, 30, True),        # 6.9, 13.3
    (879, 56, 320, 1, 90, True),         # 4.3, 10.2
    (396, 52, 1040, 2, 70, True),        # 4.5, 7.9
    (1286, 32, 720, 4, 90, True),        # 4.1, 8.5
    (49, 1296, 256, 8, 0, True),         # 7.3, 11.3
    (34, 1472, 160, 16, 0, True),        # 7.4, 13.6
    (392, 640, 232, 4, 50, True),        # 7.6, 7.8
    (733, 512, 512, 16, 70, True),       # 8.9, 10.9
    (171, 428, 576, 4, 30, True),        # 7.0, 7.6
])
def test_the_faster_kernel_is_picked(m, cin, cout, g, pct, tensor):
    d = WL.single_conv_inputs(1, 1, 1, cin, cout, 1, g, pct, 3, 0.05, 0.05)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
    ld = (m + 3) // 4 * 4
    sbnn.conv1x1_gs_cm(p, torch.zeros((cin, ld), device="cuda"), ld, torch.empty((cout, ld), device="cuda"), ld, m, sbnn.SBNN_RELU | sbnn.SBNN_OUT_CM)
    assert (sbnn.debug_last_route()[0] != 0) == tensor
    p.free()


# 45 tiles of 64 channels fit the device in clusters of 3, but not behind another launch (10.3 us; unshared 7.5), 12.0 (of 2: 9.6);
# 42 tiles of 15 steps: 9.8 us in clusters of 3, 11.6 of 2
@gpu
@pytest.mark.parametrize("m,cin,cout,fits", [(1072, 384, 288, False), (621, 608, 576, False), (349, 608, 912, False), (1674, 940, 176, True)])
def test_clusters_that_fit_behind_another_launch(m, cin, cout, fits):
    d = WL.single_conv_inputs(1, 1, 1, cin, cout, 1, 4, 0, 3, 0.05, 0.05)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], 4)
    ld = (m + 3) // 4 * 4
    sbnn.conv1x1_gs_cm(p, torch.zeros((cin, ld), device="cuda"), ld, torch.empty((cout, ld), device="cuda"), ld, m, sbnn.SBNN_RELU | sbnn.SBNN_OUT_CM)
    tile, split = sbnn.debug_last_route()
    assert tile == 64 and (split == 3) == fits
    p.free()
