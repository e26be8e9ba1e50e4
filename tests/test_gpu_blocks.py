"""Blocks of the network (depthwise and pointwise layer) in one launch on the tensor-core kernel.

Tolerance of a block: the pointwise layer's own (see test_gpu_routes.py) on the depthwise output, and what the depthwise output may be
off by, ten roundings of 2^-24 of its magnitude and one more for storing the oracle's in fp32, taken through the weights' magnitudes.
"""
import ctypes
import functools

import numpy as np
import pytest
import torch

import paper_2310_19509_b200 as sbnn
from oracle import reference as R
from sbnn_inputs import mobilenet_v1_inputs

pytestmark = pytest.mark.gpu
# one tile width and split after the other; block 1 has one step of 32 channels, block 5 four of 64
INSTANCES = [(1, 64, 1), (2, 64, 1), (2, 128, 1), (3, 64, 1), (3, 128, 1), (3, 64, 2), (4, 64, 1), (4, 128, 1), (4, 256, 1), (4, 64, 2),
             (5, 64, 1), (5, 128, 1), (5, 256, 1), (5, 64, 3), (5, 64, 4)]


@functools.lru_cache(maxsize=None)
def layers():
    return mobilenet_v1_inputs(1, 50, 4, seed=2)[1]


@pytest.fixture(scope="module")
def net():
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    pack = lambda L: sbnn.pack_weights(L["w"], L["mask"], L["bias"], L["g"])  # noqa: E731
    of = lambda kind: [L for L in layers() if L["kind"] == kind]  # noqa: E731
    net = sbnn.MobileNetV1([pack(L) for L in of("pw")], pack(of("fc")[0]), [t(L["w"]) for L in of("dw")], [t(L["bias"]) for L in of("dw")],
                           t(layers()[0]["w"]), t(layers()[0]["bias"]), 3)
    yield net
    net.free()


@functools.lru_cache(maxsize=None)
def block(b, n):
    """Input, oracle result and tolerance of block b on n images."""
    side, c, _, _ = sbnn.mobilenet_v1_layer_shape(2 * b - 1)
    x = np.random.default_rng(10 * b + n).standard_normal((n, side, side, c), dtype=np.float32)
    dw, pw = layers()[2 * b - 1], layers()[2 * b]
    mid, s_mid = R.dwconv3x3(x, dw["w"], dw["bias"], stride=dw["stride"], relu=True)
    ref, s = R.conv2d(mid.astype(np.float32), pw["w"], pw["mask"], pw["bias"], relu=True)
    off, _ = R.conv2d((11 * 2.0 ** -24 * s_mid).astype(np.float32), np.abs(pw["w"]), pw["mask"], None, relu=False)
    steps = (c + 63) // 64
    return x, ref, (4 * 2.0 ** -23 + (steps + 3) * 2.0 ** -24) * s + off


def planes(a):
    """NHWC as the network keeps activations, [C][pixels]."""
    return torch.from_numpy(np.ascontiguousarray(a.reshape(-1, a.shape[-1]).T)).cuda()


def run(net, b, x, tile, split):
    n = len(x)
    _, _, side, cout = sbnn.mobilenet_v1_layer_shape(2 * b)
    y = torch.full((cout * n * side * side + 512,), float("nan"), device="cuda")
    net.debug_block(b, planes(x), y[256:], n, tile, split)
    sbnn.get_async_status()
    assert bool(torch.isnan(y[:256]).all()) and bool(torch.isnan(y[-256:]).all())
    return y[256:-256].view(cout, -1).cpu().numpy().T.reshape(n, side, side, cout)


@pytest.mark.parametrize("n", [1, 3])
@pytest.mark.parametrize("b,tile,split", INSTANCES)
def test_block_in_one_launch(net, b, tile, split, n):
    x, ref, tol = block(b, n)
    err = np.abs(run(net, b, x, tile, split).astype(np.float64) - ref)
    assert np.all(err <= tol), np.max(err / tol)


@pytest.mark.parametrize("b,tile", [(1, 64), (2, 128), (3, 128), (4, 256), (5, 256)])
def test_bad_activations_as_in_two_launches(net, b, tile):
    """An infinity or a NaN reaches the pixels around it, and of those only the outputs that keep its channel, as in two launches."""
    x, _, tol = block(b, 1)
    x = x.copy()
    x[0, 5, 9, 3], x[0, 0, 0, 17], x[0, -1, -1, 1], x[0, 20, 13, 8:12] = np.inf, -np.inf, np.nan, np.inf
    _, _, side, cout = sbnn.mobilenet_v1_layer_shape(2 * b)
    mid, want = torch.empty((x.shape[-1], side * side), device="cuda"), torch.empty((cout, side * side), device="cuda")
    net.run_layer_cm(2 * b - 1, planes(x), mid, 1)
    net.run_layer_cm(2 * b, mid, want, 1)
    want = want.cpu().numpy().T.reshape(1, side, side, cout)
    got = run(net, b, x, tile, 1)
    assert np.isinf(want).any() and np.array_equal(np.isinf(got), np.isinf(want)) and not np.isnan(got).any()
    finite = np.isfinite(want)
    err = np.abs(got.astype(np.float64) - np.where(finite, want, 0))
    assert np.all(err[finite] <= 2 * np.maximum(tol, 1e-5 * np.abs(want))[finite])


def test_forward_runs_the_blocks_that_it_says(net):
    """The last layer of a prefix gets the same values whether the layers before it ran one by one or as forward launches them."""
    x = torch.rand((3, 224, 224, 3), device="cuda")
    for n in (1, 3):
        for last in (2, 4, 6, 8, 10):
            assert net.debug_launches(n, last) in (net.debug_launches(n, last - 2) + 1, net.debug_launches(n, last - 2) + 2)
            _, _, side, cout = sbnn.mobilenet_v1_layer_shape(last)
            ld = (n * side * side + 3) // 4 * 4
            got, want = torch.zeros((cout, ld), device="cuda"), torch.zeros((cout, ld), device="cuda")
            net.forward_prefix(x, got, n, last)
            mid = torch.empty((sbnn.mobilenet_v1_layer_shape(last)[1], ld), device="cuda")
            net.forward_prefix(x, mid, n, last - 1)
            net.run_layer_cm(last, mid, want, n)
            sbnn.get_async_status()
            assert float((got - want).norm() / want.norm()) < 1e-6      # (2-norm of an fp32 layer's error: below 5.5e-7 on any kernel)


# Which blocks run in one launch: what each saves of the time of the network is in csrc/conv_tc.cu.  (At 9 images the third would cost 0.6 us.)
JOINED = {1: [1], 2: [1, 2], 4: [1, 2, 3], 6: [1, 2, 3], 9: [1, 2], 12: [1, 2, 3, 4], 16: [1, 2, 3, 4, 5], 40: [1, 2, 3, 4, 5], 64: [1, 2, 3, 4, 5]}


def make_net(batch, limit=None):
    """The network of `net` for up to `batch` images; limit: bytes of the first pointwise layer's images for the tensor cores."""
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    of = lambda kind: [L for L in layers() if L["kind"] == kind]  # noqa: E731
    pw, (fc,) = ([sbnn.pack_weights(L["w"], L["mask"], L["bias"], L["g"]) for L in of(kind)] for kind in ("pw", "fc"))
    if limit is not None:
        sbnn.debug_limit_images(pw[0], limit)
    return sbnn.MobileNetV1(pw, fc, [t(L["w"]) for L in of("dw")], [t(L["bias"]) for L in of("dw")], t(layers()[0]["w"]), t(layers()[0]["bias"]), batch)


def test_the_blocks_that_are_joined():
    big = make_net(64)
    for n, blocks in JOINED.items():
        got = [b for b in range(1, 14) if big.debug_launches(n, 2 * b) == big.debug_launches(n, 2 * b - 2) + 1]
        assert got == blocks, n
    big.free()


def launched(net, n, last):
    """Kernel launches of the first layers, counted in a graph of them."""
    x = torch.rand((n, 224, 224, 3), device="cuda")
    _, _, side, cout = sbnn.mobilenet_v1_layer_shape(last)
    out = torch.empty(max(cout * ((n * side * side + 3) // 4 * 4), 1024 * 4), device="cuda")
    net.forward_prefix(x, out, n, last)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        net.forward_prefix(x, out, n, last)
    count = ctypes.c_size_t()
    nodes = ctypes.CDLL("libcudart.so.12").cudaGraphGetNodes
    assert nodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(count)) == 0
    return count.value


@pytest.mark.parametrize("limit", [None, 1000])
def test_launches_are_those_of_the_forward_pass(limit):
    """Also where a block could run in one launch, but its pointwise layer's images have no room on the device (limit)."""
    net = make_net(6, limit)
    for n in (1, 6):
        for last in (1, 2, 4, 6, 28):
            assert net.debug_launches(n, last) == launched(net, n, last), (n, last)
    assert net.debug_launches(6, 2) == (2 if limit is None else 3)
    net.free()


@pytest.mark.parametrize("tile,split", [(128, 2), (256, 4), (64, 0), (64, -1), (64, 9), (96, 1), (0, 1), (64, 5)])
def test_tiles_that_there_are_not(net, tile, split):
    """Refused, and not run in some other way (block 5 has four steps to share)."""
    x, ref, _ = block(5, 1)
    with pytest.raises(sbnn.SbnnError):
        net.debug_block(5, planes(x), torch.empty(ref.size, device="cuda"), 1, tile, split)


@pytest.mark.parametrize("b,tile", [(1, 64), (2, 128), (3, 128), (4, 256), (5, 256)])
def test_bad_depthwise_weights_as_in_two_launches(b, tile):
    """Infinities and NaN in the depthwise weights and biases spoil the same outputs in one launch as in two: zeros outside the image are
    multiplied by them, ReLU turns NaN into 0, and an infinity that is left reaches the outputs that keep its channel."""
    x, _, tol = block(b, 1)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    of = lambda kind: [L for L in layers() if L["kind"] == kind]  # noqa: E731
    pw, (fc,) = ([sbnn.pack_weights(L["w"], L["mask"], L["bias"], L["g"]) for L in of(kind)] for kind in ("pw", "fc"))
    dw_w, dw_b = [L["w"].copy() for L in of("dw")], [L["bias"].copy() for L in of("dw")]
    w, bias = dw_w[b - 1].reshape(3, 3, -1), dw_b[b - 1]
    w[0, 0, 3], w[1, 1, 9], w[2, 1, 14], bias[20], bias[25] = np.inf, np.nan, -np.inf, np.inf, np.nan
    bad = sbnn.MobileNetV1(pw, fc, [t(a) for a in dw_w], [t(a) for a in dw_b], t(layers()[0]["w"]), t(layers()[0]["bias"]), 1)
    _, _, side, cout = sbnn.mobilenet_v1_layer_shape(2 * b)
    mid, want = torch.empty((x.shape[-1], side * side), device="cuda"), torch.empty((cout, side * side), device="cuda")
    bad.run_layer_cm(2 * b - 1, planes(x), mid, 1)
    bad.run_layer_cm(2 * b, mid, want, 1)
    want = want.cpu().numpy().T.reshape(1, side, side, cout)
    got = run(bad, b, x, tile, 1)
    assert np.isinf(want).any() and np.isfinite(want).any()
    assert np.array_equal(np.isinf(got), np.isinf(want)) and np.array_equal(np.isnan(got), np.isnan(want))
    finite = np.isfinite(want)
    err = np.abs(got.astype(np.float64) - np.where(finite, want, 0))
    assert np.all(err[finite] <= 2 * np.maximum(tol, 1e-5 * np.abs(want))[finite])
    bad.free()
