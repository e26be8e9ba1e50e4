"""Layers on a kernel that the test names: every instance of the tensor-core kernel, and the FMA kernels at shapes that the
library's own choice gives to the tensor cores.

Tolerance of the tensor-core kernel, per output: |gpu - ref| <= (4 * 2^-23 + (steps + 3) * 2^-24) * S, S = |b| + sum |w*x|.  A
64-channel step adds its products in 24 MMAs of 16 channels, each of which cuts off less than a unit in the last place of the
running sum; the 20 of them that add the small products have sums below 2^-7 S, so four count.  Steps are added in fp32,
rounded to nearest; the three omitted products and the scale of the weights are within the remaining 3 * 2^-24.
Over a whole output the 2-norm of the error is at most 4e-7 of the result's: measured 0.3e-7 to 0.9e-7 for 4 to 1024
channels; without any one of the six products it is above 8e-7 (see test_a_missing_product_would_be_seen).
FMA kernels: 1e-5 * S, as in their own tests (one rounding per kept product).
"""
import functools

import numpy as np
import pytest
import torch

import paper_2310_19509_b200 as sbnn
from oracle import reference as R
from sbnn_inputs import tap_pattern_mask
from sbnn_inputs import workloads as WL

gpu = pytest.mark.gpu
RMS = 4e-7


@functools.lru_cache(maxsize=None)
def inputs(n, h, w, cin, cout, k, g, pct, bf16=False):
    d = WL.single_conv_inputs(n, h, w, cin, cout, k, g, pct, 11, 0.05, 0.05)
    ref, s = R.conv2d(d["x"], d["w"], d["mask"], d["bias"], relu=False, bf16=bf16)
    return d, ref, s


def run(p, d, layout, tile, split, flags=0):
    """layout: 'nhwc', 'cm' (channel-major in, rows out) or 'cm-cm'.  Output as [M][Cout]; guards and padding are checked."""
    n, h, w, cin = d["x"].shape
    m, cout = n * h * w, d["w"].shape[0]
    x = torch.from_numpy(d["x"]).cuda()
    if layout == "nhwc":
        y = torch.full((m * cout + 512,), float("nan"), device="cuda")
        sbnn.debug_conv_gs(p, x, 0, y[256:], 0, n, h, w, flags, tile, split)
        assert bool(torch.isnan(y[:256]).all()) and bool(torch.isnan(y[-256:]).all())
        out = y[256:-256].view(m, cout)
    else:
        ld = (m + 3) // 4 * 4 + 8
        xt = torch.full((cin, ld), float("nan"), device="cuda")
        xt[:, :m] = x.reshape(m, cin).T
        cm = layout == "cm-cm"
        y = torch.full((cout, ld) if cm else (m, cout), float("nan"), device="cuda")
        sbnn.debug_conv_gs(p, xt, ld, y, ld if cm else cout, n, h, w, flags | (sbnn.SBNN_OUT_CM if cm else 0), tile, split)
        if cm:
            assert bool(torch.isnan(y[:, m:]).all())
        out = y[:, :m].T if cm else y
    assert sbnn.debug_last_route() == ((tile, split) if tile else (0, 0))
    sbnn.get_async_status()
    return out.cpu().numpy()


def check_tc(got, ref, s, steps):
    ref, s = ref.reshape(got.shape), s.reshape(got.shape)
    err = np.abs(got.astype(np.float64) - ref)
    assert np.all(err <= (4 * 2.0 ** -23 + (steps + 3) * 2.0 ** -24) * s)
    assert np.linalg.norm(err) <= RMS * np.linalg.norm(ref)


INSTANCES = [(64, 1), (128, 1), (256, 1)] + [(64, split) for split in range(2, 9)]
# ragged pixels, channels and output channels; nine steps for the splits; more tiles than SMs at every tile width
SHAPES_1X1 = [(3, 17, 19, 516, 260, 4, 50), (7, 61, 63, 100, 516, 4, 30)]
SHAPES_3X3 = [(2, 13, 14, 132, 260, 4, 50), (48, 14, 15, 132, 300, 4, 30)]


@gpu
@pytest.mark.parametrize("layout", ["nhwc", "cm", "cm-cm"])
@pytest.mark.parametrize("k,shape,tile,split", [(k, s, *i) for k, shapes in ((1, SHAPES_1X1), (3, SHAPES_3X3)) for s in shapes for i in INSTANCES
                                                if k == 3 or (s[3] + 63) // 64 >= i[1]])
def test_every_tensor_core_instance(k, shape, tile, split, layout):
    d, ref, s = inputs(*shape[:5], k, *shape[5:])
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], d["g"])
    steps = (shape[3] + 63) // 64 * k * k
    check_tc(run(p, d, layout, tile, split), ref, s, steps)
    check_tc(run(p, d, layout, tile, split, sbnn.SBNN_RELU), np.maximum(ref, 0), s, steps)


@gpu
@pytest.mark.parametrize("tile,split", INSTANCES)
def test_every_bf16_instance(tile, split):
    """Operands rounded to bf16, exact products, sums cut off at most 4 * steps times: 36 * 2^-23 = 4.3e-6 of S."""
    d, ref, s = inputs(*SHAPES_1X1[0][:5], 1, *SHAPES_1X1[0][5:], bf16=True)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], d["g"])
    got = run(p, d, "nhwc", tile, split, sbnn.SBNN_BF16_TC)
    assert np.all(np.abs(got.astype(np.float64) - ref.reshape(got.shape)) <= 1e-5 * s.reshape(got.shape))


@gpu
@pytest.mark.parametrize("k,layout", [(1, "nhwc"), (1, "cm"), (3, "nhwc"), (3, "cm")])
@pytest.mark.parametrize("tile,split", INSTANCES)
def test_same_bits_on_every_run(k, layout, tile, split):
    """Stages, images and accumulators change hands hundreds of times in a launch; a reader that ran ahead would show."""
    d, _, _ = inputs(48, 14, 15, 516, 140, 1, 4, 50) if k == 1 else inputs(*SHAPES_3X3[1][:5], 3, *SHAPES_3X3[1][5:])
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], d["g"])
    first = run(p, d, layout, tile, split)
    for _ in range(5):
        assert np.array_equal(first, run(p, d, layout, tile, split))


@gpu
@pytest.mark.parametrize("tile,split", [(64, 1), (64, 4), (256, 1)])
def test_layers_back_to_back_on_two_buffers(tile, split):
    """Depthwise and pointwise layers that write in turn what the other has just read, launched without a pause: each may start
    early, but must not touch a buffer before the launch in front of it, and the one before that, are done with it."""
    n, hw, c = 2, 14, 512
    d, _, _ = inputs(n, hw, hw, c, c, 1, 4, 50)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], 4)
    m = n * hw * hw
    dw_w, dw_b = torch.randn((3, 3, c), device="cuda") / 3, torch.zeros(c, device="cuda")
    first = torch.rand((c, m), device="cuda")

    def chain(pause):
        a, b = first.clone(), torch.zeros((c, m), device="cuda")
        for _ in range(12):
            sbnn.dwconv3x3_cm(dw_w, dw_b, a, m, b, m, n, hw, hw, c, 1)
            if pause:
                torch.cuda.synchronize()
            sbnn.debug_conv_gs(p, b, m, a, m, n, hw, hw, sbnn.SBNN_RELU | sbnn.SBNN_OUT_CM, tile, split)
            if pause:
                torch.cuda.synchronize()
        return a

    want = chain(True)
    assert bool(torch.isfinite(want).all()) and float(want.abs().max()) > 0
    for _ in range(20):
        assert torch.equal(chain(False), want)
    sbnn.get_async_status()


@gpu
@pytest.mark.parametrize("cin", [32, 64])
def test_weights_that_stay_in_shared_memory(cin):
    """One channel tile and no more steps than weight stages: the weights are loaded once and serve every tile."""
    for tile, cout in ((64, 60), (128, 124), (256, 252)):
        d, ref, s = inputs(7, 61, 63, cin, cout, 1, 4, 50)
        p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], d["g"])
        for layout in ("nhwc", "cm-cm"):
            check_tc(run(p, d, layout, tile, 1), ref, s, 1)


@gpu
@pytest.mark.parametrize("scale", [2.0 ** -60, 2.0 ** 60])
def test_small_and_large_operands_keep_their_bits(scale):
    """A pixel whose activations are all small (or large) must be as exact as any other: its own sum is the measure."""
    d, ref, s = inputs(3, 17, 19, 516, 260, 1, 4, 50)
    x = d["x"].copy()
    x[:, 5, :, :] *= np.float32(scale)
    d = dict(d, x=x, bias=np.zeros_like(d["bias"]))
    ref, s = R.conv2d(d["x"], d["w"], d["mask"], d["bias"], relu=False)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], d["g"])
    got = run(p, d, "nhwc", 128, 1).reshape(ref.shape)
    check_tc(got[:, 5], ref[:, 5], s[:, 5], 9)
    check_tc(got, ref, s, 9)


@gpu
@pytest.mark.parametrize("exponent", [-100, -120, -140])
def test_operands_near_the_end_of_bf16(exponent):
    """Down to 2^-109 an operand keeps all its bits; below, each of its three images is rounded to multiples of 2^-133, which
    leaves at most 2^-134 of it out (and a smaller operand whole)."""
    d, _, _ = inputs(3, 17, 19, 516, 260, 1, 4, 50)
    x, w = np.ldexp(d["x"], exponent).astype(np.float32), np.ldexp(d["w"], 60).astype(np.float32)
    d = dict(d, x=x, w=w, bias=np.zeros_like(d["bias"]))
    ref, s = R.conv2d(x, w, d["mask"], d["bias"], relu=False)
    p = sbnn.pack_weights(w, d["mask"], d["bias"], d["g"])
    got = run(p, d, "nhwc", 128, 1)
    if exponent == -100:
        check_tc(got, ref, s, 9)
    lost = 2.0 ** -133 * np.abs(w * d["mask"]).astype(np.float64).reshape(260, -1).sum(1)
    err = np.abs(got.astype(np.float64) - ref.reshape(got.shape))
    assert np.all(err <= lost + (4 * 2.0 ** -23 + 12 * 2.0 ** -24) * s.reshape(got.shape))


def bf16_images(v):
    """Three bf16 numbers whose sum is v, each rounded to nearest even."""
    out, r = [], np.asarray(v, np.float32)
    for _ in range(3):
        u = r.view(np.uint32)
        h = ((u + 0x7FFF + ((u >> 16) & 1)) & np.uint32(0xFFFF0000)).astype(np.uint32).view(np.float32)
        out.append(h.astype(np.float64))
        r = (r - h).astype(np.float32)
    return out


@pytest.mark.parametrize("cin", [100, 516])
def test_a_missing_product_would_be_seen(cin):
    """The bound on the 2-norm is below the error of a sum without any one of the six products (a model in fp64)."""
    rng = np.random.default_rng(cin)
    x = rng.random((200, cin), dtype=np.float32)
    w = rng.standard_normal((64, cin), dtype=np.float32) * np.float32(0.05) * (rng.random((64, cin)) < 0.5)
    ref = x.astype(np.float64) @ w.astype(np.float64).T
    xi, wi = bf16_images(x), bf16_images(w.astype(np.float32))
    six = [(2, 0), (0, 2), (1, 1), (1, 0), (0, 1), (0, 0)]
    err = lambda kept: np.linalg.norm(sum(xi[a] @ wi[b].T for a, b in kept) - ref) / np.linalg.norm(ref)  # noqa: E731
    assert err(six) < RMS / 10
    for gone in six:
        assert err([q for q in six if q != gone]) > 2 * RMS


# ---- the FMA 3x3 kernels: split tiles, tap lists, both numbers of rows per lane, every group size -----------------------
@gpu
@pytest.mark.parametrize("g,n,h,w,cin,cout", [
    (4, 40, 14, 28, 64, 64), (4, 9, 7, 28, 40, 96), (8, 12, 14, 28, 64, 128), (2, 30, 8, 56, 32, 24), (1, 20, 10, 28, 24, 40),
    (16, 6, 28, 28, 48, 64), (4, 200, 14, 28, 16, 32), (4, 20, 14, 28, 40, 72), (4, 3, 56, 56, 24, 120), (16, 20, 16, 8, 16, 32),
    (4, 2, 5, 5, 20, 48), (8, 2, 9, 13, 20, 48), (2, 2, 14, 14, 20, 48), (4, 2, 3, 57, 20, 48), (8, 2, 6, 100, 20, 48), (4, 1, 5, 252, 20, 24),
])
def test_3x3_on_the_fma_kernels(g, n, h, w, cin, cout):
    d, ref, s = inputs(n, h, w, cin, cout, 3, g, 50)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
    for layout in ("nhwc", "cm", "cm-cm") if w <= 224 else ("nhwc",):
        got = run(p, d, layout, 0, 1)
        assert np.all(np.abs(got.astype(np.float64) - ref.reshape(got.shape)) <= 1e-5 * s.reshape(got.shape))
        assert np.array_equal(got, run(p, d, layout, 0, 1))             # split tiles are summed in the same order every time


@gpu
@pytest.mark.parametrize("g", [1, 4, 8, 16])
@pytest.mark.parametrize("taps", [2, 4, 7])
def test_3x3_patterns_on_the_fma_kernels(g, taps):
    """Tap lists (few taps) and the whole-kernel loop (many) on whole and odd heights."""
    for n, h in ((6, 28), (5, 7)):
        d = dict(inputs(n, h, 28, 40, 64, 3, g, 30)[0])
        d["mask"] = tap_pattern_mask(2, 19, d["mask"][::g, 0, 0, :].astype(bool), g, taps)
        p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g, tap_patterns=True)
        ref, s = R.conv2d(d["x"], d["w"], d["mask"], d["bias"], relu=False)
        for tile in (0, 64):
            got = run(p, d, "nhwc", tile, 1)
            assert np.all(np.abs(got.astype(np.float64) - ref.reshape(got.shape)) <= 1e-5 * s.reshape(got.shape))


@gpu
def test_the_library_s_own_choice():
    """Wide and half-pruned layers run on the tensor cores, nearly empty ones and non-finite ones on the FMA kernels; a first
    call during a capture cannot build the images and runs on the FMA kernels."""
    def route(n, hw, cin, cout, k, g, pct, poke=None):
        d = WL.single_conv_inputs(1, 1, 1, cin, cout, k, g, pct, 3, 0.05, 0.05)
        if poke is not None:
            d["w"][0, 0, 0, np.argmax(d["mask"][0, 0, 0])] = poke
        p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
        x, y = torch.zeros((n, hw, hw, cin), device="cuda"), torch.empty((n, hw, hw, cout), device="cuda")
        (sbnn.conv1x1_gs if k == 1 else sbnn.conv3x3_gs)(p, x, y, n, hw, hw)
        return sbnn.debug_last_route()

    assert route(64, 14, 1024, 1024, 1, 4, 50)[0] in (128, 256)
    assert route(8, 28, 256, 256, 3, 4, 50)[0] in (64, 128, 256)
    assert route(5, 7, 512, 512, 3, 8, 70)[1] > 1
    assert route(32, 28, 256, 256, 3, 8, 90) == (0, 0)
    assert route(64, 14, 1024, 1024, 1, 4, 50, np.inf) == (0, 0)

    d, ref, s = inputs(7, 61, 63, 64, 124, 1, 4, 50)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], 4)
    x, y = torch.from_numpy(d["x"]).cuda(), torch.empty(ref.shape, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        sbnn.conv1x1_gs(p, x, y, 7, 61, 63, 0)
        assert sbnn.debug_last_route() == (0, 0)
    graph.replay()
    torch.cuda.synchronize()
    assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - ref) <= 1e-5 * s)
    sbnn.conv1x1_gs(p, x, y, 7, 61, 63, 0)
    assert sbnn.debug_last_route()[0] != 0


@gpu
@pytest.mark.parametrize("value", [-np.inf, np.inf, np.nan])
def test_a_bias_that_is_not_finite_costs_nothing(value):
    """A channel switched off by its bias: the layer runs on the FMA kernels, where such a bias is a number like any other (on
    the tensor cores it would look like a bad activation in every pixel, and have every pixel summed again)."""
    d, ref, s = inputs(7, 61, 63, 64, 124, 1, 4, 50)
    bias = d["bias"].copy()
    bias[0] = value
    p = sbnn.pack_weights(d["w"], d["mask"], bias, 4)
    x, y = torch.from_numpy(d["x"]).cuda(), torch.empty(ref.shape, device="cuda")
    sbnn.conv1x1_gs(p, x, y, 7, 61, 63, 0)
    assert sbnn.debug_last_route() == (0, 0)
    got = y.cpu().numpy()
    assert np.array_equal(got[..., 0], np.full(got.shape[:-1], value, np.float32), equal_nan=True)
    assert np.all(np.abs(got[..., 1:].astype(np.float64) - ref[..., 1:]) <= 1e-5 * s[..., 1:])


# ---- infinities, NaN and sums beyond fp32 ------------------------------------------------------------------------------
def same_kind(got, want, s):
    """NaN where `want` (the FMA kernels' result) has NaN, the same infinities, the rest within both kernels' bounds."""
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    f = np.isfinite(want)
    assert np.all(np.abs(got[f].astype(np.float64) - want[f]) <= 2e-5 * s[f])


def spoil(x, how):
    rng = np.random.default_rng(5)
    x = x.copy().reshape(-1, x.shape[-1])
    if how == "all":
        x[:] = np.nan
    elif how == "one per pixel":
        x[np.arange(len(x)), rng.integers(0, x.shape[1], len(x))] = np.inf
    elif how == "both signs":
        bad = rng.random(x.shape) < 0.01
        x[bad] = np.where(rng.random(x.shape) < 0.5, np.inf, -np.inf)[bad]
    else:
        x[len(x) // 3, 1], x[len(x) // 2, 0], x[-1, -1] = np.nan, np.inf, -np.inf
    return x


@gpu
@pytest.mark.parametrize("how", ["three", "one per pixel", "both signs", "all"])
@pytest.mark.parametrize("k,layout,tile,split", [(1, "nhwc", 256, 1), (1, "cm-cm", 128, 1), (1, "cm", 64, 4), (3, "nhwc", 128, 1), (3, "cm-cm", 64, 1),
                                                 (3, "nhwc", 64, 8), (1, "cm-cm", 64, 3), (3, "nhwc", 64, 7), (3, "cm", 64, 5)])
def test_bad_activations_spoil_what_they_touch_and_little_time(k, layout, tile, split, how):
    """The same outputs are infinite or NaN as on the FMA kernels, the others keep their values, and the call does not take
    many times what it takes there (at most seven times, when every pixel has a bad channel; summed by a thread a pixel it was a hundred times)."""
    n, h, w, cin, cout, g = (6, 25, 31, 1024, 516, 4) if k == 1 else (12, 28, 27, 260, 136, 8)
    if split > 1:
        n, h, w = 1, 17, 19
    d = WL.single_conv_inputs(n, h, w, cin, cout, k, g, 50, 11, 0.05, 0.05)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
    d = dict(d, x=spoil(d["x"], how).reshape(d["x"].shape))
    want = run(p, d, layout, 0, 1)
    s = np.broadcast_to(np.abs(d["bias"]) + np.abs(d["w"] * d["mask"]).reshape(cout, -1).sum(1), want.shape)      # (activations are below 1)
    for flags in (0, sbnn.SBNN_RELU):
        same_kind(run(p, d, layout, tile, split, flags), np.fmax(want, 0) if flags else want, s)
    m = n * h * w
    xt = torch.from_numpy(d["x"].reshape(m, cin)).cuda()
    cm = layout != "nhwc"
    ld = (m + 3) // 4 * 4
    x = torch.zeros((cin, ld), device="cuda") if cm else xt
    if cm:
        x[:, :m] = xt.T
    y = torch.empty(max(ld, m) * cout, device="cuda")
    ldy = (ld if layout == "cm-cm" else cout) if cm else 0

    def us(tile, split):
        best = 1e30
        for _ in range(3):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sbnn.debug_conv_gs(p, x, ld if cm else 0, y, ldy, n, h, w, sbnn.SBNN_OUT_CM if layout == "cm-cm" else 0, tile, split)
            b.record()
            b.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
        return best

    base, bad = us(0, 1), us(tile, split)
    print(f"{k} {layout} {tile} {split} {how}: FMA {base:.0f} us, tensor cores {bad:.0f} us")
    assert bad <= 10 * base
    sbnn.get_async_status()


@gpu
@pytest.mark.parametrize("taps", [4, 7])
@pytest.mark.parametrize("layout,tile,split", [("nhwc", 128, 1), ("cm-cm", 64, 1), ("nhwc", 64, 4)])
def test_bad_activations_under_pruned_taps(layout, tile, split, taps):
    """What a pruned tap sees: nothing in layers that run from tap lists (4 taps), its product with zero in others (7)."""
    d, _, s = inputs(6, 28, 28, 40, 64, 3, 4, 30)
    d = dict(d, mask=tap_pattern_mask(2, 19, d["mask"][::4, 0, 0, :].astype(bool), 4, taps), x=spoil(d["x"], "one per pixel").reshape(d["x"].shape))
    d["x"].reshape(-1, 40)[::3] = 0.25
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], 4, tap_patterns=True)
    want = run(p, d, layout, 0, 1)
    assert np.isfinite(want).any() and not np.isfinite(want).all()
    same_kind(run(p, d, layout, tile, split), want, s.reshape(want.shape))


@gpu
@pytest.mark.parametrize("layout,tile,split", [("nhwc", 64, 1), ("nhwc", 256, 1), ("cm-cm", 128, 1), ("nhwc", 64, 2), ("nhwc", 64, 3),
                                               ("cm-cm", 64, 6)])
def test_sums_that_overflow_on_the_way(layout, tile, split):
    """fp32 sums depend on their order near the end of the range: where the tensor cores' order overflows in any channel, the
    order of the FMA kernels (products ascending, bias last) decides."""
    d = WL.single_conv_inputs(3, 27, 29, 516, 260, 1, 4, 0, 3, 0.05, 0.05)       # (from 2048 pixels on the NHWC route adds the bias last, too)
    w, x, bias = np.zeros_like(d["w"]), np.ones_like(d["x"]), np.zeros(260, np.float32)
    for o in (5, 70, 131, 258):                                # 3e38 + (1e38 - 3e38): not finite from the left
        w[o, 0, 0, 3], w[o, 0, 0, 300], bias[o] = 1e38, -3e38, 3e38
    d = dict(d, w=w, x=x, bias=bias)
    p = sbnn.pack_weights(w, d["mask"], bias, 4)
    want = run(p, d, layout, 0, 1)
    assert np.isfinite(want).all()
    assert np.allclose(run(p, d, layout, tile, split), want, rtol=1e-5, atol=0)


@gpu
@pytest.mark.parametrize("k", [1, 3])
def test_images_that_do_not_fit_the_device(k):
    """The images of a sparse layer can be many times its stored weights: without room for them it runs as it is stored."""
    n, h, w, cin, cout, g, pct = SHAPES_3X3[1] if k == 3 else (7, 61, 63, 100, 516, 4, 30)
    d, ref, s = inputs(n, h, w, cin, cout, k, g, pct)
    p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
    x, y = torch.from_numpy(d["x"]).cuda(), torch.empty(ref.shape, device="cuda")
    call = sbnn.conv1x1_gs if k == 1 else sbnn.conv3x3_gs
    call(p, x, y, n, h, w, 0)
    assert sbnn.debug_last_route()[0] != 0
    q = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
    sbnn.debug_limit_images(q, 1000)
    sbnn.prepare(q, n, h, w)
    call(q, x, y, n, h, w, 0)
    assert sbnn.debug_last_route() == (0, 0)
    assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - ref) <= 1e-5 * s)
    if k == 1:
        call(q, x, y, n, h, w, sbnn.SBNN_BF16_TC)
        assert sbnn.debug_last_route() == (0, 0)
        assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - ref) <= 1e-2 * s)


@gpu
def test_prepared_calls_build_nothing():
    """A call prepared for some number of pixels runs the same way in a capture, where nothing can be built, as outside, for
    every smaller number.  (The choice follows whole rounds of tiles: 96 -> 512 at 90 % gains on 2443 and 18749 pixels, say, but
    not on 19256, nor a half or a quarter of that.)"""
    for cin, cout, g, pct, top in ((96, 512, 4, 90, 19256), (80, 512, 8, 90, 4964), (96, 96, 8, 90, 37915)):
        d = WL.single_conv_inputs(1, 1, 1, cin, cout, 1, g, pct, 3, 0.05, 0.05)
        p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
        sbnn.prepare(p, 1, 1, top)
        ld = (top + 3) // 4 * 4
        x, y = torch.zeros((cin, ld), device="cuda"), torch.empty((cout, ld), device="cuda")
        for m in range(1, top, 331):
            captured = []
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
                sbnn.conv1x1_gs_cm(p, x, ld, y, ld, m, sbnn.SBNN_OUT_CM)
                captured.append(sbnn.debug_last_route())
            del graph
            sbnn.conv1x1_gs_cm(p, x, ld, y, ld, m, sbnn.SBNN_OUT_CM)
            assert [sbnn.debug_last_route()] == captured, m
        torch.cuda.synchronize()
