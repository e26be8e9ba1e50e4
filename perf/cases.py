"""Performance cases: what programs that use this library ask of it, through the package's public functions.

A program converts its pruned layers once (`pack_weights`), lets the library set itself up (`prepare`, `MobileNetV1`),
and then calls layers or the whole network on device tensors.  A case is one such call.  Shapes come from the
benchmark configurations and the test suite: the layers of MobileNet-v1 at 224 x 224, the sparsity sweep on 1024 -> 1024
channels, 3x3 layers of ImageNet networks; densities from dense to 90 % pruned; groups of 4 and 8 output channels.
"""
import math

import numpy as np
import torch

import paper_2310_19509_b200 as sbnn


def listed():
    return [
        # One thin layer of one image: the smallest call, where launch and host latency count.
        dict(name="pw-b1-56-64-128-s50", op="pw", n=1, hw=56, cin=64, cout=128, g=4, pct=50),
        # A wide layer of a large batch, half pruned: the middle of the sparsity sweep.
        dict(name="pw-b256-14-1024-1024-s50", op="pw", n=256, hw=14, cin=1024, cout=1024, g=4, pct=50),
        # Layers chained on the device in the channel-major layout, heavily pruned, an odd batch.
        dict(name="pwcm-b101-14-1024-512-s90", op="pwcm", n=101, hw=14, cin=1024, cout=512, g=8, pct=90),
        # The bf16 mode of the wide layer, for programs that accept bf16 operands.
        dict(name="pwbf16-b256-14-1024-1024-s50", op="pwbf16", n=256, hw=14, cin=1024, cout=1024, g=8, pct=50),
        # A group-sparse 3x3 layer in the middle of a residual network, a serving batch.
        dict(name="c3-b32-28-256-256-s50", op="c3", n=32, hw=28, cin=256, cout=256, g=4, pct=50),
        # A deep 3x3 layer on a small odd map, a few images.
        dict(name="c3-b5-7-512-512-s70", op="c3", n=5, hw=7, cin=512, cout=512, g=8, pct=70),
        # A thin 3x3 layer on a large map, channel-major on both sides.
        dict(name="c3cm-b8-56-64-64-s30", op="c3cm", n=8, hw=56, cin=64, cout=64, g=4, pct=30),
        # A 3x3 layer pruned by connectivity and by four-tap kernel patterns.
        dict(name="c3pat-b32-28-256-256-s50", op="c3pat", n=32, hw=28, cin=256, cout=256, g=4, pct=50),
        # A dense depthwise layer in NHWC between layers of the caller's own.
        dict(name="dw-b64-56-128", op="dw", n=64, hw=56, c=128, stride=1),
        # The network on one image (interactive use), lightly pruned.
        dict(name="mbv1-b1-s30", op="mbv1", n=1, g=4, pct=30),
        # The network on an odd, small batch, strongly pruned.
        dict(name="mbv1-b9-s70", op="mbv1", n=9, g=4, pct=70),
        # The network at the serving batch of the benchmark.
        dict(name="mbv1-b64-s50", op="mbv1", n=64, g=4, pct=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_one(rng):
    op = rng.choice(["pw", "pw", "pwcm", "pwcm", "pwbf16", "c3", "c3", "c3cm", "c3pat", "dw", "mbv1", "mbv1"])
    g, pct = rng.choice([4, 4, 8]), rng.choice([0, 30, 50, 50, 70, 90])
    if op == "mbv1":
        return dict(op=op, n=_log_int(rng, 1, 64), g=4, pct=rng.choice([0, 30, 50, 70]))
    n, hw = _log_int(rng, 1, 256), rng.choice([7, 13, 14, 14, 28, 28, 56, 112])
    if op == "dw":
        return dict(op=op, n=n, hw=hw, c=8 * _log_int(rng, 4, 128), stride=rng.choice([1, 2]))
    cin, cout = 4 * _log_int(rng, 8, 256), 8 * _log_int(rng, 4, 128)
    if op.startswith("c3"):
        cin, cout, hw = 4 * _log_int(rng, 8, 128), 8 * _log_int(rng, 4, 64), min(hw, 56)
    return dict(op=op, n=n, hw=hw, cin=cin, cout=cout, g=g, pct=pct)


def draw(rng):
    most = {c["name"]: work(c) for c in listed()}
    while True:
        case = _draw_one(rng)
        w, cap = work(case), most["mbv1-b64-s50" if case["op"] == "mbv1" else "pw-b256-14-1024-1024-s50"]
        if all(w[k] <= cap[k] for k in w):
            return case


# ---- sizes ----------------------------------------------------------------------------------------

def _kept_counts(groups, cin, pct):
    """Kept input channels per group when pct % of all (group, channel) units are removed evenly."""
    removed = (pct * groups * cin + 50) // 100
    base, extra = divmod(removed, groups)
    return [cin - base - (1 if i < extra else 0) for i in range(groups)]


def _network_layers():
    """(layer, input side, input channels, output side, output channels) of the network's 29 layers."""
    return [(i, *sbnn.mobilenet_v1_layer_shape(i)) for i in range(29)]


def _conv_work(m, cin, cout, g, pct, taps, kept_taps):
    units = sum(_kept_counts(cout // g, cin, pct))
    weights = units * (4 + 4 * g * kept_taps + (2 if kept_taps != taps else 0)) + 4 * cout + 4 * (cout // g + 1)
    return {"bytes": 4 * m * (cin + cout) + weights, "flops": 2 * units * g * kept_taps * m}


def work(case):
    op = case["op"]
    if op == "dw":
        n, hw, c, s = case["n"], case["hw"], case["c"], case["stride"]
        ho = (hw - 1) // s + 1
        return {"bytes": 4 * n * c * (hw * hw + ho * ho) + 40 * c, "flops": 18 * n * ho * ho * c}
    if op == "mbv1":
        # Layer by layer: every activation is an input and an output of layers that a program can also call singly.
        n, total = case["n"], {"bytes": 0, "flops": 0}
        for i, hin, cin, hout, cout in _network_layers():
            if i == 0:
                w = {"bytes": 4 * n * (hin * hin * cin + hout * hout * cout), "flops": 54 * n * hout * hout * cout}
            elif i == 27:
                w = {"bytes": 4 * n * cin * (hin * hin + 1), "flops": n * cin * hin * hin}
            elif i == 28:
                w = _conv_work(n, cin, cout, 4, 0, 1, 1)
            elif i % 2:
                w = {"bytes": 4 * n * cin * (hin * hin + hout * hout), "flops": 18 * n * hout * hout * cin}
            else:
                w = _conv_work(n * hin * hin, cin, cout, case["g"], case["pct"], 1, 1)
            total = {k: total[k] + w[k] for k in total}
        return total
    taps = 9 if op.startswith("c3") else 1
    return _conv_work(case["n"] * case["hw"] ** 2, case["cin"], case["cout"], case["g"], case["pct"], taps,
                      4 if op == "c3pat" else taps)


def tolerance(case):
    # About four times the distance of the results from the same sums taken in 64 bits: fp32 layers show rel 0.6e-7 to
    # 5.5e-7 (max 6e-6), the network 2.4e-7 (max 1e-6).  The bf16 mode defines how operands are rounded, so against sums
    # of the rounded operands it shows 5.8e-7 (max 4.3e-6) as well.
    return {"rel": 3e-6 if case["op"] == "pwbf16" else 2.2e-6, "max": 2.5e-5}


# ---- inputs ---------------------------------------------------------------------------------------

def _unit_mask(rng, groups, cin, pct):
    """Per group a uniform-random set of kept input channels, as connectivity pruning leaves them."""
    order = np.argsort(rng.random((groups, cin), dtype=np.float32), axis=1)
    kept = np.asarray(_kept_counts(groups, cin, pct))
    mask = np.zeros((groups, cin), bool)
    np.put_along_axis(mask, order, np.arange(cin)[None, :] < kept[:, None], axis=1)
    return mask


def _packed(rng, cin, cout, g, pct, k=1, sigma=0.05, b_sigma=0.05, four_taps=False):
    w = rng.standard_normal((cout, k, k, cin), dtype=np.float32) * np.float32(sigma)
    bias = rng.standard_normal(cout, dtype=np.float32) * np.float32(b_sigma)
    unit = _unit_mask(rng, cout // g, cin, pct)
    taps = np.broadcast_to(unit[:, None, None, :], (cout // g, k, k, cin))
    if four_taps:  # the centre and three of the other eight, the same for the filters of a group
        rank = np.argsort(np.argsort(rng.random((cout // g, cin, 8), dtype=np.float32), axis=2), axis=2)
        keep = np.insert(rank < 3, 4, True, axis=2)
        taps = taps & keep.transpose(0, 2, 1).reshape(cout // g, 3, 3, cin)
    mask = np.repeat(taps, g, axis=0).astype(np.uint8)
    return sbnn.pack_weights(w, mask, bias, g, tap_patterns=four_taps)


def _network(rng, n, g, pct):
    def device(shape, sigma):
        return torch.from_numpy(rng.standard_normal(shape, dtype=np.float32) * np.float32(sigma)).cuda()

    layers = _network_layers()
    pw = []
    for _, _, cin, _, cout in layers[2:27:2]:
        kept = cin * (100 - pct) / 100
        pw.append(_packed(rng, cin, cout, g, pct, sigma=math.sqrt(2 / kept), b_sigma=0.01))
    dw_w = [device((3, 3, cin), math.sqrt(2 / 9)) for _, _, cin, _, _ in layers[1:27:2]]
    dw_b = [device((cin,), 0.01) for _, _, cin, _, _ in layers[1:27:2]]
    fc = _packed(rng, 1024, 1000, 4, 0, sigma=math.sqrt(1 / 1024), b_sigma=0.01)
    return sbnn.MobileNetV1(pw, fc, dw_w, dw_b, device((32, 3, 3, 3), math.sqrt(2 / 27)), device((32,), 0.01), n)


def _round4(v):
    return (v + 3) // 4 * 4


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gpu = torch.Generator(device="cuda").manual_seed(seed)
    op, n = case["op"], case["n"]

    def activations(*shape):
        return torch.rand(shape, generator=gpu, device="cuda")

    if op == "mbv1":
        return dict(op=op, n=n, net=_network(rng, n, case["g"], case["pct"]), x=activations(n, 224, 224, 3),
                    y=torch.empty((n, 1000), device="cuda"))
    hw = case["hw"]
    if op == "dw":
        c, s = case["c"], case["stride"]
        ho = (hw - 1) // s + 1
        return dict(op=op, n=n, hw=hw, c=c, stride=s, x=activations(n, hw, hw, c), y=torch.empty((n, ho, ho, c), device="cuda"),
                    w=torch.randn((3, 3, c), generator=gpu, device="cuda") * math.sqrt(2 / 9),
                    b=torch.randn((c,), generator=gpu, device="cuda") * 0.01)
    cin, cout, m = case["cin"], case["cout"], n * hw * hw
    layer = _packed(rng, cin, cout, case["g"], case["pct"], 3 if op.startswith("c3") else 1,
                    sigma=0.02 if op.startswith("c3") or cin > 512 else 0.05, four_taps=op == "c3pat")
    sbnn.prepare(layer, n, hw, hw, sbnn.SBNN_BF16_TC if op == "pwbf16" else 0)
    state = dict(op=op, n=n, hw=hw, layer=layer)
    if op in ("pwcm", "c3cm"):
        ld = _round4(m)
        return dict(state, m=m, ld=ld, x=activations(cin, ld), y=torch.zeros((cout, ld), device="cuda"))
    return dict(state, x=activations(n, hw, hw, cin), y=torch.empty((n, hw, hw, cout), device="cuda"))


def run(state):
    op, n, x, y = state["op"], state["n"], state["x"], state["y"]
    if op == "mbv1":
        state["net"].forward(x, y, n)
        return y
    hw = state["hw"]
    if op == "pw":
        sbnn.conv1x1_gs(state["layer"], x, y, n, hw, hw)
    elif op == "pwbf16":
        sbnn.conv1x1_gs(state["layer"], x, y, n, hw, hw, sbnn.SBNN_RELU | sbnn.SBNN_BF16_TC)
    elif op == "pwcm":
        sbnn.conv1x1_gs_cm(state["layer"], x, state["ld"], y, state["ld"], state["m"], sbnn.SBNN_RELU | sbnn.SBNN_OUT_CM)
        return y[:, :state["m"]]
    elif op == "c3cm":
        sbnn.conv3x3_gs_cm(state["layer"], x, state["ld"], y, state["ld"], n, hw, hw, sbnn.SBNN_RELU | sbnn.SBNN_OUT_CM)
        return y[:, :state["m"]]
    elif op == "dw":
        sbnn.dwconv3x3(state["w"], state["b"], x, y, n, hw, hw, state["c"], state["stride"])
    else:
        sbnn.conv3x3_gs(state["layer"], x, y, n, hw, hw)
    return y
