#!/usr/bin/env python
"""Benchmark of the group-sparse convolution path on B200.

Default workload: MobileNet-v1 (width 1.0, 224x224x3, fp32), batch 64 per GPU, the 13 pointwise
layers group-sparse with G=4 at 50 % sparsity, synthetic seeded weights and images.  One step is
one forward pass of the whole chain.  Prints ONE JSON line (rank 0).

  python bench.py --gpus 1 --steps 20 --warmup 5
  python -m torch.distributed.run --nproc-per-node N ... bench.py --gpus N ...   (batch-sharded replicas)
  python bench.py --impl reference       (the CPU oracle on a bounded sample, host cores)
  python bench.py --sweep                (extra lines: single-layer configs and dense library baselines)
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

FP32_PEAK_TFLOPS = 148 * 128 * 2 * 1.965e9 / 1e12   # 148 SMs x 128 FP32 lanes x 2 flop x max SM clock
HBM_FALLBACK_GBS = 6650.0
BF16_FALLBACK_TFLOPS = 1590.0
METRIC = "mobilenet_v1_images_per_s"
# DRAM bytes (read + write) of the 13 pointwise launches (five of them with a depthwise layer) of one default step, from the ncu capture summarised in
# profiles/bench_mobilenet_v1_b64_s50_launch_list.md, and the SHA-1 of the kernel source the capture was taken with:
# the figure is reported only while the kernel source still has that hash.
PW_DRAM_BYTES_PER_STEP = 1018.8e6
PW_DRAM_KERNEL_SHA1 = "f95dfd04ebd49c5efc51b9ca5c73fad2cb143e5c"
PW_KERNEL_SOURCES = tuple("paper_2310_19509_b200/csrc/" + f for f in ("conv_tc.cu", "tcgen05.cuh", "conv1x1_cm.cu", "pipeline.cuh"))


def kernel_source_sha1():
    import hashlib
    h = hashlib.sha1()
    for rel in PW_KERNEL_SOURCES:
        with open(os.path.join(ROOT, rel), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


def measured_peaks():
    """(HBM GB/s, bf16 dense TFLOP/s burst, 'measured' | 'fallback')."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        try:
            d = json.load(open(p))
            return float(d["hbm_gbs"]), float(d.get("bf16_tflops", BF16_FALLBACK_TFLOPS)), "measured"
        except Exception:
            pass
    return HBM_FALLBACK_GBS, BF16_FALLBACK_TFLOPS, "fallback"


# ------------------------------------------------------------------------------------------
# algorithmic work of a layer (flops on kept weights only; every activation read/written once)
# ------------------------------------------------------------------------------------------
def layer_work(L, batch):
    kind, hin, ci, co, s = L["kind"], L["hin"], L["cin"], L["cout"], L["stride"]
    ho = hin // s if kind in ("conv0", "dw") else (1 if kind in ("pool", "fc") else hin)
    m = batch * ho * ho
    if kind == "conv0":
        return 2.0 * m * 27 * co, 4.0 * (batch * hin * hin * ci + m * co + 27 * co + co)
    if kind == "dw":
        return 2.0 * m * 9 * ci, 4.0 * (batch * hin * hin * ci + m * ci + 10 * ci)
    if kind in ("pw", "fc"):
        g = L["g"]
        units = int(L["mask"].sum()) // g
        return 2.0 * m * g * units, 4.0 * (m * (ci + co) + units * (1 + g) + co + co // g + 1)
    return float(batch * 49 * ci), 4.0 * (batch * 49 * ci + batch * ci)   # pool


class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index, self.proc = index, None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.15)
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out = ""
        sm, mx, reasons = [], [], set()
        for line in out.splitlines():
            f = [t.strip() for t in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for name, v in zip(("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"), f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "samples": len(sm), "reasons": sorted(reasons)}


# ------------------------------------------------------------------------------------------
# CPU oracle timing (baseline only; the oracle is never tuned for this)
# ------------------------------------------------------------------------------------------
def oracle_forward_seconds(x1, layers):
    """Wall time of the oracle's chained forward for the images in x1."""
    from oracle import reference as R
    t0 = time.perf_counter()
    R.mobilenet_v1_forward(x1, layers)
    return time.perf_counter() - t0


def cpu_baseline(x, layers):
    from oracle import reference as R
    R.num_threads()                      # loads the library outside the timed part
    n = min(len(x), 32)
    dt = oracle_forward_seconds(x[:n], layers)
    return {"value": n / dt, "unit": "images/s", "cores": R.num_threads(), "kind": "oracle",
            "sample": f"{n} images of the batch through the whole chain (error-bound pass included), {dt:.1f} s"}


def run_reference(args, rank):
    """The reference arm: the CPU oracle as it stands, on host cores, one image per step."""
    if rank != 0:
        return
    from oracle import reference as R
    from sbnn_inputs import mobilenet_v1_inputs
    x, layers = mobilenet_v1_inputs(1, args.sparsity, 4, seed=0)
    for _ in range(min(args.warmup, 1)):
        oracle_forward_seconds(x, layers)
    steps = max(1, min(args.steps, 10))
    t0 = time.perf_counter()
    for _ in range(steps):
        oracle_forward_seconds(x, layers)
    dt = (time.perf_counter() - t0) / steps
    v = 1.0 / dt
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "images/s", "n_gpus": args.gpus,
            "steps": steps, "warmup": min(args.warmup, 1), "ms_per_step": dt * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": f"MobileNet-v1 224x224x3, pointwise G=4 sparsity {args.sparsity}%, "
                                   "bounded sample: 1 image per step on host cores"},
            "cpu_baseline": {"value": v, "unit": "images/s", "cores": R.num_threads(), "kind": "oracle",
                             "sample": "1 image per step through the whole chain"},
            "e2e": {"value": v, "unit": "images/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)


# ------------------------------------------------------------------------------------------
# GPU arm
# ------------------------------------------------------------------------------------------
def build_network(sbnn, torch, layers, batch):
    pw = [sbnn.pack_weights(L["w"], L["mask"], L["bias"], L["g"]) for L in layers if L["kind"] == "pw"]
    fcL = [L for L in layers if L["kind"] == "fc"][0]
    fc = sbnn.pack_weights(fcL["w"], fcL["mask"], fcL["bias"], fcL["g"])
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    dw_w = [t(L["w"]) for L in layers if L["kind"] == "dw"]
    dw_b = [t(L["bias"]) for L in layers if L["kind"] == "dw"]
    return sbnn.MobileNetV1(pw, fc, dw_w, dw_b, t(layers[0]["w"]), t(layers[0]["bias"]), batch)


def time_layers(sbnn, torch, net, layers, batch, reps, flush):
    """Every layer alone, as forward launches it (channel-major buffers of its own shape), CUDA events, L2 flushed
    between launches."""
    res = []
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for li, L in enumerate(layers):
        hin, cin, hout, cout = sbnn.mobilenet_v1_layer_shape(li)
        r4 = lambda v: (v + 3) // 4 * 4  # noqa: E731
        if L["kind"] == "conv0":
            xin = torch.rand((batch, hin, hin, cin), device="cuda")
        else:
            xin = torch.rand((cin, r4(batch * hin * hin)), device="cuda")
        if L["kind"] == "fc":
            yout = torch.empty((batch, cout), device="cuda")
        else:
            yout = torch.empty((cout, r4(batch * hout * hout)), device="cuda")
        for _ in range(3):
            net.run_layer_cm(li, xin, yout, batch)
        ts = []
        for _ in range(reps):
            flush.add_(1.0)
            ev0.record()
            net.run_layer_cm(li, xin, yout, batch)
            ev1.record()
            ev1.synchronize()
            ts.append(ev0.elapsed_time(ev1) * 1e-3)
        fl, by = layer_work(L, batch)
        sparse = L["kind"] in ("pw", "fc")
        res.append({"name": L["name"], "kind": L["kind"], "s": float(np.median(ts)), "flops": fl, "bytes": by,
                    "tile": sbnn.debug_last_route()[0] if sparse else 0, "dense_flops": 2.0 * batch * hout * hout * cin * cout if sparse else 0.0})
        del xin, yout
    return res


def time_layers_in_chain(sbnn, torch, net, layers, batch, xd, reps):
    """Cost of every layer inside a step: T(layers 0..l) - T(layers 0..l-1), where each prefix of the chain is recorded
    into a CUDA graph (the way forward runs) and replayed back to back, CUDA events around `reps` replays, median of 3.
    A pointwise layer that runs in one launch with the depthwise layer in front gets the time of both, that layer zero.
    The 29 figures add up to the time of the whole chain, so they include what a kernel costs its neighbours (launch
    gap, cold pipeline) and nothing that a step does not pay."""
    r4 = lambda v: (v + 3) // 4 * 4  # noqa: E731
    out = torch.empty(64 * r4(batch * 112 * 112) + 4096, device="cuda")
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    prefix = []
    for l in range(len(layers)):
        net.forward_prefix(xd, out, batch, l)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            net.forward_prefix(xd, out, batch, l)
        for _ in range(3):
            g.replay()
        runs = []
        for _ in range(3):
            torch.cuda.synchronize()
            ev0.record()
            for _ in range(reps):
                g.replay()
            ev1.record()
            ev1.synchronize()
            runs.append(ev0.elapsed_time(ev1) * 1e-3 / reps)
        prefix.append(float(np.median(runs)))
        del g
    # (a difference can come out at or below zero when timing noise exceeds a very short layer: floor of 10 ns)
    times = [max(prefix[0], 1e-8)] + [max(prefix[l] - prefix[l - 1], 1e-8) for l in range(1, len(layers))]
    for l in joined_layers(net, layers, batch):
        times[l - 1], times[l] = 0.0, prefix[l] - prefix[l - 2]
    return times


def joined_layers(net, layers, batch):
    """Pointwise layers that forward runs in one launch with the depthwise layer in front of them."""
    return [l for l, L in enumerate(layers) if L["kind"] == "pw" and net.debug_launches(batch, l) == net.debug_launches(batch, l - 2) + 1]


def layer_pixels(sbnn, l):
    return sbnn.mobilenet_v1_layer_shape(l)[0] ** 2


def sweep_oracle_lines():
    """The oracle timed on the host cores for each distinct single-layer shape of the sweep (it does not skip zeros,
    so sparsity and G do not change its work): one warm-up, one timed run, on a bounded number of images and scaled
    to the configuration's batch.  A baseline beside the GPU lines, nothing more."""
    from oracle import reference as R
    from sbnn_inputs import workloads as WL
    cases = [("config1", WL.config1(), 1, 1), ("config4", WL.config4(n=4), 4, 32),
             ("config5", WL.config5(4, 50, n=8), 8, 256)]
    for name, d, n_timed, n_full in cases:
        for rep in range(2):
            t0 = time.perf_counter()
            R.conv2d(d["x"], d["w"], d["mask"], d["bias"], relu=True)
            dt = time.perf_counter() - t0
        print(json.dumps({"case": name, "impl": "oracle (fp64, dense over masked weights)", "cores": R.num_threads(),
                          "sample": f"{n_timed} of {n_full} images, scaled", "us": dt * 1e6 * n_full / n_timed}), flush=True)


def measure_fma_peak(sbnn, torch):
    """FP32 rate of the register-only packed-FMA kernel of the library (TFLOP/s), best of 5 launches of about 1 ms."""
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = 0.0
    for rep in range(7):
        ev0.record()
        flop = sbnn.selftest_fma_rate(4000)
        ev1.record()
        ev1.synchronize()
        if rep >= 2:
            best = max(best, flop / (ev0.elapsed_time(ev1) * 1e-3) / 1e12)
    return best


def _time_fn(torch, fn, reps, flush):
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(3):
        fn()
    ts = []
    for _ in range(reps):
        flush.add_(1.0)
        ev0.record()
        fn()
        ev1.record()
        ev1.synchronize()
        ts.append(ev0.elapsed_time(ev1) * 1e-3)
    return float(np.median(ts))


def dense_library_us(torch, m, cin, cout, k, shape4, reps, flush):
    """Dense library times of one layer shape, microseconds: cuDNN conv2d on channels-last tensors and, for 1x1, cuBLAS
    addmm on [M][Cin] x [Cin][Cout], each with TF32 off (like for like with the fp32 kernels) and on (context)."""
    n, h, w = shape4
    x = torch.rand((n, h, w, cin), device="cuda")
    xt = x.permute(0, 3, 1, 2)
    wt = torch.randn(cout, cin, k, k, device="cuda").contiguous(memory_format=torch.channels_last)
    b = torch.randn(cout, device="cuda")
    out = {}
    for tag, tf32 in (("fp32", False), ("tf32", True)):
        torch.backends.cudnn.allow_tf32 = tf32
        torch.backends.cuda.matmul.allow_tf32 = tf32
        out[f"cudnn_{tag}_us"] = round(_time_fn(torch, lambda: torch.relu_(torch.nn.functional.conv2d(xt, wt, b, padding=(k - 1) // 2)),
                                                reps, flush) * 1e6, 1)
        if k == 1:
            x2, w2 = x.reshape(m, cin), wt.reshape(cout, cin).t().contiguous()
            out[f"cublas_{tag}_us"] = round(_time_fn(torch, lambda: torch.relu_(torch.addmm(b, x2, w2)), reps, flush) * 1e6, 1)
    torch.backends.cudnn.allow_tf32 = False
    torch.backends.cuda.matmul.allow_tf32 = False
    return out


def single_layer_lines(sbnn, torch, flush, hbm_gbs, bf16_tflops, reps):
    """The single-layer configurations (config 1, config 4, the ten config-5 cases in fp32 and in the bf16 tensor-core
    mode) through the NHWC entry points, beside dense cuDNN / cuBLAS of the same shape.  fp32 fractions are against
    max(flops, bytes / HBM), flops = the nonzero ones / FP32 peak, or those of the unpruned layer / a sixth of the bf16 peak where
    that is less; bf16 fractions against max(nonzero flop / bf16 tensor peak, bytes / HBM)."""
    from sbnn_inputs import workloads as WL
    out, dense = [], {}

    def one(name, d, k, flags, mode, tap_mask=None):
        x = d["x"]
        n, h, w, cin = x.shape
        cout, g = d["w"].shape[0], d["g"]
        m = n * h * w
        if tap_mask is not None:     # kernels pruned tap by tap on top of the unit mask (packed with their patterns)
            p = sbnn.pack_weights(d["w"], tap_mask, d["bias"], g, tap_patterns=True)
        else:
            p = sbnn.pack_weights(d["w"], d["mask"], d["bias"], g)
        xd = torch.from_numpy(x).cuda()
        yd = torch.empty((n, h, w, cout), device="cuda")
        fn = (lambda: sbnn.conv3x3_gs(p, xd, yd, n, h, w, flags)) if k == 3 else (lambda: sbnn.conv1x1_gs(p, xd, yd, n, h, w, flags))
        t = _time_fn(torch, fn, reps, flush)
        sbnn.get_async_status()
        units = int(d["unit_mask"].sum())
        taps = k * k if tap_mask is None else int(tap_mask.sum()) / float(g * units)   # kept taps per kept kernel
        flops = 2.0 * m * g * taps * units
        byts = 4.0 * (m * (cin + cout) + units * (1 + g * taps) + cout + cout // g + 1)
        tile = sbnn.debug_last_route()[0]
        t_hbm = byts / (hbm_gbs * 1e9)
        t_fma, t_tensor = flops / (FP32_PEAK_TFLOPS * 1e12), 6 * 2.0 * m * cin * cout * k * k / (bf16_tflops * 1e12)
        t_alu = flops / (bf16_tflops * 1e12) if mode == "bf16_tc" else min(t_fma, t_tensor)
        limit = "tensor" if mode == "bf16_tc" or t_tensor < t_fma else "alu"
        rec = {"case": name, "mode": mode, "G": g, "sparsity_pct": d["sparsity_pct"], "us": round(t * 1e6, 1),
               "tflops_nonzero": round(flops / t / 1e12, 2), "roofline_us": round(max(t_alu, t_hbm) * 1e6, 1),
               "frac": round(max(t_alu, t_hbm) / t, 3), "bound": limit if t_alu > t_hbm else "hbm",
               "kernel": "FMA" if not tile and mode == "fp32" else ("gathered bf16" if not tile else f"conv_tc, {tile} channels a tile")}
        if k == 1 and mode == "fp32" and cin >= 128:
            # the same layer in the kernel's own layout (channel-major in and out, as the MobileNet chain calls it): no
            # conversion pass, row-contiguous output
            ld = (m + 3) // 4 * 4
            xt, yt = torch.empty((cin, ld), device="cuda"), torch.empty((cout, ld), device="cuda")
            sbnn.to_channel_major(xd, xt, m, cin, ld)
            tc = _time_fn(torch, lambda: sbnn.conv1x1_gs_cm(p, xt, ld, yt, ld, m, flags | sbnn.SBNN_OUT_CM), reps, flush)
            sbnn.get_async_status()
            rec["us_channel_major"] = round(tc * 1e6, 1)
            rec["frac_channel_major"] = round(max(t_alu, t_hbm) / tc, 3)
            del xt, yt
        if tap_mask is not None:
            rec["kept_taps_per_kernel"] = round(taps, 2)
        if k == 3 and w % 4 == 0 and tap_mask is None:
            # the 3x3 layer in the kernel's own layout (channel-major in and out): no conversion pass
            ld = (m + 3) // 4 * 4
            xt, yt = torch.empty((cin, ld), device="cuda"), torch.empty((cout, ld), device="cuda")
            sbnn.to_channel_major(xd, xt, m, cin, ld)
            tc = _time_fn(torch, lambda: sbnn.conv3x3_gs_cm(p, xt, ld, yt, ld, n, h, w, flags | sbnn.SBNN_OUT_CM), reps, flush)
            sbnn.get_async_status()
            rec["us_channel_major"] = round(tc * 1e6, 1)
            rec["frac_channel_major"] = round(max(t_alu, t_hbm) / tc, 3)
            del xt, yt
        key = (m, cin, cout, k)
        if key not in dense:
            dense[key] = dense_library_us(torch, m, cin, cout, k, (n, h, w), max(3, reps // 2), flush)
        rec.update(dense[key])
        out.append(rec)
        p.free()
        del xd, yd

    one("config1", WL.config1(), 1, sbnn.SBNN_RELU, "fp32")
    d4 = WL.config4()
    one("config4", d4, 3, sbnn.SBNN_RELU, "fp32")
    from sbnn_inputs import tap_pattern_mask
    one("config4_patterns_4_of_9_taps", d4, 3, sbnn.SBNN_RELU, "fp32", tap_mask=tap_pattern_mask(0, 19, d4["unit_mask"], 4, 4))
    del d4
    cases = [(g, sp) for g in (4, 8) for sp in (0, 30, 50, 70, 90)]
    for (g, sp), d in zip(cases, WL.config5_family(cases)):
        one(f"config5_G{g}_s{sp}", d, 1, sbnn.SBNN_RELU, "fp32")
        one(f"config5_G{g}_s{sp}", d, 1, sbnn.SBNN_RELU | sbnn.SBNN_BF16_TC, "bf16_tc")
    return out


def other_chain_configs(sbnn, torch, default_batch, default_sparsity):
    """The chain's other configurations (batch 64 at 70 %, batch 1 at 30 %): forward time by graph replay, inputs resident."""
    from sbnn_inputs import mobilenet_v1_inputs
    out = []
    for batch, sp in ((64, 70), (1, 30)):
        if (batch, sp) == (default_batch, default_sparsity):
            continue
        x, layers = mobilenet_v1_inputs(batch, sp, 4, seed=0)
        net = build_network(sbnn, torch, layers, batch)
        xd = torch.from_numpy(x).cuda()
        logits = torch.empty((batch, 1000), device="cuda")
        for _ in range(5):
            net.forward(xd, logits, batch)
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        reps = 100
        ev0.record()
        for _ in range(reps):
            net.forward(xd, logits, batch)
        ev1.record()
        ev1.synchronize()
        sbnn.get_async_status()
        ms = ev0.elapsed_time(ev1) / reps
        out.append({"batch": batch, "pointwise_sparsity_pct": sp, "ms_per_forward": round(ms, 4), "images_per_s": round(batch / ms * 1e3, 1)})
        net.free()
        del xd, logits
    return out


def max_over_ranks(values, world, device="cpu"):
    """Element-wise maximum of per-rank timings over the process group (the job is as slow as its slowest replica)."""
    if world <= 1:
        return [float(v) for v in values]
    import torch
    import torch.distributed as dist
    t = torch.tensor(values, device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t]


def job_throughput(per_rank_units, steps, world, seconds):
    """Whole-job rate of batch-sharded replicas: every rank processes per_rank_units per step, no exchange."""
    return per_rank_units * world * steps / seconds


def run_gpu(args, rank, world, local_rank):
    import torch
    import torch.distributed as dist

    import paper_2310_19509_b200 as sbnn
    from sbnn_inputs import mobilenet_v1_inputs

    sbnn.lib()                               # fails loudly if the CUDA library is missing
    torch.cuda.set_device(local_rank)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
    batch = args.batch
    x, layers = mobilenet_v1_inputs(batch, args.sparsity, 4, seed=rank)
    net = build_network(sbnn, torch, layers, batch)
    stream = torch.cuda.current_stream()
    xd = torch.from_numpy(x).cuda()
    logits = torch.empty((batch, 1000), device="cuda")

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    for _ in range(max(args.warmup, 3)):
        net.forward(xd, logits, batch)
    barrier()
    sampler = ClockSampler(local_rank)
    if rank == 0:
        sampler.start()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    barrier()
    ev0.record(stream)
    for _ in range(args.steps):
        net.forward(xd, logits, batch)
    ev1.record(stream)
    barrier()
    elapsed = ev0.elapsed_time(ev1) * 1e-3

    # end to end through the public binding: pinned host images in, logits back to the host, every step.  As a serving
    # loop would, the upload of step i+1 (copy stream, second input buffer) runs while step i computes.
    xh = torch.from_numpy(x).pin_memory()
    lh = [torch.empty((batch, 1000)).pin_memory() for _ in range(2)]
    xds = [xd, torch.empty_like(xd)]
    lds = [logits, torch.empty_like(logits)]
    copy_stream = torch.cuda.Stream()
    uploaded = [torch.cuda.Event() for _ in range(2)]
    consumed = [torch.cuda.Event() for _ in range(2)]

    def e2e_steps(n_steps):
        for i in range(n_steps):
            b = i & 1
            with torch.cuda.stream(copy_stream):
                if i >= 2:
                    copy_stream.wait_event(consumed[b])           # the forward that read this buffer two steps ago
                xds[b].copy_(xh, non_blocking=True)
                uploaded[b].record(copy_stream)
            stream.wait_event(uploaded[b])
            net.forward(xds[b], lds[b], batch)
            consumed[b].record(stream)
            lh[b].copy_(lds[b], non_blocking=True)

    e2e_steps(3)
    barrier()
    ev0.record(stream)
    copy_stream.wait_event(ev0)
    e2e_steps(args.steps)
    ev1.record(stream)
    barrier()
    e2e_elapsed = ev0.elapsed_time(ev1) * 1e-3
    clocks = sampler.stop() if rank == 0 else None

    elapsed, e2e_elapsed = max_over_ranks([elapsed, e2e_elapsed], world, "cuda")
    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return

    # per-layer timings for the roofline of the dominant kernel (the group-sparse 1x1)
    flush = torch.zeros(64 * 1024 * 1024, device="cuda")     # 256 MB > L2
    per = time_layers(sbnn, torch, net, layers, batch, args.layer_reps, flush)
    chain_t = time_layers_in_chain(sbnn, torch, net, layers, batch, xd, max(args.layer_reps, 10))
    for r, t in zip(per, chain_t):
        r["s_cold"], r["s"] = r["s"], t          # the roofline uses the in-step durations; the cold ones are reported beside
    step_flops = sum(r["flops"] for r in per)
    for l in joined_layers(net, layers, batch):  # one launch: the depthwise layer's output is not moved
        per[l]["bytes"] += per[l - 1]["bytes"] - 8.0 * batch * layer_pixels(sbnn, l) * sbnn.mobilenet_v1_layer_shape(l)[1]
        per[l]["s_cold"] += per[l - 1]["s_cold"]
        per[l - 1].update(bytes=0.0, flops=0.0)
    hbm_gbs, bf16_tflops, peak_kind = measured_peaks()
    fma_measured = measure_fma_peak(sbnn, torch)
    pw = [r for r in per if r["kind"] == "pw"]
    pw_t, pw_fl, pw_by = sum(r["s"] for r in pw), sum(r["flops"] for r in pw), sum(r["bytes"] for r in pw)
    pw_t_cold = sum(r["s_cold"] for r in pw)
    # Least time of a layer: its bytes, or its flops -- the kept ones on the FP32 pipe, or all of them, six bf16 products each,
    # on the tensor cores, whichever is less.
    tc_peak = bf16_tflops / 6
    t_flops = lambda r: min([r["flops"] / (FP32_PEAK_TFLOPS * 1e12)] + ([r["dense_flops"] / (tc_peak * 1e12)] if r["dense_flops"] else []))  # noqa: E731
    t_roof = lambda r: max(t_flops(r), r["bytes"] / (hbm_gbs * 1e9))  # noqa: E731
    total_layer_t = sum(r["s"] for r in per)
    on_tc, on_fma = [r for r in pw if r["tile"]], [r for r in pw if not r["tile"]]
    tc_t, tc_fl = sum(r["s"] for r in on_tc), sum(r["dense_flops"] for r in on_tc)
    tensor = tc_t > 0.5 * pw_t
    achieved, peak = (tc_fl / tc_t / 1e12, tc_peak) if tensor else (pw_fl / pw_t / 1e12, FP32_PEAK_TFLOPS)
    roofline = {
        "bound": "tensor" if tensor else "alu",
        "kernel": f"conv_tc_kernel ({len(on_tc)} of the 13 pointwise launches per step)" if tensor
                  else f"FMA kernels ({len(on_fma)} of the 13 pointwise launches per step)",
        "launches_on_tensor_cores": len(on_tc), "launches_on_fma_kernels": len(on_fma),
        "note": "tensor: flops of the unpruned layers, which is what the kernel multiplies, against a sixth of the measured bf16 rate (six "
                "bf16 products make an fp32 one), over the launches that run there, some of which compute a depthwise layer as well; alu: nonzero flops of all 13 against the FP32 FMA peak",
        "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
        "nonzero_tflops": pw_fl / pw_t / 1e12, "nonzero_frac_of_fp32_fma_peak": pw_fl / pw_t / 1e12 / FP32_PEAK_TFLOPS,
        "timing": "per layer: time of the chain's prefix up to and including the layer minus the prefix before it, each prefix a "
                  "CUDA graph replayed back to back under CUDA events (forward's launches and buffers, no flush); the 29 "
                  "figures add up to one whole forward; a pointwise layer that runs in one launch with the depthwise layer in front "
                  "(us 0) has the time of both, us_cold apart",
        "frac_cold": (sum(r["dense_flops"] for r in on_tc) / sum(r["s_cold"] for r in on_tc) if tensor else pw_fl / pw_t_cold) / 1e12 / peak,
        "frac_cold_note": "each layer launched alone after a 256 MB write has flushed L2",
        "peak_source": f"bf16 rate, {peak_kind}, divided by six" if tensor else "derived: 148 SMs x 128 FP32 lanes x 2 x 1.965 GHz",
        "fp32_fma_peak": FP32_PEAK_TFLOPS, "fp32_fma_peak_source": "derived: 148 SMs x 128 FP32 lanes x 2 x 1.965 GHz",
        "fp32_fma_measured": fma_measured,
        "fp32_fma_measured_note": "register-only fma.rn.f32x2 kernel of the library (sbnn_selftest_fma_rate) timed in this run",
        "traffic": PW_DRAM_BYTES_PER_STEP if (batch == 64 and args.sparsity == 50 and PW_DRAM_KERNEL_SHA1 == kernel_source_sha1()) else None,
        "algorithmic_bytes": pw_by,
        "mixed_frac": sum(t_roof(r) for r in pw) / pw_t,
        "mixed_note": f"sum over layers of max(min(nonzero flops/FP32 peak, flops/tensor peak), bytes/{hbm_gbs:.0f} GB/s {peak_kind}) / measured",
        "hbm_achieved_gbs": pw_by / pw_t / 1e9,
        "share_of_step": pw_t / total_layer_t,
        "whole_chain_frac": sum(t_roof(r) for r in per) / total_layer_t,
    }
    layers_out = [{"name": r["name"], "us": round(r["s"] * 1e6, 2), "us_cold": round(r["s_cold"] * 1e6, 2), "tflops": round(r["flops"] / max(r["s"], 1e-8) / 1e12, 2),
                   "gbs": round(r["bytes"] / max(r["s"], 1e-8) / 1e9, 1), "frac": round(t_roof(r) / max(r["s"], 1e-8), 3),
                   **({"tensor_core_tile": r["tile"]} if r["kind"] in ("pw", "fc") else {})} for r in per]

    if not args.no_dense:
        seen = {}
        for r, L in zip(per, layers):
            if L["kind"] != "pw":
                continue
            hin, cin, hout, cout = sbnn.mobilenet_v1_layer_shape(layers.index(L))
            key = (hout, cin, cout)
            if key not in seen:
                seen[key] = dense_library_us(torch, batch * hout * hout, cin, cout, 1, (batch, hout, hout), 5, flush)
            for lo in layers_out:
                if lo["name"] == r["name"]:
                    lo.update(seen[key])
        roofline["dense_library_us_per_step"] = {k: round(sum(lo.get(k, 0.0) for lo in layers_out if lo["name"].startswith("pw")), 1)
                                                 for k in ("cublas_fp32_us", "cublas_tf32_us", "cudnn_fp32_us", "cudnn_tf32_us")}
        roofline["pointwise_us_per_step"] = round(pw_t * 1e6, 1)
    single = single_layer_lines(sbnn, torch, flush, hbm_gbs, bf16_tflops, 7) if (world == 1 and not args.no_single) else None
    others = other_chain_configs(sbnn, torch, batch, args.sparsity) if (world == 1 and not args.no_single) else None
    cpu = cpu_baseline(x, layers) if world == 1 and not args.no_cpu else None
    imgs = batch * world * args.steps
    assert abs(job_throughput(batch, args.steps, world, elapsed) - imgs / elapsed) < 1e-6 * imgs / elapsed
    line = {
        "metric": METRIC, "value": imgs / elapsed, "unit": "images/s", "n_gpus": world, "steps": args.steps,
        "warmup": max(args.warmup, 3), "ms_per_step": elapsed / args.steps * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": f"MobileNet-v1 1.0 224x224x3 forward, batch {batch} per GPU, 13 pointwise layers "
                               f"group-sparse G=4 at {args.sparsity}% (balanced random masks), rest dense",
                   "global_batch": batch * world, "parallelism": f"batch-sharded replicas x{world}, no collective",
                   "l2": "one step streams about 2.6 GB of activations through two ping-pong buffers (far above the "
                         "126 MB L2); per-layer timings: differences of chain prefixes replayed as CUDA graphs, no flush (us, roofline), "
                         "and each layer launched alone after a 256 MB write has flushed L2 (us_cold)"},
        "effective_gflops_nonzero": step_flops / (elapsed / args.steps) / 1e9,
        "e2e": {"value": imgs / e2e_elapsed, "unit": "images/s", "h2d_bytes_per_step": int(x.nbytes),
                "d2h_bytes_per_step": int(batch * 1000 * 4)},
        "gpu_launches": net.debug_launches(batch) * args.steps,
        "clocks": clocks, "roofline": roofline, "layers": layers_out,
    }
    if single is not None:
        line["single_layer"] = single
    if others is not None:
        line["other_chain_configs"] = others
    if cpu is not None:
        line["cpu_baseline"] = cpu
    print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--batch", type=int, default=64)
    ap.add_argument("--sparsity", type=int, default=50)
    ap.add_argument("--layer-reps", type=int, default=10)
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU-oracle baseline leg")
    ap.add_argument("--no-dense", action="store_true", help="skip the dense cuDNN / cuBLAS times of the pointwise shapes")
    ap.add_argument("--no-single", action="store_true", help="skip the single-layer configurations (configs 1, 4, 5)")
    ap.add_argument("--sweep", action="store_true", help="print extra lines for the single-layer configurations")
    args = ap.parse_args()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        run_reference(args, rank)
        return
    if args.sweep:
        from paper_2310_19509_b200 import sweep
        sweep.main()
        if rank == 0 and not args.no_cpu:
            sweep_oracle_lines()
        return
    run_gpu(args, rank, world, local_rank)


if __name__ == "__main__":
    main()
