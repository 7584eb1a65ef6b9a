#!/usr/bin/env python
"""Benchmark of the quantized linear layer (Agile-Quant, Sec. 4.4) on B200.

One step = one pass of the whole path (layer absmax, activation quantization, integer
product on packed 4-bit weights, fp16 output) over the three LLaMA-7B projection shapes at
M = 2048 tokens with group-128 weight scales and int8 activations. Prints ONE JSON line.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

N > 1 is launched with torch.distributed.run, one rank per GPU; ranks run independent
copies of the workload (no collective on the data path: the layer shards by batch), a
barrier brackets the timed region and the slowest rank's time is used.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np
import torch

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2312_05693_b200 import inputs  # noqa: E402

# ncu, gemm_tensor_kernel<192, grouped>, M=2048, K=N=4096: dram__bytes_read.sum + dram__bytes_write.sum =
# 15.75 MB (whole rounds) + 10.08 MB (launch of the shared last round) per product call against 33.6 MB
# algorithmic (codes + packed weights + fp16 outputs, which stay in L2); the mean algorithmic bytes of the
# benchmark's three shapes is 57.1 MB. See profiles/.
GEMM_DRAM_BYTES_PER_LAUNCH = 25.83e6 * 57.1 / 33.6

WORKLOAD = "llama7b_prefill_w4a8"
METRIC = "w4a8_linear_tops"
UNIT = "TOPS"


def layer_ops(M, shapes):
    return sum(2.0 * M * s.K * s.N for s in shapes)


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return {"hbm_gbs": float(d["hbm_gbs"]), "bf16_tflops": float(d["bf16_tflops"]),
                "bf16_tflops_sustained": float(d.get("bf16_tflops_sustained", d["bf16_tflops"])),
                "source": "measured"}
    return {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0, "source": "fallback"}


class ClockSampler:
    """Samples SM clock and throttle reasons with nvidia-smi while the timed region runs."""
    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.rows = []
        self.proc = None
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits", "-lms", "20",
                 "-i", str(self.index)], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()
        t0 = time.perf_counter()                  # nvidia-smi takes a moment to start: have it sampling
        while not self.rows and time.perf_counter() - t0 < 5.0:      # before the region it is to cover begins
            time.sleep(0.01)

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 7:
                self.rows.append(parts)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, mx, pw = [], [], []
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in self.rows:
            try:
                sm.append(float(r[0]))
                mx.append(float(r[1]))
                pw.append(float(r[2]))
            except ValueError:
                continue
            for name, v in zip(names, r[3:7]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        busy = [c for c, p in zip(sm, pw) if p > 300.0] or sm
        return {"sm_mhz": statistics.median(busy) if busy else None,
                "sm_max_mhz": max(mx) if mx else None,
                "power_w_max": max(pw) if pw else None,
                "samples": len(sm), "reasons": sorted(reasons)}


def graph_replay_ms(launch, replays, warm=2):
    """Captures `launch()` (any number of kernel launches on torch's current stream) in a CUDA
    graph and returns the mean device time of one replay in ms (events around `replays`
    replays), so that host launch overhead is not part of the measurement."""
    launch()                                     # one-time set-up happens outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        launch()
    for _ in range(warm):
        g.replay()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a.record()
    for _ in range(replays):
        g.replay()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / replays


def max_over_ranks(values, dist, device):
    """Element-wise maximum over all ranks of a list of per-rank times (identity without a
    process group). Every rank gets the same list back."""
    t = torch.tensor(list(values), dtype=torch.float64, device=device)
    if dist is not None:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t]


def aggregate_value(world, units_per_rank_step, ms_per_step):
    """Whole-job throughput when every rank processes `units_per_rank_step` per step and the
    slowest rank needs `ms_per_step` (replicas: work per GPU is fixed as N grows)."""
    return world * units_per_rank_step / (ms_per_step * 1e-3)


def make_inputs(wl, M):
    xs, ws = [], []
    for i, s in enumerate(wl.shapes):
        xs.append(inputs.activations(M, s.K, wl.seed, wl.outlier_frac, wl.outlier_mult, sub=i))
        ws.append(inputs.weights(s.N, s.K, wl.seed, sub=i))
    return xs, ws


# ----------------------------------------------------------------------------------------
# CPU baseline: the checker as it stands, on a bounded sample of the same workload
# ----------------------------------------------------------------------------------------
def cpu_sample_step(oracle, wl, xs, wq, rows):
    t0 = time.perf_counter()
    for i, s in enumerate(wl.shapes):
        codes, sc = wq[i]
        oracle.linear(xs[i][:rows], codes, sc, wl.act_bits, wl.group_size, 0, wl.clip_shift)
    dt = time.perf_counter() - t0
    return layer_ops(rows, wl.shapes) / dt / 1e12, dt


def cpu_quantize_weights(oracle, wl, ws):
    return [oracle.quantize_weights(w, wl.group_size) for w in ws]


def cpu_baseline(wl, xs, ws, M, target_s=12.0):
    import oracle
    wq = cpu_quantize_weights(oracle, wl, ws)
    _, dt = cpu_sample_step(oracle, wl, xs, wq, 32)
    rows = int(min(M, max(32, 32 * target_s / max(dt, 1e-6))))
    tops, dt = cpu_sample_step(oracle, wl, xs, wq, rows)
    return {"value": tops, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
            "sample": f"first {rows} of {M} token rows of all {len(wl.shapes)} layer shapes, "
                      f"whole path, {dt:.1f} s"}


def run_reference(args):
    """--impl reference: the CPU checker timed on the same config, metric and unit."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import oracle
    wl = inputs.WORKLOADS[WORKLOAD]
    M = wl.Ms[0]
    xs, ws = make_inputs(wl, M)
    wq = cpu_quantize_weights(oracle, wl, ws)
    _, dt = cpu_sample_step(oracle, wl, xs, wq, 16)
    budget = 120.0 / max(args.steps + args.warmup, 1)
    rows = int(min(M, max(16, 16 * min(budget, 8.0) / max(dt, 1e-6))))
    for _ in range(args.warmup):
        cpu_sample_step(oracle, wl, xs, wq, rows)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        cpu_sample_step(oracle, wl, xs, wq, rows)
    dt = (time.perf_counter() - t0) / args.steps
    tops = layer_ops(rows, wl.shapes) / dt / 1e12
    sample = f"each step: first {rows} of {M} token rows of all {len(wl.shapes)} layer shapes, whole path"
    line = {
        "impl": "reference", "metric": METRIC, "value": tops, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "int8xint4->int32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "M": M, "shapes_KN": [[s.K, s.N] for s in wl.shapes],
                   "group_size": wl.group_size, "act_bits": wl.act_bits},
        "cpu_baseline": {"value": tops, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": tops, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))


# ----------------------------------------------------------------------------------------
# decode measurement (extra keys): weight streaming at M <= 16
# ----------------------------------------------------------------------------------------
def bench_decode(h, peaks, iters=40):
    from paper_2312_05693_b200 import binding
    wl = inputs.WORKLOADS["llama13b_decode_w4a8"]
    out = []
    for s in wl.shapes:
        wbytes = s.N * s.K // 2
        copies = max(2, int(320e6 // wbytes) + 1)          # rotate through > 2x L2 of weights
        w = torch.from_numpy(inputs.weights(s.N, s.K, wl.seed)).cuda()
        packs = []
        for c in range(copies):
            p, sc = h.aq_pack_w4(w, 0)
            packs.append((p, sc))
        for M in wl.Ms:
            x = torch.from_numpy(inputs.activations(M, s.K, wl.seed, wl.outlier_frac, wl.outlier_mult)).cuda()
            q, e = h.aq_quantize_act(x, 8)
            ws = h.alloc_workspace(M, s.K, s.N, 0)
            y = torch.empty((M, s.N), dtype=torch.float16, device="cuda")
            def launch():
                for i in range(copies):                      # a different weight copy per launch: HBM, not L2
                    h.aq_gemm_w4(q, packs[i][0], packs[i][1], s.N, 0, e, y=y, workspace=ws)
            ms = graph_replay_ms(launch, max(2, iters // copies)) / copies
            def launch_layer():                              # the whole layer call: quantize kernel + product kernel
                for i in range(copies):
                    h.aq_linear_w4a8(x, packs[i][0], packs[i][1], s.N, 0, y=y, workspace=ws)
            layer_ms = graph_replay_ms(launch_layer, max(2, iters // copies)) / copies
            # the same two sequences with the caller's promise that nothing in flight writes the weights
            # (aq_set_weights_stable): consecutive launches overlap; reported beside the default, not instead
            h.aq_set_weights_stable(True)
            try:
                ms_st = graph_replay_ms(launch, max(2, iters // copies)) / copies
                layer_ms_st = graph_replay_ms(launch_layer, max(2, iters // copies)) / copies
            finally:
                h.aq_set_weights_stable(False)
            algo = wbytes + 2 * s.N + M * s.K + 2 * M * s.N
            gbs = algo / (ms * 1e-3) / 1e9
            out.append({"K": s.K, "N": s.N, "M": M, "us": ms * 1e3, "layer_us": layer_ms * 1e3, "GBps": gbs,
                        "frac_of_hbm_peak": gbs / peaks["hbm_gbs"],
                        "weights_stable": {"us": ms_st * 1e3, "layer_us": layer_ms_st * 1e3,
                                           "frac_of_hbm_peak": algo / (ms_st * 1e-3) / 1e9 / peaks["hbm_gbs"]}})
        del packs
    return out


# ----------------------------------------------------------------------------------------
# the other prefill workloads (extra keys): int4 activations, token-pruned prefill
# ----------------------------------------------------------------------------------------
def _event_ms(fn, reps):
    """Mean device time of fn() over reps back-to-back calls (events on the current stream)."""
    fn()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(reps):
        fn()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / reps


def bench_w4a4(h, reps=30):
    wl = inputs.WORKLOADS["llama7b_prefill_w4a4"]
    M = wl.Ms[0]
    layers = []
    for s in wl.shapes:
        x = torch.from_numpy(inputs.activations(M, s.K, wl.seed, wl.outlier_frac, wl.outlier_mult)).cuda()
        p, sc = h.aq_pack_w4(torch.from_numpy(inputs.weights(s.N, s.K, wl.seed)).cuda(), wl.group_size)
        layers.append((x, p, sc, s, h.alloc_workspace(M, s.K, s.N, wl.group_size),
                       torch.empty((M, s.N), dtype=torch.float16, device="cuda")))
    def step():
        for x, p, sc, s, ws, y in layers:
            h.aq_linear_w4a4(x, p, sc, s.N, wl.group_size, clip_shift_or_exp=wl.clip_shift, y=y, workspace=ws)
    ms = _event_ms(step, reps)
    ops = sum(2.0 * M * s.K * s.N for s in wl.shapes)
    out = {"workload": wl.name, "ms_per_step": ms, "TOPS": ops / (ms * 1e-3) / 1e12,
           "note": "int4 codes travel in int8 containers: the tensor cores have no 4-bit integer kind"}
    # the same step with per-channel TRIP factors (Eq. 5-8) found on these activations, k_max = 4
    k_max = 4
    alphas, cal_us, mse = [], [], []
    for x, p, sc, s, ws, y in layers:
        alphas.append(h.aq_trip_calibrate(x, k_max)[0])
        cal_us.append(_event_ms(lambda: h.aq_trip_calibrate(x, k_max), 5) * 1e3)
        # reconstruction error of the activations (measurement only): plain 4-bit codes at this
        # workload's clip_shift against codes with factors
        xf = x.float()
        q0, e0 = h.aq_quantize_act(x, 4, clip_shift_or_exp=wl.clip_shift)
        q1, e1 = h.aq_quantize_act_trip(x, alphas[-1], k_max)
        err0 = (xf - q0.float() * 2.0 ** int(e0.item())).square().mean().item()
        err1 = (xf - q1.float() * 2.0 ** int(e1.item())).square().mean().item()
        mse.append({"plain": err0, "trip": err1})
    def step_trip():
        for (x, p, sc, s, ws, y), al in zip(layers, alphas):
            h.aq_linear_w4a4_trip(x, p, sc, s.N, wl.group_size, al, k_max, y=y, workspace=ws)
    ms_t = _event_ms(step_trip, reps)
    out["trip"] = {"k_max": k_max, "ms_per_step": ms_t, "TOPS": ops / (ms_t * 1e-3) / 1e12,
                   "calibrate_us": cal_us, "activation_mse": mse,
                   "channels_with_factor": [int((a > 0).sum().item()) for a in alphas]}
    return out


def bench_zero_point(h, reps=30):
    """The benchmark step with the unsigned quantizer and a zero point (Eq. 2, Eq. 5-7), 8-bit codes."""
    wl = inputs.WORKLOADS["llama7b_prefill_w4a8"]
    M = wl.Ms[0]
    layers = []
    for s in wl.shapes:
        x = torch.from_numpy(inputs.activations(M, s.K, wl.seed, wl.outlier_frac, wl.outlier_mult)).cuda()
        p, sc = h.aq_pack_w4(torch.from_numpy(inputs.weights(s.N, s.K, wl.seed)).cuda(), wl.group_size)
        r = h.aq_weight_offsets(p, sc, s.N, s.K, wl.group_size)          # once per weight matrix
        layers.append((x, p, sc, r, s, h.alloc_workspace(M, s.K, s.N, wl.group_size),
                       torch.empty((M, s.N), dtype=torch.float16, device="cuda")))
    def step():
        for x, p, sc, r, s, ws, y in layers:
            h.aq_linear_asym(8, x, p, sc, r, s.N, wl.group_size, y=y, workspace=ws)
    ms = _event_ms(step, reps)
    ops = sum(2.0 * M * s.K * s.N for s in wl.shapes)
    return {"workload": wl.name + " with zero point", "ms_per_step": ms, "TOPS": ops / (ms * 1e-3) / 1e12,
            "note": "range and quantize kernels (min/max; e, zp and codes); the per-channel term in the product kernel"}


def bench_chain(h, reps=30):
    """Two layers back to back (the 4096 -> 11008 -> 4096 pair of the benchmark shapes): fp16 in between
    against the chained call that hands the second layer its int8 codes directly (static exponent)."""
    wl = inputs.WORKLOADS["llama7b_prefill_w4a8"]
    M = wl.Ms[0]
    s1, s2 = wl.shapes[1], wl.shapes[2]
    x = torch.from_numpy(inputs.activations(M, s1.K, wl.seed, wl.outlier_frac, wl.outlier_mult)).cuda()
    p1, sc1 = h.aq_pack_w4(torch.from_numpy(inputs.weights(s1.N, s1.K, wl.seed)).cuda(), wl.group_size)
    p2, sc2 = h.aq_pack_w4(torch.from_numpy(inputs.weights(s2.N, s2.K, wl.seed + 1)).cuda(), wl.group_size)
    ws1 = h.alloc_workspace(M, s1.K, s1.N, wl.group_size)
    ws2 = h.alloc_workspace(M, s2.K, s2.N, wl.group_size)
    y1 = torch.empty((M, s1.N), dtype=torch.float16, device="cuda")
    y2 = torch.empty((M, s2.N), dtype=torch.float16, device="cuda")
    q1 = torch.empty((M, s1.N), dtype=torch.int8, device="cuda")
    h.aq_linear_w4a8(x, p1, sc1, s1.N, wl.group_size, y=y1, workspace=ws1)
    _, e_mid = h.aq_quantize_act(y1, 8)                       # calibration: the exponent the middle activation needs
    e_next = int(e_mid.item())
    def plain():
        h.aq_linear_w4a8(x, p1, sc1, s1.N, wl.group_size, y=y1, workspace=ws1)
        h.aq_linear_w4a8(y1, p2, sc2, s2.N, wl.group_size, y=y2, workspace=ws2)
    def chained():
        h.aq_linear_chain(8, x, p1, sc1, s1.N, wl.group_size, 8, e_next, q_next=q1, workspace=ws1)
        h.aq_gemm_w4(q1, p2, sc2, s2.N, wl.group_size, e_mid, y=y2, workspace=ws2)
    ops = 2.0 * M * (s1.K * s1.N + s2.K * s2.N)
    t_plain, t_chain = _event_ms(plain, reps), _event_ms(chained, reps)
    return {"layers_KN": [[s1.K, s1.N], [s2.K, s2.N]], "M": M,
            "fp16_between": {"us": t_plain * 1e3, "TOPS": ops / (t_plain * 1e-3) / 1e12},
            "codes_between": {"us": t_chain * 1e3, "TOPS": ops / (t_chain * 1e-3) / 1e12}}


def bench_act4(h, reps=30):
    """4-bit activation codes stored two per byte (Sec. 4.4): cost of the passes that pack them and
    widen them again before the product, on the first int4 benchmark shape."""
    wl = inputs.WORKLOADS["llama7b_prefill_w4a4"]
    M, s = wl.Ms[0], wl.shapes[0]
    x = torch.from_numpy(inputs.activations(M, s.K, wl.seed, wl.outlier_frac, wl.outlier_mult)).cuda()
    p, sc = h.aq_pack_w4(torch.from_numpy(inputs.weights(s.N, s.K, wl.seed)).cuda(), wl.group_size)
    ws = h.alloc_workspace(M, s.K, s.N, wl.group_size)
    y = torch.empty((M, s.N), dtype=torch.float16, device="cuda")
    q, e = h.aq_quantize_act(x, 4, clip_shift_or_exp=wl.clip_shift)
    q4 = h.aq_act4_pack(q)
    t_pack = graph_replay_ms(lambda: h.aq_act4_pack(q, q4), reps)
    t_plain = _event_ms(lambda: h.aq_gemm_w4(q, p, sc, s.N, wl.group_size, e, y=y, workspace=ws), reps)
    t_packed = _event_ms(lambda: h.aq_gemm_w4_act4(q4, p, sc, s.N, wl.group_size, e, y=y, workspace=ws), reps)
    # the chained layer call whose epilogue writes the next layer's 4-bit codes: one byte each / packed
    e_next = -2
    qn = torch.empty((M, s.N), dtype=torch.int8, device="cuda")
    qn4 = torch.empty((M, s.N // 2), dtype=torch.uint8, device="cuda")
    t_chain = _event_ms(lambda: h.aq_linear_chain(4, x, p, sc, s.N, wl.group_size, 4, e_next,
                                                  clip_shift_or_exp=wl.clip_shift, q_next=qn, workspace=ws), reps)
    t_chain4 = _event_ms(lambda: h.aq_linear_chain_act4(4, x, p, sc, s.N, wl.group_size, e_next,
                                                        clip_shift_or_exp=wl.clip_shift, q4_next=qn4, workspace=ws), reps)
    return {"M": M, "K": s.K, "N": s.N, "code_bytes": {"int8_containers": M * s.K, "packed": M * s.K // 2},
            "pack_us": t_pack * 1e3, "product_us": t_plain * 1e3, "product_on_packed_us": t_packed * 1e3,
            "chained_layer_us": {"codes_one_byte_each": t_chain * 1e3, "codes_packed_by_the_epilogue": t_chain4 * 1e3},
            "note": "the product widens packed codes with one extra pass; the tensor cores take 8-bit integers"}


def bench_attention(h, reps=5):
    """Softmax output as 4-bit log2 codes times int8 value codes (Eq. 3), LLaMA-7B attention shape."""
    H, M, J, D = 32, 2048, 2048, 128
    g = torch.Generator(device="cuda").manual_seed(7)
    scores = torch.randn((H, M, J), generator=g, device="cuda", dtype=torch.float32) * 3.0
    p = torch.softmax(scores, dim=2).to(torch.float16)           # synthetic attention probabilities (input only)
    del scores
    v = torch.from_numpy(inputs.activations(H * J, D, 7, 0.01, 8.0)).cuda()
    vq, ev = h.aq_quantize_act(v, 8)
    vq = vq.reshape(H, J, D)
    pc, pmax = h.aq_log2_quantize(p, 4)
    y = torch.empty((H, M, D), dtype=torch.float16, device="cuda")
    t_q = _event_ms(lambda: h.aq_log2_quantize(p, 4), reps)
    t_av = _event_ms(lambda: h.aq_attn_v_log2(pc, pmax, vq, ev, 4, y=y), reps)
    _, ws = h.aq_attn_v_log2_tc(pc, pmax, vq, ev, y=y)
    t_tc = _event_ms(lambda: h.aq_attn_v_log2_tc(pc, pmax, vq, ev, y=y, workspace=ws), 4 * reps)
    # the same with the byte factors written by the log2 kernel itself: no conversion pass over P
    pf, pfmax, _ = h.aq_log2_quantize_factors(p)
    t_qf = _event_ms(lambda: h.aq_log2_quantize_factors(p, factors=pf), reps)
    t_tcf = _event_ms(lambda: h.aq_attn_v_factors_tc(pf, pfmax, vq, ev, y=y, workspace=ws), 4 * reps)
    macs = float(H) * M * J * D
    # query x key scores on int8 codes (reduction over the head dimension); the fp16 score matrix is the traffic
    qa = torch.from_numpy(inputs.activations(H * M, D, 8, 0.01, 6.0)).cuda()
    ka = torch.from_numpy(inputs.activations(H * J, D, 9, 0.01, 6.0)).cuda()
    qc, eq = h.aq_quantize_act(qa, 8)
    kc, ek = h.aq_quantize_act(ka, 8)
    qc, kc = qc.reshape(H, M, D), kc.reshape(H, J, D)
    s_out, ws_qk = h.aq_attn_qk_tc(qc, eq, kc, ek)
    t_qk = _event_ms(lambda: h.aq_attn_qk_tc(qc, eq, kc, ek, s=s_out, workspace=ws_qk), 4 * reps)
    qk = {"us": t_qk * 1e3, "TOPS": 2.0 * macs / (t_qk * 1e-3) / 1e12,
          "GBps_scores_written": 2.0 * H * M * J / (t_qk * 1e-3) / 1e9}
    del s_out, qa, ka
    return {"H": H, "M": M, "J": J, "D": D, "qk_scores": qk,
            "log2_quantize": {"us": t_q * 1e3, "GBps": 3.0 * H * M * J / (t_q * 1e-3) / 1e9},
            "attn_v_shift": {"us": t_av * 1e3, "Gproducts_per_s": macs / (t_av * 1e-3) / 1e9,
                             "note": "CUDA-core kernel: one shift and one add per product"},
            "attn_v_tensor": {"us": t_tc * 1e3, "TOPS": 2.0 * macs / (t_tc * 1e-3) / 1e12,
                              "note": "value transpose + tcgen05 u8 x s8 kernel that turns each tile of codes into byte factors in shared memory"},
            "attn_v_tensor_on_factors": {"us": t_tcf * 1e3, "TOPS": 2.0 * macs / (t_tcf * 1e-3) / 1e12, "log2_quantize_factors_us": t_qf * 1e3,
                                         "note": "byte factors from aq_log2_quantize_factors: value transpose + tcgen05 kernel"}}


def bench_pruned(h, reps=10):
    wl = inputs.WORKLOADS["opt30b_pruned_prefill_w4a8"]
    M = wl.Ms[0]
    n_keep = wl.n_keep(M)
    scores = torch.from_numpy(inputs.token_scores(M, wl.seed)).cuda()
    out = []
    for s in wl.shapes:
        x = torch.from_numpy(inputs.activations(M, s.K, wl.seed, wl.outlier_frac, wl.outlier_mult)).cuda()
        p, sc = h.aq_pack_w4(torch.from_numpy(inputs.weights(s.N, s.K, wl.seed)).cuda(), wl.group_size)
        ws = h.alloc_workspace(n_keep, s.K, s.N, wl.group_size)
        y = torch.empty((n_keep, s.N), dtype=torch.float16, device="cuda")
        xc = torch.empty((n_keep, s.K), dtype=torch.float16, device="cuda")
        def gathered():                      # select, copy the kept rows, then the layer
            idx = h.aq_token_select(scores, n_keep)
            h.aq_token_compact(x, idx, out=xc)
            h.aq_linear_w4a8(xc, p, sc, s.N, wl.group_size, y=y, workspace=ws)
        def fused():                         # select, then the layer reads the kept rows in place
            idx = h.aq_token_select(scores, n_keep)
            h.aq_linear_w4a8(x, p, sc, s.N, wl.group_size, row_idx=idx, y=y, workspace=ws)
        q, e = h.aq_quantize_act(xc, 8)
        def product():
            h.aq_gemm_w4(q, p, sc, s.N, wl.group_size, e, y=y, workspace=ws)
        ops = 2.0 * n_keep * s.K * s.N
        r = {"K": s.K, "N": s.N, "M_in": M, "n_keep": n_keep}
        for name, fn in (("select_gather_linear", gathered), ("select_rowidx_linear", fused), ("product_only", product)):
            ms = _event_ms(fn, reps)
            r[name] = {"us": ms * 1e3, "TOPS": ops / (ms * 1e-3) / 1e12}
        out.append(r)
        del x, p, sc, ws, y, xc, q
    return out


# ----------------------------------------------------------------------------------------
# measured int8 tensor rate of this GPU (roofline denominator) and the step under sustained load
# ----------------------------------------------------------------------------------------
def bench_int8_probe(h, device_index):
    """The library's load-free tcgen05 kind::i8 loop on all SMs: a burst launch (about a millisecond, full
    clock) and launches back to back for about two seconds (the power cap acts), with the clocks seen."""
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    out = {}
    for name, from_tmem in (("a_from_tmem", True), ("both_from_smem", False)):
        iters = 4096
        h.aq_probe_int8_mma(iters, from_tmem, ws)
        torch.cuda.synchronize()
        best = None
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ops = h.aq_probe_int8_mma(iters, from_tmem, ws)
            b.record()
            torch.cuda.synchronize()
            ms = a.elapsed_time(b)
            best = ms if best is None else min(best, ms)
        entry = {"burst_TOPS": ops / (best * 1e-3) / 1e12, "burst_ms": best}
        if from_tmem:
            sampler = ClockSampler(device_index)
            sampler.start()
            big = 65536                                   # about 17 ms per launch at full clock
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            n = 0
            a.record()
            t0 = time.perf_counter()
            while time.perf_counter() - t0 < 2.0:
                for _ in range(8):
                    ops_big = h.aq_probe_int8_mma(big, from_tmem, ws)
                    n += 1
                torch.cuda.synchronize()
            b.record()
            torch.cuda.synchronize()
            ck = sampler.stop()
            ms = a.elapsed_time(b)
            entry["sustained_TOPS"] = n * ops_big / (ms * 1e-3) / 1e12
            entry["sustained_s"] = ms * 1e-3
            entry["sustained_clocks"] = ck
        st = h.aq_check_workspace(ws)
        if st != 0:
            entry["status"] = st
        out[name] = entry
    return out


def bench_sustained(step, ops_per_step, device_index, seconds=3.0):
    """The benchmark step looped for `seconds` with the clock sampler running: what the step delivers once
    the power cap has acted, with the median SM clock and time x clock."""
    sampler = ClockSampler(device_index)
    sampler.start()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    n = 0
    t0 = time.perf_counter()
    a.record()
    while time.perf_counter() - t0 < seconds:
        for _ in range(50):
            step()
            n += 1
        torch.cuda.synchronize()
    b.record()
    torch.cuda.synchronize()
    ck = sampler.stop()
    ms = a.elapsed_time(b) / n
    out = {"TOPS": ops_per_step / (ms * 1e-3) / 1e12, "ms_per_step": ms, "steps": n, "seconds": a.elapsed_time(b) * 1e-3,
           "clocks": ck}
    if ck.get("sm_mhz"):
        out["ms_x_mhz"] = ms * ck["sm_mhz"]
    return out


def bench_quantize(h, peaks, reps=20):
    """The two quantize kernels (range, codes) alone on the benchmark's activation shapes (HBM / L2 bound)."""
    wl = inputs.WORKLOADS[WORKLOAD]
    M = wl.Ms[0]
    out = []
    for K in sorted({s.K for s in wl.shapes}):
        x = torch.from_numpy(inputs.activations(M, K, wl.seed, wl.outlier_frac, wl.outlier_mult)).cuda()
        ws = torch.empty(256, dtype=torch.uint8, device="cuda")
        ms = graph_replay_ms(lambda: h.aq_quantize_act(x, wl.act_bits, workspace=ws), reps)
        algo = 5.0 * M * K          # fp16 read for the maximum, fp16 read for the codes, int8 codes written
        hbm = 3.0 * M * K           # what has to cross HBM when the second read is served on chip
        out.append({"kernel": "range_kernel + quantize_kernel", "M": M, "K": K, "us": ms * 1e3, "bound": "hbm",
                    "algorithmic_bytes": algo, "achieved": algo / (ms * 1e-3) / 1e9, "peak": peaks["hbm_gbs"],
                    "unit": "GB/s", "frac": algo / (ms * 1e-3) / 1e9 / peaks["hbm_gbs"],
                    "hbm_bytes_once": hbm, "frac_counting_x_once": hbm / (ms * 1e-3) / 1e9 / peaks["hbm_gbs"]})
    return out


# ----------------------------------------------------------------------------------------
# single-shape case (for profiling one kernel on a small or a full-size shape)
# ----------------------------------------------------------------------------------------
def run_case(args):
    """--case M,K,N,group[,bits[,kernel]]: quantize once, then time the product kernel alone."""
    from paper_2312_05693_b200 import binding
    parts = [int(v) for v in args.case.split(",")]
    M, K, N, group = parts[:4]
    bits = parts[4] if len(parts) > 4 else 8
    kernel = parts[5] if len(parts) > 5 else binding.AQ_KERNEL_AUTO
    torch.cuda.set_device(0)
    h = binding.Handle(0)
    h.aq_set_kernel(kernel)
    x = torch.from_numpy(inputs.activations(M, K, 1, 0.005, 30.0)).cuda()
    w = torch.from_numpy(inputs.weights(N, K, 1)).cuda()
    wbytes = N * K // 2
    copies = max(1, min(64, int(args.rotate_mb * 1e6 // wbytes)))
    packs = [h.aq_pack_w4(w, group) for _ in range(copies)]
    q, e = h.aq_quantize_act(x, bits)
    ws = h.alloc_workspace(M, K, N, group)
    y = torch.empty((M, N), dtype=torch.float16, device="cuda")
    def launch():
        for i in range(copies):
            h.aq_gemm_w4(q, packs[i][0], packs[i][1], N, group, e, y=y, workspace=ws)
    for _ in range(args.warmup):
        launch()
    reps = max(1, args.steps // copies)
    ts = sorted(graph_replay_ms(launch, reps) / copies for _ in range(3))
    med = ts[1]
    st = h.aq_check_workspace(ws)
    algo = wbytes + M * K + 2 * M * N
    print(json.dumps({"case": args.case, "status": st, "us": med * 1e3, "us_min": ts[0] * 1e3,
                      "TOPS": 2.0 * M * K * N / (med * 1e-3) / 1e12, "GBps": algo / (med * 1e-3) / 1e9,
                      "weight_copies": copies}))


def run_attn_case(args):
    """--attn-case H,M,J,D: time the tensor-core attention x value path on log2 codes."""
    from paper_2312_05693_b200 import binding
    H, M, J, D = [int(v) for v in args.attn_case.split(",")]
    torch.cuda.set_device(0)
    h = binding.Handle(0)
    g = torch.Generator(device="cuda").manual_seed(7)
    p = torch.softmax(torch.randn((H, M, J), generator=g, device="cuda") * 3.0, dim=2).to(torch.float16)
    v = torch.from_numpy(inputs.activations(H * J * D // 128, 128, 7, 0.01, 8.0)).cuda()
    vq, ev = h.aq_quantize_act(v, 8)
    vq = vq.reshape(H, J, D)
    pc, pmax = h.aq_log2_quantize(p, 4)
    y, ws = h.aq_attn_v_log2_tc(pc, pmax, vq, ev)
    for _ in range(args.warmup):
        h.aq_attn_v_log2_tc(pc, pmax, vq, ev, y=y, workspace=ws)
    ms = _event_ms(lambda: h.aq_attn_v_log2_tc(pc, pmax, vq, ev, y=y, workspace=ws), max(1, args.steps))
    print(json.dumps({"attn_case": args.attn_case, "status": h.aq_check_workspace(ws), "us": ms * 1e3,
                      "TOPS": 2.0 * H * M * J * D / (ms * 1e-3) / 1e12}))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=400)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-decode", action="store_true", help="skip the extra keys (rate probe, sustained leg, decode, w4a4, pruned_prefill, ...)")
    ap.add_argument("--case", default=None, help="M,K,N,group[,bits[,kernel]]: time one product kernel")
    ap.add_argument("--rotate-mb", type=float, default=0.0,
                    help="with --case: rotate through this many MB of weight copies (defeats L2)")
    ap.add_argument("--attn-case", default=None, help="H,M,J,D: time the tensor-core attention x value path")
    args = ap.parse_args()
    if args.case:
        run_case(args)
        return
    if args.attn_case:
        run_attn_case(args)
        return
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        run_reference(args)
        return

    from paper_2312_05693_b200 import binding

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (there is no CPU path)")
    torch.cuda.set_device(local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    peaks = load_peaks()
    wl = inputs.WORKLOADS[WORKLOAD]
    M = wl.Ms[0]
    h = binding.Handle(local_rank)
    xs_np, ws_np = make_inputs(wl, M)
    fn = h.aq_linear_w4a8 if wl.act_bits == 8 else h.aq_linear_w4a4

    layers = []
    for i, s in enumerate(wl.shapes):
        wd = torch.from_numpy(ws_np[i]).cuda()
        packed, scales = h.aq_pack_w4(wd, wl.group_size)
        del wd
        layers.append({
            "K": s.K, "N": s.N, "x": torch.from_numpy(xs_np[i]).cuda(), "packed": packed, "scales": scales,
            "y": torch.empty((M, s.N), dtype=torch.float16, device="cuda"),
            "ws": h.alloc_workspace(M, s.K, s.N, wl.group_size),
            "x_host": torch.from_numpy(xs_np[i]).pin_memory(),
            "y_host": torch.empty((M, s.N), dtype=torch.float16).pin_memory(),
            "scratch": torch.empty(binding.aq_linear_host_scratch_bytes(M, s.K, s.N, wl.group_size),
                                   dtype=torch.uint8, device="cuda"),
        })
    torch.cuda.synchronize()

    def step():
        for L in layers:
            fn(L["x"], L["packed"], L["scales"], L["N"], wl.group_size, binding.AQ_SCALE_DYNAMIC,
               wl.clip_shift, y=L["y"], workspace=L["ws"])

    ops_per_step = layer_ops(M, wl.shapes)
    # ---- main timed region: the public layer call, device-resident inputs
    sampler = ClockSampler(local_rank)
    sampler.start()
    for _ in range(args.warmup):
        step()
    barrier()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    barrier()
    ev0.record()
    for _ in range(args.steps):
        step()
    ev1.record()
    barrier()
    ms_total = ev0.elapsed_time(ev1)

    # ---- second pass, same kernels launched as two calls so the product kernel can be
    #      bracketed by events on the launching stream (its duration feeds the roofline)
    gemm_ev = []
    for _ in range(min(args.steps, 50)):
        for L in layers:
            q, e = h.aq_quantize_act(L["x"], wl.act_bits, binding.AQ_SCALE_DYNAMIC, wl.clip_shift,
                                     workspace=L["ws"][:256])
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            h.aq_gemm_w4(q, L["packed"], L["scales"], L["N"], wl.group_size, e, y=L["y"], workspace=L["ws"])
            b.record()
            gemm_ev.append((a, b, 2.0 * M * L["K"] * L["N"]))
    torch.cuda.synchronize()
    clocks = sampler.stop()
    gemm_ms = sum(a.elapsed_time(b) for a, b, _ in gemm_ev)
    gemm_ops = sum(o for _, _, o in gemm_ev)
    for L in layers:
        st = h.aq_check_workspace(L["ws"])
        if st != binding.AQ_OK:
            raise SystemExit(f"kernel reported {binding.status_string(st)}")

    # ---- end to end through the host-buffer entry point (H2D of x and D2H of y inside every step).
    # Every layer has its own stream and device scratch: a layer's copy in, kernels and copy out are
    # ordered on its stream, while different layers (and the same layer's next step behind it) overlap,
    # so both directions of the host link and the SMs work at the same time.
    main_stream = torch.cuda.current_stream()
    for L in layers:
        L["stream"] = torch.cuda.Stream()
    def step_host():
        for L in layers:
            with torch.cuda.stream(L["stream"]):
                h.aq_linear_host_async(wl.act_bits, L["x_host"], L["packed"], L["scales"], L["N"], wl.group_size,
                                       L["y_host"], L["scratch"], binding.AQ_SCALE_DYNAMIC, wl.clip_shift)
    def join_host():
        for L in layers:
            main_stream.wait_stream(L["stream"])
    e2e_steps = max(3, min(args.steps, 10))
    for _ in range(3):
        step_host()
    join_host()
    barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for L in layers:
        L["stream"].wait_event(e0)
    for _ in range(e2e_steps):
        step_host()
    join_host()
    e1.record()
    barrier()
    e2e_ms = e0.elapsed_time(e1) / e2e_steps

    ms_total, e2e_ms = max_over_ranks([ms_total, e2e_ms], dist, "cuda")
    ms_per_step = ms_total / args.steps
    value = aggregate_value(world, ops_per_step, ms_per_step) / 1e12
    e2e_value = aggregate_value(world, ops_per_step, e2e_ms) / 1e12

    # The product launches were event-timed in a pass of well under a second at full clock, so the measured
    # peak that applies is the burst one; the sustained and nominal fractions are printed beside it.
    gemm_pass_s = gemm_ms * 1e-3
    burst_peak = 2.0 * peaks["bf16_tflops"]              # dense int8 = 2 x dense bf16 (nominal ratio)
    sustained_peak = 2.0 * peaks["bf16_tflops_sustained"]
    timed_as = "burst" if gemm_pass_s < 1.0 else "sustained"
    int8_peak = burst_peak if timed_as == "burst" else sustained_peak
    achieved = gemm_ops / (gemm_ms * 1e-3) / 1e12
    roofline = {
        "kernel": "gemm_tensor_kernel<192, grouped> (whole rounds + shared last round)", "bound": "tensor", "achieved": achieved,
        "peak": int8_peak, "unit": "TFLOP/s", "frac": achieved / int8_peak, "traffic": GEMM_DRAM_BYTES_PER_LAUNCH,
        "traffic_note": "dram read+write of one product call (both launches) from ncu on K=N=4096 (25.8 MB, outputs stay in L2), "
                        "scaled by algorithmic bytes to the mean of the three shapes",
        "peak_source": f"2 x bf16_tflops ({timed_as}) of {peaks['source']} peaks (int8:bf16 nominal 2:1); the product launches "
                       f"were timed in a {gemm_pass_s * 1e3:.1f} ms pass",
        "frac_of_burst_peak": achieved / burst_peak, "frac_of_sustained_peak": achieved / sustained_peak,
        "frac_of_nominal_4500": achieved / 4500.0,
        "timing": "CUDA events around each aq_gemm_w4 launch in a second pass of the same steps",
        "avg_launch_us": gemm_ms * 1e3 / len(gemm_ev),
    }

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "int8xint4->int32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "M": M, "shapes_KN": [[s.K, s.N] for s in wl.shapes],
                   "group_size": wl.group_size, "act_bits": wl.act_bits, "parallelism": f"replicas x{world}",
                   "l2": "per-step footprint (x, packed w, y of 3 layers) ~210 MB exceeds the 126 MB L2"},
        "tokens_per_s": world * M * len(wl.shapes) / (ms_per_step * 1e-3),
        "e2e": {"value": e2e_value, "unit": UNIT,
                "h2d_bytes_per_step": int(sum(M * s.K * 2 for s in wl.shapes)),
                "d2h_bytes_per_step": int(sum(M * s.N * 2 for s in wl.shapes)),
                "ms_per_step": e2e_ms, "api": "aq_linear_host_async, one stream per layer"},
        # per layer: the range and quantize kernels and the product kernel, which is two launches where the tiles of a
        # partial last round are shared between CTA pairs (the workspace then has room for their partial sums)
        "gpu_launches": args.steps * sum(3 + (binding.aq_workspace_bytes(M, s.K, s.N, wl.group_size) >
                                              binding.aq_workspace_bytes(M, s.K, s.N, 0)) for s in wl.shapes),
        "clocks": clocks,
        "roofline": roofline,
    }
    if rank == 0 and world == 1 and not args.no_decode:
        try:
            probe = bench_int8_probe(h, local_rank)
            line["int8_peak_measured"] = probe
            p_burst = probe["a_from_tmem"]["burst_TOPS"]
            roofline["frac_of_int8_probe_burst"] = achieved / p_burst
            roofline["int8_probe_burst"] = p_burst
        except Exception as ex:  # report, do not hide
            line["int8_peak_measured"] = {"error": repr(ex)}
        try:
            line["sustained"] = bench_sustained(step, ops_per_step, local_rank)
            probe = line["int8_peak_measured"]
            if "a_from_tmem" in probe and "sustained_TOPS" in probe["a_from_tmem"]:
                line["sustained"]["frac_of_int8_probe_sustained"] = line["sustained"]["TOPS"] / probe["a_from_tmem"]["sustained_TOPS"]
            line["sustained"]["frac_of_2x_bf16_sustained"] = line["sustained"]["TOPS"] / sustained_peak
        except Exception as ex:
            line["sustained"] = {"error": repr(ex)}
        try:
            line["quantize_roofline"] = bench_quantize(h, peaks)
        except Exception as ex:
            line["quantize_roofline"] = {"error": repr(ex)}
    if rank == 0 and world == 1 and not args.no_decode:
        try:
            line["decode"] = bench_decode(h, peaks)
            fr = [d["frac_of_hbm_peak"] for d in line["decode"]]
            line["decode_roofline"] = {
                "kernel": "gemm_decode_stream_kernel", "bound": "hbm", "unit": "GB/s", "peak": peaks["hbm_gbs"],
                "achieved": statistics.mean(d["GBps"] for d in line["decode"]), "frac": statistics.mean(fr),
                "frac_min": min(fr), "frac_max": max(fr),
                "algorithmic_bytes": "N*K/2 + 2*N + M*K + 2*M*N per launch", "cases": len(fr)}
            fs = [d["weights_stable"]["frac_of_hbm_peak"] for d in line["decode"]]
            # the same launches under the caller's promise that nothing in flight writes the weights (off by default)
            line["decode_roofline"]["with_weights_stable_promise"] = {"frac": statistics.mean(fs), "frac_min": min(fs),
                                                                      "frac_max": max(fs)}
        except Exception as ex:  # report, do not hide
            line["decode"] = {"error": repr(ex)}
    if rank == 0 and world == 1 and not args.no_decode:
        for key, fn in (("w4a4", bench_w4a4), ("zero_point", bench_zero_point), ("chain", bench_chain), ("act4_storage", bench_act4),
                        ("attention_log2", bench_attention), ("pruned_prefill", bench_pruned)):
            try:
                line[key] = fn(h)
            except Exception as ex:  # report, do not hide
                line[key] = {"error": repr(ex)}
    if isinstance(line.get("pruned_prefill"), list):
        # the per-channel prefill product of the token-pruned workload (tiles of 256 channels), as a roofline entry
        pr = line["pruned_prefill"]
        ach = statistics.mean(r["product_only"]["TOPS"] for r in pr)
        ent = {"kernel": "gemm_wide_kernel<192> (one scale per channel, 256-channel tiles)", "bound": "tensor", "unit": "TFLOP/s",
               "workload": "opt30b_pruned_prefill_w4a8, product kernel, mean of the two shapes", "achieved": ach,
               "peak": burst_peak, "frac": ach / burst_peak, "frac_of_nominal_4500": ach / 4500.0,
               "per_shape_TOPS": [r["product_only"]["TOPS"] for r in pr],
               "timing": "event-timed back-to-back launches (a fraction of a second at full clock: burst peak)"}
        probe = line.get("int8_peak_measured", {})
        if "a_from_tmem" in probe:
            ent["frac_of_int8_probe_burst"] = ach / probe["a_from_tmem"]["burst_TOPS"]
        line["perchannel_roofline"] = ent
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(wl, xs_np, ws_np, M)
    if rank == 0:
        print(json.dumps(line))
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
