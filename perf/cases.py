"""Performance cases of the quantized linear layer: the work a program that runs quantized transformer
layers has this library do, through `paper_2312_05693_b200.binding`.

A case is one pass of one of these:

* kind "layers": the linear layers of a part of a transformer, in order, each one library call on fp16
  activations (quantize, integer product, fp16 output), with weights that were packed before;
* kind "attention": the three products' inputs quantized, query x key scores, the log2 codes of a given softmax
  output as byte factors, and attention x value on them (the softmax itself is outside the library).

Layer shapes are those of `inputs.WORKLOADS` (OPT-125M, LLaMA-7B, LLaMA-13B, OPT-30B), activations follow its
recipe (N(0, 1) with a few fixed outlier channels), weights are N(0, 0.02).
"""
import math

import torch

from paper_2312_05693_b200 import binding

# Case fields (kind "layers"): m token rows; hidden, ffn: the model's widths; part: which layers (see _shapes);
# group: 0 = one weight scale per output channel, 128 = one per 128 inputs; bits: activation codes; mode:
# "plain", "asym" (zero point), "trip" (per-channel factors), "codes" (4-bit codes packed two per byte between the
# two layers of an MLP); keep: share of the tokens kept by score before the layers; stable: the program has made
# the library's promise that nothing in flight writes the weights.
_LAYERS = {"kind": "layers", "group": 0, "bits": 8, "mode": "plain", "keep": 1.0, "stable": False}


def _layers(name, **kw):
    return dict(_LAYERS, name=name, **kw)


def listed():
    return [
        # the smallest layer: one 768 x 768 projection of a small model, 16 tokens of a batch
        _layers("opt125m_layer_m16", m=16, hidden=768, ffn=3072, part="square"),
        # generating one token: the seven linear layers of a block, one activation row (per-channel scales)
        _layers("decode_13b_m1", m=1, hidden=5120, ffn=13824, part="block", stable=True),
        # the same for a batch of 16 sequences
        _layers("decode_13b_m16", m=16, hidden=5120, ffn=13824, part="block", stable=True),
        # generating one token with weights in groups of 128
        _layers("decode_7b_g128_m1", m=1, hidden=4096, ffn=11008, part="block", group=128, stable=True),
        # the same for six sequences
        _layers("decode_7b_g128_m6", m=6, hidden=4096, ffn=11008, part="block", group=128, stable=True),
        # a batch beyond the few-row range (or a very short prompt), 4-bit activations that clip their outliers
        _layers("batch_7b_g128_w4a4_m48", m=48, hidden=4096, ffn=11008, part="block", group=128, bits=4),
        # a prompt of ordinary, ragged length, per-channel scales
        _layers("prompt_13b_m333", m=333, hidden=5120, ffn=13824, part="shapes"),
        # prefill of a long prompt with weights in groups of 128
        _layers("prefill_7b_g128_m2048", m=2048, hidden=4096, ffn=11008, part="shapes", group=128),
        # an MLP whose 4-bit codes stay packed between its two layers
        _layers("mlp_13b_w4a4_codes_m1024", m=1024, hidden=5120, ffn=13824, part="mlp", bits=4, mode="codes"),
        # one-sided activations (behind a ReLU-like function): codes with a zero point
        _layers("prompt_7b_asym_g128_m509", m=509, hidden=4096, ffn=11008, part="shapes", group=128, mode="asym"),
        # prefill after token pruning: 2458 of 4096 tokens kept by score, the largest layers
        _layers("prefill_opt30b_pruned", m=4096, hidden=7168, ffn=28672, part="opt", keep=0.6),
        # attention of one layer over a long prompt
        {"name": "attention_h32_2048", "kind": "attention", "heads": 32, "m": 2048, "j": 2048, "d": 128},
    ]


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def draw(rng):
    most = 0.9 * max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= most:
            return c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    if rng.random() < 0.15:
        return {"kind": "attention", "heads": rng.choice([12, 16, 32, 40, 56]), "m": _log_int(rng, 100, 2048),
                "j": 16 * _log_int(rng, 8, 128), "d": 128}
    group = rng.choice([0, 128])
    step = 128 if group else 32
    bits = rng.choice([8, 8, 4])
    mode = rng.choice(["plain", "plain", "plain", "asym"] + (["trip", "codes"] if bits == 4 else []))
    m = _log_int(rng, 1, 3000)
    hidden = step * max(1, _log_int(rng, 768, 7168) // step)
    ffn = step * max(1, int(hidden * rng.uniform(2.0, 4.0)) // step)
    part = "mlp" if mode == "codes" else rng.choice(["square", "block", "shapes", "mlp", "opt"])
    keep = round(rng.uniform(0.3, 0.9), 2) if m > 256 and mode == "plain" and rng.random() < 0.3 else 1.0
    return dict(_LAYERS, m=m, hidden=hidden, ffn=ffn, part=part, group=group, bits=bits, mode=mode, keep=keep,
                stable=m <= 16)


def _shapes(case):
    """(K, N, index of the activation it reads) of the layers of one pass."""
    h, f = case["hidden"], case["ffn"]
    return {
        "square": [(h, h, 0)],
        # query, key, value, attention output, gate, up, down
        "block": [(h, h, 0), (h, h, 0), (h, h, 0), (h, h, 1), (h, f, 2), (h, f, 2), (f, h, 3)],
        "shapes": [(h, h, 0), (h, f, 1), (f, h, 2)],
        "opt": [(h, h, 0), (h, f, 1)],
        "mlp": [(h, f, 0), (f, h, 1)],
    }[case["part"]]


def _kept(case):
    return case["m"] if case["keep"] >= 1.0 else int(math.ceil(case["keep"] * case["m"]))


def _clip(case):
    return 4 if case["bits"] == 4 and case["mode"] in ("plain", "codes") else 0     # outlier channels saturate at 4 bits


def _activations(gen, m, k, one_sided):
    x = torch.randn((m, k), generator=gen, device="cuda")
    n_out = max(1, k // 200)                                     # 0.5 % of the channels, the same in every row
    at = torch.randperm(k, generator=gen, device="cuda")[:n_out]
    x[:, at] *= 30.0
    if one_sided:
        x = torch.where(x < 0, 0.1 * x, x)
    return x.to(torch.float16)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    h = binding.Handle(0)
    if case["kind"] == "attention":
        return _prepare_attention(case, gen, h)
    shapes, m, rows, group = _shapes(case), case["m"], _kept(case), case["group"]
    mode, bits = case["mode"], case["bits"]
    xs = {}
    for k, _, i in shapes:
        if i not in xs and not (mode == "codes" and i > 0):
            xs[i] = _activations(gen, m, k, mode == "asym")
    layers = []
    for k, n, i in shapes:
        w = (torch.randn((n, k), generator=gen, device="cuda") * 0.02).to(torch.float16)
        packed, scales = h.aq_pack_w4(w, group)
        layer = {"n": n, "x": xs.get(i), "packed": packed, "scales": scales}
        if mode == "asym":
            layer["offsets"] = h.aq_weight_offsets(packed, scales, n, k, group)
        if mode == "trip":
            layer["alpha"] = h.aq_trip_calibrate(xs[i], 4)[0]
        layers.append(layer)
    nbytes = max(binding.aq_workspace_bytes(rows, k, n, group) for k, n, _ in shapes)
    state = {"case": case, "h": h, "layers": layers, "workspace": torch.empty(nbytes, dtype=torch.uint8, device="cuda")}
    if case["keep"] < 1.0:
        state["scores"] = torch.rand(m, generator=gen, device="cuda")
        state["n_keep"] = rows
    if mode == "codes":
        # the exponent of the codes between the layers comes from calibration: here from rows of the same input
        up = layers[0]
        y = h.aq_linear_w4a4(up["x"][: min(m, 64)], up["packed"], up["scales"], up["n"], group, clip_shift_or_exp=_clip(case))
        state["next_exp"] = int(h.aq_quantize_act(y, 4)[1].item()) - 1
        state["scale_exp"] = torch.tensor([state["next_exp"]], dtype=torch.int32, device="cuda")
    h.aq_set_weights_stable(bool(case["stable"]))
    return state


def _prepare_attention(case, gen, h):
    H, M, J, D = case["heads"], case["m"], case["j"], case["d"]
    st = {"case": case, "h": h}
    st["q"] = _activations(gen, H * M, D, False)
    st["k"] = _activations(gen, H * J, D, False)
    st["v"] = _activations(gen, H * J, D, False)
    p = torch.empty((H, M, J), dtype=torch.float16, device="cuda")
    for i in range(H):                                           # the softmax output, head by head
        p[i] = torch.softmax(3.0 * torch.randn((M, J), generator=gen, device="cuda"), dim=-1).to(torch.float16)
    st["p"] = p
    st["quant_ws"] = torch.empty(256, dtype=torch.uint8, device="cuda")
    st["workspace"] = torch.empty(binding.load().aq_attn_workspace_bytes(H, M, J, D), dtype=torch.uint8, device="cuda")
    return st


def run(state):
    case, h = state["case"], state["h"]
    if case["kind"] == "attention":
        H, M, J, D = case["heads"], case["m"], case["j"], case["d"]
        ws = state["quant_ws"]
        qc, qe = h.aq_quantize_act(state["q"], 8, workspace=ws)
        kc, ke = h.aq_quantize_act(state["k"], 8, workspace=ws)
        vc, ve = h.aq_quantize_act(state["v"], 8, workspace=ws)
        s, _ = h.aq_attn_qk_tc(qc.view(H, M, D), qe, kc.view(H, J, D), ke, workspace=ws)
        f, mx, _ = h.aq_log2_quantize_factors(state["p"], workspace=ws)
        y, _ = h.aq_attn_v_factors_tc(f, mx, vc.view(H, J, D), ve, workspace=state["workspace"])
        return {"scores": s, "factors": f, "y": y}
    group, bits, mode, ws, clip = case["group"], case["bits"], case["mode"], state["workspace"], _clip(case)
    out = []
    idx = None
    if "scores" in state:
        idx = h.aq_token_select(state["scores"], state["n_keep"])
        out.append(idx)
    if mode == "codes":
        up, down = state["layers"]
        q4 = h.aq_linear_chain_act4(bits, up["x"], up["packed"], up["scales"], up["n"], group, state["next_exp"],
                                    clip_shift_or_exp=clip, workspace=ws)
        y = h.aq_gemm_w4_act4(q4, down["packed"], down["scales"], down["n"], group, state["scale_exp"], workspace=ws)
        return [q4, y]
    linear = h.aq_linear_w4a8 if bits == 8 else h.aq_linear_w4a4
    for l in state["layers"]:
        if mode == "asym":
            y = h.aq_linear_asym(bits, l["x"], l["packed"], l["scales"], l["offsets"], l["n"], group, workspace=ws)
        elif mode == "trip":
            y = h.aq_linear_w4a4_trip(l["x"], l["packed"], l["scales"], l["n"], group, l["alpha"], 4, workspace=ws)
        else:
            y = linear(l["x"], l["packed"], l["scales"], l["n"], group, clip_shift_or_exp=clip, row_idx=idx, workspace=ws)
        out.append(y)
    return out


def work(case):
    """Inputs once, outputs once; two operations per multiply-add."""
    if case["kind"] == "attention":
        H, M, J, D = case["heads"], case["m"], case["j"], case["d"]
        # q, k, v and P in (fp16); scores, byte factors and y out
        return {"bytes": 2.0 * H * D * (M + 2 * J) + 2.0 * H * M * J + 2.0 * H * M * J + 1.0 * H * M * J + 2.0 * H * M * D,
                "flops": 2.0 * 2.0 * H * M * J * D}
    rows, total, flops, seen = _kept(case), 0.0, 0.0, set()
    for i, (k, n, x) in enumerate(_shapes(case)):
        groups = k // 128 if case["group"] else 1
        total += 0.5 * n * k + 2.0 * groups * n                 # codes and scales of the weights
        if case["mode"] == "codes":
            total += 2.0 * rows * k + 0.5 * rows * n if i == 0 else 0.5 * rows * k + 2.0 * rows * n
        else:
            total += 2.0 * rows * n + (2.0 * rows * k if x not in seen else 0.0)
        seen.add(x)
        flops += 2.0 * rows * n * k
    if case["keep"] < 1.0:
        total += 4.0 * case["m"] + 4.0 * rows
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # Integer sums are exact; what is left is fp32 scaling and one rounding to fp16. Against the same layer in 64
    # bits rounded once to fp16, at most 4.7 % of the outputs were seen to differ, by one unit in the last place
    # (rel 6.7e-5, max 9.8e-4: zero point, K = 11008); the plain layers and attention not at all. Four times that.
    # Behind packed 4-bit codes a tie of such an output may move a code by one: one term of a 5120-term sum or more
    # in that row's outputs.
    if case.get("mode") == "codes":
        return {"rel": 3e-4, "max": 3e-2, "differ": 1e-5}
    return {"rel": 3e-4, "max": 4e-3, "differ": 0.0}
