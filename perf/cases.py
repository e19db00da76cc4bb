"""What the library is timed on: the calls a program makes that runs a Visual-Mamba backbone with quantized linears.

Offline, such a program takes static parameters from a few calibration images (``calibrate``) and may refine the
activation steps by a grid search (``search_act_step``).  From then on it calls ``PtqLinear.forward`` for every
linear of every block, one image at a time in a serving loop or a batch at a time.  A case is a list of layers
(``layers``, see ``parse_layers``), repeated over ``blocks`` blocks with weights and activations of their own, and
one pass calls the entry point once for each of them in the order of the model.

``op``      "forward", or one of the offline steps "calibrate" and "search"
``scheme``  "pts" (static steps per token position), "asym" (with zero offsets), "dynamic" (steps measured at run
            time), "w4a4" (4-bit codes, packed weights); forward passes only
``call``    how a forward pass gets its memory: "buffers" (outputs and one workspace for all layers kept by the
            caller), "static" (``forward_static``: kept outputs, no workspace), "plain" (``y = layer.forward(x)``)
"""
import math

import numpy as np
import torch

import paper_2412_20386_b200 as ptq

CALIB_IMAGES = 8                      # images from which the forward cases take their static parameters
N_GRID, J_LO = 100, 20                # the step search's grid: 81 candidates
VIM_TI = "192x768,384x44,12x384+bias,384x192"                        # in_proj, x_proj, dt_proj, out_proj
VIM_S = "384x1536,768x384"                                           # in_proj, out_proj
VIM_B = "768x3072,1536x768"
STAGES = ("96x384@3136,192x96@3136,192x768@784,384x192@784,"         # VMamba-like: in_proj and out_proj of the
          "384x1536@196,768x384@196,768x3072@49,1536x768@49")        # four stages at 224 x 224
RAGGED = "129x257@5,40x300@3,16x1000@1,1536x768@49,520x600@197"      # sizes that fill no tile, of the parity tests


def _case(layers, B, T=197, op="forward", scheme="pts", call="buffers", blocks=1, df=3.0, outliers=4, gain=20.0):
    return {"op": op, "scheme": scheme, "call": call, "layers": layers, "T": T, "B": B, "blocks": blocks, "df": df,
            "outliers": outliers, "gain": gain}


def listed():
    heavy = dict(df=2.5, outliers=8, gain=50.0)
    return [
        # one call on one image: what the latency of a single layer is
        dict(_case("384x192", 1), name="vim-ti out_proj, 1 image"),
        # serving: one image through all 24 blocks, 96 calls one after the other, no device memory allocated
        dict(_case(VIM_TI, 1, call="static", blocks=24), name="vim-ti model, 1 image"),
        # the same model on a batch: medium layers, many calls
        dict(_case(VIM_TI, 64, blocks=24), name="vim-ti model, batch 64"),
        # one block's two large linears of the middle model
        dict(_case(VIM_S, 128), name="vim-s block, batch 128"),
        # the largest: long reductions, wide outputs, a heavy tail and strong outliers
        dict(_case(VIM_B, 256, **heavy), name="vim-b block, batch 256"),
        # a hierarchical backbone: from many tokens and few channels to few tokens and many channels
        dict(_case(STAGES, 64), name="vmamba stages, batch 64"),
        # sizes that are multiples of nothing, outputs allocated by the call
        dict(_case(RAGGED, 57, call="plain"), name="ragged layers, batch 57"),
        # zero offsets per token position
        dict(_case(VIM_S, 32, scheme="asym", call="plain"), name="vim-s block asymmetric, batch 32"),
        # 4-bit codes at the batch size of the paper's latency table
        dict(_case(STAGES, 32, scheme="w4a4"), name="vmamba stages w4a4, batch 32"),
        # the dynamic alternative
        dict(_case(VIM_B, 32, scheme="dynamic", **heavy), name="vim-b block dynamic, batch 32"),
        # offline: static parameters of a block's linears from 8 images
        dict(_case(VIM_TI + "," + VIM_S + "," + VIM_B, CALIB_IMAGES, op="calibrate"), name="calibration, 8 images"),
        # offline: refining the steps of a block's linears
        dict(_case(VIM_S, CALIB_IMAGES, op="search"), name="step search, 8 images"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a block of some width, token count and batch, or layers of any odd size."""
    op = rng.choices(["forward", "calibrate", "search"], [8, 1, 1])[0]
    scheme = rng.choices(["pts", "asym", "dynamic", "w4a4"], [5, 1, 1, 1])[0] if op == "forward" else "pts"
    call = rng.choice(["buffers", "buffers", "plain", "static"]) if op == "forward" and scheme != "dynamic" else "buffers"
    while True:
        T = rng.choice([197, 49, 196, 784, 3136, _log(rng, 1, 3136)])
        B = _log(rng, 1, 256) if op == "forward" else rng.randint(2, 16)
        if rng.random() < 0.25:
            layers = ",".join("%dx%d%s" % (_log(rng, 8, 1600), _log(rng, 8, 3072), rng.choice(["", "+bias"]))
                              for _ in range(rng.randint(1, 4)))
        else:
            d = rng.choice([96, 192, 384, 768, 8 * _log(rng, 8, 96)])
            r = (d + 15) // 16
            parts = ["%dx%d" % (d, 4 * d), "%dx%d" % (2 * d, r + 32), "%dx%d+bias" % (r, 2 * d), "%dx%d" % (2 * d, d)]
            layers = ",".join(parts if rng.random() < 0.5 else [parts[0], parts[3]])
        blocks = rng.choice([1, 1, 2, _log(rng, 1, 12)]) if op == "forward" else 1
        case = _case(layers, B, T=T, op=op, scheme=scheme, call=call, blocks=blocks, df=rng.choice([2.5, 3.0]),
                     outliers=rng.choice([4, 8]), gain=rng.choice([20.0, 50.0]))
        w = work(case)
        codes = max(B * t * ((K + 15) // 16 * 16) for K, N, t, bias in parse_layers(case))
        if w["bytes"] > 6e8 or w["flops"] > (3e9 if op == "search" else 3e11) or (call == "static" and codes > ptq.binding.STATIC_SCRATCH_BYTES):
            continue
        return case


def parse_layers(case):
    """"KxN[+bias][@T]" items -> (K, N, T, bias), with the case's T where an item names none."""
    out = []
    for item in case["layers"].split(","):
        shape, _, t = item.partition("@")
        shape, _, bias = shape.partition("+")
        K, N = shape.split("x")
        out.append((int(K), int(N), int(t) if t else case["T"], bias == "bias"))
    return out


def _activations(gen, B, T, K, case, structure):
    """sat_fp16(StudentT(df) * g[t] * o[k]), the library's own workload recipe; one-sided and shifted positions
    where the layer has zero offsets."""
    g, o = structure
    x = torch.empty((B, T, K), dtype=torch.float16, device="cuda")
    df, step = case["df"], max(1, (1 << 24) // (T * K))
    for b in range(0, B, step):
        n = min(step, B - b)
        shape = (n, T, K)
        v = torch.randn(shape, generator=gen, device="cuda")
        chi2 = 2.0 * torch._standard_gamma(torch.full(shape, 0.5 * df, device="cuda"), generator=gen)
        v = v * torch.rsqrt(chi2.clamp_min_(1e-12) / df) * (g[:, None] * o[None, :])
        if case["scheme"] == "asym":
            v = v + (0.75 * g * torch.cos(torch.arange(T, device="cuda", dtype=torch.float32)))[None, :, None]
            v[:, ::7] = v[:, ::7].abs()
        x[b:b + n] = v.clamp_(-65504.0, 65504.0)
    return x


def _structure(gen, T, K, case):
    g = torch.exp(0.5 * torch.randn(T, generator=gen, device="cuda"))
    if T == 197:
        g[98] *= 0.1                                                 # the class token
    o = torch.ones(K, device="cuda")
    o[torch.randperm(K, generator=gen, device="cuda")[:case["outliers"]]] = case["gain"]
    return g, o


def _weights(gen, K, N, bias, w4a4):
    dw = torch.empty(N, device="cuda").uniform_(1e-3, 1e-2, generator=gen).cpu().numpy()
    b = torch.randn(N, generator=gen, device="cuda").cpu().numpy() if bias else None
    if not w4a4:
        return torch.randint(-127, 128, (N, K), generator=gen, device="cuda").to(torch.int8).cpu().numpy(), dw, b
    w = torch.randint(-7, 8, (N, K + K % 2), generator=gen, device="cuda")
    w[:, K:] = 0
    return ((w[:, 1::2] << 4) | (w[:, 0::2] & 15)).bitwise_and_(255).to(torch.uint8).cpu().numpy(), dw, b


def prepare(case, seed):
    shapes, B = parse_layers(case), case["B"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    calls, scheme = [], case["scheme"]
    ys = [torch.zeros((case["blocks"], B, T, N), dtype=torch.float16, device="cuda") if case["call"] != "plain" else None
          for K, N, T, bias in shapes] if case["op"] == "forward" else []
    for block in range(case["blocks"]):
        for i, (K, N, T, bias) in enumerate(shapes):
            structure = _structure(gen, T, K, case)
            wq, dw, b = _weights(gen, K, N, bias, scheme == "w4a4")
            x = _activations(gen, B, T, K, case, structure)
            if case["op"] == "calibrate":
                calls.append((x, wq, dw))
                continue
            if case["op"] == "search":
                calls.append((x,) + ptq.calibrate(x, wq, dw))
                continue
            xcal = _activations(gen, CALIB_IMAGES, T, K, case, structure)
            if scheme == "w4a4":
                s, dx = ptq.calibrate_w4a4(xcal, wq, K, dw)
                layer = ptq.PtqLinear(wq, dw, s, dx, b, packed4_K=K)
            elif scheme == "asym":
                s, dx, z = ptq.calibrate_asym(xcal, wq, dw)
                layer = ptq.PtqLinear(wq, dw, s, dx, b, act_zero=z)
            else:
                s, dx = ptq.calibrate(xcal, wq, dw)
                layer = ptq.PtqLinear(wq, dw, s, dx, b)
            calls.append((layer, x, None if ys[i] is None else ys[i][block]))
    ws = None
    if case["op"] == "forward" and case["call"] == "buffers":
        need = max(layer.workspace_bytes_dynamic(B) if scheme == "dynamic" else layer.workspace_bytes(B) for layer, x, y in calls)
        ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
    return {"op": case["op"], "scheme": scheme, "call": case["call"], "calls": calls, "ys": ys, "ws": ws}


def run(state):
    calls = state["calls"]
    if state["op"] == "calibrate":
        return [ptq.calibrate(x, wq, dw) for x, wq, dw in calls]
    if state["op"] == "search":
        return [ptq.search_act_step(x, s, base, N_GRID, J_LO)[:2] for x, s, base in calls]
    ws, call = state["ws"], state["call"]
    if state["scheme"] == "dynamic":
        for layer, x, y in calls:
            layer.forward_dynamic(x, y=y, workspace=ws)
    elif call == "static":
        for layer, x, y in calls:
            layer.forward_static(x, y)
    elif call == "buffers":
        for layer, x, y in calls:
            layer.forward(x, y=y, workspace=ws)
    else:
        return [layer.forward(x) for layer, x, y in calls]
    return state["ys"]


def work(case):
    bytes_, flops = 0.0, 0.0
    for K, N, T, bias in parse_layers(case):
        M = case["B"] * T
        if case["op"] == "calibrate":                 # x and the weights once, s and dx; |x|, a division and two maxima
            bytes_ += 2 * M * K + N * K + 4 * N + 4 * K + 4 * T
            flops += 4.0 * M * K
        elif case["op"] == "search":                  # x once; quotient, rounding, error and square for every candidate
            bytes_ += 2 * M * K + 4 * K + 12 * T
            flops += 5.0 * M * K * (N_GRID - J_LO + 1)
        else:                                         # x, weights and parameters once, y once
            weights = N * (K + 1) // 2 if case["scheme"] == "w4a4" else N * K
            bytes_ += 2 * M * K + weights + 4 * (N + K + T) + 2 * M * N
            flops += 2.0 * M * K * N
    return {"bytes": bytes_ * case["blocks"], "flops": flops * case["blocks"]}


def tolerance(case):
    # calibration and search return the only correct values (maxima and integer choices, each step correctly rounded)
    if case["op"] != "forward":
        return "exact"
    # the epilogue in 64 bits instead of 32, rounded once: 4e-6 to 6e-6 over the listed layers, at most one binary16 ulp
    return {"rel": 2.5e-5, "max": 2e-3}
