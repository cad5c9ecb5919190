"""What the speed of this library is measured on: the work that a program quantizing and running a diffusion
U-Net has it do, through the binding's public calls.

Layer shapes are those of the Stable-Diffusion-v1-style U-Net (width 320, levels 1/2/4/4, 64 x 64 latent), the
DDIM-CIFAR-style and the LDM-4-style convolutions of paper_2408_06995_b200/inputs.py.  A program keeps a layer's
prepared weights, its scales, its output buffer and one workspace; a pass gets them and the FP32 activations.
"""
import math

import torch

import paper_2408_06995_b200 as fpq

FORMATS = {"e4m3": fpq.E4M3, "e5m2": fpq.E5M2, "e2m1": fpq.E2M1, "e1m2": fpq.E1M2, "e3m4": fpq.E3M4, "e2m5": fpq.E2M5}
# the encodings that the search visits, with the paper's clipping value
SEARCH = {"fp8": [fpq.Format(2, 5, 2), fpq.Format(3, 4, 4), fpq.Format(4, 3, 7), fpq.Format(5, 2, 15)],
          "fp4": [fpq.E1M2, fpq.E2M1]}
CLIPS = 111


def listed():
    return [
        # the smallest call: a residual block's time-embedding projection, one row per image of a batch of two
        {"name": "linear_time_embed", "kind": "linear", "M": 2, "K": 1280, "N": 1280, "fx": "e4m3", "fw": "e2m1"},
        # self-attention QKV at the 64 x 64 level, batch 2, FP8 weights
        {"name": "linear_qkv", "kind": "linear", "M": 8192, "K": 320, "N": 960, "fx": "e4m3", "fw": "e4m3"},
        # feed-forward input at the 64 x 64 level, batch 16 (throughput serving): the largest output
        {"name": "linear_geglu_batch16", "kind": "linear", "M": 65536, "K": 320, "N": 2560, "fx": "e4m3", "fw": "e2m1"},
        # feed-forward output at the 32 x 32 level with an encoding that the search selects for weights
        {"name": "linear_ffn_out_e3m4", "kind": "linear", "M": 2048, "K": 2560, "N": 640, "fx": "e4m3", "fw": "e3m4"},
        # DDIM-CIFAR-style 3 x 3 convolution, a sampling batch of 64 images, FP8
        {"name": "conv_ddim_w8a8", "kind": "conv", "B": 64, "C": 128, "H": 32, "W": 32, "Co": 128, "R": 3, "stride": 1,
         "fx": "e4m3", "fw": "e4m3"},
        # LDM-4-style 3 x 3 convolution, FP4 weights with learned rounding
        {"name": "conv_ldm_w4a8", "kind": "conv", "B": 16, "C": 256, "H": 32, "W": 32, "Co": 256, "R": 3, "stride": 1,
         "fx": "e4m3", "fw": "e2m1"},
        # deepest level of the U-Net at batch 2: little work, a long reduction, latency counts
        {"name": "conv_deep_8x8", "kind": "conv", "B": 2, "C": 1280, "H": 8, "W": 8, "Co": 1280, "R": 3, "stride": 1,
         "fx": "e4m3", "fw": "e2m1"},
        # a downsampling convolution of an image whose sizes are not powers of two
        {"name": "conv_down_ragged", "kind": "conv", "B": 3, "C": 320, "H": 45, "W": 77, "Co": 320, "R": 3, "stride": 2,
         "fx": "e4m3", "fw": "e4m3"},
        # decoder residual block: skip connection and previous output quantized with their own scales
        {"name": "conv_concat_64x64", "kind": "split", "B": 2, "C1": 640, "C2": 320, "H": 64, "W": 64, "Co": 320, "R": 3,
         "fx": "e4m3", "fw": "e2m1"},
        # the nine layers of one transformer block at the 32 x 32 level, batch 2, in execution order
        {"name": "block_640_32x32", "kind": "block", "B": 2, "C": 640, "res": 32, "fx": "e4m3", "fw": "e2m1"},
        # choosing a layer's weight encoding and bias: 4 x 111 candidates on a 640 x 640 3 x 3 convolution
        {"name": "search_fp8_weights", "kind": "search", "n": 640 * 640 * 9, "set": "fp8", "law": "weights"},
        # learning a layer's FP4 rounding: one evaluation and descent step on 4096 calibration rows
        {"name": "learn_qkv_step", "kind": "learn", "M": 4096, "N": 960, "K": 320, "fw": "e2m1"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    # most widths are multiples of 32; some are not even multiples of 4
    c = _log(rng, lo, hi)
    return c if rng.random() < 0.2 else max(32, c // 32 * 32)


def draw(rng):
    """One more layer (or offline step) of the ranges above."""
    largest = work(listed()[2])["bytes"]
    fmts = {"fx": rng.choice(["e4m3"] * 10 + ["e5m2", "e3m4"]), "fw": rng.choice(["e4m3"] * 4 + ["e2m1"] * 5 + ["e1m2", "e3m4", "e5m2"])}
    while True:
        kind = rng.choice(["linear"] * 5 + ["conv"] * 5 + ["split", "block", "search", "learn"])
        if kind == "linear":
            c = {"kind": kind, "M": _log(rng, 1, 65536), "K": _channels(rng, 64, 5120), "N": _channels(rng, 64, 10240), **fmts}
        elif kind == "conv":
            res = _log(rng, 7, 64)
            image = rng.choice([3, 4] + 8 * [0])   # the U-Net's first convolution reads the image itself
            c = {"kind": kind, "B": _log(rng, 1, 64), "C": image or _channels(rng, 64, 1920), "H": res,
                 "W": rng.choice([res, res, rng.randint(7, 96)]), "Co": _channels(rng, 64, 1280), "R": rng.choice([1, 3, 3]),
                 "stride": rng.choice([1, 1, 1, 1, 2]), **fmts}
        elif kind == "split":
            res = rng.choice([8, 16, 32, 64, rng.randint(8, 64)])
            c = {"kind": kind, "B": rng.randint(1, 4), "C1": 320 * rng.randint(1, 4), "C2": 320 * rng.randint(1, 4), "H": res,
                 "W": res, "Co": 320 * rng.randint(1, 4), "R": 3, "fx": "e4m3", "fw": rng.choice(["e4m3", "e2m1"])}
        elif kind == "block":
            lvl = rng.randint(0, 3)
            c = {"kind": kind, "B": rng.choice([1, 2, 2, 3, 4]), "C": (320, 640, 1280, 1280)[lvl],
                 "res": (64, 32, 16, 8)[lvl] + rng.choice([0, 0, 1, -1]), "fx": "e4m3", "fw": rng.choice(["e4m3", "e2m1"])}
        elif kind == "search":
            c = {"kind": kind, "n": _log(rng, 4096, 1 << 24), "set": rng.choice(["fp8", "fp4"]),
                 "law": rng.choice(["weights", "silu", "outliers"])}
        else:
            c = {"kind": kind, "M": _log(rng, 64, 8192), "N": _channels(rng, 128, 2560), "K": _channels(rng, 128, 2560),
                 "fw": rng.choice(["e2m1", "e2m1", "e1m2"])}
        w = work(c)
        if w["bytes"] <= largest / 2 and w["flops"] <= (4e10 if kind == "learn" else 2e11):
            return c


# ---- inputs ------------------------------------------------------------------------------------------------------


def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)


def _activations(gen, *shape):
    """What a layer of the U-Net reads: SiLU outputs, with the few large entries that transformer layers have."""
    x = torch.nn.functional.silu(_normal(gen, *shape))
    at = torch.randint(x.numel(), (max(1, x.numel() // 2000),), generator=gen, device="cuda")
    x.view(-1)[at] *= 10.0
    return x


def _act_scale(x, fx):
    return fpq.fpq_scale_from_max(float(x.abs().max()), fx)


def _codes(gen, N, K, fw):
    """Encoded weights [N][K] and their scale per output channel; FP4 weights have learned rounding decisions."""
    w = _normal(gen, N, K) * 0.02
    scale = (w.abs().amax(dim=1) / fpq.fpq_format_max(fw)).contiguous()
    bits = None
    if fw.four_bit:
        bits = torch.randint(256, (N, (K + 7) // 8), generator=gen, device="cuda", dtype=torch.uint8)
    return fpq.fpq_quantize_weight(w, scale, fw, bits), scale


def _bias(gen, N):
    return _normal(gen, N) * 0.01


def _linear(gen, M, K, N, fx, fw):
    x = _activations(gen, M, K)
    codes, scale = _codes(gen, N, K, fw)
    return {"kind": "linear", "x": x, "w": fpq.fpq_prepare_weight(codes, fw, fpq.LINEAR, N, K), "scale": scale,
            "x_scale": _act_scale(x, fx), "fx": fx, "fw": fw, "bias": _bias(gen, N), "N": N,
            "y": torch.empty(M, N, device="cuda"), "ws": fpq.fpq_linear_workspace_size(M, N, K, fx, fw)}


def _out(n, R, stride):
    return (n + 2 * (R // 2) - R) // stride + 1


def _conv(gen, B, C, H, W, Co, R, stride, fx, fw):
    x = _activations(gen, B, C, H, W)
    codes, scale = _codes(gen, Co, C * R * R, fw)
    return {"kind": "conv", "x": x, "w": fpq.fpq_prepare_weight(codes, fw, fpq.CONV2D, Co, C, R, R), "scale": scale,
            "x_scale": _act_scale(x, fx), "fx": fx, "fw": fw, "bias": _bias(gen, Co), "Co": Co, "R": R, "pad": R // 2,
            "stride": stride, "y": torch.empty(B, Co, _out(H, R, stride), _out(W, R, stride), device="cuda"),
            "ws": fpq.fpq_conv2d_workspace_size(B, C, H, W, Co, R, R, R // 2, stride, fx, fw)}


def _block_layers(c):
    """(kind, rows or resolution, inputs, outputs) of a transformer block; 77 text tokens of width 768."""
    C, res, T = c["C"], c["res"], c["B"] * c["res"] ** 2
    return [("conv", res, C, C), ("linear", T, C, 3 * C), ("linear", T, C, C), ("linear", T, C, C),
            ("linear", c["B"] * 77, 768, 2 * C), ("linear", T, C, C), ("linear", T, C, 8 * C), ("linear", T, 4 * C, C),
            ("conv", res, C, C)]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "search":
        n = case["n"]
        if case["law"] == "weights":
            x = _normal(gen, n) * 0.02
        elif case["law"] == "silu":
            x = torch.nn.functional.silu(_normal(gen, n))
        else:
            x = _activations(gen, n) * 3.0
        encs = SEARCH[case["set"]]
        clip = fpq.fpq_search_clip_candidates(float(x.abs().max()), CLIPS).cuda()
        return {"kind": kind, "x": x, "encs": encs, "clip": clip,
                "mse": torch.empty(len(encs), CLIPS, dtype=torch.float64, device="cuda"),
                "best": torch.empty(2, dtype=torch.int32, device="cuda"),
                "workspace": torch.empty(fpq.fpq_search_workspace_size(len(encs), CLIPS), dtype=torch.uint8, device="cuda")}
    fw = FORMATS[case["fw"]]
    if kind == "learn":
        M, N, K = case["M"], case["N"], case["K"]
        w = _normal(gen, N, K) * 0.02
        return {"kind": kind, "w": w, "scale": (w.abs().amax(dim=1) / fpq.fpq_format_max(fw)).contiguous(), "fmt": fw,
                "start": _normal(gen, N, K) * 0.5, "alpha": torch.empty(N, K, device="cuda"), "a": _activations(gen, M, K),
                "grad": torch.empty(N, K, device="cuda"), "loss": torch.empty(2, dtype=torch.float64, device="cuda"),
                "workspace": torch.empty(fpq.fpq_round_learn_workspace_size(M, N, K), dtype=torch.uint8, device="cuda")}
    fx = FORMATS[case["fx"]]
    if kind == "split":
        B, C1, C2, H, W, Co, R = (case[k] for k in ("B", "C1", "C2", "H", "W", "Co", "R"))
        x1, x2 = _activations(gen, B, C1, H, W), _normal(gen, B, C2, H, W) * 3.0
        codes, scale = _codes(gen, Co, (C1 + C2) * R * R, fw)
        ws = fpq.fpq_conv2d_split_workspace_size(B, C1, C2, H, W, Co, R, R, R // 2, 1, fx, fw)
        return {"kind": kind, "x1": x1, "x2": x2, "s1": _act_scale(x1, fx), "s2": _act_scale(x2, fx), "fx": fx, "fw": fw,
                "w": fpq.fpq_prepare_weight_split(codes, fw, Co, C1, C2, R, R), "scale": scale, "bias": _bias(gen, Co), "R": R,
                "y": torch.empty(B, Co, H, W, device="cuda"), "workspace": torch.empty(ws, dtype=torch.uint8, device="cuda")}
    if kind == "linear":
        layers = [_linear(gen, case["M"], case["K"], case["N"], fx, fw)]
    elif kind == "conv":
        layers = [_conv(gen, *(case[k] for k in ("B", "C", "H", "W", "Co", "R", "stride")), fx, fw)]
    else:
        layers = [_conv(gen, case["B"], cin, m, m, cout, 1, 1, fx, fw) if what == "conv" else _linear(gen, m, cin, cout, fx, fw)
                  for what, m, cin, cout in _block_layers(case)]
    # one workspace for all layers of a model
    ws = torch.empty(max(256, max(L["ws"] for L in layers)), dtype=torch.uint8, device="cuda")
    return {"kind": "layers", "layers": layers, "workspace": ws}


# ---- the pass ----------------------------------------------------------------------------------------------------


def run(state):
    kind = state["kind"]
    if kind == "layers":
        out = []
        for L in state["layers"]:
            if L["kind"] == "linear":
                out.append(fpq.fpq_linear(L["x"], L["w"], L["scale"], L["x_scale"], L["fx"], L["fw"], L["bias"], L["N"], L["y"],
                                          state["workspace"]))
            else:
                out.append(fpq.fpq_conv2d(L["x"], L["w"], L["scale"], L["x_scale"], L["fx"], L["fw"], L["bias"], L["Co"], L["R"],
                                          L["R"], L["pad"], L["stride"], L["y"], state["workspace"]))
        return out
    s = state
    if kind == "split":
        return fpq.fpq_conv2d_split(s["x1"], s["s1"], s["x2"], s["s2"], s["w"], s["scale"], s["fx"], s["fw"], s["bias"], s["y"],
                                    s["R"], s["R"], s["R"] // 2, 1, s["workspace"])
    if kind == "search":
        return fpq.fpq_search_format(s["x"], s["encs"], s["clip"], s["mse"], s["best"], s["workspace"])
    # a descent step from the same start each time, so that a pass can be repeated
    s["alpha"].copy_(s["start"])
    grad, loss = fpq.fpq_round_learn_step(s["w"], s["scale"], s["fmt"], s["alpha"], s["a"], 1e-6, 1e6, s["grad"], s["loss"],
                                          s["workspace"])
    return {"grad": grad, "loss": loss, "alpha": s["alpha"]}


def work(case):
    """Each input read once, each output written once; multiply-adds count two operations."""
    kind = case["kind"]
    if kind == "search":
        # (how often the data has to be looked at per candidate depends on the method: only the data itself is counted)
        return {"bytes": 4 * case["n"] + 12 * CLIPS * len(SEARCH[case["set"]]), "flops": 0}
    if kind == "learn":
        M, N, K = case["M"], case["N"], case["K"]
        # weights, alpha in and out, gradient; calibration rows; the layer-output error and its product with the rows
        return {"bytes": 4 * (4 * N * K + M * K), "flops": 4 * M * N * K}
    bits = 4 if FORMATS[case["fw"]].four_bit else 8

    def layer(n_in, n_out, N, K, M):
        return {"bytes": 4 * n_in + N * K * bits // 8 + 4 * n_out + 8 * N, "flops": 2 * M * N * K}

    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        return layer(M * K, M * N, N, K, M)
    if kind == "block":
        ws = []
        for what, m, cin, cout in _block_layers(case):
            rows = case["B"] * m * m if what == "conv" else m
            ws.append(layer(rows * cin, rows * cout, cout, cin, rows))
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    stride = case.get("stride", 1)
    B, H, W, Co, R = (case[k] for k in ("B", "H", "W", "Co", "R"))
    C = case["C"] if kind == "conv" else case["C1"] + case["C2"]
    pixels = B * _out(H, R, stride) * _out(W, R, stride)
    return layer(B * C * H * W, pixels * Co, Co, C * R * R, pixels)


def tolerance(case):
    """Products are exact in every layer and sums are FP32, so the order of the additions is all that may differ: against
    64-bit sums the layers show up to 2e-7 (largest single difference 1e-6), the loss of the learning step 4e-6 and the
    search, whose error terms are single FP32 roundings, 5e-8 at its largest size and more at small ones."""
    if case["kind"] == "learn":
        return {"rel": 2e-5, "max": 4e-4}
    return {"rel": 2e-6, "max": 2e-5}
