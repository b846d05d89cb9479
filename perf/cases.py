"""Workloads of the library as a user's program runs them, for timing one build against another.

Five kinds of work, each through the public entry points of `paper_2501_04304_b200.binding` with their
default buffers:

  linear  a group-quantized layer on fp16 activations: `quantize_act` followed by `linear`;
  conv    the same for a 3x3 convolution: zero-centred codes and an implicit GEMM;
  cross   cross-attention with log2-quantized scores and a prompt-specific scale;
  self    self-attention with log2-quantized scores;
  setup   what a program does once per layer when it loads a model: calibrate the groups on recorded
          activations, fill the parameter row of a second timestep, prepare the weight, and take the tables and
          codes out to store them.

Calibrated groups, prepared weights and biases are made by `prepare`, as a program that serves a model keeps
them; a pass then covers everything from the fp16 input to the fp16 output.  A layer's outlier positions and
calibration recordings are the model's and the same for every seed (so is the shape of its code rows); weights
and inputs are drawn from the seed.  Inputs follow the recipe of
`synth.py` (normal activations with channel and pixel outliers, a dominant <start> key), drawn on the GPU.
"""
import math

import torch

from paper_2501_04304_b200 import binding as b


def listed():
    return [
        # The smallest call: one 16x16 latent (256 tokens) through a 320 -> 320 projection with static tables over
        # pixel and channel groups (the paper's mode), where launches and the host path count.
        _linear("linear_256x320_320_w8_static", 256, 1, 320, 320, 8, 8, 4, "static", "both"),
        # Cross-attention k/v projection of the text context: 8 prompts of 77 tokens, ragged rows, 4-bit weights.
        _linear("linear_616x768_1280_w4", 77, 8, 768, 1280, 8, 4, 8, "dynamic", "channel"),
        # Stacked q/k/v projection of the 64x64 level at batch 2 (classifier-free guidance), W8A8.
        _linear("linear_8192x320_960_w8", 4096, 2, 320, 960, 8, 8, 8, "dynamic", "channel"),
        # Feed-forward of the 16x16 level at batch 8: a long reduction, 4-bit weights.
        _linear("linear_2048x5120_1280_w4", 256, 8, 5120, 1280, 8, 4, 8, "dynamic", "channel"),
        # GEGLU feed-forward of the 64x64 level, wide outputs: batch 2 W8A8 ...
        _linear("linear_8192x320_2560_w8", 4096, 2, 320, 2560, 8, 8, 8, "dynamic", "channel"),
        # ... and batch 8 W4A8, the layer with the largest output.
        _linear("linear_32768x320_2560_w4", 4096, 8, 320, 2560, 8, 4, 8, "dynamic", "channel"),
        # ResBlock 3x3 convolutions, W4A6 with 16 groups: the 64x64 level at batch 2, the 16x16 level at batch 8.
        _conv("conv_2x64x64x320_320", 2, 64, 64, 320, 320, 16),
        _conv("conv_8x16x16x1280_1280", 8, 16, 16, 1280, 1280, 16),
        # Cross-attention of the 64x64 level at batch 2, 8-bit scores, and of the 32x32 level at batch 8 with 4-bit
        # scores.
        _cross("cross_2x4096x8x40", 2, 8, 4096, 77, 40, 8, "prompt", 0),
        _cross("cross_8x1024x8x80_4bit", 8, 8, 1024, 77, 80, 4, "prompt", 0),
        # Self-attention of the 64x64 level at batch 2: the heaviest attention of a denoising step.
        _self("self_2x4096x8x40", 2, 8, 4096, 40, 8, False),
        # Loading one layer: the 640 -> 5120 feed-forward of the 32x32 level, 4-bit weights, 8 groups.
        _setup("setup_640_5120_w4", 1024, 4, 640, 5120, 8, 4, 8, "channel", False),
    ]


def _linear(name, tokens, batch, c, n, act_bits, w_bits, groups, mode, dim):
    return dict(name=name, kind="linear", tokens=tokens, batch=batch, c=c, n=n, act_bits=act_bits, w_bits=w_bits,
                groups=groups, mode=mode, dim=dim)


def _conv(name, images, h, w, c, n, groups, w_bits=4, act_bits=6):
    return dict(name=name, kind="conv", images=images, h=h, w=w, c=c, n=n, groups=groups, w_bits=w_bits,
                act_bits=act_bits)


def _cross(name, batch, heads, nq, nk, d, bits, scale, v_bits):
    return dict(name=name, kind="cross", batch=batch, heads=heads, nq=nq, nk=nk, d=d, bits=bits, scale=scale,
                v_bits=v_bits)


def _self(name, batch, heads, tokens, d, bits, fixed):
    return dict(name=name, kind="self", batch=batch, heads=heads, tokens=tokens, d=d, bits=bits, fixed=fixed)


def _setup(name, tokens, samples, c, n, act_bits, w_bits, groups, dim, conv):
    return dict(name=name, kind="setup", tokens=tokens, samples=samples, c=c, n=n, act_bits=act_bits, w_bits=w_bits,
                groups=groups, dim=dim, conv=conv)


# ------------------------------------------------------------------------------------------ further cases
def _log_int(rng, lo, hi, step=1):
    """An integer between lo and hi, a multiple of step, spread over the logarithm of the range."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, int(round(v / step)) * step))


def draw(rng):
    """One more case.  Half the widths are the UNet's own channel counts, the others any multiple of 8; token and
    query counts are any integer."""
    def width(lo, hi):
        own = [v for v in (320, 640, 768, 960, 1280, 2048, 2560, 5120) if lo <= v <= hi]
        return rng.choice(own) if rng.random() < 0.5 else _log_int(rng, lo, hi, 8)

    kind = rng.choice(["linear"] * 5 + ["conv"] * 2 + ["cross"] * 3 + ["self"] * 2 + ["setup"])
    while True:
        if kind == "linear":
            mode = rng.choice(["dynamic", "static"])
            c = _linear("", _log_int(rng, 16, 4096), rng.randint(1, 8), width(64, 5120), width(64, 5120),
                        rng.choice([8, 8, 6]), rng.choice([8, 4]), rng.choice([4, 8, 16]), mode,
                        rng.choice(["channel", "both", "auto"]) if mode == "static" else "channel")
            m = c["tokens"] * c["batch"]
            ok = m * c["c"] * c["n"] <= 32768 * 320 * 2560 and m * (c["c"] + c["n"]) <= 32768 * 2880 and \
                c["c"] * c["n"] <= 5120 * 1280
        elif kind == "conv":
            # image widths that divide a 128-row tile, heights that fill it (square and wide or tall images)
            w = rng.choice([8, 16, 32, 64])
            h = max(w, 128 // w) if rng.random() < 0.5 else (128 // w) * rng.randint(1, 24)
            if w == 8 and rng.random() < 0.3:
                h = 8
            c = _conv("", rng.randint(1, 8), h, w, width(64, 1280), width(64, 1280), rng.choice([8, 16]))
            m = c["images"] * h * w
            ok = m * c["c"] * c["n"] <= 2048 * 1280 * 1280 and m * (c["c"] + c["n"]) <= 32768 * 640
        elif kind == "cross":
            c = _cross("", rng.randint(1, 8), rng.choice([5, 8, 10, 20]), _log_int(rng, 16, 4096),
                       77 if rng.random() < 0.7 else rng.randint(2, 128), rng.choice([40, 64, 80, 160]),
                       rng.choice([8, 4]), rng.choice(["prompt", "prompt", "head", "call"]), rng.choice([0, 0, 8]))
            ok = c["batch"] * c["heads"] * c["nq"] * c["d"] <= 8 * 8 * 4096 * 40
        elif kind == "self":
            c = _self("", rng.randint(1, 8), rng.choice([5, 8, 10, 20]), _log_int(rng, 48, 4096),
                      rng.choice([40, 64, 80, 160]), rng.choice([8, 4]), rng.random() < 0.25)
            ok = c["batch"] * c["heads"] * c["tokens"] ** 2 * c["d"] <= 2 * 8 * 4096 ** 2 * 40
        else:
            conv = rng.random() < 0.3
            c = _setup("", _log_int(rng, 64, 4096), rng.randint(1, 4), width(64, 1280), width(64, 5120),
                       6 if conv else 8, 4 if conv else rng.choice([8, 4]), rng.choice([8, 16]),
                       "channel" if conv else rng.choice(["channel", "both", "auto"]), conv)
            ok = c["c"] * c["n"] * (9 if conv else 1) <= 640 * 5120 and c["tokens"] * c["samples"] * c["c"] <= 4096 * 640
        if ok:
            del c["name"]
            return c


# ------------------------------------------------------------------------------------------ inputs
_DIM = {"auto": b.DIM_AUTO, "channel": b.DIM_CHANNEL, "both": b.DIM_BOTH}
_SCALE = {"prompt": b.SCALE_PER_PROMPT, "head": b.SCALE_PER_PROMPT_HEAD, "call": b.SCALE_PER_CALL}


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda")


class _Activations:
    """fp16 activations [samples * tokens, c]: normal, x30 on 1 % of the channels, x20 on 0.5 % of the pixel
    positions; the outlier positions stay the same from draw to draw, as they do from prompt to prompt."""

    def __init__(self, gen, tokens, c, pixel_outliers=True):
        self.tokens, self.c = tokens, c
        self.gain_c = torch.ones(c, device="cuda")
        self.gain_c[torch.randperm(c, generator=gen, device="cuda")[:math.ceil(0.01 * c)]] = 30.0
        self.gain_t = torch.ones(tokens, 1, device="cuda")
        if pixel_outliers:
            n = max(1, round(0.005 * tokens))
            self.gain_t[torch.randperm(tokens, generator=gen, device="cuda")[:n]] = 20.0

    def draw(self, gen, samples, gain=1.0):
        x = _normal(gen, samples, self.tokens, self.c) * (self.gain_c * gain)
        return (x * self.gain_t).half().reshape(samples * self.tokens, self.c)


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind in ("linear", "conv"):
        conv = None
        tokens, samples = case.get("tokens"), case.get("batch")
        if kind == "conv":
            tokens, samples = case["h"] * case["w"], case["images"]
            conv = (case["images"], case["h"], case["w"], case["c"])
        model = _generator(1)
        act = _Activations(model, tokens, case["c"], pixel_outliers=kind == "linear")
        groups = b.calibrate_groups(act.draw(model, 2), tokens, case["act_bits"], case["groups"],
                                    _DIM["channel" if kind == "conv" else case["dim"]])
        w = (_normal(gen, case["n"], (9 if conv else 1) * case["c"]) * 0.02).half()
        return dict(kind=kind, groups=groups, conv=conv, x=act.draw(gen, samples),
                    weight=b.weight_prepare(groups, w, case["w_bits"], conv=conv),
                    bias=(_normal(gen, case["n"]) * 0.01).half(),
                    mode=b.MODE_DYNAMIC_TOKEN if case.get("mode") == "dynamic" else b.MODE_STATIC,
                    layout=b.CODES_S8_CENTRED if conv else b.CODES_U8)
    if kind == "cross":
        B, H, nq, nk, d = (case[k] for k in ("batch", "heads", "nq", "nk", "d"))
        q = _normal(gen, B, nq, H, d)
        ctx = _normal(gen, B * nk, 768)
        k = (ctx @ (_normal(gen, 768, H * d) * 0.02)).reshape(B, nk, H, d)
        v = (ctx @ (_normal(gen, 768, H * d) * 0.02)).reshape(B, nk, H, d)
        q[..., d - 1] = 1.0          # the <start> key's logit bias of about +6
        k[:, 0, :, d - 1] = 6.0 * math.sqrt(d)
        k[:, 1:, :, d - 1] = 0.0
        return dict(kind=kind, q=q.half(), k=k.half(), v=v.half(), bits=case["bits"], scale=_SCALE[case["scale"]],
                    v_bits=case["v_bits"])
    if kind == "self":
        q, k, v = (_normal(gen, case["batch"], case["tokens"], case["heads"], case["d"]).half() for _ in range(3))
        fixed = torch.full((case["batch"],), 0.25, device="cuda") if case["fixed"] else None
        return dict(kind=kind, q=q, k=k, v=v, bits=case["bits"], fixed=fixed)
    act = _Activations(gen, case["tokens"], case["c"], pixel_outliers=not case["conv"])
    conv = (1, 1, case["tokens"], case["c"]) if case["conv"] else None
    return dict(kind=kind, x0=act.draw(gen, case["samples"]), x1=act.draw(gen, case["samples"], 1.5), conv=conv,
                w=(_normal(gen, case["n"], (9 if conv else 1) * case["c"]) * 0.02).half(), tokens=case["tokens"],
                act_bits=case["act_bits"], w_bits=case["w_bits"], groups=case["groups"], dim=_DIM[case["dim"]])


# ------------------------------------------------------------------------------------------ one pass
def run(state):
    s = state
    if s["kind"] in ("linear", "conv"):
        xq, scale, zp = b.quantize_act(s["groups"], s["x"], mode=s["mode"], layout=s["layout"])
        y = b.linear(s["groups"], s["weight"], xq, mode=s["mode"], layout=s["layout"], dyn_scale=scale, dyn_zp=zp,
                     bias=s["bias"], conv=s["conv"])
        return dict(codes=xq, scale=scale, zp=zp, y=y)
    if s["kind"] == "cross":
        o, scale, _ = b.cross_attn_logq(s["q"], s["k"], s["v"], s["bits"], s["scale"], want_scale=True,
                                        v_bits=s["v_bits"])
        return dict(o=o, scale=scale)
    if s["kind"] == "self":
        return b.self_attn_logq(s["q"], s["k"], s["v"], s["bits"], fixed_scale=s["fixed"])[0]
    cfg = dict(rows_per_sample=s["tokens"], act_bits=s["act_bits"], n_groups=s["groups"], dim_select=s["dim"],
               n_timesteps=2)
    groups = b.calibrate_groups(s["x0"], timestep=0, **cfg)
    b.calibrate_groups(s["x1"], timestep=1, groups=groups, **cfg)
    weight = b.weight_prepare(groups, s["w"], s["w_bits"], conv=s["conv"])
    codes, w_scale = weight.export()
    tables = groups.export()
    return dict(col_group=tables["col_group"], row_group=tables["row_group"], scale=tables["scale"], zp=tables["zp"],
                codes=codes, w_scale=w_scale)


# ------------------------------------------------------------------------------------------ what a pass needs
def work(case):
    kind = case["kind"]
    if kind in ("linear", "conv"):
        m = case["images"] * case["h"] * case["w"] if kind == "conv" else case["tokens"] * case["batch"]
        c, n = case["c"], case["n"]
        k = 9 * c if kind == "conv" else c
        # input, codes, weight, bias and output once each; (scale, zero-point) of every token and group
        params = 8 * m * case["groups"] if case.get("mode") == "dynamic" else 0
        return {"bytes": 2 * m * c + m * c + n * k * case["w_bits"] // 8 + 2 * n + 2 * m * n + params,
                "flops": 2 * m * n * k}
    if kind in ("cross", "self"):
        B, H, d = case["batch"], case["heads"], case["d"]
        nq = case["nq"] if kind == "cross" else case["tokens"]
        nk = case["nk"] if kind == "cross" else nq
        return {"bytes": 4 * B * H * nq * d + 4 * B * H * nk * d, "flops": 4 * B * H * nq * nk * d}
    k = (9 if case["conv"] else 1) * case["c"]
    # both calibration sets and the fp16 weight are read, the codes are written
    return {"bytes": 4 * case["tokens"] * case["samples"] * case["c"] + 3 * case["n"] * k, "flops": 0}


def tolerance(case):
    kind = case["kind"]
    if kind == "setup":
        return "exact"      # codes, tables and layouts
    if kind in ("linear", "conv"):
        # Codes and zero-points are exact.  Outputs are fp16: integer products and fp32 sums in another order may
        # round to the neighbouring fp16 value.
        return {"rel": 3e-4, "max": 2e-3, "differ": 0.0}
    # fp16 outputs, and a score on a rounding boundary may take the neighbouring power of two, which moves its
    # row's output by half that score's contribution (at most 1e-4 of the scores do).
    return {"rel": 2e-3, "max": 0.5}
