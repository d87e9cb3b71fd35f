"""Workloads that the speed of the mixers is judged on.

A case is a plain dict.  ``path`` says which public calls a pass makes:

* ``mixers``: one mixer (a schedule of one letter: ``linear_attn``, ``window_attn`` or ``full_attn``) or a stack of
  them (``hybrid_mixers``) on query, key and value tensors that are there already;
* ``block``: a whole token-mixing block, ``qkv_proj`` -> mixer -> ``out_proj``, from token-major activations.

Sizes are those of the configurations, tests and benchmark of this repository (16 x 16 up to 128 x 128 tokens, 6 to 24
heads of 64 or 8 of 128 channels, 0 / 1 / 5 prefix tokens) and the ranges between them.  Outputs and scratch are
allocated once, as a program that runs the same model on one image after the other keeps them.
"""
import torch

from paper_2605_26636_b200 import inputs
from paper_2605_26636_b200 import jetvit as jv

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(path, schedule, B, H, Hg, Wg, D=64, dtype="bf16", win=16, prefix=0, dwc="none", layout="bhnd"):
    return {"path": path, "schedule": schedule, "B": B, "H": H, "Hg": Hg, "Wg": Wg, "D": D, "dtype": dtype, "win": win,
            "prefix": prefix, "dwc": dwc, "layout": layout}


def listed():
    """The listed cases, smallest work first within each group."""
    named = {
        # One layer of each kind on the 16 x 16 oracle-check grid in fp32: three tiny calls, launch latency and host work.
        "tiny_f32": _case("mixers", "LWF", 1, 6, 16, 16, dtype="f32", win=8),
        # fp32 as an accuracy check of a model runs it: one 512 x 512 image at patch 16, base-size heads.
        "image_f32": _case("mixers", "LWF", 1, 12, 32, 32, dtype="f32", win=16, dwc="squeeze"),
        # One 518 x 518 image at patch 14 (37 x 37 tokens and the class token) through a short stack of a small model:
        # what an interactive user waits for.
        "small_image": _case("mixers", "LWLWLF", 1, 6, 37, 37, prefix=1, dwc="squeeze"),
        # Many 256 x 256 images at once (16 x 16 tokens each), q, k and v left in the fused activation of a QKV layer.
        "lowres_batch": _case("mixers", "LWF", 32, 12, 16, 16, win=8, dwc="squeeze", layout="fused"),
        # The linear block alone, without and with its convolution, at 1024 x 1024 / 16, eight images, 16 heads.
        "linear_64x64": _case("mixers", "L", 8, 16, 64, 64),
        "linear_dwc_64x64": _case("mixers", "L", 8, 16, 64, 64, dwc="squeeze"),
        # Window attention at the same shape, without and with five prefix tokens (class token and four registers).
        "window_64x64": _case("mixers", "W", 8, 16, 64, 64),
        "window_64x64_prefix": _case("mixers", "W", 8, 16, 64, 64, prefix=5),
        # Full attention on a grid that no tile divides: 1022 x 1022 / 14.
        "full_73x73": _case("mixers", "F", 4, 16, 73, 73),
        # A whole linear block of a base-size model on 1024 x 2048 images: projections either side of the mixer.
        "block_64x128": _case("block", "L", 2, 12, 64, 128, dwc="squeeze"),
        # Heads of 128 channels, one layer of each kind.
        "head128_64x64": _case("mixers", "LWF", 2, 8, 64, 64, D=128),
        # The 24-layer hybrid stack at 2048 x 2048 / 16: the largest call.
        "hybrid24_128x128": _case("mixers", inputs.HYBRID_SCHEDULE, 1, 16, 128, 128, dwc="squeeze"),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _grid(rng, lo, hi, most):
    """A token grid, ragged more often than not, sides in [lo, hi] and at most ``most`` tokens."""
    while True:
        Hg, Wg = _log_uniform(rng, lo, hi), _log_uniform(rng, lo, hi)
        if rng.random() < 0.3:
            Wg = Hg
        if Hg * Wg <= most:
            return Hg, Wg


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["f32", "stack", "stack", "lowres", "linear", "linear", "window", "window", "full", "block", "head128"])
    prefix = rng.choice([0, 0, 1, 5])
    dwc = rng.choice(["none", "static", "squeeze", "squeeze"])
    heads = rng.choice([6, 12, 16, 24])
    if kind == "f32":
        Hg, Wg = _grid(rng, 12, 40, 1400)
        return _case("mixers", rng.choice(["L", "W", "F", "LWF"]), rng.randint(1, 2), rng.choice([6, 12]), Hg, Wg, dtype="f32",
                     win=rng.choice([8, 16]), prefix=prefix, dwc=dwc)
    if kind == "stack":                       # one image through a few layers, small model to large
        Hg, Wg = _grid(rng, 14, 128, 9000)
        return _case("mixers", rng.choice(["LWF", "LWLWLF", "LLWLLF"]), 1, heads, Hg, Wg, prefix=prefix, dwc=dwc)
    if kind == "lowres":                      # many small images
        Hg, Wg = _grid(rng, 12, 24, 576)
        return _case("mixers", rng.choice(["L", "W", "F", "LWF"]), _log_uniform(rng, 8, 64), rng.choice([6, 12]), Hg, Wg,
                     win=rng.choice([8, 16]), dwc=dwc, layout=rng.choice(["bhnd", "fused"]))
    if kind == "linear":
        Hg, Wg = _grid(rng, 24, 128, 10000)
        layout = rng.choice(["bhnd", "bhnd", "fused"])
        return _case("mixers", "L", rng.randint(1, 8), heads, Hg, Wg, prefix=0 if layout == "fused" else prefix, dwc=dwc,
                     layout=layout)
    if kind == "window":
        Hg, Wg = _grid(rng, 24, 128, 10000)
        layout = rng.choice(["bhnd", "bhnd", "fused"])
        return _case("mixers", "W", rng.randint(1, 8), heads, Hg, Wg, win=rng.choice([8, 16, 16]),
                     prefix=0 if layout == "fused" else prefix, layout=layout)
    if kind == "full":
        Hg, Wg = _grid(rng, 24, 90, 7000)
        return _case("mixers", "F", rng.randint(1, 4), heads, Hg, Wg, prefix=prefix)
    if kind == "block":
        Hg, Wg = _grid(rng, 24, 128, 9000)
        return _case("block", rng.choice(["L", "L", "W"]), rng.randint(1, 3), heads, Hg, Wg, prefix=prefix, dwc=dwc)
    Hg, Wg = _grid(rng, 20, 64, 4096)
    return _case("mixers", rng.choice(["L", "W", "F", "LWF"]), rng.randint(1, 3), 8, Hg, Wg, D=128)


def _seeded(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(gen, shape, std=1.0, dtype=torch.float32):
    return (torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32) * std).to(dtype)


def _dwc(gen, case):
    """The convolution of one linear layer: a generator of C / 8 hidden units, or static kernels; centre taps of 0.1
    as ``inputs.dwc_weights`` has them."""
    if case["dwc"] == "none":
        return None
    C = case["H"] * case["D"]
    b2 = torch.zeros(C, 3, 3, device="cuda")
    b2[:, 1, 1] = 0.1
    if case["dwc"] == "static":
        return {"k": 3, "R": 0, "b2": (b2 + _normal(gen, (C, 3, 3), 0.2)).reshape(-1).contiguous()}
    R = C // 8
    return {"k": 3, "R": R, "W1": _normal(gen, (R, C), C ** -0.5), "b1": torch.zeros(R, device="cuda"),
            "W2": _normal(gen, (C * 9, R), R ** -0.5), "b2": b2.reshape(-1)}


def prepare(case, seed):
    gen = _seeded(seed)
    dt = DTYPES[case["dtype"]]
    B, H, D = case["B"], case["H"], case["D"]
    N = case["prefix"] + case["Hg"] * case["Wg"]
    n = len(case["schedule"])
    dwc = [_dwc(gen, case) if m == "L" else None for m in case["schedule"]]
    s = {"case": case, "dwc": dwc}
    if case["path"] == "block":
        C = H * D
        s["x"] = _normal(gen, (B, N, C), dtype=dt)
        s["w_qkv"], s["b_qkv"] = _normal(gen, (3 * C, C), C ** -0.5, dt), _normal(gen, (3 * C,), 0.1)
        s["w_o"], s["b_o"] = _normal(gen, (C, C), C ** -0.5, dt), _normal(gen, (C,), 0.1)
        s["qkv"] = tuple(torch.empty((B, H, N, D), dtype=dt, device="cuda") for _ in range(3))
        s["y"] = torch.empty((B, N, C), dtype=dt, device="cuda")
        q = [s["qkv"][0]]
    elif case["layout"] == "fused":
        acts = [_normal(gen, (B, N, 3, H, D), dtype=dt) for _ in range(n)]
        q, k, v = ([a[:, :, i].permute(0, 2, 1, 3) for a in acts] for i in range(3))
        s["qkv"] = (q, k, v)
    else:
        q, k, v = ([_normal(gen, (B, H, N, D), dtype=dt) for _ in range(n)] for _ in range(3))
        s["qkv"] = (q, k, v)
    s["out"] = [torch.empty((B, H, N, D), dtype=dt, device="cuda") for _ in range(n)]
    shape = jv.make_shape(q[0], case["Hg"], case["Wg"], case["prefix"])
    has_l = "L" in case["schedule"]
    s["ws"] = jv.alloc_workspace("L", shape, jv.make_dwc(next((d for d in dwc if d), None), "cuda"), "cuda") if has_l else None
    return s


def _mixer(s, q, k, v, out):
    c = s["case"]
    if c["schedule"] == "L":
        return jv.linear_attn(q, k, v, c["Hg"], c["Wg"], dwc=s["dwc"][0], out=out, ws=s["ws"], prefix=c["prefix"])
    if c["schedule"] == "W":
        return jv.window_attn(q, k, v, c["Hg"], c["Wg"], c["win"], c["win"], out=out, prefix=c["prefix"])
    return jv.full_attn(q, k, v, out=out)


def run(s):
    c = s["case"]
    if c["path"] == "block":
        q, k, v = jv.qkv_proj(s["x"], s["w_qkv"], s["b_qkv"], c["H"], c["Hg"], c["Wg"], out=s["qkv"], prefix=c["prefix"])
        o = _mixer(s, q, k, v, s["out"][0])
        return jv.out_proj(o, s["w_o"], s["b_o"], c["Hg"], c["Wg"], out=s["y"], prefix=c["prefix"])
    q, k, v = s["qkv"]
    if len(c["schedule"]) == 1:
        return _mixer(s, q[0], k[0], v[0], s["out"][0])
    return jv.hybrid_mixers(c["schedule"], q, k, v, c["Hg"], c["Wg"], c["win"], c["win"], dwc=s["dwc"], out=s["out"], ws=s["ws"],
                            prefix=c["prefix"])


def work(case):
    """Bytes: every input tensor (weights among them) read once, every output of a public call written once.  Operations:
    two per multiply-add; the two contractions with the state in L, query-key and probability-value products over the
    pairs that attend each other in W and F, the projections."""
    B, H, D, P = case["B"], case["H"], case["D"], case["prefix"]
    Hg, Wg, win = case["Hg"], case["Wg"], case["win"]
    N, C = P + Hg * Wg, H * D
    esz = 4 if case["dtype"] == "f32" else 2
    tensor = B * N * C * esz
    nbytes = flops = 0
    for m in case["schedule"]:
        nbytes += 4 * tensor
        if m == "L":
            flops += 4 * B * N * C * D
            if case["dwc"] != "none":
                flops += 2 * 9 * B * Hg * Wg * C
                nbytes += 4 * 9 * C
            if case["dwc"] == "squeeze":
                R = C // 8
                nbytes += 4 * (R * C + 9 * C * R + R)
                flops += 2 * B * (R * C + 9 * C * R)
        elif m == "F":
            flops += 4 * B * C * N * N
        else:
            rows = [min(win, Hg - y) for y in range(0, Hg, win)]
            cols = [min(win, Wg - x) for x in range(0, Wg, win)]
            pairs = P * N + sum(r * c * (r * c + P) for r in rows for c in cols)
            flops += 4 * B * C * pairs
    if case["path"] == "block":
        nbytes += (tensor + 3 * C * C * esz + 12 * C + 3 * tensor) + (tensor + C * C * esz + 4 * C + tensor)
        flops += 2 * B * N * C * 4 * C
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times what the formulas evaluated in fp64 show against the kernels.  bf16 (stored results, probabilities,
    convolution kernels and states rounded to 8 bits): 1.7e-3 to 3.0e-3 in the norm, up to 1.6e-2 of one value.  fp32 (sums
    of up to 1400 terms, exponentials): up to 6.5e-7 and 4.8e-6."""
    if case["dtype"] == "f32":
        return {"rel": 3e-6, "max": 2e-5}
    return {"rel": 1e-2, "max": 6e-2}
