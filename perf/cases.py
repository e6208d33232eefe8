"""The work this library is timed on: what a program that uses it has it do, through the public binding.

Every case is one of the uses below.  ``listed`` holds a named case or two of each; ``draw`` gives more of the same uses with
other sizes.  Types are drawn uniformly (tokens of packed sequences at arbitrary positions) unless the handle's schedule fixes
them; activations are N(0, 1), as a normalisation layer leaves them, and weights N(0, 0.02^2), the usual initialisation.

    proj           one projection, eager call
    ffn, gated     one feed-forward layer over a batch of tokens (prefill, or the forward half of training), eager call
    decode         one decode step of a model of ``layers`` blocks: every block's FFN on the rows of the tokens being generated,
                   all calls in one CUDA graph (each block's rows come from its own attention and norm, so they are separate
                   inputs); ``gated`` says which FFN
    train          the three products of a training step of one projection: forward, gradient of the input, gradient of the weight
"""
import math

import torch

from paper_2609_32814_b200 import binding

# (width, hidden width) of the feed-forward layers whose groups number 32
WIDE_SHAPES = ((2048, 6144), (2560, 9728), (4096, 12288), (2048, 768), (7168, 2048))


def _case(use, q, d, f, m, *, dtype="bf16", schedule="explicit", table="qq", gated=False, layers=1, period=0):
    return {"use": use, "q": q, "d": d, "f": f, "m": m, "dtype": dtype, "schedule": schedule, "table": table, "gated": gated,
            "layers": layers, "period": period}


def listed():
    named = {
        # the smallest call: one fp32 projection of a few hundred rows, where the latency of a call is what counts
        "proj_f32": _case("proj", 2, 256, 1024, 512, dtype="f32"),
        # one token of one user through a small decoder with two groups
        "decode_m1": _case("decode", 2, 768, 3072, 1, layers=12),
        # the same decoder with a batch of users; 40 is no multiple of a tile
        "decode_m40": _case("decode", 2, 768, 3072, 40, layers=12),
        # one token through SwiGLU layers split 32 ways
        "decode_gated_q32": _case("decode", 32, 2048, 6144, 1, gated=True, layers=12),
        # prefill of whole sequences: type = position mod 2 is the handle's schedule
        "ffn_q2_cyclic": _case("ffn", 2, 768, 3072, 8192, schedule="cyclic"),
        # a prompt of odd length with explicit types
        "ffn_q2_ragged": _case("ffn", 2, 768, 3072, 1777),
        # prefill with eight groups of 128, types from the batch
        "ffn_q8": _case("ffn", 8, 1024, 4096, 16384),
        # the largest: a wide layer over many tokens
        "ffn_q4_wide": _case("ffn", 4, 4096, 16384, 32768),
        # SwiGLU under the tensor-square law, types in runs of 192 positions
        "gated_interval": _case("gated", 4, 768, 1536, 12288, schedule="interval", table="q2pow", gated=True, period=768),
        # SwiGLU prefill split 32 ways: about 64 rows of a type, groups of 64 and 192
        "gated_q32": _case("gated", 32, 2048, 6144, 2048, gated=True),
        # forward and both gradients of a projection on packed sequences (a batch that is no multiple of anything)
        "train_q2": _case("train", 2, 768, 3072, 8003),
        # one projection with blocks of 40 x 200 (q grows with the matrix), rows of a type contiguous
        "proj_q128": _case("proj", 128, 5120, 25600, 2048, schedule="interval"),
    }
    return [dict(case, name=name) for name, case in named.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("proj_f32", "decode", "decode_gated", "ffn_cyclic", "ffn", "ffn_wide", "gated_interval", "gated_q32", "train",
                       "proj_large"))
    if kind == "proj_f32":
        q, s = rng.choice((2, 4)), 4 * rng.randint(8, 40)
        return _case("proj", q, q * s, q * s * rng.choice((2, 3, 4)), _log(rng, 64, 4096), dtype="f32")
    if kind == "decode":
        d = rng.choice((512, 768, 1024))
        return _case("decode", 2, d, 4 * d, _log(rng, 1, 64), layers=rng.randint(8, 16))
    if kind == "decode_gated":
        d, f = rng.choice(WIDE_SHAPES)
        return _case("decode", 32, d, f, _log(rng, 1, 4), gated=True, layers=rng.randint(8, 12))
    if kind == "ffn_cyclic":
        q, d = rng.choice((2, 4)), rng.choice((512, 768, 1024))
        return _case("ffn", q, d, 4 * d, q * (_log(rng, 512, 16384) // q), schedule="cyclic")
    if kind == "ffn":
        q = rng.choice((2, 4, 8))
        d = rng.choice((512, 1024)) if q > 2 else rng.choice((512, 768, 1024))
        return _case("ffn", q, d, 4 * d, _log(rng, 100, 16384))
    if kind == "ffn_wide":
        d = rng.choice((2048, 4096))
        return _case("ffn", rng.choice((4, 8, 16)), d, 4 * d, _log(rng, 2048, 32768))
    if kind == "gated_interval":
        return _case("gated", 4, 768, 1536, 768 * _log(rng, 2, 32), schedule="interval", table="q2pow", gated=True, period=768)
    if kind == "gated_q32":
        d, f = rng.choice(WIDE_SHAPES)
        return _case("gated", 32, d, f, _log(rng, 256, 4096), gated=True)
    if kind == "train":
        q = rng.choice((2, 4))
        d = rng.choice((512, 1024)) if q > 2 else rng.choice((512, 768, 1024))
        return _case("train", q, d, 4 * d, _log(rng, 500, 16384))
    q = rng.choice((32, 64, 128, 256))
    d, f = rng.choice(((5120, 25600), (25600, 5120)))
    return _case("proj", q, d, f, q * max(1, _log(rng, 1024, 8192) // q), schedule="interval")


def _normal(gen, shape, dtype, std=1.0):
    return (torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32) * std).to(dtype)


def prepare(case, seed):
    c = dict(case)
    q, d, f, m = c["q"], c["d"], c["f"], c["m"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    dw, fw = [d // q] * q, [f // q] * q
    kw = {"table": c["table"], "schedule": c["schedule"]}
    s = {"case": c, "layers": []}
    types = None
    if c["schedule"] == "explicit":
        # a token sits at a position drawn from the context, its type is the position mod q
        types = (torch.randint(0, 2048, (m,), generator=gen, device="cuda") % q).to(torch.int32)
    s["types"] = types
    if c["use"] in ("proj", "train"):
        s["X"] = _normal(gen, (m, d), dt)
        s["W"] = _normal(gen, (d, f), dt, 0.02)
        s["proj"] = binding.Proj(dw, fw, dtype=c["dtype"], **kw)
        if s["proj"].packed_weight_bytes() > 0:   # weights are laid out once, when they are loaded
            s["W"] = s["proj"].pack_weight(s["W"]).view(q * (-(-(d // q) // 8) * 8), -1)
            s["proj"].set_option("weight_packed", 1)
        if c["use"] == "train":
            s["G"] = _normal(gen, (m, f), dt)
            s["grad"] = binding.ProjGrad(dw, fw, **kw)
        return s
    ffn = (binding.GatedFFN if c["gated"] else binding.FFN)(dw, fw, **kw)
    if c["period"]:
        ffn.set_option("interval_period", c["period"])
    s["ffn"] = ffn
    for _ in range(c["layers"]):
        s["layers"].append({"X": _normal(gen, (m, d), dt), "W_up": _normal(gen, (d, 2 * f if c["gated"] else f), dt, 0.02),
                            "W_down": _normal(gen, (f, d), dt, 0.02)})
    if c["use"] == "decode":
        for layer in s["layers"]:
            layer["out"] = torch.empty((m, d), dtype=dt, device="cuda")
        s["workspace"] = torch.empty(ffn.workspace_bytes(m), dtype=torch.uint8, device="cuda")
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            _decode_step(s, stream)
        stream.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], stream=stream):
            _decode_step(s, stream)
    return s


def _decode_step(s, stream):
    for layer in s["layers"]:
        s["ffn"].forward(layer["X"], s["types"], layer["W_up"], layer["W_down"], out=layer["out"], workspace=s["workspace"], stream=stream)


def run(s):
    use = s["case"]["use"]
    if use == "decode":
        s["graph"].replay()
        return [layer["out"] for layer in s["layers"]]
    if use == "proj":
        return s["proj"].forward(s["X"], s["types"], s["W"])
    if use == "train":
        return {"Y": s["proj"].forward(s["X"], s["types"], s["W"]),
                "dX": s["grad"].grad_input(s["G"], s["types"], s["W"]),
                "dW": s["grad"].grad_weight(s["X"], s["G"], s["types"])}
    layer = s["layers"][0]
    return s["ffn"].forward(layer["X"], s["types"], layer["W_up"], layer["W_down"])


def work(case):
    q, d, f, m, n = case["q"], case["d"], case["f"], case["m"], case["layers"]
    e = 4 if case["dtype"] == "f32" else 2
    kept = (3 / 4) ** round(math.log2(q)) if case["table"] == "q2pow" else (2 * q - 1) / q ** 2
    types = q * (1 - (1 - 1 / q) ** m) if case["schedule"] == "explicit" else q   # expected number of types among the rows
    bank = 1.0 if case["table"] == "q2pow" else (types * q + q - types) / q ** 2    # share of the bank that some row needs
    macs = m * d * f * kept
    if case["use"] == "proj":
        return {"bytes": e * (m * d + d * f * bank + m * f), "flops": 2 * macs}
    if case["use"] == "train":
        return {"bytes": e * (m * d + d * f + m * f) + e * (m * f + m * d) + 4 * d * f, "flops": 6 * macs}
    maps = 3 if case["gated"] else 2
    return {"bytes": n * e * (2 * m * d + maps * d * f * bank), "flops": n * 2 * maps * macs}


def tolerance(case):
    """About four times what this library's results differ by from the same products in 64 bits (operands as given): 2.6e-7 and
    2.6e-6 (relative 2-norm, largest) for fp32, 1.7e-3 and 3.9e-3 for one rounding to bf16, 2.4e-3 and 1.7e-2 where the hidden
    state is rounded to bf16 as well."""
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 1e-5}
    if case["use"] in ("proj", "train"):
        return {"rel": 7e-3, "max": 1.6e-2}
    return {"rel": 1e-2, "max": 6e-2}
