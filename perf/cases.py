"""Performance cases: the calls a rollout engine and a trainer make through ``binding.Context``.

``listed()`` names the cases, ``draw()`` gives more of the same ranges, ``prepare()`` makes what a
program holds before the call, ``run()`` is one pass.  Layer sizes are those of the benchmark
(hidden 2048, expert intermediate 768, 128 experts, top-8, QKV 2048 -> 5120, output projection
4096 -> 2048); drawn cases also vary them.

kind            one pass
linear          dense FP8 projection of bf16 activations (weights already quantized)
moe             live routing and the FP8 expert layer (weights already quantized)
moe4            the expert layer on 4-bit weights already quantized, routing given
train_fwd       the masters quantized and published, then the FP8 expert layer
train4_fwd      the masters quantized to 4 bits, then the expert layer on them
linear_bwd      gradients of a dense projection
train_step      the masters quantized, the FP8 expert layer keeping activations, and its backward
tbpo            sequence-level loss and per-token gradient of a packed batch of responses
"""
import math

import numpy as np
import torch

from paper_2604_07853_b200 import binding

H, I, E, K = 2048, 768, 128, 8

_context = None


def context():
    """The one library context a program keeps."""
    global _context
    if _context is None:
        _context = binding.Context(0)
    return _context


def listed():
    layer = {"H": H, "I": I, "E": E, "k": K}
    return [
        # one sequence being decoded: QKV projection of a single token
        {"name": "qkv_decode_1", "kind": "linear", "M": 1, "N": 5120, "K": 2048},
        # a ragged prefill: output projection of one prompt
        {"name": "o_proj_prefill_777", "kind": "linear", "M": 777, "N": 2048, "K": 4096},
        # training forward: QKV projection of two 4096-token sequences
        {"name": "qkv_train_8192", "kind": "linear", "M": 8192, "N": 5120, "K": 2048},
        # one sequence being decoded: router and experts of a single token
        {"name": "moe_decode_1", "kind": "moe", "M": 1, **layer},
        # a full decode batch of the rollout engine
        {"name": "moe_decode_256", "kind": "moe", "M": 256, **layer},
        # a prefill chunk, or a large decode batch with an odd number of sequences
        {"name": "moe_prefill_1501", "kind": "moe", "M": 1501, **layer},
        # decode on the 4-bit rollout format of larger models
        {"name": "w4a16_decode_96", "kind": "moe4", "fmt": "w4", "M": 96, **layer},
        # the forward of a training step at the benchmark's size (8 x 4096 tokens, skewed experts)
        {"name": "train_fwd_32768", "kind": "train_fwd", "M": 32768, "zipf": 1.1, **layer},
        # the same with a 4-bit format, one sequence
        {"name": "fp4_train_fwd_4096", "kind": "train4_fwd", "fmt": "fp4", "M": 4096, "zipf": 1.1, **layer},
        # backward of the QKV projection, a ragged packed batch
        {"name": "qkv_backward_4100", "kind": "linear_bwd", "M": 4100, "N": 5120, "K": 2048},
        # a whole training step of the expert layer, two sequences
        {"name": "train_step_8192", "kind": "train_step", "M": 8192, "zipf": 1.1, **layer},
        # loss of one optimizer step: 1024 responses of 4096 tokens on average
        {"name": "tbpo_1024", "kind": "tbpo", "B": 1024, "T": 1024 * 4096},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _draw_layer(rng):
    if rng.random() < 0.5:
        return {"H": H, "I": I, "E": E, "k": K}
    while True:
        h, i = rng.choice((1024, 1536, 2048, 3072, 4096)), rng.choice((384, 512, 768, 1024, 1536))
        e, k = rng.choice((16, 32, 64, 96, 128)), rng.choice((2, 4, 6, 8))
        if e * h * i <= E * H * I:
            return {"H": h, "I": i, "E": e, "k": k}


def draw(rng):
    kind = rng.choice(("linear", "linear", "linear", "moe", "moe", "moe", "moe4", "moe4", "train_fwd", "train4_fwd",
                       "linear_bwd", "train_step", "tbpo"))
    if kind == "linear":
        n, k = rng.choice(((5120, 2048), (2048, 4096), (128 * rng.randint(4, 48), 128 * rng.randint(4, 48))))
        return {"kind": kind, "M": _log_int(rng, 1, 8192), "N": n, "K": k}
    if kind == "linear_bwd":
        n, k = rng.choice(((5120, 2048), (2048, 4096), (128 * rng.randint(4, 40), 128 * rng.randint(4, 40))))
        return {"kind": kind, "M": _log_int(rng, 512, 8192), "N": n, "K": k}
    if kind == "tbpo":
        b = _log_int(rng, 64, 2048)
        return {"kind": kind, "B": b, "T": b * rng.randint(512, 6144)}
    layer = _draw_layer(rng)
    scale = E * H * I * K / (layer["H"] * layer["I"] * layer["k"] * E)  # tokens of the same work
    if kind == "moe":
        return {"kind": kind, "M": _log_int(rng, 1, 4096), **layer}
    if kind == "moe4":
        return {"kind": kind, "fmt": rng.choice(("w4", "fp4")), "M": _log_int(rng, 1, 2048), **layer}
    most = {"train_fwd": 32768, "train4_fwd": 8192, "train_step": 8192}[kind]
    m = _log_int(rng, 1024, int(min(most, most * scale)))
    case = {"kind": kind, "M": m, "zipf": rng.choice((0.0, 1.1)), **layer}
    if kind == "train4_fwd":
        case["fmt"] = rng.choice(("w4", "fp4"))
    return case


# ------------------------------------------------------------------------------------- inputs
def _weight(g, *shape):
    """bf16 N(0, 0.02^2)."""
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=g)


def _acts(g, m, h):
    """bf16 N(0, 1) with 1 % of the entries times 50."""
    x = torch.randn((m, h), device="cuda", generator=g)
    x = torch.where(torch.rand((m, h), device="cuda", generator=g) < 0.01, x * 50.0, x)
    return x.to(torch.bfloat16)


def _routing(g, m, e, k, zipf):
    """Top-k ids and softmax weights of N(0, 1) logits, biased to a Zipf popularity if zipf > 0."""
    logits = torch.randn((m, e), device="cuda", generator=g)
    if zipf > 0:
        rank = torch.randperm(e, device="cuda", generator=g).float() + 1.0
        logits += -zipf * rank.log()
    top, ids = logits.topk(k, dim=1)
    return ids.to(torch.int32), torch.softmax(top, dim=1)


def _quantize4(ctx, fmt, w, out=None):
    return ctx.quantize_weight_w4(w, out=out) if fmt == "w4" else ctx.quantize_weight_fp4(w, out=out)


def prepare(case, seed):
    ctx = context()
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    s = {"ctx": ctx, "case": case}
    if kind == "linear":
        s["x"] = _acts(g, case["M"], case["K"])
        s["w"] = ctx.quantize_weight(_weight(g, case["N"], case["K"]))
    elif kind == "linear_bwd":
        s["x"] = _acts(g, case["M"], case["K"])
        s["w"] = _weight(g, case["N"], case["K"])
        s["dy"] = torch.empty((case["M"], case["N"]), dtype=torch.bfloat16, device="cuda").normal_(0.0, 1e-3, generator=g)
    elif kind == "tbpo":
        s.update(_tbpo_inputs(g, seed, case["B"], case["T"]))
    else:
        m, h, i, e, k = (case[n] for n in ("M", "H", "I", "E", "k"))
        s["x"] = _acts(g, m, h)
        w13, w2 = _weight(g, e, 2 * i, h), _weight(g, e, h, i)
        if kind == "moe":
            s["router"] = _weight(g, e, h)
            s["w13"], s["w2"] = ctx.quantize_weight(w13), ctx.quantize_weight(w2)
            return s
        s["ids"], s["wts"] = _routing(g, m, e, k, case.get("zipf", 0.0))
        if kind == "moe4":
            s["w13"], s["w2"] = _quantize4(ctx, case["fmt"], w13), _quantize4(ctx, case["fmt"], w2)
            return s
        s["w13"], s["w2"] = w13, w2
        if kind == "train4_fwd":
            s["q13"], s["q2"] = _quantize4(ctx, case["fmt"], w13), _quantize4(ctx, case["fmt"], w2)
            return s
        s["q13"], s["q2"] = ctx.quantize_weight(w13), ctx.quantize_weight(w2)
        if kind == "train_fwd":  # the rollout engine's weight buffers
            s["pub13"], s["pub2"] = ([torch.empty_like(t) for t in q] for q in (s["q13"], s["q2"]))
        else:
            s["dout"] = torch.empty((m, h), dtype=torch.bfloat16, device="cuda").normal_(0.0, 1e-3, generator=g)
            s["save"] = {"gate_up": torch.empty((m * k, 2 * i), dtype=torch.bfloat16, device="cuda"),
                         "h": torch.empty((m * k, i), dtype=torch.bfloat16, device="cuda")}
            s["grads"] = {"dx": torch.empty((m, h), dtype=torch.bfloat16, device="cuda"),
                          "dw13": torch.empty((e, 2 * i, h), device="cuda"),
                          "dw2": torch.empty((e, h, i), device="cuda"), "dwts": None}
    return s


def _tbpo_inputs(g, seed, b, t):
    """Log-probs of b packed responses of t tokens in all: lengths lognormal (sigma 0.8), at least
    16; the learner one small step away from the sampler, so that ratios straddle the trust bands."""
    share = np.random.default_rng(seed).lognormal(0.0, 0.8, size=b)
    ends = np.cumsum(share) / share.sum()
    offsets = np.concatenate([[0], np.arange(1, b + 1) * 16 + np.rint(ends * (t - 16 * b)).astype(np.int64)])
    offsets = torch.from_numpy(offsets.astype(np.int64)).cuda()

    def normal(n, std):
        return torch.empty(n, device="cuda").normal_(0.0, std, generator=g)

    sampler = -normal(t, 1.5).abs() - 0.01
    learner = sampler + normal(t, 0.02)
    shift = normal(b, 5e-4).repeat_interleave(offsets[1:] - offsets[:-1], output_size=t)
    return {"cur": learner + shift + normal(t, 1e-3), "learner": learner, "sampler": sampler, "offsets": offsets,
            "adv": normal(b, 1.0)}


# --------------------------------------------------------------------------------------- passes
def run(s):
    ctx, kind = s["ctx"], s["case"]["kind"]
    if kind == "linear":
        return ctx.linear_fwd(s["x"], *s["w"])
    if kind == "moe":
        logits, ids, wts = ctx.router_fwd(s["x"], s["router"], s["case"]["k"])
        return logits, ids, wts, ctx.moe_fwd(s["x"], ids, wts, *s["w13"], *s["w2"])
    if kind == "moe4":
        fwd = ctx.moe_fwd_w4a16 if s["case"]["fmt"] == "w4" else ctx.moe_fwd_fp4a16
        return fwd(s["x"], s["ids"], s["wts"], s["w13"], s["w2"])
    if kind == "train_fwd":
        ctx.quantize_weight_publish(s["w13"], *s["q13"], *s["pub13"])
        ctx.quantize_weight_publish(s["w2"], *s["q2"], *s["pub2"])
        y = ctx.moe_fwd(s["x"], s["ids"], s["wts"], *s["q13"], *s["q2"])
        return y, s["q13"], s["q2"], s["pub13"], s["pub2"]
    if kind == "train4_fwd":
        fmt = s["case"]["fmt"]
        _quantize4(ctx, fmt, s["w13"], s["q13"])
        _quantize4(ctx, fmt, s["w2"], s["q2"])
        fwd = ctx.moe_fwd_w4a16 if fmt == "w4" else ctx.moe_fwd_fp4a16
        return fwd(s["x"], s["ids"], s["wts"], s["q13"], s["q2"]), s["q13"], s["q2"]
    if kind == "linear_bwd":
        dx, _, dw = ctx.linear_bwd(s["dy"], s["x"], s["w"])
        return dx, dw
    if kind == "train_step":
        ctx.quantize_weight(s["w13"], *s["q13"])
        ctx.quantize_weight(s["w2"], *s["q2"])
        y = ctx.moe_fwd(s["x"], s["ids"], s["wts"], *s["q13"], *s["q2"], save=s["save"])
        ctx.moe_bwd(s["x"], s["ids"], s["wts"], s["w13"], s["w2"], s["save"]["gate_up"], s["save"]["h"], s["dout"],
                    out=s["grads"])
        return y, s["q13"], s["q2"], s["save"], s["grads"]
    return ctx.tbpo_loss(s["cur"], s["learner"], s["sampler"], s["offsets"], s["adv"])


# ------------------------------------------------------------------------------- what it takes
def work(case):
    kind = case["kind"]
    if kind in ("linear", "linear_bwd"):
        m, n, k = case["M"], case["N"], case["K"]
        if kind == "linear":
            return {"bytes": 2 * m * k + n * k + 4 * n * k // 16384 + 2 * m * n, "flops": 2 * m * n * k}
        return {"bytes": 2 * (m * n + 2 * m * k + n * k) + 4 * n * k, "flops": 4 * m * n * k}
    if kind == "tbpo":
        return {"bytes": 16 * case["T"] + 40 * case["B"], "flops": 6 * case["T"]}
    m, h, i, e, k = (case[n] for n in ("M", "H", "I", "E", "k"))
    active = e if case.get("zipf") else e * (1.0 - (1.0 - k / e) ** m)  # experts that some token goes to
    weights = 3 * h * i
    tokens = 4 * m * h + 8 * m * k
    flops = 6 * m * k * h * i
    fp8, four = 1 + 4 / 16384, 0.5 + (3 if case.get("fmt") == "w4" else 2) / 128
    if kind == "moe":
        return {"bytes": tokens + 2 * e * h + 4 * m * e + active * weights * fp8, "flops": flops + 2 * m * e * h}
    if kind == "moe4":
        return {"bytes": tokens + active * weights * four, "flops": flops}
    if kind == "train_fwd":
        return {"bytes": tokens + e * weights * (2 + 2 * fp8), "flops": flops}
    if kind == "train4_fwd":
        return {"bytes": tokens + e * weights * (2 + four), "flops": flops}
    saved = 2 * m * k * 3 * i
    return {"bytes": tokens + 4 * m * h + saved + e * weights * (2 + fp8 + 4), "flops": 3 * flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "tbpo":  # double arithmetic on fp32 inputs; the gradient is rounded to fp32
        return {"rel": 1e-6}
    if kind == "moe":  # near-ties of the router's logits may fall either way
        return {"rel": 1e-2, "differ": 2e-3}
    if kind in ("linear", "linear_bwd"):  # one rounding to bf16
        return {"rel": 4e-3}
    return {"rel": 1e-2}  # bf16 (and FP8) intermediates
