"""The work that users of the Mixture-of-Channels FFN have it do, as cases to be timed.

Three kinds of pass, each through the entry point that a program of that kind calls:

  train    one forward and one backward of the layer through `autograd.moc_ffn`: the output and all four gradients
  prefill  the forward of a prompt with nothing kept (`moc_ffn_forward(save=False)`), output and workspace owned by the caller
  decode   one generation step for a batch of sequences, one token each: `moc_ffn_decode`, or with "block" the FFN half of a
           pre-norm layer, `moc_ffn_decode_block` (RMSNorm in front, the residual added); buffers owned by the caller

A case: kind, tokens, d_model, d_ff, pad (zero rows behind the d_ff channels of each weight array), k, dtype, and the options
grouped (2 of every 8 channels), recompute (the up values are formed again in backward) and block.  Widths are those of the
benchmark configurations (128/512, 768/2048, 2048/5461 padded to 5504, 2048/5504, 4096/11008); k is an eighth of the channels
unless the case says otherwise.  The Top-K after the activation (`post_silu`) is an ablation and is not timed.
"""
import math

import torch

from paper_2511_09323_b200 import binding
from paper_2511_09323_b200.autograd import moc_ffn

RMS_EPS = 1e-5
# the largest listed case's tokens * d_model * d_ff
MOST_WORK = 65536 * 2048 * 5504


def _case(name, kind, tokens, d_model, d_ff, k, pad=0, dtype="bf16", grouped=False, recompute=False, block=False):
    case = {"kind": kind, "tokens": tokens, "d_model": d_model, "d_ff": d_ff, "pad": pad, "k": k, "dtype": dtype,
            "grouped": grouped, "recompute": recompute, "block": block}
    return dict(case, name=name) if name else case


def listed():
    return [
        # one sequence on a small model: nothing but latency, launches and the host's part of the call
        _case("decode 1, 768x2048", "decode", 1, 768, 2048, 256),
        # one sequence on the decode configuration's layer, the way a layer calls it
        _case("decode 1 block, 4096x11008", "decode", 1, 4096, 11008, 1376, block=True),
        # the decode configuration's two other batches
        _case("decode 4, 4096x11008", "decode", 4, 4096, 11008, 1376),
        _case("decode 16 block, 4096x11008", "decode", 16, 4096, 11008, 1376, block=True),
        # continuous batching: however many sequences are running
        _case("decode 61, 4096x11008", "decode", 61, 4096, 11008, 1376),
        # a short and a long prompt
        _case("prefill 307, 4096x11008", "prefill", 307, 4096, 11008, 1376),
        _case("prefill 2048, 4096x11008", "prefill", 2048, 4096, 11008, 1376),
        # the 32-bit configuration
        _case("train 256 f32, 128x512", "train", 256, 128, 512, 64, dtype="f32"),
        # a micro-batch of unpadded text on the 5461-channel layer
        _case("train 1111, 2048x5461", "train", 1111, 2048, 5461, 688, pad=43),
        # the small layer's pre-training batch
        _case("train 16384, 768x2048", "train", 16384, 768, 2048, 256),
        # the 2-of-8 mask on the larger layer
        _case("train 16384 2of8, 2048x5504", "train", 16384, 2048, 5504, 1376, grouped=True),
        # the largest pre-training batch of one GPU
        _case("train 65536, 2048x5504", "train", 65536, 2048, 5504, 688),
    ]


def _between(rng, low, high):
    """A whole number from low to high, spread over its logarithm."""
    return min(high, max(low, round(math.exp(rng.uniform(math.log(low), math.log(high))))))


def draw(rng):
    kind = rng.choice(("decode", "decode", "prefill", "train", "train", "train f32"))
    dtype = "f32" if kind == "train f32" else "bf16"
    kind = kind.split()[0]
    d_model = 8 * _between(rng, *((8, 96) if dtype == "f32" else (48, 640)))
    # 8/3 of d_model is the usual width of a gated layer; some have four times
    d_ff = round(d_model * rng.choice((8 / 3, 8 / 3, 8 / 3, 4)))
    if rng.random() < 0.5:
        d_ff = 64 * max(1, round(d_ff / 64))
    pad = -d_ff % 64
    if kind == "decode":
        tokens = _between(rng, 1, 256)
    elif kind == "prefill":
        tokens = _between(rng, 257, 4096)
    elif dtype == "f32":
        tokens = _between(rng, 32, 4096)
    else:
        tokens = _between(rng, 64, 65536)
    tokens = max(1, min(tokens, MOST_WORK // (d_model * (d_ff + pad))))
    grouped = dtype == "bf16" and d_ff % 8 == 0 and rng.random() < 0.25
    k = d_ff // 4 if grouped else max(1, d_ff // rng.choice((16, 8, 8, 4)))
    recompute = kind == "train" and dtype == "bf16" and not grouped and rng.random() < 0.15
    block = kind == "decode" and rng.random() < 0.4
    return _case(None, kind, tokens, d_model, d_ff, k, pad, dtype, grouped, recompute, block)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dtype = {"bf16": torch.bfloat16, "f32": torch.float32}[case["dtype"]]
    tokens, d, rows = case["tokens"], case["d_model"], case["d_ff"] + case["pad"]

    def normal(*shape, std=1.0):
        return (torch.randn(*shape, generator=gen, device="cuda") * std).to(dtype)

    weights = [normal(rows, d, std=0.02) for _ in range(3)]
    for w in weights:
        w[case["d_ff"]:] = 0
    x = normal(tokens, d)
    state = {"case": case, "x": x, "weights": weights}
    if case["kind"] == "train":
        state["grad_out"] = normal(tokens, d)
        state["leaves"] = [t.requires_grad_() for t in (x, *weights)]
        return state
    # inference: the server owns the output and the workspace
    op = binding.MOC_OP_FORWARD if case["kind"] == "prefill" else \
        binding.MOC_OP_DECODE_BLOCK if case["block"] else binding.MOC_OP_DECODE
    desc = binding.make_desc(tokens, d, case["d_ff"], case["k"], dtype, d_ff_ld=rows,
                             flags=binding.MOC_FLAG_SELECT_2_OF_8 if case["grouped"] else 0)
    state["workspace"] = binding.alloc_workspace(desc, op)
    state["out"] = torch.empty_like(x)
    if case["block"]:
        state["rms_weight"] = (1 + 0.1 * torch.randn(d, generator=gen, device="cuda")).to(dtype)
    return state


def run(state):
    case, x, weights = state["case"], state["x"], state["weights"]
    options = {"d_ff": case["d_ff"], "grouped": case["grouped"]}
    if case["kind"] == "train":
        out = moc_ffn(x, *weights, case["k"], recompute_up=case["recompute"], **options)
        return (out.detach(), *torch.autograd.grad(out, state["leaves"], state["grad_out"]))
    options.update(out=state["out"], workspace=state["workspace"])
    if case["kind"] == "prefill":
        return binding.moc_ffn_forward(x, *weights, case["k"], save=False, **options)[0]
    if case["block"]:
        return binding.moc_ffn_decode_block(x, state["rms_weight"], RMS_EPS, *weights, case["k"], **options)
    return binding.moc_ffn_decode(x, *weights, case["k"], **options)


def work(case):
    """Every input read once and every output written once; the gate projection is dense, all else runs on the kept channels."""
    e = 2 if case["dtype"] == "bf16" else 4
    tokens, d, d_ff, k = case["tokens"], case["d_model"], case["d_ff"], case["k"]
    if case["kind"] == "train":
        return {"bytes": e * d * (4 * tokens + 6 * d_ff), "flops": 2 * tokens * d * (d_ff + 8 * k)}
    used = 1 - (1 - k / d_ff) ** tokens  # share of the channels that at least one token keeps
    return {"bytes": e * d * (2 * tokens + d_ff * (1 + 2 * used)), "flops": 2 * tokens * d * (d_ff + 2 * k)}


def tolerance(case):
    """Sums of bf16 products rounded to bf16 (rel 1e-2), or fp32 sums (rel 1e-5); and the Top-K cut.

    Two correct implementations add the gate projection in different orders.  Where a token's K-th and next gate values lie
    closer than the last bits of those sums (2e-7 of their standard deviation), they keep different channels: with some
    d_ff / 4 channels per standard deviation at the cut, that is to be expected of tokens * d_ff * 5e-8 tokens of a call.
    Such a token's output, and its part of the gradients, differ by two terms of k, which is sqrt(2 / k) of them; the largest
    element lies some five standard deviations out.  Calls in which it happens less than once in a hundred are held to the
    sums alone.
    """
    base = 1e-2 if case["dtype"] == "bf16" else 1e-5
    tokens, k = case["tokens"], case["k"]
    expected = tokens * case["d_ff"] * 5e-8
    if expected < 0.01:
        return {"rel": base, "max": 4 * base}
    return {"rel": min(0.03, base + math.sqrt(2 * (1 + expected) / (tokens * k))), "max": min(0.9, 4 * base + 5 * math.sqrt(2 / k))}
