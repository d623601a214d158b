"""Workloads of the Switch FFN layer whose time is followed: one pass is what a user's program asks of the library.

A case says the layer's shape (T tokens, d_model, d_ff, E experts, capacity factor), the activation type, the direction
("fwd": inference, one switch_moe_fwd; "train": switch_moe_fwd and switch_moe_bwd) and the options that are on.  Inputs
are drawn on the GPU from the seed with the distributions of `paper_2101_03961_b200/inputs.py`: x and dy ~ N(0, 1),
weights truncated normal with sigma sqrt(0.1 / fan_in), an optional per-expert router bias that skews the routing.
"""
from __future__ import annotations

import math

import torch

from paper_2101_03961_b200 import switch_moe as sm

_DEFAULTS = {
    "dtype": "bf16", "pass": "train", "cf": 1.25, "residual": False, "geglu": False, "top2": False, "reroute": 0,
    "groups": 1, "bias_std": 0.0, "noise": 0.0, "jitter": 0.0, "dropout": 0.0,
}


def _case(T, d, f, E, **kw):
    c = {"T": T, "d_model": d, "d_ff": f, "E": E}
    c.update(_DEFAULTS)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest training step: a float32 layer of unit-test size, all latency and launches
        _case(512, 64, 256, 8, cf=1.0, dtype="f32", name="tiny_f32_train"),
        # a float32 layer of ordinary size: the full-precision run that a bfloat16 recipe is compared with
        _case(4096, 512, 2048, 16, dtype="f32", name="layer_f32_train"),
        # inference, a handful of tokens through a small layer
        _case(96, 256, 1024, 8, cf=2.0, residual=True, **{"pass": "fwd"}, name="small_fwd"),
        # one decoding step of a batch of sequences: few tokens per expert, every expert's weights are read
        _case(256, 768, 3072, 128, cf=2.0, residual=True, **{"pass": "fwd"}, name="decode_fwd"),
        # prefill: a ragged number of prompt tokens through the same kind of layer with fewer experts
        _case(6001, 768, 3072, 60, cf=2.0, **{"pass": "fwd"}, name="prefill_fwd"),
        # one training step of the Switch-Base-shaped layer, the size the benchmark quotes
        _case(32768, 768, 3072, 128, name="switch_base_train"),
        # skewed routing: a third of the tokens overflow their expert and are offered to their second choice
        _case(32768, 768, 3072, 64, cf=1.0, bias_std=0.10, reroute=1, name="overflow_reroute_train"),
        # GEGLU experts inside the residual connection
        _case(32768, 768, 2048, 128, geglu=True, residual=True, name="geglu_base_train"),
        # top-2 routing, every slot of every expert full
        _case(16384, 768, 3072, 64, top2=True, residual=True, name="top2_train"),
        # many small experts, an odd number of tokens, exploration noise on the router's logits
        _case(20011, 512, 1536, 200, noise=0.01, name="many_experts_train"),
        # many tokens through a narrow layer, eight routing groups
        _case(65536, 256, 512, 128, groups=8, jitter=0.01, name="long_batch_train"),
        # the largest: wide experts, 5.4 GB of weights in each direction of the layer
        _case(16384, 4096, 10240, 64, name="wide_train"),
    ]


def _log_int(rng, lo, hi, step=1):
    return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step)


def draw(rng):
    while True:
        kind = rng.choice(["fwd", "train", "train", "train", "f32"])
        d = _log_int(rng, 128, 2048, 64)
        f = _log_int(rng, 256, 6144, 64)
        E = _log_int(rng, 4, 256)
        cf = rng.choice([1.0, 1.25, 1.25, 2.0])
        if kind == "f32":
            T, d, f, E = _log_int(rng, 300, 8192), _log_int(rng, 64, 768, 8), _log_int(rng, 128, 3072, 8), _log_int(rng, 4, 64)
            kw = {"dtype": "f32", "residual": rng.random() < 0.5, "pass": rng.choice(["fwd", "train", "train"])}
            limit = 8e10
        elif kind == "fwd":
            T, cf = _log_int(rng, 64, 32768), 2.0
            kw = {"pass": "fwd", "residual": rng.random() < 0.5, "geglu": rng.random() < 0.3}
            limit = 4e12
        else:
            T = _log_int(rng, 1024, 65536)
            kw = {"residual": rng.random() < 0.5, "bias_std": rng.choice([0.0, 0.0, 0.1])}
            option = rng.choice(["plain", "plain", "geglu", "geglu_dropout", "top2", "reroute", "groups", "noise", "jitter"])
            if option.startswith("geglu"):
                kw["geglu"] = True
            if option == "geglu_dropout":
                kw["dropout"] = 0.4
            if option == "top2":
                kw["top2"], T = True, max(1024, T // 2 // 256 * 256)
            if option == "reroute":
                kw["reroute"] = rng.choice([1, 1, 2])
            if option == "groups":
                kw["groups"] = rng.choice([2, 4, 8])
                T = max(1, T // (256 * kw["groups"])) * 256 * kw["groups"]
            if option == "noise":
                kw["noise"] = 0.01
            if option == "jitter":
                kw["jitter"] = 0.01
            limit = 4e12
        c = _case(T, d, f, E, cf=cf, **kw)
        w = work(c)
        if (T // c["groups"]) * cf / E >= 1 and w["flops"] <= limit and w["bytes"] <= 1.2e10:
            return c


def _make_config(case):
    return sm.make_config(
        case["T"], case["d_model"], case["d_ff"], case["E"], case["cf"], 0.01,
        dtype=sm.F32 if case["dtype"] == "f32" else sm.BF16, residual=case["residual"], groups=case["groups"],
        reroute=case["reroute"] > 0, reroute_stages=max(1, case["reroute"]), input_jitter=case["jitter"] > 0,
        geglu=case["geglu"], top2=case["top2"], expert_dropout=case["dropout"] or None)


def _truncated_normal(shape, fan_in, dtype, gen):
    """Normal cut at two standard deviations, sigma = sqrt(0.1 / fan_in), drawn expert by expert."""
    out = torch.empty(shape, dtype=dtype, device="cuda")
    bound = math.erf(math.sqrt(2.0))
    for part in (out if len(shape) == 3 else [out]):
        u = torch.empty(part.shape, dtype=torch.float32, device="cuda").uniform_(-bound, bound, generator=gen)
        part.copy_(u.erfinv_().mul_(math.sqrt(2.0) * math.sqrt(0.1 / fan_in)))
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    T, d, f, E = case["T"], case["d_model"], case["d_ff"], case["E"]
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16

    def normal(*shape):
        return torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=gen)

    def around_one(eps, shape, dt):
        return torch.empty(shape, dtype=torch.float32, device="cuda").uniform_(1 - eps, 1 + eps, generator=gen).to(dt)

    s = {"train": case["pass"] == "train", "cfg": _make_config(case)}
    cfg = s["cfg"]
    s["x"] = normal(T, d)
    s["W_r"] = _truncated_normal((d, E), d, torch.float32, gen)
    s["bias"] = None
    if case["bias_std"] > 0:
        s["bias"] = torch.empty(E, device="cuda").normal_(0.0, case["bias_std"], generator=gen)
    s["W_in"] = _truncated_normal((E, d, 2 * f if case["geglu"] else f), d, dtype, gen)
    s["W_out"] = _truncated_normal((E, f, d), f, dtype, gen)
    if case["noise"] > 0:
        s["noise"] = around_one(case["noise"], (T, E), torch.float32)
        cfg.router_noise = s["noise"].data_ptr()
    if case["jitter"] > 0:
        s["jitter"] = around_one(case["jitter"], (T, d), dtype)
        cfg.router_jitter = s["jitter"].data_ptr()
    if case["dropout"] > 0:
        rows = E * sm.switch_moe_capacity(cfg)
        word = torch.zeros((rows, f // 32), dtype=torch.int64, device="cuda")
        for bit in range(32):
            keep = torch.empty(word.shape, device="cuda").uniform_(generator=gen) >= case["dropout"]
            word += keep.to(torch.int64) << bit
        s["keep"] = torch.where(word >= 1 << 31, word - (1 << 32), word).to(torch.int32)
        cfg.expert_keep = s["keep"].data_ptr()
    s["y"] = torch.empty_like(s["x"])
    s["aux"] = torch.empty(1, dtype=torch.float32, device="cuda")
    if s["train"]:
        s["dy"] = normal(T, d)
        for k in ("x", "W_r", "W_in", "W_out"):
            s["d" + k] = torch.empty_like(s[k])
    s["ws"] = sm.allocate_workspace(cfg)
    return s


def run(s):
    sm.switch_moe_fwd(s["cfg"], s["x"], s["W_r"], s["bias"], s["W_in"], s["W_out"], s["y"], s["aux"], s["ws"])
    if not s["train"]:
        return {"y": s["y"], "aux": s["aux"]}
    sm.switch_moe_bwd(s["cfg"], s["dy"], 1.0, s["x"], s["W_r"], s["W_in"], s["W_out"], s["y"], s["ws"], s["dx"],
                      s["dW_r"], s["dW_in"], s["dW_out"])
    return {k: s[k] for k in ("y", "aux", "dx", "dW_r", "dW_in", "dW_out")}


def work(case):
    """Inputs read once, outputs written once, multiplications of the tokens that an expert can hold (an expected
    number of experts has any: the weights of the others are not needed, their gradients are still written)."""
    T, d, f, E = case["T"], case["d_model"], case["d_ff"], case["E"]
    elt = 4 if case["dtype"] == "f32" else 2
    train = case["pass"] == "train"
    slots = E * case["groups"] * max(1, int(T // case["groups"] * case["cf"] / E))
    rows = min(T * (2 if case["top2"] else 1), slots)
    used = E * (1.0 - (1.0 - 1.0 / E) ** rows)
    fin = 2 * f if case["geglu"] else f
    expert = (fin + f) * d
    nbytes = elt * (2 * T * d + used * expert) + 4 * d * E
    nbytes += 4 * T * E * (case["noise"] > 0) + elt * T * d * (case["jitter"] > 0) + slots * f / 8 * (case["dropout"] > 0)
    flops = 2.0 * rows * expert + 2.0 * T * d * E
    if train:
        nbytes += elt * (2 * T * d + E * expert) + 4 * d * E
        flops *= 3
    return {"bytes": float(nbytes), "flops": float(flops)}


def tolerance(case):
    """Measured between the library's tensor-core and FP32-FMA paths (bfloat16) and against float64 (float32), times
    about four.  Forward outputs differ by accumulation order alone: 7e-7 (float32), 3e-4 with a largest element of
    8e-3 (bfloat16: a last-bit rounding).  In training the sign of a pre-activation next to zero also decides whether a
    token's whole term enters dx and dW_in, so the same pair of paths differs there by 8e-4 (float32) and, with the
    saved GEGLU factors and near-ties of the routing, by 4e-3 (bfloat16), and a single element by up to its own size."""
    if case["pass"] == "fwd":
        return {"rel": 4e-6, "max": 4e-5} if case["dtype"] == "f32" else {"rel": 2e-3, "max": 4e-2}
    return {"rel": 3e-3 if case["dtype"] == "f32" else 1e-2, "max": 0.99}
