"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one call pattern of the public Python entry points (``Model`` and its methods) at one size:

* ``train``: what a training program runs per update — the batch comes from pinned host memory, the n-wise step
  (or its micro-batches) is enqueued, AdamW follows where the program uses the built-in optimiser, and the head
  losses are read back, as ``bench.py`` does in its end-to-end measurement.
* ``eval``: scoring of a batch — forward of every component, every head's loss, the losses and the last head's
  per-token losses read back.

Shapes are the repository's own configurations (``workloads.CONFIGS``), those of its tests, and generic ones between
them; weights and tokens follow the same laws as ``workloads`` (N(0, 0.02^2), gains around one, Zipf(1.1) tokens), drawn
on the GPU because the states are made many times.
"""
import gc
import math

import numpy as np
import torch

from paper_2010_04116_b200 import Model

# A learning rate of early warm-up: a case may be run thousands of times on one batch, and the weights must stay where
# a training run has them.
ADAMW = {"lr": 1e-6, "beta1": 0.9, "beta2": 0.98, "eps": 1e-9, "weight_decay": 0.01}


def _case(name, **kw):
    c = {"kind": "train", "K": 2, "Lc": 1, "d": 128, "H": 4, "F": 512, "V": 512, "B": 1, "T": 64, "n": 1, "rule": "sum",
         "Lh": 0, "M": 1, "adamw": True, "head_mode": "stored", "attn_bwd": "one_sweep"}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    small = {"d": 768, "H": 12, "F": 3072, "V": 50257}      # GPT-2-small widths
    medium = {"d": 1024, "H": 16, "F": 4096, "V": 50257}    # GPT-2-medium widths
    return [
        # a unit-test or debugging-sized model: a step is a few hundred tiny kernels
        _case("tiny_train", K=2, Lc=2, d=128, H=4, F=512, V=512, B=4, T=64, n=2),
        # the same with everything odd: ragged tiles, a weighted rule, a block inside every head, gradients only
        # (the program has an optimiser of its own)
        _case("tiny_ragged_mean_rule", K=4, Lc=1, d=256, H=4, F=1000, V=1003, B=2, T=129, n=3, rule="mean", Lh=1, adamw=False),
        # fine-tuning on one short sequence at a time: full-size matrices, few rows
        _case("one_short_sequence", K=4, Lc=3, B=1, T=256, n=2, **small),
        # local learning of a mid-sized model on an odd batch, head that never holds the [tokens, vocabulary] matrix
        _case("local_learning_ragged_recompute", K=4, Lc=2, d=512, H=16, F=2048, V=32003, B=5, T=501, n=1, head_mode="recompute"),
        # long sequence, heads of 128, reproducible attention backward
        _case("long_sequence_two_kernels", K=2, Lc=2, d=1024, H=8, F=4096, V=8192, B=1, T=4096, n=2, attn_bwd="two_kernels"),
        # the GPT-2-small-shaped configuration at n = K (backpropagation of the summed head losses), gradients only
        _case("small_full_backprop", K=4, Lc=3, B=8, T=1024, n=4, adamw=False, **small),
        # the headline: GPT-2-medium-shaped 2-wise step with AdamW
        _case("medium_2wise", K=8, Lc=3, B=8, T=1024, n=2, **medium),
        # the widths of the 2.7B-shaped configuration (heads of 80), two one-layer components
        _case("wide_2wise", K=2, Lc=1, d=2560, H=32, F=10240, V=50257, B=2, T=2048, n=2),
        # the paper's Transformer shape: heads of 256, 128-token sequences, two blocks inside every auxiliary head, the
        # mean rule, four micro-batches per update
        _case("paper_shape_micro_batches", K=4, Lc=6, d=1024, H=4, F=4096, V=50257, B=256, T=128, n=2, rule="mean", Lh=2, M=4),
        # scoring a validation batch
        _case("eval_small_batch", kind="eval", K=4, Lc=3, B=8, T=1024, n=2, **small),
        # scoring one short text
        _case("eval_one_text", kind="eval", K=2, Lc=4, d=1024, H=8, F=4096, V=50257, B=1, T=200, n=1),
    ]


def _params(c):
    layer = 4 * c["d"] ** 2 + 2 * c["d"] * c["F"] + 9 * c["d"] + c["F"]
    return (c["V"] + c["T"]) * c["d"] + c["K"] * ((c["Lc"] + c["Lh"]) * layer + (c["V"] + 2) * c["d"])


def _streams(c, k):
    """Gradient tensors that component k has to carry: one per distinct stopping level of the heads that cross it (sum
    rule), or the parameter gradient's combination and one per head that continues below (weighted rules)."""
    K, n = c["K"], c["n"]
    top = min(k + n - 1, K - 1)
    if c["rule"] == "sum":
        return len({max(h - n + 1, 0) for h in range(k, top + 1)})
    used = 1
    far_alone = c["rule"] == "far" or top == k
    for h in range(k, top + 1):
        if k > 0 and h < k + n - 1 and not (far_alone and h == top):
            used += 1
    return used


def work(c):
    N, d, F, T = c["B"] * c["T"], c["d"], c["F"], c["T"]
    gemm = 2.0 * (4 * d * d + 2 * d * F)             # per token and block, one product with every matrix
    att = 2.0 * T * d                                # causal scores and mix, per token
    head = 2.0 * d * c["V"]
    flops = c["K"] * ((c["Lc"] + c["Lh"]) * (gemm + att) + head)
    if c["kind"] == "train":
        for k in range(c["K"]):
            s = _streams(c, k)
            flops += c["Lc"] * (gemm + s * (gemm + 2 * att)) + c["Lh"] * (2 * gemm + 2 * att) + 2 * head
    flops *= N
    P = _params(c)
    if c["kind"] == "eval":
        nbytes = 2.0 * (P - c["V"] * d) + 4.0 * N * d                     # bf16 weights, the batch's embedding rows
    else:
        nbytes = (24.0 if c["adamw"] else 8.0) * P                        # weights in, gradients out; AdamW: p, m, v in and out
    return {"bytes": nbytes + 8.0 * N, "flops": flops}


def _device_bytes(c):
    N, d, F = c["B"] // c["M"] * c["T"], c["d"], c["F"]
    layer = N * (2 * (6 * d + 2 * F) + 8 * d)
    s = max(_streams(c, k) for k in range(c["K"])) if c["rule"] == "sum" else c["n"]
    chunk = c["V"] + 64 if c["head_mode"] == "stored" else 8192
    return _params(c) * 18 + c["K"] * ((c["Lc"] + c["Lh"]) * layer + s * N * (2 * F + 16 * d) + N * (2 * chunk + 12 * d))


def draw(rng):
    """One more case of the ranges above: sizes over their logarithm, odd ones among them, options as users set them."""
    limit = work(listed()[6])["flops"]

    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        dh = rng.choice([32, 64, 64, 64, 80, 128, 256])
        H = max(1, round(logint(128, 2560) / dh))
        d = H * dh
        K = rng.choice([1, 2, 2, 3, 4, 4, 6, 8])
        M = rng.choice([1, 1, 1, 2, 4])
        T = logint(16, 2048)
        B = logint(1, 64)
        c = _case(None, kind=rng.choice(["train", "train", "train", "eval"]), K=K, Lc=rng.choice([1, 2, 3, 4]), d=d, H=H,
                  F=rng.choice([4 * d, 4 * d, 3 * d, (8 * d // 3 + 7) // 8 * 8]), V=logint(300, 50257), T=T, B=B,
                  n=rng.randint(1, min(K, 4)), rule=rng.choice(["sum", "sum", "sum", "mean", "far"]),
                  Lh=rng.choice([0, 0, 0, 1, 2]), adamw=rng.random() < 0.7,
                  head_mode=rng.choice(["stored", "stored", "recompute"]),
                  attn_bwd=rng.choice(["one_sweep", "one_sweep", "two_kernels"]))
        if c["kind"] == "train" and M > 1:
            c["M"], c["B"] = M, (B + M - 1) // M * M
        if c["B"] // c["M"] * T <= 16384 and work(c)["flops"] <= limit and _device_bytes(c) < 40e9:
            return c


def _draw_tokens(c, gen):
    p = torch.arange(1, c["V"] + 1, dtype=torch.float64, device="cuda").pow(-1.1)
    cdf = torch.cumsum(p, 0)
    u = torch.rand(c["B"], c["T"] + 1, dtype=torch.float64, device="cuda", generator=gen) * cdf[-1]
    ids = torch.searchsorted(cdf, u).clamp(max=c["V"] - 1).to(torch.int32)
    return ids[:, :-1].contiguous(), ids[:, 1:].contiguous()


def prepare(case, seed):
    """A model with its weights loaded and a batch in pinned host memory."""
    gc.collect()                    # a model that is no longer used gives its memory back before the next is made
    c = dict(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    m = Model(c["K"], c["Lc"], c["d"], c["H"], c["F"], c["V"], c["n"], c["B"] // c["M"], c["T"], head_layers=c["Lh"],
              head_mode=c["head_mode"], attn_bwd=c["attn_bwd"])
    if c["rule"] != "sum":
        m.set_rule(c["rule"])
    if c["M"] > 1:
        m.set_micro_batches(c["M"])
    staging = torch.empty(max(int(np.prod(s)) for s in m.shapes.values()), dtype=torch.float32, pin_memory=True)
    for name in m.names:
        shape = m.shapes[name]
        w = torch.randn(shape, dtype=torch.float32, device="cuda", generator=gen) * 0.02
        if name.endswith(".g"):
            w += 1.0
        host = staging[:w.numel()].view(shape)
        host.copy_(w)
        m.set_param(name, host.numpy())
    tokens, targets = (t.cpu().pin_memory() for t in _draw_tokens(c, gen))
    # The model's parameters, gradients and Adam moments: the first four blocks it took from torch's allocator, fp32
    # in registry order.
    flat = [b.view(torch.float32) for b in list(m._blocks.values())[:4]]
    return {"case": c, "model": m, "tokens": tokens, "targets": targets, "flat": flat}


def run(state):
    m, c = state["model"], state["case"]
    if c["kind"] == "eval":
        m.set_batch(state["tokens"], state["targets"])
        for k in range(c["K"]):
            m.forward_component(k)
            m.aux_head_loss(k)
        losses = m.get_losses()
        return {"losses": losses, "token_losses": m.get_token_losses(c["K"] - 1, c["B"] * c["T"])}
    hp = ADAMW if c["adamw"] else None
    if c["M"] > 1:
        if hp is None:
            m.set_micro_batches(c["M"])          # no update follows: start the next accumulation
        m.train_minibatch(state["tokens"], state["targets"], c["M"], adamw=hp)
    else:
        m.train_step(state["tokens"], state["targets"], adamw=hp)
    out = {"losses": m.get_losses(), "gradients": state["flat"][1]}
    if hp:
        out.update(weights=state["flat"][0], adam_m=state["flat"][2], adam_v=state["flat"][3])
    return out


def tolerance(case):
    # bf16 operands, fp32 sums.  Losses: a bf16 rounding (2^-9) of a logit of order one against a loss of order ln V.
    # Gradients: four times what the other head mode and the other attention backward give on the same inputs (up to
    # 2.3e-3, single values up to 0.58 of the root mean square).
    if case["kind"] == "eval":
        return {"rel": 5e-4, "max": 5e-3}
    return {"rel": 1e-2, "max": 0.9}
