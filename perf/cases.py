"""The work that users of this framework have it do, as cases that can be timed and compared.

Four kinds, all through the public Python entry points (`binding.Mira`, `binding.NativeStack`):

  layer     one MoE layer on compressed experts, `Mira.moe_layer`: decode batches, mixed batches, prefill
  quantize  full-precision experts to compressed ones, `Mira.quantize_experts`: once per checkpoint
  predict   the expert predictor of a decode or prefill step, `Mira.predict` (linear head) or
            `Mira.predict_mixture` (mixture head on the router's by-products)
  stack     one decode step of a stack of layers over a small expert cache, `NativeStack.layer_step`

Shapes are those of `paper_2609_38090_b200.inputs`: Mixtral-8x7B's and 8x22B's layer, a fine-grained layer with
shared experts, and (drawn cases) layers of generic sizes between them. Values follow the recipe of that module
(activations N(0, 1), weights 0.02 N(0, 1), a Zipf-skewed router bias), drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_38090_b200 import binding, inputs

_SHAPES = {s.name: s for s in (inputs.MIXTRAL, inputs.MIXTRAL22, inputs.FINE)}


def _layer(shape: str, tokens: int, name: str | None = None, fmt: int = 0, act_on_w1: bool = False) -> dict:
    s = _SHAPES[shape]
    c = dict(kind="layer", hidden=s.C, ffn=s.R, experts=s.E, shared=s.n_shared, top_k=s.k, zipf=s.zipf_a, tokens=tokens,
             fmt=fmt, act_on_w1=act_on_w1)
    return dict(c, name=name) if name else c


def listed() -> list[dict]:
    fine = _SHAPES["fine_grained"]
    return [
        # one user typing: the step that latency is judged by
        _layer("mixtral8x7b", 1, "mixtral-decode-1"),
        # a handful of users on the larger model, weights in the standard per-matrix format, checkpoint convention
        # for the activated matrix; an odd batch as continuous batching leaves it
        _layer("mixtral8x22b", 13, "mixtral22-decode-13", fmt=1, act_on_w1=True),
        # the framework's headline step: a full decode batch
        _layer("mixtral8x7b", 32, "mixtral-decode-32"),
        # decode batch plus a chunk of somebody's prompt
        _layer("mixtral8x7b", 200, "mixtral-mixed-200"),
        # a long prompt
        _layer("mixtral8x7b", 2048, "mixtral-prefill-2048"),
        # beam search of width 4 on a model of many small experts
        _layer("fine_grained", 4, "fine-decode-4"),
        # a full decode batch there
        _layer("fine_grained", 64, "fine-decode-64"),
        # a prompt there, of no particular length
        _layer("fine_grained", 1000, "fine-prefill-1000"),
        # converting a checkpoint: one layer's experts, stored as bf16
        dict(kind="quantize", hidden=fine.C, ffn=fine.R, experts=fine.n_experts_total, dtype="bf16", fmt=0,
             name="fine-quantize-layer"),
        # which experts to stage, asked once per layer of a beam-4 decode step: the smallest call
        dict(kind="predict", hidden=fine.C, experts=fine.E, tokens=4, k_pred=4, mixture=False, name="fine-predict-4"),
        # the same question put to the mixture head for a full decode batch
        dict(kind="predict", hidden=fine.C, experts=fine.E, tokens=64, k_pred=4, mixture=True, name="fine-mixture-64"),
        # memory-limited decoding: beam 4, a quarter of the experts resident, the others fetched over PCIe
        dict(kind="stack", hidden=fine.C, ffn=fine.R, experts=fine.E, shared=fine.n_shared, top_k=fine.k, zipf=fine.zipf_a,
             tokens=4, layers=6, hot=12, stage=3, k_pred=4, name="fine-stack-beam4"),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    u = rng.random()
    if u < 0.68:
        v = rng.random()
        if v < 0.35:
            c = _layer("mixtral8x7b", _log_int(rng, 1, 2048))
        elif v < 0.45:
            c = _layer("mixtral8x22b", _log_int(rng, 1, 1024))
        elif v < 0.8:
            c = _layer("fine_grained", _log_int(rng, 1, 4096))
        else:  # layers of other sizes; a layer's experts together are at most as large as the 8x7B's
            hidden, ffn = 64 * _log_int(rng, 12, 80), 64 * _log_int(rng, 10, 160)
            experts = min(rng.choice([8, 16, 32, 64, 96, 128]), max(8, int(1.4e9 / (3 * hidden * ffn))))
            c = dict(kind="layer", hidden=hidden, ffn=ffn, experts=experts, shared=rng.choice([0, 0, 1, 2]),
                     top_k=rng.randint(1, min(8, experts)), zipf=1.1, tokens=_log_int(rng, 1, 2048))
            flops = 6.0 * hidden * ffn * (c["top_k"] + c["shared"])
            c["tokens"] = max(1, min(c["tokens"], int(1.4e12 / flops)))
        c["fmt"], c["act_on_w1"] = int(rng.random() < 0.2), rng.random() < 0.5
        c["zipf"] = rng.choice([0.0, c["zipf"], c["zipf"]])
        return c
    if u < 0.80:
        s = _SHAPES[rng.choice(["mixtral8x7b", "fine_grained", "mixtral8x22b"])]
        most = {"mixtral8x7b": 4, "mixtral8x22b": 2, "fine_grained": 64}[s.name]
        return dict(kind="quantize", hidden=s.C, ffn=s.R, experts=_log_int(rng, 1, most), dtype=rng.choice(["bf16", "fp32"]),
                    fmt=int(rng.random() < 0.2))
    if u < 0.93:
        s = _SHAPES[rng.choice(["mixtral8x7b", "fine_grained"])]
        return dict(kind="predict", hidden=s.C, experts=s.E, tokens=_log_int(rng, 1, 2048), k_pred=min(s.E, rng.choice([2, 4, 8])),
                    mixture=rng.random() < 0.4)
    s = _SHAPES["fine_grained"]
    return dict(kind="stack", hidden=s.C, ffn=s.R, experts=s.E, shared=s.n_shared, top_k=s.k, zipf=s.zipf_a,
                tokens=rng.choice([1, 2, 3, 4, 5, 6, 8]), layers=rng.choice([3, 4, 5, 6]), hot=rng.choice([12, 18, 21, 30, 45, 60]),
                stage=rng.choice([3, 4]), k_pred=rng.choice([0, 4, 4]))


# ----------------------------------------------------------------------------------------------- what a program holds
class _Draws:
    """Random tensors on the GPU, from the seed alone."""

    def __init__(self, seed: int):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(1_000_003 * seed + 17)
        self.host = np.random.Generator(np.random.PCG64([seed, 29]))

    def normal(self, *dims, scale=1.0, dtype=torch.bfloat16):
        return (torch.randn(dims, generator=self.g, device="cuda") * scale).to(dtype)

    def bias(self, experts: int, zipf: float):
        p = (1 + self.host.permutation(experts)).astype(np.float64) ** (-zipf)
        return torch.from_numpy(np.log(p / p.sum()).astype(np.float32))


def _weights(d: _Draws, n: int, hidden: int, ffn: int, dtype):
    return [d.normal(n, *s, scale=0.02, dtype=dtype) for s in ((ffn, hidden), (hidden, ffn), (ffn, hidden))]


def _compressed(d: _Draws, m, n: int, hidden: int, ffn: int, out) -> None:
    step = max(1, int(2e8 / (hidden * ffn)))
    for e in range(0, n, step):
        out[e:e + step] = m.quantize_experts(*_weights(d, min(step, n - e), hidden, ffn, torch.float32))


def prepare(case: dict, seed: int) -> dict:
    d, kind, C = _Draws(seed), case["kind"], case["hidden"]
    if kind == "quantize":
        m = binding.Mira(C, case["ffn"], case["experts"], max_tokens=1, max_top_k=1, fmt=case["fmt"])
        dtype = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
        return dict(kind=kind, m=m, w=_weights(d, case["experts"], C, case["ffn"], dtype))
    E, T = case["experts"], case["tokens"]
    if kind == "predict":
        m = binding.Mira(C, 64, E, n_layers=24, max_tokens=T, max_top_k=min(E, 4))
        s = dict(kind=kind, m=m, x=d.normal(T, C), k_pred=case["k_pred"], mixture=case["mixture"])
        if case["mixture"]:
            k = min(E, 4)
            s["head"] = dict(wa_h=d.normal(E, C, scale=0.02), wa_l=d.normal(E, E, scale=0.3), wh_c=d.normal(E, E, scale=2.0),
                             wh_t=d.normal(E, E, scale=0.3), g_h=d.normal(C, scale=0.02), g_l=d.normal(E, scale=0.3),
                             g_c=d.normal(E), b_a=d.normal(E, scale=0.02, dtype=torch.float32),
                             b_h=d.normal(E, scale=0.02, dtype=torch.float32), b_g=0.1)
            r = m.route(s["x"], d.normal(E, C, scale=0.02), d.bias(E, 1.1).cuda(), k)
            s.update(logits=r["logits"], count=r["count"], k_top=k)
        else:
            s.update(w=d.normal(E, C, scale=0.02), b=d.normal(E, scale=0.02, dtype=torch.float32))
        return s
    R, ns, k = case["ffn"], case["shared"], case["top_k"]
    if kind == "layer":
        m = binding.Mira(C, R, E, n_shared=ns, max_tokens=T, max_top_k=k, act_on_w1=case["act_on_w1"], fmt=case["fmt"])
        blobs = torch.empty((E + ns, m.expert_bytes), dtype=torch.uint8, device="cuda")
        _compressed(d, m, E + ns, C, R, blobs)
        return dict(kind=kind, m=m, x=d.normal(T, C), w=d.normal(E, C, scale=0.02), b=d.bias(E, case["zipf"]).cuda(), k=k,
                    blobs=blobs, slots=binding.slot_table(blobs), slot_map=torch.arange(E + ns, dtype=torch.int32, device="cuda"))
    L, hot = case["layers"], case["hot"]
    m = binding.Mira(C, R, E, n_shared=ns, n_layers=L, max_tokens=T, max_top_k=k)
    host = torch.empty((L, E + ns, m.expert_bytes), dtype=torch.uint8, pin_memory=True)
    blobs = torch.empty((E + ns, m.expert_bytes), dtype=torch.uint8, device="cuda")
    for layer in range(L):
        _compressed(d, m, E + ns, C, R, blobs)
        host[layer].copy_(blobs)
    bias = [d.bias(E, case["zipf"]) for _ in range(L)]
    mem = torch.empty((L, ns + hot + case["stage"], m.expert_bytes), dtype=torch.uint8, device="cuda")
    stack = binding.NativeStack(m, host, mem, [sorted(torch.argsort(-v)[:hot].tolist()) for v in bias], hot, case["stage"],
                                case["k_pred"], torch.cuda.Stream())
    return dict(kind=kind, m=m, stack=stack, k=k, k_pred=case["k_pred"], x=[d.normal(T, C) for _ in range(L)],
                w=[d.normal(E, C, scale=0.02) for _ in range(L)], b=[v.cuda() for v in bias])


def run(state: dict):
    kind, m = state["kind"], state["m"]
    if kind == "layer":
        return m.moe_layer(state["x"], state["w"], state["b"], state["slots"], state["slot_map"], state["k"])
    if kind == "quantize":
        return m.quantize_experts(*state["w"])
    if kind == "predict":
        if state["mixture"]:
            return m.predict_mixture(0, state["x"], state["logits"], state["count"], state["k_top"], state["head"], state["k_pred"])
        return m.predict(0, state["x"], state["w"], state["b"], k_pred=state["k_pred"])
    outs, w, b = [], state["w"], state["b"]
    L = len(w)
    # What enters a layer comes from the attention block before it, which this framework does not have: it is in hand.
    # The head that scores the experts of layer + 2 is that layer's router, as in the stack harness.
    for layer, x in enumerate(state["x"]):
        ahead = layer + 2 if state["k_pred"] and layer + 2 < L else None
        y = state["stack"].layer_step(layer, x, w[layer], b[layer], state["k"], None if ahead is None else w[ahead],
                                      None if ahead is None else b[ahead])
        outs.append(binding.residual_rmsnorm(x, y))
    return outs


# ----------------------------------------------------------------------------------------- what cannot be done without
def _distinct(experts: int, top_k: int, tokens: int, zipf: float, spread: float) -> float:
    """Distinct routed experts of a batch: the mean of a few simulated ones (logits N(0, spread^2) plus the Zipf bias)."""
    g, n = np.random.Generator(np.random.PCG64([experts, top_k, tokens])), max(1, 64 // tokens)
    logits = spread * g.standard_normal((n, tokens, experts)) - zipf * np.log(np.arange(1, experts + 1))
    best = np.argpartition(-logits, top_k - 1, axis=2)[:, :, :top_k]
    return float(np.mean([len(np.unique(b)) for b in best]))


def _expert_bytes(case: dict) -> int:
    return int(binding.mira_expert_bytes_format(case["ffn"], case["hidden"], case.get("fmt", 0)))


def work(case: dict) -> dict:
    kind, C, E = case["kind"], case["hidden"], case["experts"]
    if kind == "quantize":
        n = 3 * case["ffn"] * C
        return dict(bytes=E * (n * (4 if case["dtype"] == "fp32" else 2) + _expert_bytes(case)), flops=E * 2.0 * n)
    T = case["tokens"]
    if kind == "predict":
        if case["mixture"]:
            return dict(bytes=2 * T * C + 4 * T * E + 2 * E * C + 6 * E * E + 2 * C, flops=T * C + 2.0 * E * C + 6.0 * E * E)
        return dict(bytes=2 * T * C + 2 * E * C, flops=2.0 * T * C * E)
    active = _distinct(E, case["top_k"], T, case["zipf"], 0.02 * math.sqrt(C)) + case["shared"]
    one = dict(bytes=active * _expert_bytes(case) + 4 * T * C + 2 * E * C,
               flops=6.0 * T * (case["top_k"] + case["shared"]) * C * case["ffn"] + 2.0 * T * C * E)
    if kind == "layer":
        return one
    heads = (case["layers"] - 2 if case["k_pred"] else 0) * 2 * E * C
    return dict(bytes=case["layers"] * (one["bytes"] + 6 * T * C) + heads, flops=case["layers"] * one["flops"])


def tolerance(case: dict):
    if case["kind"] == "quantize":
        return "exact"      # codes and scales are defined bit for bit
    if case["kind"] == "predict":
        # 32-bit sums; against 64-bit ones 0.6e-7 to 1.7e-7 at 4 and 64 tokens, and the mean over thousands of
        # tokens is a small number left of larger ones
        return dict(rel=1e-5, max=1e-4, differ=0.0)
    # bf16 outputs of 32-bit sums over a 16-bit intermediate: a value next to a rounding boundary moves by one unit in
    # the last place (2^-8 to 2^-7 of itself). The two kernel families on the same inputs: rel 2.1e-4 to 3.5e-4, max 7.8e-3
    return dict(rel=1.4e-3, max=2e-2)
