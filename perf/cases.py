"""Performance cases of the MoE layer: what a program that uses this package has it do.

Every case is one pass through the public entry points (``binding.Plan``): the whole layer on device buffers
(``entry = "layer"``), the four steps called one after the other on the caller's own buffers (``"stages"``), or a
stream of batches in pinned host memory with two steps in flight (``"host"``).  Shapes are the workloads of
``inputs.py`` (the Mixtral-, Phi-3.5-, Qwen- and DeepSeek-V3-like layers, the identity-expert dispatch / combine
sweep and the tiny fp32 layer) with the token counts of decoding (1 to some hundred) and of prefill (thousands), and
generic ragged ones.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_05888_b200 import binding as B

# H, E, R, K, F, renormalised weights
SHAPES = {
    "mixtral": dict(H=4096, E=8, R=8, K=2, F=14336, renorm=1),
    "phi35": dict(H=4096, E=16, R=8, K=2, F=6400, renorm=1),
    "qwen": dict(H=2048, E=60, R=4, K=4, F=1408, renorm=0),
    "deepseek": dict(H=7168, E=256, R=32, K=8, F=2048, renorm=1),
    "sweep": dict(H=7168, E=256, R=32, K=8, F=0, renorm=0),      # identity experts: dispatch and combine only
}
HOST_BATCHES = 4  # batches of one "host" pass


def _case(entry, dtype, T, H, E, R, K, F, renorm=0, zipf=0.0):
    return dict(entry=entry, dtype=dtype, T=T, H=H, E=E, R=R, K=K, F=F, renorm=renorm, zipf=zipf)


def listed():
    S = SHAPES
    cases = {
        # the smallest layer: latency and launches; fp32, where every sum has to be fp32
        "tiny_fp32": _case("layer", "fp32", T=256, H=128, E=8, R=2, K=2, F=256),
        # a small model served or checked in fp32, ragged token count
        "ragged_fp32": _case("layer", "fp32", T=1000, H=1024, E=16, R=4, K=2, F=2048),
        # decoding one sequence: four experts' weights once, nothing to batch
        "qwen_decode_1": _case("layer", "bf16", T=1, **S["qwen"]),
        # decoding a small batch with a few large experts: weight streaming
        "mixtral_decode_24": _case("layer", "bf16", T=24, **S["mixtral"]),
        # a decode-shaped batch over many small experts
        "qwen_512": _case("layer", "bf16", T=512, **S["qwen"]),
        # decoding a batch over 256 experts with skewed popularity: nearly all weights for a thousand rows
        "deepseek_decode_128": _case("layer", "bf16", T=128, zipf=1.0, **S["deepseek"]),
        # a ragged prefill chunk through the four steps on the caller's buffers
        "qwen_stages_2777": _case("stages", "bf16", T=2777, **S["qwen"]),
        # a prefill chunk from and to host memory, two steps in flight
        "phi35_host_1023": _case("host", "bf16", T=1023, **S["phi35"]),
        # large prefill, few experts: tensor-core bound
        "mixtral_4096": _case("layer", "bf16", T=4096, **S["mixtral"]),
        # large prefill, many experts, skewed load: the largest layer
        "deepseek_8192": _case("layer", "bf16", T=8192, zipf=1.0, **S["deepseek"]),
        # routing, dispatch and combine alone (the experts are someone else's), small and large
        "sweep_256": _case("stages", "bf16", T=256, **S["sweep"]),
        "sweep_16384": _case("stages", "bf16", T=16384, zipf=1.2, **S["sweep"]),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp32", "qwen", "mixtral", "phi35", "deepseek", "sweep", "generic", "generic"])
    if kind == "fp32":
        E = rng.choice([4, 8, 16, 32, 60])
        return _case("layer", "fp32", T=_log_int(rng, 16, 1024), H=4 * _log_int(rng, 16, 256), E=E, R=4, K=rng.randint(1, 4),
                     F=4 * _log_int(rng, 16, 512), renorm=rng.randint(0, 1), zipf=rng.choice([0.0, 1.0]))
    if kind == "generic":
        E, R = rng.choice([(8, 2), (12, 4), (32, 4), (64, 8), (96, 8), (128, 8)])
        return _case(rng.choice(["layer", "layer", "stages"]), "bf16", T=_log_int(rng, 1, 4096), H=8 * _log_int(rng, 64, 512), E=E, R=R,
                     K=rng.choice([1, 2, 3, 4, 6, 8]), F=8 * _log_int(rng, 32, 512), renorm=rng.randint(0, 1), zipf=rng.choice([0.0, 1.0]))
    top = {"qwen": 8192, "mixtral": 6000, "phi35": 8192, "deepseek": 8000, "sweep": 32768}[kind]
    low = {"deepseek": 8, "sweep": 128}.get(kind, 1)
    entry = "stages" if kind == "sweep" else rng.choice(["layer", "layer", "stages", "host"])
    if kind == "deepseek":
        entry = "layer"
    elif entry == "host":
        top //= HOST_BATCHES
    zipf = {"deepseek": rng.choice([0.0, 1.0]), "sweep": rng.choice([0.0, 1.2])}.get(kind, 0.0)
    return _case(entry, "bf16", T=_log_int(rng, low, top), zipf=zipf, **SHAPES[kind])


def _elem(case):
    return 2 if case["dtype"] == "bf16" else 4


def _dispatch_mode(case):
    """Large dispatches use the token-ordered scheme, others the default (paged) one, as bench.py does."""
    moved = case["T"] * case["H"] * _elem(case) * (1 + case["K"])
    return B.DISPATCH_ATOMIC_ORDERED if moved >= 512e6 else B.DISPATCH_ATOMIC_PAGED


def prepare(case, seed):
    c = case
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    T, H, E, K, F = c["T"], c["H"], c["E"], c["K"], c["F"]
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape, std=1.0):
        return torch.empty(shape, dtype=dt, device="cuda").normal_(0.0, std, generator=g)

    s = {"entry": c["entry"], "identity": F == 0}
    s["wr"] = normal(E, H, std=0.02)
    s["bias"] = None
    if c["zipf"] > 0.0:
        order = torch.randperm(E, device="cuda", generator=g).to(torch.float32)
        s["bias"] = -c["zipf"] * torch.log1p(order)
    s["wg"] = normal(E, F, H, std=0.02) if F else None
    s["wu"] = normal(E, F, H, std=0.02) if F else None
    s["wd"] = normal(E, H, F, std=0.02) if F else None
    plan = B.Plan(B.make_config(T, H, E, c["R"], K, F, B.DTYPE_BF16 if c["dtype"] == "bf16" else B.DTYPE_FP32, renormalize=c["renorm"],
                                dispatch_mode=_dispatch_mode(c), identity_experts=int(F == 0)))
    s["plan"] = plan
    if c["entry"] == "host":
        s["x"] = [normal(T, H).cpu().pin_memory() for _ in range(HOST_BATCHES)]
        s["y"] = [torch.empty(T, H, dtype=dt).pin_memory() for _ in range(HOST_BATCHES)]
        return s
    s["x"] = normal(T, H)
    s["y"] = torch.empty(T, H, dtype=dt, device="cuda")
    if c["entry"] == "layer":
        # the layer's picks, weights and rows per expert, where the plan keeps them
        s["idx"], s["w"], s["count"] = (plan.layer_tensor(i) for i in (0, 1, 3))
        return s
    rows = plan.P * B.TILE_ROWS

    def ints(*shape):
        return torch.empty(shape, dtype=torch.int32, device="cuda")

    s["idx"], s["w"] = ints(T, K), torch.empty(T, K, dtype=torch.float32, device="cuda")
    s["recv"] = torch.empty(rows, H, dtype=dt, device="cuda")
    s["out_rows"] = torch.empty(rows, H, dtype=dt, device="cuda") if F else s["recv"]
    s["count"], s["tile_expert"], s["src"], s["slot"] = ints(E), ints(plan.P), ints(rows), ints(T, K)
    s["tile_count"], s["rows_done"] = ints(plan.P), ints(1)
    return s


def run(s):
    p = s["plan"]
    if s["entry"] == "layer":
        p.moe_layer(s["x"], s["wr"], s["bias"], s["wg"], s["wu"], s["wd"], s["y"])
    elif s["entry"] == "stages":
        p.moe_route(s["x"], s["wr"], s["bias"], s["idx"], s["w"])
        p.moe_dispatch(s["x"], s["idx"], s["recv"], s["count"], s["tile_expert"], s["src"], s["slot"], s["tile_count"], s["rows_done"])
        if not s["identity"]:
            p.moe_expert_ffn(s["recv"], s["tile_expert"], s["wg"], s["wu"], s["wd"], s["out_rows"], s["tile_count"], s["rows_done"])
        p.moe_combine(s["out_rows"], s["slot"], s["w"], s["y"])
    else:
        tickets = []
        for x, y in zip(s["x"], s["y"]):
            if len(tickets) >= 2:
                p.moe_layer_host_wait(tickets[-2])
            tickets.append(p.moe_layer_host_submit(x, s["wr"], s["bias"], s["wg"], s["wu"], s["wd"], y))
        for t in tickets[-2:]:
            p.moe_layer_host_wait(t)
        return {"y": s["y"]}
    return {"y": s["y"], "idx": s["idx"], "w": s["w"], "count": s["count"]}


def _experts_used(case):
    """Experts that at least one token picks: simulated, as the logits are (near) normal."""
    T, H, E, K = case["T"], case["H"], case["E"], case["K"]
    rng = np.random.default_rng(1)
    logits = rng.standard_normal((min(T, 4096), E)) * (0.02 * math.sqrt(H))
    if case["zipf"] > 0.0:
        logits = logits - case["zipf"] * np.log1p(rng.permutation(E))
    return len(np.unique(np.argpartition(-logits, K - 1, axis=1)[:, :K]))


def work(case):
    c, b = case, _elem(case)
    T, H, E, K, F = c["T"], c["H"], c["E"], c["K"], c["F"]
    passes = HOST_BATCHES if c["entry"] == "host" else 1
    nbytes = E * H * b + passes * 2 * T * H * b
    if c["entry"] == "stages":
        # the steps hand rows over in the caller's buffers: each is an output of one and an input of the next
        nbytes += 2 * T * K * H * b * (2 if F else 1) + 4 * T * K * 8
    if F:
        nbytes += passes * 3 * _experts_used(c) * F * H * b  # more than L2 holds: every batch streams them
    return {"bytes": float(nbytes), "flops": float(passes * (2 * T * H * E + 6 * T * K * H * F))}


def tolerance(case):
    # About four times what the path is away from itself in 64 bits: fp32 up to 1.3e-6 (largest 1.1e-5, H 1024,
    # F 2048), bf16 2.9e-3 (1.8e-2): the intermediate, the expert rows and y are each rounded to bf16 once.
    if case["dtype"] == "fp32":
        return {"rel": 6e-6, "max": 6e-5}
    return {"rel": 1e-2, "max": 6e-2}
