"""The calls that a program built on this framework makes, with the sizes and values it makes them at.

Every case goes through the public entry points of `paper_2608_15383_b200.binding`.  Three kinds:

  layer   device tensors: per layer `exmoe_route` (Eq. 1) and then `Cache.forward`, for `steps` consecutive steps through
          `layers` sparse layers.  The dense parts between the layers are not this framework's, so each layer's hidden
          states are given.  `slots` below `experts` is the offloaded cache over the pinned host bank.
  host    the same layers through `Cache.forward_host`: host tensors in and out, one synchronous call per layer.
  pack    `pack_bank`: the offline conversion of one layer's BF16 experts into the pinned int4 bank.

Weights N(0, 0.02), hidden states N(0, 1), router weights N(0, 0.02) and a Zipf bias of strength `alpha`, as in `synth`.
A step walks a stack of layers, as decoding does, so the weights of small batches come from HBM and not from L2.
"""
import math

import numpy as np
import torch

from paper_2608_15383_b200 import binding, synth

SIZES = ("d_model", "d_ff", "experts", "top_k")
OLMOE = (2048, 1024, 64, 8)     # synth.OLMOE
WIDE_FF = (2048, 1408, 60, 4)   # the block of the shared-expert test: 11 blocks of 128, no power of two
MID = (512, 256, 16, 4)         # synth.MID
TINY = (256, 128, 8, 2)         # synth.TINY
BANKS = 2                       # distinct banks of a stack; resident layers copy theirs into slots of their own


def _layer(sizes, tokens, layers, slots=None, alpha=0.5, steps=1, kind="layer"):
    return dict(zip(SIZES, sizes), kind=kind, tokens=tokens, layers=layers, slots=slots or sizes[2], alpha=alpha, steps=steps)


def listed():
    return [
        # the smallest layer anybody runs (a unit test, a toy model, a draft model's block): launches and host time only
        dict(_layer(TINY, 16, 1, alpha=0.0), name="tiny_16"),
        # one user's decode step through all 16 sparse layers of the 64-expert top-8 model, everything resident
        dict(_layer(OLMOE, 1, 16), name="decode_1"),
        # the same step by a serving process whose tensors live on the host
        dict(_layer(OLMOE, 1, 16, kind="host"), name="decode_1_host"),
        # a few users, or a few speculated tokens, at an odd count
        dict(_layer(OLMOE, 5, 16), name="decode_5"),
        # ordinary batched decode
        dict(_layer(OLMOE, 16, 8), name="decode_16"),
        # large batched decode: every expert active with a handful of rows
        dict(_layer(OLMOE, 64, 4), name="decode_64"),
        # batched decode of another geometry, whose block counts are not powers of two
        dict(_layer(WIDE_FF, 24, 8), name="wide_ff_24"),
        # the paper's memory-bound setting: 16 of 64 experts on the GPU, misses fetched from the host bank
        dict(_layer(OLMOE, 16, 2, slots=16, alpha=1.0, steps=4), name="offload_16"),
        # a short prompt of odd length (or one chunk of a chunked prefill)
        dict(_layer(OLMOE, 333, 2), name="prefill_333"),
        # an ordinary prompt, uniform routing
        dict(_layer(OLMOE, 2048, 1, alpha=0.0), name="prefill_2048"),
        # the largest prefill batch, skewed routing
        dict(_layer(OLMOE, 8192, 1, alpha=1.0), name="prefill_8192"),
        # converting a checkpoint, one layer at a time
        dict(zip(SIZES, OLMOE), kind="pack", name="pack_64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(("decode", "decode", "prefill", "prefill", "other", "host", "offload", "pack"))
    alpha = rng.choice((0.0, round(rng.uniform(0.1, 1.5), 2)))
    if what == "decode":
        T = _log_int(rng, 1, 128)
        return _layer(OLMOE, T, rng.randint(8, 16) if T < 20 else rng.randint(3, 8), alpha=alpha)
    if what == "prefill":
        return _layer(OLMOE, _log_int(rng, 128, 8192), 1, alpha=alpha)
    if what == "other":
        sizes = rng.choice((TINY, MID, WIDE_FF, (128 * rng.randint(4, 16), 128 * rng.randint(2, 12), 4 * rng.randint(4, 24), rng.randint(2, 8))))
        return _layer(sizes, _log_int(rng, 1, 1024), rng.randint(1, 8), alpha=alpha)
    if what == "host":
        return _layer(OLMOE, _log_int(rng, 1, 512), rng.randint(4, 16), alpha=alpha, kind="host")
    if what == "offload":
        return _layer(OLMOE, _log_int(rng, 1, 64), 2, slots=rng.choice((16, 24, 32, 48)), alpha=round(rng.uniform(0.3, 2.0), 2), steps=4)
    return dict(d_model=128 * rng.randint(4, 16), d_ff=128 * rng.randint(2, 12), experts=rng.randint(8, 64), top_k=2, kind="pack")


def _shape(case):
    return synth.Shape(*(case[k] for k in SIZES))


def prepare(case, seed):
    shape = _shape(case)
    seed = 1000 * (seed % 1_000_003)
    if case["kind"] == "pack":
        return {"kind": "pack", "shape": shape, "weights": synth.expert_weights(shape, seed, device="cuda")}
    L, T, steps = case["layers"], case["tokens"], case["steps"]
    banks = [binding.pack_bank(shape, *synth.expert_weights(shape, seed + b, device="cuda")) for b in range(min(L, BANKS))]
    state = {"kind": case["kind"], "shape": shape, "steps": steps, "layers": L,
             "cache": binding.Cache(shape, [banks[l % BANKS] for l in range(L)], case["slots"], T),
             "router": [synth.router_weights(shape, seed + 100 + l, device="cuda") for l in range(L)],
             "bias": [synth.zipf_bias(shape.num_experts, case["alpha"], seed + 200 + l).cuda() if case["alpha"] else None for l in range(L)]}
    state["hidden"] = [[synth.hidden_states(shape, T, seed + 300 + s * L + l, device="cuda") for l in range(L)] for s in range(steps)]
    if case["kind"] == "host":
        # a host-side serving loop has its activations, ids and mixture weights in page-locked memory
        calls = []
        for l, hidden in enumerate(state["hidden"][0]):
            ids, weights = binding.exmoe_route(shape, hidden, state["router"][l], state["bias"][l])
            calls.append(tuple(x.cpu().pin_memory() for x in (hidden, ids, weights)))
        state["calls"] = calls
        state["out"] = [torch.empty_like(c[0]).pin_memory() for c in calls]
    return state


def run(state):
    shape = state["shape"]
    if state["kind"] == "pack":
        return binding.pack_bank(shape, *state["weights"])
    cache = state["cache"]
    if state["kind"] == "host":
        return [cache.forward_host(l, *call, out=state["out"][l]) for l, call in enumerate(state["calls"])]
    outs = []
    for step in state["hidden"]:
        for l, hidden in enumerate(step):
            ids, weights = binding.exmoe_route(shape, hidden, state["router"][l], state["bias"][l])
            outs.append((ids, weights, cache.forward(l, hidden, ids, weights)))
    return outs


def _active_experts(case):
    """Distinct experts that `tokens` tokens select, on average: inclusion frequencies of a sample of routed tokens."""
    E, k, T = case["experts"], case["top_k"], case["tokens"]
    rng = np.random.default_rng(0)
    logits = 0.02 * math.sqrt(case["d_model"]) * rng.standard_normal((2048, E)) - case["alpha"] * 1.1 * np.log(np.arange(1, E + 1))
    chosen = np.argpartition(-logits, k - 1, axis=1)[:, :k] if k < E else np.tile(np.arange(E), (2048, 1))
    share = np.bincount(chosen.ravel(), minlength=E) / 2048
    return float(np.sum(1.0 - (1.0 - share) ** T))


def work(case):
    H, I, E, k = (case[x] for x in SIZES)
    packed = 3 * I * H * (4 / 8 + 2 / 128)
    if case["kind"] == "pack":
        return {"bytes": E * (3 * I * H * 2 + packed), "flops": 0}
    T, calls = case["tokens"], case["layers"] * case["steps"]
    route = case["kind"] != "host"
    # per call: active experts' packed bytes, hidden in, output, ids and mixture weights (and the router's matrix)
    per = _active_experts(case) * packed + 2 * T * H * 2 + T * k * 8 + (2 * H * E if route else 0)
    return {"bytes": calls * per, "flops": calls * (6 * T * k * I * H + (2 * T * H * E if route else 0))}


def tolerance(case):
    if case["kind"] == "pack":
        return "exact"
    # BF16 products, one BF16 rounding between the GEMMs (some kernels round the scaled weights to BF16 too) and one of
    # the output; an expert id may differ where two logits tie in binary32
    return {"rel": 1e-2, "max": 5e-2, "differ": 1e-3}
