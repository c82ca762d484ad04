"""What this library is timed on: the calls its users make, over the range of sizes they make them at.

A case names a call of the public interface (``kind``), the layer it is made on (``shape``, the
kept experts, skipping on or off) and the number of tokens.  Shapes: ``mixtral`` (h 4096, f 14336,
8 experts, top-2) and ``tiny`` (h 128, f 448, 8 experts) are the two configured layers of
``paper_2402_14800_b200.synth``; ``wide`` (h 2048, f 4096, 16 experts) is a generic layer of many
smaller experts for the general top-k call.  Inputs are the seeded synthetic weights and hidden
states that the tests and the benchmark use.

``skip`` runs with beta = the median of w1/w0 over a separate calibration batch, as the paper
calibrates it; without it beta is 0.  ``kept`` = r keeps experts 0 .. r-1.
"""
from __future__ import annotations

import itertools

import numpy as np
import torch

from paper_2402_14800_b200 import binding, synth

DEV = "cuda:0"
SHAPES = {"mixtral": synth.MIXTRAL, "tiny": synth.TINY, "wide": dict(h=2048, f=4096, E=16)}
CAL_TOKENS = 4096      # hidden states beta is calibrated on
TOPK_BETA = 0.1        # share of the selected mass the generalised skipping rule may drop


def listed():
    return [
        # batch-1 decoding on the unpruned layer: one token, two experts, nothing but weight streaming
        dict(name="decode_1", kind="forward", shape="mixtral", tokens=1, kept=8, skip=False, record=False),
        # a handful of concurrent sequences, an odd number of them: most experts touched, few tokens each
        dict(name="decode_9", kind="forward", shape="mixtral", tokens=9, kept=8, skip=False, record=False),
        # a full decode batch on the layer pruned to 4 experts with skipping on, the routing record
        # kept for monitoring (the paper's two methods together)
        dict(name="decode_128_r4_skip", kind="forward", shape="mixtral", tokens=128, kept=4, skip=True, record=True),
        # a chunk of a prompt (or prompts mixed with decoding): more tokens than a decode batch, ragged
        # expert groups of one to two row tiles
        dict(name="chunk_611", kind="forward", shape="mixtral", tokens=611, kept=8, skip=False, record=False),
        # prompt processing of a batch of prompts on the unpruned layer
        dict(name="prefill_8192", kind="forward", shape="mixtral", tokens=8192, kept=8, skip=False, record=False),
        # a model of several layers (RMSNorm, residual) pruned to 6 experts with skipping on, at an
        # ordinary prompt length
        dict(name="stack_2000_r6_skip", kind="stack", shape="mixtral", tokens=2000, kept=6, skip=True, layers=4),
        # the general top-k call with the generalised skipping rule: 16 smaller experts, 4 per token
        dict(name="topk_333_k4", kind="topk", shape="wide", tokens=333, kept=16, skip=True, k=4),
        # the tiny layer of the first configuration: launches and latency are everything
        dict(name="tiny_256", kind="forward", shape="tiny", tokens=256, kept=8, skip=True, record=False),
        # the pruning search on the tiny layer, both subset sizes
        dict(name="search_tiny_256", kind="search", shape="tiny", tokens=256, r4=True),
        # the layer-wise pruning search at full size, subsets of 6 and of 4 in one call: the largest work
        dict(name="search_32768", kind="search", shape="mixtral", tokens=32768, r4=True),
        # calibrating beta on a batch of hidden states of the unpruned layer
        dict(name="calibrate_16384", kind="calibrate", shape="mixtral", tokens=16384),
        # the call on host buffers, end to end: copy in, layer, copy out
        dict(name="host_1500", kind="host", shape="mixtral", tokens=1500, kept=8, skip=False),
    ]


def _size(rng, lo, hi):
    """A whole number from lo .. hi, spread over its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "stack", "topk", "tiny", "search_tiny", "search",
                       "calibrate", "host"])
    kept, skip = rng.choice([8, 8, 6, 4]), rng.random() < 0.5
    if kind == "forward":
        return dict(kind="forward", shape="mixtral", tokens=_size(rng, 2, 32768), kept=kept, skip=skip,
                    record=rng.random() < 0.25)
    if kind == "stack":
        return dict(kind="stack", shape="mixtral", tokens=_size(rng, 1, 4096), kept=kept, skip=skip,
                    layers=rng.randint(2, 4))
    if kind == "topk":
        return dict(kind="topk", shape="wide", tokens=_size(rng, 2, 4096), kept=16, skip=skip, k=rng.randint(2, 6))
    if kind == "tiny":
        return dict(kind="forward", shape="tiny", tokens=_size(rng, 2, 2048), kept=kept, skip=skip, record=False)
    if kind == "search_tiny":
        return dict(kind="search", shape="tiny", tokens=_size(rng, 64, 2048), r4=rng.random() < 0.5)
    if kind == "search":
        return dict(kind="search", shape="mixtral", tokens=_size(rng, 512, 32768), r4=rng.random() < 0.5)
    if kind == "calibrate":
        return dict(kind="calibrate", shape="mixtral", tokens=_size(rng, 128, 32768))
    return dict(kind="host", shape="mixtral", tokens=_size(rng, 2, 8192), kept=kept, skip=skip)


def _layer(shape, kept, seed):
    s = SHAPES[shape]
    W = synth.make_layer_weights(s["h"], s["f"], s["E"], seed=seed, device=DEV)
    return binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2, (1 << kept) - 1)


def _beta(layer, seed):
    return layer.calibrate_beta(synth.make_tokens(CAL_TOKENS, layer.h, seed=seed, device=DEV))


def prepare(case, seed):
    kind, T = case["kind"], case["tokens"]
    kept = case.get("kept", SHAPES[case["shape"]]["E"])
    base = 1000 * seed
    state = dict(case=case)
    n_layers = case.get("layers", 1)
    state["layers"] = [_layer(case["shape"], kept, base + i) for i in range(n_layers)]
    layer = state["layer"] = state["layers"][0]
    x = state["x"] = synth.make_tokens(T, layer.h, seed=base + 500, device=DEV)
    if kind == "topk":
        state["beta"] = TOPK_BETA if case["skip"] else 0.0
    elif case.get("skip"):
        state["betas"] = [_beta(l, base + 600 + i) for i, l in enumerate(state["layers"])]
        state["beta"] = state["betas"][0]
    else:
        state["betas"], state["beta"] = None, 0.0
    if kind in ("forward", "stack", "host"):
        layer.reserve(T)   # scratch grown at start-up, as a serving loop does
    if kind in ("forward", "stack", "topk"):
        state["y"] = torch.empty_like(x)
    if case.get("record"):
        state["stats"] = binding.RoutingStats(T, layer.E, DEV)
    if kind == "host":
        state["x_host"] = x.cpu().pin_memory()
        state["y_host"] = torch.empty_like(state["x_host"]).pin_memory()
    return state


def run(state):
    case, layer = state["case"], state["layer"]
    kind = case["kind"]
    if kind == "forward":
        stats = state.get("stats")
        layer.forward(state["x"], state["beta"], y=state["y"], stats=stats)
        if stats is None:
            return state["y"]
        return {"y": state["y"], "idx": stats.idx, "wn": stats.wn, "skipped": stats.skipped, "count": stats.count}
    if kind == "stack":
        return binding.stack_forward(state["layers"], state["x"], betas=state["betas"], y=state["y"])
    if kind == "topk":
        y, idx, wn, n_active = layer.forward_topk(state["x"], case["k"], state["beta"], y=state["y"], record=True)
        return {"y": y, "idx": idx, "wn": wn, "n_active": n_active}
    if kind == "search":
        found = layer.prune_search_multi(state["x"], [6, 4] if case["r4"] else [6])
        return {"losses": [np.array(losses, np.float32) for losses, _ in found],
                "best": np.array([best for _, best in found], np.int64)}
    if kind == "calibrate":
        return layer.calibrate_beta(state["x"])
    return layer.forward_host(state["x_host"], state["beta"], state["y_host"])


def _touched(E, pairs):
    """Experts that `pairs` independent, equally likely choices of E are expected to touch."""
    return E * (1.0 - (1.0 - 1.0 / E) ** pairs)


def work(case):
    s = SHAPES[case["shape"]]
    h, f, E = s["h"], s["f"], s["E"]
    kind, T, L = case["kind"], case["tokens"], case.get("layers", 1)
    kept = case.get("kept", E)
    rows = 2.0 * h * T                      # bytes of the hidden states, once
    if kind == "calibrate":
        return {"bytes": rows + 2.0 * E * h, "flops": 2.0 * E * h * T}
    if kind == "search":
        # a subset of r experts always routes a token to two of its E - r + 2 top-ranked ones
        pairs = T * (E - (4 if case["r4"] else 6) + 2)
        touched = E
    elif kind == "topk":
        # the rule drops at most a tenth of the mass: between three and four experts of four stay
        pairs = T * case["k"] * (0.85 if case["skip"] else 1.0)
        touched = _touched(kept, pairs)
    else:
        pairs = T * (1.5 if case["skip"] else 2.0)   # the median beta skips the second expert of half the tokens
        touched = max(_touched(kept, pairs), 2.0 if not case["skip"] else 1.0)
    out = 0.0 if kind == "search" else rows
    return {"bytes": L * (touched * 6.0 * h * f + 2.0 * kept * h) + rows + out, "flops": L * pairs * 6.0 * h * f}


def tolerance(case):
    """About four times what two of the path's own kernels with different orders of their sums
    (matrix-vector / weight-major / token-major / CUDA-core) differ by on the same inputs."""
    kind = case["kind"]
    if kind == "calibrate":
        return {"rel": 1e-5}                 # a ratio of softmax numerators, fp32 logits
    if kind == "search":
        return {"rel": 1e-5, "max": 1e-4}    # fp32 sums of squares (seen: 6.9e-7)
    if kind == "stack":
        return {"rel": 1e-2, "max": 0.085}   # bf16 states through several layers (seen: 2.7e-3, 0.021)
    return {"rel": 4e-3, "max": 0.032}       # bf16 outputs (seen: 8.4e-4, 0.0078 = one bf16 step)


def _exact_weights(shape, seed):
    s = SHAPES[shape]
    return synth.make_layer_weights(s["h"], s["f"], s["E"], seed=seed, device=DEV)


def _exact_logits(W, x, kept):
    """Logits [T][E] over the first `kept` experts; the others cannot be chosen."""
    logits = x.double() @ W.W_gate.double().T
    logits[:, kept:] = -torch.inf
    return logits


def _exact_ranked(W, x, kept):
    """The logits in descending order and their experts, ties to the lower index."""
    return _exact_logits(W, x, kept).sort(dim=1, descending=True, stable=True)


def _exact_expert(W, e, x):
    x = x.double()
    act = torch.nn.functional.silu(x @ W.W1[e].double().T) * (x @ W.W3[e].double().T)
    return act @ W.W2[e].double().T


def _exact_ratio_median(W, x, kept):
    ranked, _ = _exact_ranked(W, x, kept)
    ratio = torch.exp(ranked[:, 1] - ranked[:, 0]).sort().values
    T = ratio.numel()
    return float((ratio[(T - 1) // 2] + ratio[T // 2]) / 2)


def _exact_mix(W, x, idx, wn):
    """sum_m wn[:, m] E_idx[:, m](x); an expert of weight 0 is not run."""
    z = torch.zeros(x.shape, dtype=torch.float64, device=x.device)
    for e in range(W.E):
        t, m = torch.nonzero((idx == e) & (wn > 0), as_tuple=True)
        if t.numel():
            z[t] += wn[t, m, None] * _exact_expert(W, e, x[t])   # a token has an expert once
    return z


def _exact_top2(W, x, kept, beta):
    ranked, order = _exact_ranked(W, x, kept)
    p = torch.exp(ranked[:, :2] - ranked[:, :1])
    p[:, 1] *= ~(p[:, 1] < beta)
    return order[:, :2], p / p.sum(1, keepdim=True)


def _exact_topk(W, x, k, beta):
    ranked, order = _exact_ranked(W, x, W.E)
    p = torch.exp(ranked[:, :k] - ranked[:, :1])
    tail = p.flip(1).cumsum(1).flip(1) - p                        # mass after rank m
    n_active = (tail > beta * p.sum(1, keepdim=True)).sum(1) + 1   # the first i whose tail is small enough
    p = p * (torch.arange(k, device=p.device)[None] < n_active[:, None])
    return order[:, :k], p / p.sum(1, keepdim=True)


def _exact_search(W, x, sizes):
    logits = _exact_logits(W, x, W.E)
    Y = torch.stack([_exact_expert(W, e, x) for e in range(W.E)], dim=1)
    rows = torch.arange(x.shape[0], device=x.device)

    def mixed(subset):
        ranked, order = logits[:, subset].sort(dim=1, descending=True, stable=True)
        p = torch.softmax(ranked[:, :2], dim=1)
        order = torch.tensor(subset, device=x.device)[order]
        return p[:, :1] * Y[rows, order[:, 0]] + p[:, 1:] * Y[rows, order[:, 1]]

    full = mixed(list(range(W.E)))
    return [np.array([float((mixed(list(c)) - full).norm()) for c in itertools.combinations(range(W.E), r)])
            for r in sizes]


def exact(case, seed):
    """What ``run`` returns, computed in 64 bits from the same inputs without any intermediate rounding;
    None for whole-number outputs."""
    kind, T, base = case["kind"], case["tokens"], 1000 * seed
    kept = case.get("kept", SHAPES[case["shape"]]["E"])
    W = _exact_weights(case["shape"], base)
    x = synth.make_tokens(T, W.h, seed=base + 500, device=DEV)

    def beta(W, i=0):
        if not case.get("skip"):
            return 0.0
        return _exact_ratio_median(W, synth.make_tokens(CAL_TOKENS, W.h, seed=base + 600 + i, device=DEV), kept)

    if kind == "calibrate":
        return _exact_ratio_median(W, x, kept)
    if kind == "search":
        return {"losses": _exact_search(W, x, [6, 4] if case["r4"] else [6]), "best": None}
    if kind == "topk":
        idx, wn = _exact_topk(W, x, case["k"], TOPK_BETA if case["skip"] else 0.0)
        return {"y": _exact_mix(W, x, idx, wn), "idx": None, "wn": wn, "n_active": None}
    if kind == "stack":
        state = x.double()
        for i in range(case["layers"]):
            W = W if i == 0 else _exact_weights(case["shape"], base + i)
            xn = state * torch.rsqrt(state.square().mean(1, keepdim=True) + 1e-5)
            state = state + _exact_mix(W, xn, *_exact_top2(W, xn, kept, beta(W, i)))
        return state
    idx, wn = _exact_top2(W, x, kept, beta(W))
    y = _exact_mix(W, x, idx, wn)
    if case.get("record"):
        return {"y": y, "idx": None, "wn": wn, "skipped": None, "count": None}
    return y.cpu() if kind == "host" else y
