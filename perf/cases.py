"""The calls this layer is used for, as measurable cases: inputs, one pass through the public entry points, the work
a pass cannot do without, and how far two correct implementations may differ.

The layer is the MoE FFN of a reranker.  Scoring runs the forward-only call on anything from one query-passage pair
(about 256 tokens) to large batches; training runs forward + backward on 1000 to 65536 tokens per GPU; a window of
micro-batches accumulates fp32 gradients; adapters are trained on frozen experts.  Shapes are those of the
repository's configurations (`paper_2608_00916_b200.synth.CONFIGS`)."""
import math

import torch

from paper_2608_00916_b200.binding import FLAG_ROUTER_FP32, MoELayer
from paper_2608_00916_b200.synth import CONFIGS, GAP

QWEN = {"d": 2048, "E": 128, "k": 8, "f": 768, "x_std": 1.0}
D_AUX = 0.01  # coefficient of the load-balance loss


def _case(name, mode, T, zipf=0.0, router_fp32=False, rank=0, **shape):
    return {"name": name, "mode": mode, "T": T, **(shape or QWEN), "zipf": zipf, "router_fp32": router_fp32, "rank": rank}


def _config(name):
    s, _, x_std, _ = CONFIGS[name]
    return {"d": s.d, "E": s.E, "k": s.k, "f": s.f, "x_std": x_std}


def listed():
    return [
        # scoring: one query-passage pair of an odd length, one query with eight passages of 256 tokens, a full batch
        _case("score_pair", "score", 241),
        _case("score_query", "score", 2048),
        _case("score_batch", "score", 16384),
        # the smallest training step (unit tests, debugging runs): launches and host work are all there is
        _case("train_tiny", "train", 256, **_config("tiny")),
        # training steps of growing micro-batches, ragged token counts among them; 16384 = 8 queries x 8 passages x 256
        _case("train_1000", "train", 1000),
        _case("train_4096", "train", 4096),
        _case("train_8191", "train", 8191),
        _case("train_16384", "train", 16384),
        # the same batch when the router has collapsed onto a few experts (Zipf 1.2 loads, some experts empty)
        _case("train_skewed", "train", 16384, zipf=1.1),
        # few wide experts
        _case("train_coarse", "train", 16384, **_config("coarse")),
        # one micro-batch of an accumulation window: fp32 main gradients, router weight kept in fp32
        _case("accumulate_16384", "accumulate", 16384, router_fp32=True),
        # adapter training: rank 16 on frozen experts
        _case("lora_8192", "lora", 8192, rank=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["score", "score", "train", "train", "train", "skewed", "coarse", "small", "accumulate", "lora"])
    if kind == "score":
        c = _case("", "score", _log_int(rng, 128, 32768))
    elif kind == "train":
        c = _case("", "train", _log_int(rng, 512, 65536))
    elif kind == "skewed":
        c = _case("", rng.choice(["train", "score"]), _log_int(rng, 2048, 32768), zipf=round(rng.uniform(0.3, 1.3), 2))
    elif kind == "coarse":
        c = _case("", rng.choice(["train", "score"]), _log_int(rng, 512, 16383), **_config("coarse"))
    elif kind == "small":
        c = _case("", "train", _log_int(rng, 16, 2048), d=64 * rng.randint(2, 12), E=8 * rng.randint(1, 8), k=rng.randint(1, 4),
                  f=64 * rng.randint(2, 12), x_std=1.0)
    elif kind == "accumulate":
        c = _case("", "accumulate", _log_int(rng, 1000, 32768), router_fp32=rng.random() < 0.5)
    else:
        c = _case("", "lora", _log_int(rng, 1000, 32768), rank=8 * rng.randint(1, 8))
    del c["name"]
    return c


def _normal(g, shape, std, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)


def _tokens(g, T, d, std, W_r, b_r, k):
    """Hidden states whose k + 1 largest logits are at least GAP apart: which experts a token takes must not hang on
    the rounding of a sum, or two correct implementations could not be compared."""
    x = _normal(g, (T, d), std)
    W = W_r.double()
    bad = torch.arange(T, device="cuda")
    for _ in range(64):
        l = x[bad].double() @ W
        if b_r is not None:
            l += b_r.double()
        top = l.topk(min(k + 1, l.shape[1]), dim=1).values
        bad = bad[((top[:, :-1] - top[:, 1:]) < GAP).any(dim=1)]
        if bad.numel() == 0:
            return x
        x[bad] = _normal(g, (bad.numel(), d), std)
    raise RuntimeError("no well separated tokens found")


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    mode, T, d, E, k, f = (case[n] for n in ("mode", "T", "d", "E", "k", "f"))
    flags = FLAG_ROUTER_FP32 if case["router_fp32"] else 0
    s = {"mode": mode, "layer": MoELayer(d, E, f, k, flags)}
    s["W_r"] = _normal(g, (d, E), 0.02, torch.float32 if flags else torch.bfloat16)
    s["W_gate"], s["W_up"], s["W_down"] = (_normal(g, shape, 0.02) for shape in ((E, d, f), (E, d, f), (E, f, d)))
    s["b_r"] = None
    if case["zipf"] > 0:
        # a bias under which the experts' loads follow a Zipf law of exponent 1.2 in a random order
        sigma = 0.02 * case["x_std"] * math.sqrt(d)
        order = torch.randperm(E, generator=g, device="cuda")
        s["b_r"] = (-1.2 * case["zipf"] * sigma) * torch.log(1.0 + order.float())
    s["x"] = _tokens(g, T, d, case["x_std"], s["W_r"], s["b_r"], k)
    if mode != "score":
        s["dy"] = _normal(g, (T, d), 1.0)
    if mode == "train":  # gradient buffers live as long as the weights
        s["grads"] = {"dW_r": torch.zeros(d, E, device="cuda"), **{"d" + n: torch.zeros_like(s[n]) for n in ("W_gate", "W_up", "W_down")}}
    elif mode == "accumulate":  # the window's fp32 gradients, some micro-batches in
        s["acc"] = {"d" + n: _normal(g, tuple(s[n].shape), 1.0, torch.float32) for n in ("W_r", "W_gate", "W_up", "W_down")}
    elif mode == "lora":
        r = case["rank"]
        shapes = {"A1": (E, d, r), "B1_gate": (E, r, f), "B1_up": (E, r, f), "A2": (E, f, r), "B2": (E, r, d)}
        s["adapters"] = {n: _normal(g, shape, 0.05) for n, shape in shapes.items()}
        s["scale"] = 2.0
    return s


def run(state):
    s = state
    layer, weights = s["layer"], (s["W_r"], s["W_gate"], s["W_up"], s["W_down"])
    if s["mode"] == "score":
        return layer.forward(s["x"], *weights, b_r=s["b_r"], inference=True)
    if s["mode"] == "lora":
        out = layer.lora_forward(s["x"], *weights, s["adapters"], s["scale"], b_r=s["b_r"])
        return [out, layer.lora_backward(s["dy"], D_AUX)]
    out = layer.forward(s["x"], *weights, b_r=s["b_r"])
    if s["mode"] == "accumulate":
        return [out, layer.backward_accumulate(s["dy"], D_AUX, s["acc"]), s["acc"]]
    return [out, layer.backward(s["dy"], D_AUX, grads=s["grads"])]


def work(case):
    mode, T, d, E, k, f, r = (case[n] for n in ("mode", "T", "d", "E", "k", "f", "rank"))
    R, router = T * k, d * E * (4 if case["router_fp32"] else 2)
    weights = 3 * E * d * f * 2 + router
    forward = weights + 4 * T * d + 12 * R + 4 * E  # x in, y out, indices, gates, order, counts
    flops = 6 * R * d * f + 2 * T * d * E
    if mode == "score":
        return {"bytes": forward, "flops": flops}
    backward = weights + 6 * T * d + 4 * d * E  # x and dy in, dx and the router gradient out
    flops += 4 * T * d * E
    if mode == "lora":
        adapters = 2 * E * r * (3 * d + 3 * f)
        return {"bytes": forward + backward + 3 * adapters, "flops": flops + 6 * R * d * f + 6 * R * r * (2 * d + 3 * f)}
    grads = 3 * E * d * f * (8 if mode == "accumulate" else 2)  # accumulation reads and writes fp32
    return {"bytes": forward + backward + grads, "flops": flops + 12 * R * d * f}


def exact(case, seed):
    """What run() returns for these inputs, by the layer's definition in float64 (plain torch, one expert at a time)."""
    s = prepare(case, seed)
    mode, T, E, k = (case[n] for n in ("mode", "T", "E", "k"))
    x, W_r = s["x"].double(), s["W_r"].double()
    logits = x @ W_r if s["b_r"] is None else x @ W_r + s["b_r"].double()
    p = logits.softmax(dim=1)
    idx = logits.topk(k, dim=1).indices  # no ties: _tokens keeps the logits apart
    gates = p.gather(1, idx)
    gates = gates / gates.sum(dim=1, keepdim=True)
    counts = torch.bincount(idx.reshape(-1), minlength=E)
    perm = torch.sort(idx.reshape(-1), stable=True).indices
    share = counts.double() / (T * k)
    aux = (E * (share * p.mean(dim=0)).sum()).reshape(1)
    dy = s["dy"].double() if mode != "score" else None
    y, dx = torch.zeros_like(x), torch.zeros_like(x)
    dg = torch.zeros_like(gates)
    grads = {}

    def add(name, e, value):  # gradients of expert e
        if name not in grads:
            grads[name] = torch.zeros((E, *value.shape), dtype=torch.float64, device="cuda")
        grads[name][e] = value

    first = 0
    for e, n in enumerate(counts.tolist()):
        rows = perm[first:first + n]
        first += n
        tok, slot = rows // k, rows % k
        Wg, Wu, Wd = (s[w][e].double() for w in ("W_gate", "W_up", "W_down"))
        if mode == "lora":
            c = s["scale"]
            A1, B1g, B1u, A2, B2 = (s["adapters"][w][e].double() for w in ("A1", "B1_gate", "B1_up", "A2", "B2"))
            Wg, Wu, Wd = Wg + c * A1 @ B1g, Wu + c * A1 @ B1u, Wd + c * A2 @ B2
        xe, g = x[tok], gates[tok, slot][:, None]
        hg, hu = xe @ Wg, xe @ Wu
        sig = torch.sigmoid(hg)
        act = hg * sig * hu
        o = act @ Wd
        y.index_add_(0, tok, g * o)
        if mode == "score":
            continue
        dye = dy[tok]
        dg[tok, slot] = (dye * o).sum(dim=1)
        da = g * (dye @ Wd.T)
        dhg, dhu = da * hu * sig * (1.0 + hg * (1.0 - sig)), da * hg * sig
        dx.index_add_(0, tok, dhg @ Wg.T + dhu @ Wu.T)
        dWg, dWu, dWd = xe.T @ dhg, xe.T @ dhu, act.T @ (g * dye)
        if mode == "lora":
            for name, v in (("dA1", dWg @ B1g.T + dWu @ B1u.T), ("dB1_gate", A1.T @ dWg), ("dB1_up", A1.T @ dWu), ("dA2", dWd @ B2.T), ("dB2", A2.T @ dWd)):
                add(name, e, c * v)
        else:
            for name, v in (("dW_gate", dWg), ("dW_up", dWu), ("dW_down", dWd)):
                add(name, e, v)
    out = {"y": y, "idx": idx.int(), "gates": gates, "counts": counts.int(), "aux": aux}
    if mode != "lora":
        out.update(perm=perm.int(), logits=None)
    if mode == "score":
        return out
    # gates are a softmax over the selected logits; the loss term reaches the logits through the mean probabilities
    dl = torch.zeros_like(p).scatter_(1, idx, gates * (dg - (gates * dg).sum(dim=1, keepdim=True)))
    dp = (D_AUX * E / T) * share
    dl += p * (dp - (p * dp).sum(dim=1, keepdim=True))
    dx += dl @ W_r.T
    dW_r = x.T @ dl
    if mode == "accumulate":
        return [out, dx, {n: s["acc"][n].double() + (dW_r if n == "dW_r" else grads[n]) for n in s["acc"]}]
    grads.update(dx=dx, dW_r=dW_r)
    if mode == "train":
        grads["db_r"] = None
    return [out, grads]


def tolerance(case):
    # bf16 intermediates (pre-activations, activation, expert outputs, their gradients) and bf16 results.  Measured
    # against the same layer in float64: 2.3e-3 to 3.5e-3 (adapters, whose products are rounded once more: 3.3e-3 to
    # 4.4e-3), single values up to 0.047 of the root mean square, up to 0.12 where a skewed router leaves most of a
    # gradient nearly zero.  Which experts a token takes is exact (see _tokens).
    return {"rel": 1.5e-2 if case["mode"] == "lora" else 1e-2, "max": 0.4 if case["zipf"] > 0 else 0.2, "differ": 0.0}
