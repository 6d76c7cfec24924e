"""The work that users of this library have it do, as cases that can be timed: decode steps and prefills through
one MoTE layer or a stack of them, the host-buffer call, and the offline weight quantizer.

Shapes are those of workloads/synth.py (FFN sizes of the 0.5B / 1.5B / 3B models, 4 to 16 routed experts, top-1 with
the probability of Eq. 3 or top-2 renormalised, bf16 / INT8 / INT4 shared expert) and, for drawn cases, other widths that
are multiples of 128.  Weights are N(0, 0.02^2) and tokens N(0, 1), with 1 % outlier channels where a case says so.  Stacks
hold 2 to 8 of a model's 24 to 36 layers: more than the L2 cache, and quick to draw; what enters them is a residual stream
sixteen times as large as one layer's update, as in the middle of a model.
"""
import math

import torch

import paper_2506_14435_b200 as mote

MODELS = {                                  # d, f
    "tiny": (256, 512),
    "0.5B": (896, 4864),
    "1.5B": (1536, 8960),
    "3B": (2048, 11008),
}


def _layer(name, model, T, E, k, *, kind="layer", layers=1, bits=16, norm=True, outliers=False, bias="none", residual=True):
    d, f = MODELS[model]
    return dict(name=name, kind=kind, d=d, f=f, E=E, k=k, T=T, layers=layers, shared_bits=bits, norm_topk=norm,
                outliers=outliers, bias=bias, residual=residual)


def listed():
    return [
        # smallest call: a toy layer on 64 tokens, as in unit tests and demos; launches are all there is to it
        _layer("tiny-64", "tiny", 64, 4, 2, residual=False),
        # one user's decode step through consecutive layers of the 3B shape (norm, layer, residual)
        _layer("stack-decode-1", "3B", 1, 16, 2, kind="stack", layers=8),
        # the same with the paper's own routing (4 experts, top-1, gate = P(x)_i) and its smallest memory point
        _layer("stack-decode-1-int4", "3B", 1, 4, 1, kind="stack", layers=8, bits=4, norm=False),
        # a small decode batch, unevenly loaded experts
        _layer("decode-8", "1.5B", 8, 8, 2, bias="zipf"),
        # a decode batch of a busy server: nearly every expert is touched
        _layer("stack-decode-32", "3B", 32, 16, 2, kind="stack", layers=8),
        # a large decode batch or a short prompt
        _layer("decode-64", "1.5B", 64, 8, 2, bias="zipf"),
        # a prompt of odd length, INT8 shared expert, the paper's routing
        _layer("prompt-333-int8", "1.5B", 333, 4, 1, bits=8, norm=False),
        # prefill of an image and its text, small model
        _layer("prefill-4096", "0.5B", 4096, 4, 2, outliers=True),
        # the largest call: a long batched prefill with imbalanced experts
        _layer("prefill-8192", "3B", 8192, 16, 2, outliers=True, bias="normal"),
        # a training-length sequence through consecutive layers
        _layer("stack-prefill-2048", "3B", 2048, 16, 2, kind="stack", layers=4),
        # a long prefill whose tokens arrive in, and leave to, pinned host memory
        _layer("host-prefill-8192", "3B", 8192, 16, 2, kind="host", outliers=True, bias="normal", residual=False),
        # up-cycling a checkpoint: the three matrices of one expert, fp32 master weights to 2-bit codes
        dict(name="ternarize-expert", kind="ternarize", d=2048, f=11008, dtype="float32"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    d, f = rng.choice(list(MODELS.values())) if rng.random() < 0.6 else (128 * rng.randint(2, 16), 128 * rng.randint(4, 86))
    kind = rng.choice(["layer", "layer", "layer", "stack", "stack", "host", "ternarize"])
    if kind == "ternarize":
        return dict(kind=kind, d=d, f=f, dtype=rng.choice(["float32", "bfloat16"]))
    E = rng.choice([4, 4, 8, 16])
    k = rng.choice([1, 2])
    T = _log_int(rng, 1, 2048 if kind == "stack" else 8192)
    layers = 1
    if kind == "stack":
        layers = rng.randint(2, 8 if T <= 64 else 4)
    return dict(kind=kind, d=d, f=f, E=E, k=k, T=T, layers=layers, shared_bits=rng.choice([16, 16, 8, 4]),
                norm_topk=rng.choice([True, False]), outliers=rng.choice([True, False]),
                bias=rng.choice(["none", "zipf", "normal"]), residual=kind != "host" and rng.choice([True, False]))


def _generator(seed, *ids):
    g = torch.Generator(device="cuda")
    n = seed
    for i in ids:
        n = n * 1009 + i
    g.manual_seed(n & (2 ** 62 - 1))
    return g


def _make_layer(c, seed, index):
    """One layer's weights, drawn on the device and quantized the way a loader does it, once."""
    d, f, E = c["d"], c["f"], c["E"]
    ids = dict(gate=0, up=1, down=2, sh_gate=3, sh_up=4, sh_down=5, Wr=6, bias=7)

    def make(name, expert=0):
        g = _generator(seed, index, expert, ids[name])
        if name == "bias":
            if c["bias"] == "zipf":                         # expert load ~ (e + 1)^-1.1
                p = torch.arange(1, E + 1, device="cuda", dtype=torch.float64) ** -1.1
                return torch.log(p / p.sum()).float()
            return torch.randn(E, generator=g, device="cuda") * 0.5 if c["bias"] == "normal" else None
        shape = (E, d) if name == "Wr" else (d, f) if name in ("down", "sh_down") else (f, d)
        w = torch.randn(shape, generator=g, device="cuda").mul_(0.02)
        if name == "Wr":
            return w.bfloat16().float()
        return w.bfloat16() if name.startswith("sh_") else w

    layer = mote.MoteLayer.from_device_draws(d, f, E, c["k"], int(c["norm_topk"]), make)
    return layer if c["shared_bits"] == 16 else layer.quantize_shared(c["shared_bits"])


def _tokens(c, seed):
    g = _generator(seed, 8)
    x = torch.randn(c["T"], c["d"], generator=g, device="cuda")
    if c["outliers"]:
        x[:, torch.randperm(c["d"], generator=g, device="cuda")[:max(1, round(0.01 * c["d"]))]] *= 20.0
    if c["kind"] == "stack":
        x *= 16.0
    return x.bfloat16()


def prepare(case, seed):
    c = case
    if c["kind"] == "ternarize":
        dtype = getattr(torch, c["dtype"])
        mats = []
        for i, shape in enumerate(((c["f"], c["d"]), (c["f"], c["d"]), (c["d"], c["f"]))):
            mats.append((torch.randn(shape, generator=_generator(seed, i), device="cuda") * 0.02).to(dtype))
        return dict(kind="ternarize", mats=mats)
    layers = [_make_layer(c, seed, i) for i in range(c["layers"])]
    x = _tokens(c, seed)
    state = dict(kind=c["kind"], layer=layers[0])
    if c["kind"] == "host":
        state["x"] = x.cpu().pin_memory()
        state["out"] = torch.empty_like(state["x"]).pin_memory()
    else:
        state["x"] = x
        if c["kind"] == "stack":
            state["stack"] = mote.MoteStack(layers)
        elif c["residual"]:                                 # the residual stream that x is the norm of
            state["residual"] = torch.randn(c["T"], c["d"], generator=_generator(seed, 9), device="cuda").bfloat16()
    return state


def run(state):
    if state["kind"] == "ternarize":
        return [mote.mote_ternarize_pack(w) for w in state["mats"]]
    if state["kind"] == "host":
        return mote.mote_moe_forward_host(state["layer"], state["x"], state["out"])
    if state["kind"] == "stack":
        return mote.mote_stack_forward(state["stack"], state["x"])
    return mote.mote_moe_forward(state["layer"], state["x"], residual=state.get("residual"))


def work(case):
    c = case
    mat = c["d"] * c["f"]
    if c["kind"] == "ternarize":
        return dict(bytes=3.0 * mat * ((4 if c["dtype"] == "float32" else 2) + 0.25), flops=0.0)
    touched = c["E"] * (1.0 - (1.0 - c["k"] / c["E"]) ** c["T"])        # expected experts that receive tokens
    weights = 3.0 * mat * (c["shared_bits"] / 8.0 + touched / 4.0) + 4.0 * c["E"] * c["d"]
    tokens = 2.0 * c["T"] * c["d"] * (3 if c["residual"] and c["kind"] == "layer" else 2)
    return dict(bytes=c["layers"] * weights + tokens, flops=c["layers"] * 6.0 * mat * c["T"] * (1 + c["k"]))


def tolerance(case):
    """Codes and scales of the quantizer are fixed bit for bit.  The layer's integer stages are too; its bf16 matmuls and
    the combine leave the summation order open.  Measured: the three implementations of the layer (CUDA cores, tcgen05, weight
    stream) against one another, over the listed cases, drawn ones and several seeds.  One layer: rel at most 8.6e-4, max one unit
    in the last place of bf16 (7.8e-3).  A stack carries a rounding that fell the other way on into the next layer's int8 codes:
    rel at most 3.4e-3 over 8 layers, 1.5e-3 over 4; max 0.05.  Stated: four times that."""
    if case["kind"] == "ternarize":
        return "exact"
    if case["kind"] == "stack":
        return dict(rel=max(3.5e-3, 1.7e-3 * case["layers"]), max=0.2)
    return dict(rel=3.5e-3, max=3.2e-2)
