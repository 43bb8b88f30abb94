"""What the framework's users have it do, as cases whose time and results can be measured.

A case is one pass through the public entry points of `paper_2609_33977_gb300.groupsparse`:

  linear   y = x (W (.) M)^T for one packed layer, one `linear` call (a model that runs layer by layer);
  block    the projections of a Transformer block that share a token count, one `linear_batched_into` call;
  export   selector logits -> mask -> packed layer -> dense check copy (deploying a learned mask);
  sample   one Gumbel-Sigmoid sample of a whole stack's selectors (the start of a mask-training step);
  train    one mask-training step of one layer: sample, pack, forward, straight-through backward.

Weights, activations and logits are drawn as the workload module describes them (W ~ N(0, 0.02^2),
x ~ N(0, 1), optionally 1 % outlier channels x20, per-layer densities spread around a global one).
"""
from __future__ import annotations

import math

import torch

from paper_2609_33977_gb300 import groupsparse as gs
from paper_2609_33977_gb300 import workload as wk

BLOCKS = {"llama2-7b": wk.LLAMA2_7B_BLOCK, "llama2-13b": wk.LLAMA2_13B_BLOCK, "qwen2.5-7b": wk.QWEN25_7B_BLOCK}
GROUPS = ((1, 256), (1, 128), (16, 16), (32, 32), (64, 64), (128, 128))
TAU = 0.4   # temperature of the relaxation


def listed():
    return [
        # the smallest call: one small layer for a few tokens, where latency is all
        {"name": "linear_1024_t8", "kind": "linear", "layers": "1024x1024", "g_out": 1, "g_in": 256, "T": 8,
         "density": 0.5, "spread": 0.0, "outliers": False},
        # generating one token at a time with a 7B model, one call per block
        {"name": "block7b_t1", "kind": "block", "layers": "llama2-7b", "g_out": 1, "g_in": 256, "T": 1,
         "density": 0.5, "spread": 0.2, "outliers": False},
        # the same for 16 concurrent sequences of a 13B model
        {"name": "block13b_t16", "kind": "block", "layers": "llama2-13b", "g_out": 1, "g_in": 256, "T": 16,
         "density": 0.5, "spread": 0.3, "outliers": False},
        # the finer row groups of the granularity study, a handful of sequences
        {"name": "block7b_1x128_t4", "kind": "block", "layers": "llama2-7b", "g_out": 1, "g_in": 128, "T": 4,
         "density": 0.5, "spread": 0.2, "outliers": False},
        # square groups of the granularity study, decoding 16 sequences
        {"name": "qwen_32x32_t16", "kind": "block", "layers": "qwen2.5-7b", "g_out": 32, "g_in": 32, "T": 16,
         "density": 0.5, "spread": 0.2, "outliers": False},
        # a short prompt (or a large decode batch) through a 13B block
        {"name": "block13b_t128", "kind": "block", "layers": "llama2-13b", "g_out": 1, "g_in": 256, "T": 128,
         "density": 0.5, "spread": 0.3, "outliers": False},
        # a long prompt through a 7B block, activations with outlier channels
        {"name": "block7b_t2048", "kind": "block", "layers": "llama2-7b", "g_out": 1, "g_in": 256, "T": 2048,
         "density": 0.5, "spread": 0.3, "outliers": True},
        # one layer at a time, a prompt of no round length, finer groups, denser keep ratio
        {"name": "linear_up_1x128_t777", "kind": "linear", "layers": "18944x3584", "g_out": 1, "g_in": 128, "T": 777,
         "density": 0.7, "spread": 0.0, "outliers": False},
        # prompt processing with square groups
        {"name": "block7b_64x64_t512", "kind": "block", "layers": "llama2-7b", "g_out": 64, "g_in": 64, "T": 512,
         "density": 0.5, "spread": 0.2, "outliers": False},
        # deploying a learned mask: the down projection of a 13B block
        {"name": "export_13b_down", "kind": "export", "layers": "5120x13824", "g_out": 1, "g_in": 256, "T": 0,
         "density": 0.5, "spread": 0.0, "outliers": False},
        # drawing every selector of a 7B stack (32 blocks) for one training step
        {"name": "sample_7b_stack", "kind": "sample", "layers": "25296896", "g_out": 1, "g_in": 256, "T": 0,
         "density": 0.5, "spread": 0.0, "outliers": False},
        # one mask-training step of a 7B block's gate projection over a 2048-token sequence
        {"name": "train_7b_gate_t2048", "kind": "train", "layers": "11008x4096", "g_out": 1, "g_in": 256, "T": 2048,
         "density": 0.5, "spread": 0.0, "outliers": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _seconds(case):
    """A rough lower bound of a pass, for keeping drawn cases below the largest listed one."""
    w = work(case)
    return max(w["bytes"] / 6.0e12, w["flops"] / 7.0e14)


def draw(rng):
    """One more case: any kind, any group shape, sizes over the listed cases' range."""
    most = max(_seconds(c) for c in listed())
    while True:
        kind = rng.choice(["linear", "linear", "block", "block", "export", "sample", "train"])
        case = {"kind": kind, "g_out": 1, "g_in": 256, "T": 0, "density": round(rng.uniform(0.3, 0.7), 3),
                "spread": 0.0, "outliers": False}
        if kind == "sample":
            case["layers"] = str(_log_int(rng, 65536, 49561600))
        else:
            row_groups = rng.random() < 0.6
            g_out, g_in = rng.choice(GROUPS[:2] if row_groups else GROUPS[2:])
            case.update(g_out=g_out, g_in=g_in)
            if kind == "block" and rng.random() < 0.5:
                case["layers"] = rng.choice(sorted(BLOCKS))
                case["spread"] = 0.2
            else:
                n = rng.randint(2, 6) if kind == "block" else 1
                shapes = []
                for _ in range(n):
                    out = max(1, _log_int(rng, 512, 20000) // g_out) * g_out   # 1 x n groups: any row count
                    inp = max(1, _log_int(rng, 1024, 16000) // g_in) * g_in
                    shapes.append("%dx%d" % (out, inp))
                case["layers"] = " ".join(shapes)
            if kind in ("linear", "block"):
                case["T"] = _log_int(rng, 1, 2048)
                case["outliers"] = rng.random() < 0.25
            elif kind == "train":
                case["T"] = _log_int(rng, 128, 2048)
        if kind == "train":   # its tokens are rows of 16-byte aligned bf16 tensors in the layer's own GEMMs
            out, inp = _shapes(case)[0]
            case["layers"] = "%dx%d" % (max(1, out // 128) * 128, max(1, inp // 256) * 256)
        if _seconds(case) <= most:
            return case


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _shapes(case):
    if case["layers"] in BLOCKS:
        return [(o, i) for _, o, i in BLOCKS[case["layers"]]]
    return [tuple(map(int, s.split("x"))) for s in case["layers"].split()]


def _densities(case, n):
    """Per-layer densities around the case's: evenly spaced, from the two ends inwards."""
    if n == 1:
        return [case["density"]]
    rank = [i // 2 if i % 2 == 0 else n - 1 - i // 2 for i in range(n)]
    return [case["density"] + case["spread"] * (2.0 * r / (n - 1) - 1.0) for r in rank]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _randn(g, shape, scale):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).mul_(scale).to(torch.bfloat16)


def _mask(g, out, inp, case, density):
    shape = (out // case["g_out"], inp // case["g_in"])
    return (torch.rand(shape, generator=g, device="cuda") < density).to(torch.uint8)


def _x(g, T, inp, case):
    x = _randn(g, (T, inp), 1.0)
    if case["outliers"]:
        ch = torch.randperm(inp, generator=g, device="cuda")[: max(1, inp // 100)]
        x[:, ch] = x[:, ch] * 20.0
    return x


def _logits(g, shape, case):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32) + wk.logit_mean(case["density"])


def _noise(g, shape):
    u = torch.rand(shape, generator=g, device="cuda", dtype=torch.float32).clamp_(1e-7, 1.0 - 1e-6)
    return torch.log(u) - torch.log1p(-u)


def _inputs(case, seed):
    """The drawn tensors of a case (the same ones for `prepare` and `exact`)."""
    g = _generator(seed)
    kind = case["kind"]
    if kind == "sample":
        n = int(case["layers"])
        return {"logits": _logits(g, (n,), case), "noise": _noise(g, (n,))}
    shapes = _shapes(case)
    if kind in ("linear", "block"):
        layers = []
        for (out, inp), d in zip(shapes, _densities(case, len(shapes))):
            W = _randn(g, (out, inp), 0.02)
            layers.append((W, _mask(g, out, inp, case, d), _x(g, case["T"], inp, case)))
        return {"layers": layers}
    out, inp = shapes[0]
    sel = (out // case["g_out"], inp // case["g_in"])
    d = {"W": _randn(g, (out, inp), 0.02), "logits": _logits(g, sel, case)}
    if kind == "train":
        d.update(noise=_noise(g, sel), x=_x(g, case["T"], inp, case), dy=_randn(g, (case["T"], out), 1e-2))
    return d


def _pack(W, mask, case):
    if (case["g_out"], case["g_in"]) == (1, 256):
        return gs.pack(W, mask)
    return gs.pack_groups(W, mask, case["g_out"], case["g_in"])


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    if case["kind"] in ("linear", "block"):
        # a serving program keeps the packed weights and its activation buffers, not the dense weights
        layers = s.pop("layers")
        s["ps"] = [_pack(W, m, case) for W, m, _ in layers]
        s["xs"] = [x for _, _, x in layers]
        if case["kind"] == "block":
            s["ys"] = [torch.empty((case["T"], W.shape[0]), dtype=torch.bfloat16, device="cuda") for W, _, _ in layers]
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "linear":
        return gs.linear(state["xs"][0], state["ps"][0])
    if kind == "block":
        gs.linear_batched_into(state["xs"], state["ps"], state["ys"])
        return state["ys"]
    if kind == "sample":
        mask, dsdl, kept = gs.gumbel_select(state["logits"], state["noise"], TAU)
        return {"mask": mask, "dsdl": dsdl, "kept": kept}
    if kind == "export":
        mask, kept = gs.select_groups(state["logits"])
        p = _pack(state["W"], mask, case)
        return {"mask": mask, "kept": kept, "W_hat": gs.unpack(p)}
    mask, dsdl, kept = gs.gumbel_select(state["logits"], state["noise"], TAU)
    p = _pack(state["W"], mask, case)
    y = gs.linear(state["x"], p)
    dlogits, dx = gs.masked_linear_backward(state["x"], state["W"], p, state["dy"], dsdl)
    return {"mask": mask, "dsdl": dsdl, "kept": kept, "y": y, "dlogits": dlogits, "dx": dx}


# --------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct results lie apart
# --------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "sample":
        return {"bytes": 13.0 * int(case["layers"]) + 8, "flops": 0.0}   # logits, noise, ds/dl, mask, count
    shapes = _shapes(case)
    ds = _densities(case, len(shapes))
    T = case["T"]
    dense = [float(o) * i for o, i in shapes]
    kept = [d * w for d, w in zip(ds, dense)]
    if kind in ("linear", "block"):
        return {"bytes": sum(2.0 * k + 2.0 * T * (o + i) for k, (o, i) in zip(kept, shapes)),
                "flops": sum(2.0 * T * k for k in kept)}
    out, inp = shapes[0]
    n = out // case["g_out"] * (inp // case["g_in"])
    if kind == "export":   # logits, mask; kept weights read and packed; the dense check copy
        return {"bytes": 5.0 * n + 4.0 * kept[0] + 2.0 * dense[0] + 8, "flops": 0.0}
    # logits, noise, ds/dl, mask, dL/dl; W (every group gets a gradient); x, y, dy, dx
    return {"bytes": 17.0 * n + 2.0 * dense[0] + 4.0 * T * (out + inp) + 8,
            "flops": 2.0 * T * (2.0 * kept[0] + dense[0])}


def tolerance(case):
    if case["kind"] == "export":
        return "exact"
    if case["kind"] == "sample":
        return {"rel": 5e-7, "max": 1e-5}   # float32, a few roundings each
    # bf16 results of float32 sums: one rounding, 2^-9 of the value at most
    return {"rel": 6.6e-3, "max": 1.6e-2}


# --------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# --------------------------------------------------------------------------

def _expand(mask, case):
    return mask.bool().repeat_interleave(case["g_out"], 0).repeat_interleave(case["g_in"], 1)


def _exact_linear(x, W, mask, case):
    return x.double() @ (W.double() * _expand(mask, case)).T


def _exact_sample(logits, noise):
    z32 = logits + noise                  # the float32 sum is part of the definition
    z = z32.double().abs() / TAU_F32
    t = torch.exp(-z)
    mask = (z32 > 0).to(torch.uint8)
    return {"mask": mask, "dsdl": t / (1.0 + t) ** 2 / TAU_F32, "kept": mask.sum(dtype=torch.int64).reshape(1)}


TAU_F32 = float(torch.tensor(TAU, dtype=torch.float32))


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "linear":
        W, m, x = s["layers"][0]
        return _exact_linear(x, W, m, case)
    if kind == "block":
        return [_exact_linear(x, W, m, case) for W, m, x in s["layers"]]
    if kind == "sample":
        return _exact_sample(s["logits"], s["noise"])
    if kind == "export":
        mask = (s["logits"] > 0).to(torch.uint8)
        return {"mask": mask, "kept": mask.sum(dtype=torch.int64).reshape(1),
                "W_hat": s["W"].double() * _expand(mask, case)}
    r = _exact_sample(s["logits"], s["noise"])
    W, x, dy = s["W"].double(), s["x"].double(), s["dy"].double()
    m = _expand(r["mask"], case)
    dW = dy.T @ x
    out, inp = W.shape
    go, gi = case["g_out"], case["g_in"]
    dB = (W * dW).reshape(out // go, go, inp // gi, gi).sum((1, 3))
    r.update(y=x @ (W * m).T, dlogits=dB * r["dsdl"], dx=dy @ (W * m))
    return r
