"""Timed workloads of the factorized-layer library, through its public Python entry points.

A case is one pass that a training or inference program makes: a layer's forward, or its forward and
backward, or the exchange of gradients through the flat buffer.  Tensors are contiguous, as a program
gets them from its framework, so ragged widths mean ragged row pitches.  Shapes are those of the
benchmark configurations (factors at a quarter of the width and around it) and generic ones.
"""
from __future__ import annotations

import math

import torch

import paper_2103_03936_b200 as pf

_TORCH = {"bf16": torch.bfloat16, "f32": torch.float32}


# ------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest training step: a narrow fp32 layer on a small batch, all launches and host time
        _linear("fp32 tiny", "f32", 64, 256, 256, 32),
        # one time step of a recurrent layer (batch 20) with the gate biases: generation, few rows, ragged widths
        _linear("lstm step", "bf16", 20, 1500, 6000, 375, train=False, bias=True),
        # all time steps of a truncated-backpropagation window (batch 20 x 35): input-to-hidden training step
        _linear("lstm gates", "bf16", 700, 1500, 6000, 375),
        # the same layer with one factor pair per gate matrix (input and hidden gates), one shared input
        _grouped("lstm per gate", 8, 700, 1500, 1500, 375, shared=True),
        # first feed-forward layer of a Transformer block, with its bias: 64 sequences x 128 tokens
        _linear("ffn up", "bf16", 8192, 512, 2048, 128, bias=True),
        # second feed-forward layer
        _linear("ffn down", "bf16", 8192, 2048, 512, 128),
        # the same feed-forward layer trained in single precision on a smaller batch
        _linear("fp32 ffn", "f32", 2048, 512, 2048, 128),
        # a wide layer on a large batch at a small rank (bound by memory) ...
        _linear("wide r64", "bf16", 16384, 4096, 4096, 64),
        # ... and at a quarter of its width (bound by the tensor cores): the largest case
        _linear("wide r1024", "bf16", 16384, 4096, 4096, 1024),
        # 3 x 3 convolution of a residual network's middle stage, then its two gradients into the flat buffer
        _conv("conv 32x32", "bf16", 128, 32, 32, 256, 64, 256),
        # the strided convolution that opens a stage: twice the channels at half the resolution
        _conv("conv stride 2", "bf16", 128, 32, 32, 128, 64, 256, stride=2),
        # a whole network's factor gradients through the flat buffer and back
        {"name": "flat buffer", "kind": "flat", "dtype": "bf16", "tensors": 176, "small": 65536, "large": 262144},
    ]


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choices(("train", "infer", "grouped", "conv", "flat"), (5, 2, 2, 5, 1))[0]
    if kind == "flat":
        small = _log(rng, 256, 65536)
        large = _log(rng, small, 1 << 20)
        tensors = _log(rng, 2, 400)
        tensors = max(2, min(tensors, 2 * 26_000_000 // (small + large)))
        return {"kind": "flat", "dtype": rng.choice(("bf16", "bf16", "f32")), "tensors": tensors, "small": small, "large": large}
    if kind == "conv":
        f32 = rng.random() < 0.15
        most = 4e9 if f32 else 33.6e6 * 2304
        while True:
            C = rng.choice((64, 96, 128, 160, 192, 256, 256, 320, 512))
            stride = rng.choice((1, 1, 1, 2))
            O = C if stride == 1 and rng.random() < 0.6 else 2 * C
            R = rng.choice((C // 4, C // 4, C // 2, _multiple(rng, 8, C // 8, C // 2)))
            H = _log(rng, 4, 56)
            W = H if rng.random() < 0.8 else max(4, H - rng.randrange(1, 4))
            N = _log(rng, 1, 256)
            pixels = N * H * W
            if pixels * max(C, O // stride ** 2) <= (4e6 if f32 else 34e6) and pixels * R * (9 * C + O) / stride ** 2 <= most / 3:
                break
        c = _conv("", "f32" if f32 else "bf16", N, H, W, C, R, O, stride=stride, train=rng.random() < 0.8)
        del c["name"]
        return c
    if kind == "grouped":
        groups = rng.choice((2, 3, 4, 4, 8))
        k, r = _widths(rng, 64, 2048)
        n = k if rng.random() < 0.6 else _width(rng, 64, 2048)
        r = min(r, n)
        shared = rng.random() < 0.5
        m = min(_log(rng, 32, 8192), int(40e6 / (groups * max(k, n))))
        c = _grouped("", groups, max(1, m), k, n, r, shared=shared)
        del c["name"]
        return c
    f32 = rng.random() < 0.2
    train = kind == "train"
    while True:
        k, r = _widths(rng, 64, 4096)
        n = rng.choice((k, 4 * k, max(64, k // 4), _width(rng, 64, 6000)))
        m = _log(rng, 16, 16384) if train else _log(rng, 1, 4096)
        if n <= 8192 and r <= n and 6.0 * m * r * (k + n) <= (12e9 if f32 else 800e9) and m * (k + n) <= 130e6:
            break
    c = _linear("", "f32" if f32 else "bf16", m, k, n, r, train=train, bias=rng.random() < 0.4, relu=not train and rng.random() < 0.5)
    del c["name"]
    return c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _multiple(rng, step, lo, hi):
    return max(step, int(round(rng.uniform(lo, hi) / step)) * step)


def _width(rng, lo, hi):
    """A layer width: mostly a multiple of 64 or 8, else ragged (any multiple of 4, or any number)."""
    w = _log(rng, lo, hi)
    step = rng.choice((64, 64, 64, 8, 8, 4, 1))
    return max(step, w // step * step)


def _widths(rng, lo, hi):
    """A layer width and a rank around a quarter of it, mostly even."""
    k = _width(rng, lo, hi)
    r = max(8, int(k * math.exp(rng.uniform(math.log(1 / 32), math.log(1 / 2))))) if rng.random() < 0.4 else max(8, k // 4)
    step = rng.choice((16, 16, 8, 1))
    return k, max(8, min(1024, r // step * step))


def _linear(name, dtype, m, k, n, r, *, train=True, bias=False, relu=False):
    return {"name": name, "kind": "linear", "dtype": dtype, "m": m, "k": k, "n": n, "r": r, "train": train, "bias": bias, "relu": relu}


def _grouped(name, groups, m, k, n, r, *, shared):
    return {"name": name, "kind": "grouped", "dtype": "bf16", "groups": groups, "m": m, "k": k, "n": n, "r": r, "shared": shared}


def _conv(name, dtype, N, H, W, C, R, O, *, stride=1, train=True):
    return {"name": name, "kind": "conv", "dtype": dtype, "N": N, "H": H, "W": W, "C": C, "R": R, "O": O, "stride": stride, "train": train}


def _flat_sizes(c):
    """Element counts of the tensors of a flat-buffer case: spread between the two bounds, few of them round."""
    t = c["tensors"]
    return [int(c["small"] * (c["large"] / c["small"]) ** (((i * 37) % t) / max(1, t - 1))) + i % 3 for i in range(t)]


# ------------------------------------------------------------------------------------ inputs
class _Source:
    """Seeded values made on the GPU."""

    def __init__(self, seed, dtype):
        self.g = torch.Generator(device="cuda").manual_seed(seed)
        self.dtype = _TORCH[dtype]

    def normal(self, *shape, scale=1.0):
        return (torch.randn(shape, generator=self.g, device="cuda") * scale).to(self.dtype)

    def uniform(self, *shape):
        return (torch.rand(shape, generator=self.g, device="cuda") * 2 - 1).to(self.dtype)

    def relu(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda").clamp_(min=0).to(self.dtype)


def prepare(case, seed):
    c, s = case, _Source(seed, case["dtype"])
    st = {"case": c}
    if c["kind"] == "flat":
        sizes = _flat_sizes(c)
        st["grads"] = [s.normal(n) for n in sizes]
        st["flat"] = torch.empty(sum(sizes), dtype=s.dtype, device="cuda")
        st["arena"] = torch.zeros(sum(sizes), dtype=s.dtype, device="cuda")     # the optimiser's gradients, one after the other
        st["back"] = list(torch.split(st["arena"], sizes))
    elif c["kind"] == "conv":
        Ho, Wo = (c["H"] - 1) // c["stride"] + 1, (c["W"] - 1) // c["stride"] + 1
        st["x"] = s.relu(c["N"], c["H"], c["W"], c["C"])                         # activations after max(0, .)
        st["U"] = s.normal(3, 3, c["C"], c["R"], scale=math.sqrt(2.0 / (9 * c["C"])))
        st["V"] = s.normal(c["O"], c["R"], scale=math.sqrt(2.0 / c["R"]))
        if c["train"]:
            st["dY"] = s.normal(c["N"], Ho, Wo, c["O"])
            st["flat"] = torch.empty(st["U"].numel() + st["V"].numel(), dtype=s.dtype, device="cuda")
    else:
        g = (c["groups"],) if c["kind"] == "grouped" else ()
        m, k, n, r = c["m"], c["k"], c["n"], c["r"]
        x_shape = (m, k) if c.get("shared") else (*g, m, k)
        st["x"] = s.uniform(*x_shape) if k % 8 else s.normal(*x_shape)
        st["U"] = s.normal(*g, k, r, scale=k ** -0.5)
        st["V"] = s.normal(*g, n, r, scale=k ** -0.5)
        if c.get("bias"):
            st["bias"] = s.normal(n, scale=0.1)
        if c.get("train", True):
            st["dY"] = s.normal(*g, m, n)
    return st


# ------------------------------------------------------------------------------------ one pass
def run(st):
    c = st["case"]
    if c["kind"] == "flat":
        pf.pf_pack_factor_grads(st["grads"], flat=st["flat"])
        pf.pf_unpack_factor_grads(st["flat"], st["back"])
        return {"flat": st["flat"], "grads": st["arena"]}
    x, U, V = st["x"], st["U"], st["V"]
    if c["kind"] == "conv":
        if not c["train"]:
            return pf.pf_lowrank_conv_fwd(x, U, V, stride=c["stride"])
        y, T = pf.pf_lowrank_conv_fwd(x, U, V, stride=c["stride"], want_stash=True)
        dX, dU, dV = pf.pf_lowrank_conv_bwd(x, U, V, st["dY"], stride=c["stride"], T_stash=T)
        flat, _ = pf.pf_pack_factor_grads([dU, dV], flat=st["flat"])
        return {"y": y, "dX": dX, "dU": dU, "dV": dV, "flat": flat}
    if c["kind"] == "grouped":
        y, T = pf.pf_lowrank_linear_grouped_fwd(x, U, V, want_stash=True)
        dX, dU, dV = pf.pf_lowrank_linear_grouped_bwd(x, U, V, st["dY"], T_stash=T)
        return {"y": y, "dX": dX, "dU": dU, "dV": dV}
    plain = not c["bias"] and not c["relu"]
    act = pf.PF_ACT_RELU if c["relu"] else pf.PF_ACT_NONE
    if not c["train"]:
        return pf.pf_lowrank_linear_fwd(x, U, V) if plain else pf.pf_lowrank_linear_fwd_act(x, U, V, bias=st.get("bias"), act=act)
    if plain:
        y, T = pf.pf_lowrank_linear_fwd(x, U, V, want_stash=True)
        db = None
    else:
        y, T = pf.pf_lowrank_linear_fwd_act(x, U, V, bias=st["bias"], act=act, want_stash=True)
        db = pf.pf_bias_act_bwd(y, st["dY"], act=act)
    dX, dU, dV = pf.pf_lowrank_linear_bwd(x, U, V, st["dY"], T_stash=T)
    return {"y": y, "dX": dX, "dU": dU, "dV": dV, "db": db}


# ------------------------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c, size = case, 2 if case["dtype"] == "bf16" else 4
    if c["kind"] == "flat":
        return {"bytes": 4.0 * size * sum(_flat_sizes(c)), "flops": 0.0}       # read and written, twice
    train = c.get("train", True)
    if c["kind"] == "conv":
        rows_in = c["N"] * c["H"] * c["W"]
        rows = c["N"] * ((c["H"] - 1) // c["stride"] + 1) * ((c["W"] - 1) // c["stride"] + 1)
        factors = c["R"] * (9 * c["C"] + c["O"])
        x, y, flops = rows_in * c["C"], rows * c["O"], 2.0 * rows * factors
    else:
        g = c.get("groups", 1)
        factors = g * c["r"] * (c["k"] + c["n"])
        x, y = (1 if c.get("shared") else g) * c["m"] * c["k"], g * c["m"] * c["n"]
        flops = 2.0 * c["m"] * factors
    if not train:
        return {"bytes": float(size * (x + y + factors)), "flops": flops}
    packed = 2 * factors if c["kind"] == "conv" else 0
    return {"bytes": float(size * (2 * x + 2 * y + 2 * factors + packed)), "flops": 3 * flops}


def tolerance(case):
    if case["kind"] == "flat":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    # the intermediate is rounded to bf16 before the second product, the results once more
    return {"rel": 1e-2, "max": 0.1}
