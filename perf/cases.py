"""The work that users of this library have it do, as measurable cases.

A case is a dict of plain values.  `kind` names the call a user's program makes:

  train    autograd.dsa3d, forward and backward: a training step of the operator with learned offsets
  sample   autograd.dsa3d without gradients: inference / diffusion sampling
  fixed    autograd.dsa3d_fixed_window, forward and backward: the fixed window of the offsets ablation
  bounded  binding.dsa3d_forward_bounded_offsets and its backward: offsets that are small perturbations of
           the window (every component below 1 in size), with the workspace that a program keeps
  layer    layer.DeformableSlideAttention3D, forward and backward with all its parameters: Eq. 1 whole, the
           two depthwise convolutions and the offset predictor's linear layer included
  host     binding.dsa3d_step_host: forward and backward from page-locked host buffers and back

Grids, head shapes, windows and offset spreads are those of paper_2607_22696_b200/inputs.py (latent-video grids
of 480p, 720p and 1080p video, the offset / window sweep, the paper's own window), cut in frames where the whole
clip would not fit the card several times over.
"""
import math

import torch

from paper_2607_22696_b200 import autograd as ops
from paper_2607_22696_b200 import binding
from paper_2607_22696_b200.layer import DeformableSlideAttention3D

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(kind, grid, heads, d, window, offsets, sigma, dtype="bf16", name=None):
    c = {"kind": kind, "T": grid[0], "H": grid[1], "W": grid[2], "heads": heads, "d": d, "kt": window[0],
         "kh": window[1], "kw": window[2], "offsets": offsets, "sigma": sigma, "dtype": dtype}
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # the smallest call: unit tests, toy models, the first step of a port; 256 tokens, so launches and the
        # host path are all there is
        _case("train", (4, 8, 8), 2, 32, (3, 3, 3), "normal", 0.5, "f32", name="tiny_f32_train"),
        # fp32 storage in earnest: numerics studies and gradient checks of a model on a 480p-class grid
        _case("train", (8, 30, 52), 8, 64, (3, 3, 3), "normal", 1.0, "f32", name="480p_8f_f32_train"),
        # sampling from a trained model at 480p: forward only, heads of 64 channels
        _case("sample", (16, 30, 52), 16, 64, (3, 3, 3), "normal", 1.0, name="480p_16f_sample"),
        # a training step at 720p, 64 latent frames: the largest tensors
        _case("train", (64, 45, 80), 24, 128, (3, 3, 3), "normal", 1.5, name="720p_64f_train"),
        # the 32 heads of 64 channels of the paper's 1B model on a 1080p grid, offsets with the spread of the
        # headline workload
        _case("train", (16, 68, 120), 32, 64, (3, 3, 3), "normal", 2.0, name="1080p_16f_h32d64_train"),
        # the window the paper itself runs, (3,7,7), with learned offsets: the most arithmetic
        _case("train", (8, 68, 120), 16, 128, (3, 7, 7), "normal", 2.0, name="1080p_8f_w377_train"),
        # the corner of the offset / window sweep with the smallest window and integer displacements
        _case("train", (64, 45, 80), 16, 128, (2, 2, 2), "int", 0.0, name="sweep_w222_int_train"),
        # the ablation's fixed window: the usual (3,3,3), and the paper's own
        _case("fixed", (64, 45, 80), 16, 128, (3, 3, 3), "zero", 0.0, name="sweep_w333_fixed"),
        _case("fixed", (64, 45, 80), 16, 128, (3, 7, 7), "zero", 0.0, name="sweep_w377_fixed"),
        # offsets early in training, or held small by a regulariser
        _case("bounded", (64, 45, 80), 16, 128, (3, 3, 3), "small", 0.4, name="sweep_w333_bounded"),
        # Eq. 1 as a layer of a model: hidden size 1024
        _case("layer", (16, 30, 52), 16, 64, (3, 3, 3), "learned", 1.0, name="480p_16f_layer"),
        # tensors that live in host memory (activation offloading): the step with its copies both ways
        _case("host", (8, 45, 80), 16, 128, (3, 3, 3), "normal", 2.0, name="720p_8f_host_step"),
    ]


def draw(rng):
    kind = rng.choice(["train", "train", "train", "train", "sample", "sample", "fixed", "fixed", "bounded", "layer", "host"])
    dtype = "f32" if kind == "train" and rng.random() < 0.25 else "bf16"
    d = rng.choice([32, 64, 128]) if kind in ("train", "sample") and rng.random() < 0.3 else rng.choice([64, 128])
    if kind in ("bounded", "layer", "host"):
        window = (3, 3, 3)
    elif kind == "fixed":
        window = rng.choice([(2, 2, 2), (3, 3, 3), (3, 3, 3), (3, 5, 5), (3, 7, 7)])
    else:
        window = rng.choice([(2, 2, 2), (3, 3, 3), (3, 3, 3), (3, 3, 3), (3, 5, 5), (3, 7, 7)])
    P = window[0] * window[1] * window[2]
    # (token, head) items: from a toy problem to the cost of the largest listed case; samples count, and fp32 rows
    # and the copies of the host step weigh more
    most = {"train": 5.0e6, "sample": 5.0e6, "fixed": 3.6e6, "bounded": 3.6e6, "layer": 1.0e6, "host": 6.0e5}[kind]
    if kind in ("train", "sample"):
        most *= min(1.0, 27.0 / P)
    if dtype == "f32":
        most = min(most, 5.0e5) * min(1.0, 64.0 / d)
    items = math.exp(rng.uniform(math.log(512.0), math.log(most)))
    heads = rng.choice([h for h in (1, 2, 3, 4, 8, 12, 16, 24, 32) if h * 64 <= items and h * d <= 4096])
    tokens = items / heads
    # a grid of the aspect of video: frames as the cube root with some spread, then rows and columns about 9 : 16
    T = max(1, min(96, round(tokens ** (1.0 / 3.0) * math.exp(rng.uniform(-0.9, 0.3)))))
    H = max(1, min(68, round(math.sqrt(tokens / T * 9.0 / 16.0) * math.exp(rng.uniform(-0.2, 0.2)))))
    W = max(1, min(160, int(tokens / (T * H))))
    if kind in ("train", "sample", "host"):
        offsets = rng.choice(["normal", "normal", "normal", "int"]) if kind != "host" else "normal"
        sigma = round(rng.uniform(0.5, 3.0), 2) if offsets == "normal" else 0.0
    else:
        offsets, sigma = {"fixed": ("zero", 0.0), "bounded": ("small", round(rng.uniform(0.1, 0.4), 2)),
                          "layer": ("learned", round(rng.uniform(0.5, 2.0), 2))}[kind]
    return _case(kind, (T, H, W), heads, d, window, offsets, sigma, dtype)


def _shape(c):
    return c["T"], c["H"], c["W"], c["heads"], c["d"], (c["kt"], c["kh"], c["kw"])


def _points(c):
    return c["kt"] * c["kh"] * c["kw"]


def prepare(case, seed):
    T, H, W, heads, d, window = _shape(case)
    dt, P, kind = DTYPES[case["dtype"]], _points(case), case["kind"]
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape, sigma=1.0, dtype=torch.float32):
        t = torch.randn(*shape, generator=g, device="cuda", dtype=dtype)
        return t if sigma == 1.0 else t.mul_(sigma)

    s = {"case": case, "window": window}
    for name in ("q", "k", "v", "dout"):
        if name != "dout" or kind != "sample":
            s[name] = normal(T, H, W, heads, d, dtype=dt)
    if case["offsets"] == "normal":
        s["offsets"] = normal(T, H, W, heads, P, 3, sigma=case["sigma"])
    elif case["offsets"] == "small":
        s["offsets"] = normal(T, H, W, heads, P, 3, sigma=case["sigma"]).clamp_(-0.999, 0.999)
    elif case["offsets"] == "int":
        s["offsets"] = torch.randint(-2, 3, (T, H, W, heads, P, 3), generator=g, device="cuda").float()

    if kind in ("train", "fixed", "layer"):
        for name in ("q", "k", "v", "offsets"):
            if name in s:
                s[name].requires_grad_()
    if kind == "bounded":
        # outputs and workspace that the program allocates once
        s["out"], s["dq"], s["dk"], s["dv"] = (torch.empty_like(s["q"]) for _ in range(4))
        s["lse"] = torch.empty(T, H, W, heads, device="cuda")
        s["doffsets"] = torch.empty_like(s["offsets"])
        n = binding.dsa3d_backward_bounded_offsets_workspace_bytes(T, H, W, heads, d, window, dt)
        s["workspace"] = torch.empty(max(n, 16), dtype=torch.uint8, device="cuda")
    elif kind == "layer":
        # a module some way into training: its predictor yields offsets of about `sigma`
        s["layer"] = DeformableSlideAttention3D(heads, d, window, seed=seed)
        with torch.no_grad():
            w = s["layer"].offset_weight
            w.copy_(normal(*w.shape, sigma=case["sigma"] / math.sqrt(heads * d)))
        s["x"] = normal(T, H, W, heads * d, dtype=dt).requires_grad_()
        s["leaves"] = [s["x"], s["q"], s["k"], s["v"], *s["layer"].parameters()]
    elif kind == "host":
        for name in ("q", "k", "v", "offsets", "dout"):
            t = s[name]
            s[name] = torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)
        for name, like in (("out", "q"), ("dq", "q"), ("dk", "q"), ("dv", "q"), ("doffsets", "offsets")):
            s[name] = torch.empty(s[like].shape, dtype=s[like].dtype, pin_memory=True)
        s["lse"] = torch.empty(T, H, W, heads, pin_memory=True)
        n = binding.dsa3d_step_host_arena_bytes(T, H, W, heads, d, window, dt)
        s["arena"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    return s


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind == "train":
        out = ops.dsa3d(s["q"], s["k"], s["v"], s["offsets"], s["window"])
        return (out.detach(), *torch.autograd.grad(out, [s["q"], s["k"], s["v"], s["offsets"]], s["dout"]))
    if kind == "sample":
        with torch.no_grad():
            return ops.dsa3d(s["q"], s["k"], s["v"], s["offsets"], s["window"])
    if kind == "fixed":
        out = ops.dsa3d_fixed_window(s["q"], s["k"], s["v"], s["window"])
        return (out.detach(), *torch.autograd.grad(out, [s["q"], s["k"], s["v"]], s["dout"]))
    if kind == "layer":
        out = s["layer"](s["x"], s["q"], s["k"], s["v"])
        return (out.detach(), *torch.autograd.grad(out, s["leaves"], s["dout"]))
    shape = _shape(s["case"])
    if kind == "bounded":
        binding.dsa3d_forward_bounded_offsets(s["q"], s["k"], s["v"], s["offsets"], *shape, s["out"], s["lse"])
        binding.dsa3d_backward_bounded_offsets(s["q"], s["k"], s["v"], s["offsets"], s["lse"], s["dout"], *shape,
                                               s["dq"], s["dk"], s["dv"], s["doffsets"], s["workspace"])
    else:
        binding.dsa3d_step_host(s["q"], s["k"], s["v"], s["offsets"], s["dout"], *shape, s["out"], s["lse"], s["dq"],
                                s["dk"], s["dv"], s["doffsets"], s["arena"])
    return tuple(s[name] for name in ("out", "lse", "dq", "dk", "dv", "doffsets"))


def work(case):
    """Each input read once, each output written once; multiply-adds of the definition (interpolation of K and V,
    dot products, weighted sums; about twice that again for the gradients)."""
    T, H, W, heads, d, _ = _shape(case)
    P, elt, kind = _points(case), 4 if case["dtype"] == "f32" else 2, case["kind"]
    items, hidden = T * H * W * heads, heads * d
    row = d * elt
    corners = {"zero": 1, "int": 1}.get(case["offsets"], 8)
    sample = 2 * d * (corners + 1)                       # one interpolated row and its dot product or weighted sum
    fwd_bytes, fwd_flops = 4 * row + 12 * P + 4, 2 * P * sample
    bwd_bytes, bwd_flops = 7 * row + 24 * P + 4, 5 * P * sample
    if kind == "sample":
        return {"bytes": items * (fwd_bytes - 4), "flops": items * fwd_flops}
    if kind == "fixed":                                  # no offsets, no gradient of them
        return {"bytes": items * (4 * row + 7 * row + 8), "flops": items * (fwd_flops + bwd_flops)}
    total = {"bytes": items * (fwd_bytes + bwd_bytes), "flops": items * (fwd_flops + bwd_flops)}
    if kind == "layer":
        n, outputs = T * H * W, heads * P * 3
        # x, q, k, v and dout in; out, their gradients, the parameters and their gradients out; the rest is internal
        total["bytes"] = n * hidden * elt * (5 + 1 + 4) + outputs * hidden * 2 * elt
        total["flops"] += 3 * 2 * n * hidden * outputs + 2 * 3 * 2 * n * hidden * 27
    return total


def tolerance(case):
    if case["dtype"] == "f32":
        # fp32 sums of a few hundred terms; dk and dv sum several hundred contributions in any order
        return {"rel": 1e-5, "max": 2e-4}
    if case["kind"] == "layer":
        # the convolution's output is rounded to bf16 before the linear layer and doffsets before its backward
        return {"rel": 1e-2}
    # every bf16 result is one rounding of an fp32 value: results differ by one step (2^-8) where it falls on a tie
    return {"rel": 5e-3, "max": 2e-2}
