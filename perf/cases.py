"""The work that a user of this library has it do, as cases for timing: sizes, inputs, one pass, its cost, its tolerance.

The public entry points are the four forwards of the binding: hard inference on device buffers (`FFFLayer.forward_infer`)
and on host buffers (`forward_infer_host`), the training-time forward (`forward_train`) and a stack of layers
(`FFFStack.forward`); a case's "path" names the one it takes.  Sizes are those of the configurations in
paper_2308_14711_b200/workloads.py and of the benchmark's further legs, at the batches that such layers meet: one
image, a serving batch, the benchmark's whole batch.  Values follow the same recipe as workloads.py (variances of the
weights, kinds of tokens), drawn on the GPU.

Routing is a comparison of a float32 sum with zero.  As in the parity tests, tokens with a routing logit close to zero
are redrawn (here: within 1e-3), so that the order of a sum does not decide where a token goes.  In a stack the later layers
route on values that went through bf16 several times, so there every layer's logits are kept away from zero, by 2e-2.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_14711_b200 import binding
from paper_2308_14711_b200 import workloads as wl

IMAGE = 197              # tokens of one image (14 x 14 patches and a class token): the batches below are whole images
MARGIN = 1e-3
STACK_MARGIN = 2e-2
LN_EPS = 1e-5


def _case(name, path, D, O, depth, l, act, dtype, B, x, **more):
    return dict(name=name, path=path, D=D, O=O, depth=depth, l=l, act=act, dtype=dtype, B=B, x=x, **more)


def listed():
    return [
        # ---- hard inference, inputs and outputs in device memory
        # one request of a vision transformer: a single image's tokens; launches and latency count
        _case("vit_one_image", "infer", 768, 768, 8, 12, "gelu", "bf16", IMAGE, "layernorm"),
        # a serving batch of 16 images
        _case("vit_batch_16", "infer", 768, 768, 8, 12, "gelu", "bf16", 16 * IMAGE, "layernorm"),
        # the benchmark's batch of 256 images: throughput
        _case("vit_batch_256", "infer", 768, 768, 8, 12, "gelu", "bf16", 256 * IMAGE, "layernorm"),
        # a wide layer that stands in for a very large feedforward layer, tokens spread over all leaves
        _case("wide_uniform", "infer", 1024, 1024, 11, 32, "gelu", "bf16", 65536, "normal"),
        # the same layer when a few leaves receive most tokens
        _case("wide_skewed", "infer", 1024, 1024, 11, 32, "gelu", "bf16", 65536, "clusters"),
        # many one-neuron leaves: about one token per leaf, a gather of weights
        _case("deep_thin", "infer", 768, 768, 15, 1, "gelu", "bf16", 16384, "normal"),
        # a small classifier of 28 x 28 images in float32 (ten outputs, rows of y that are no multiple of 16 bytes)
        _case("digits_f32", "infer", 784, 10, 3, 32, "relu", "f32", 2048, "normal"),
        # the transformer layer kept in float32, 32 images
        _case("vit_f32_batch_32", "infer", 768, 768, 8, 12, "gelu", "f32", 32 * IMAGE, "layernorm"),
        # leaf weights stored as 8-bit floats: the wide layer at half the memory
        _case("wide_w8", "infer", 1024, 1024, 11, 32, "gelu", "w8", 65536, "normal"),
        # ---- the other entry points
        # tokens that start and end in pinned host memory
        _case("vit_host_256", "host", 768, 768, 8, 12, "gelu", "bf16", 256 * IMAGE, "layernorm"),
        # the forward half of a training step, with the mixture weights and the entropies that the losses need
        _case("vit_train_256", "train", 768, 768, 8, 12, "gelu", "bf16", 256 * IMAGE, "layernorm"),
        # the feedforward layers of four transformer blocks with layer norm and residual connections, 64 images
        _case("vit_stack_64", "stack", 768, 768, 8, 12, "gelu", "bf16", 64 * IMAGE, "layernorm", layers=4),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the ranges above: every path at sizes around and between the listed ones, odd batches among them."""
    kind = rng.choice(["layer", "layer", "layer", "thin", "small_f32", "layer_f32", "w8", "host", "train", "stack"])
    act = rng.choice(["gelu", "gelu", "relu", "silu", "gelu_tanh"])
    x = rng.choice(["layernorm", "normal", "normal", "clusters"])
    D = 64 * rng.randint(4, 16)                    # 256 .. 1024: model widths
    if rng.random() < 0.3:
        D -= 8 * rng.randint(1, 7)                 # and widths that are no multiple of 64
    wide = D // 16 * 16
    if kind == "layer":
        depth, l = rng.randint(4, 11), rng.randint(8, 40)
        return _case("", "infer", D, wide, depth, l, act, "bf16", _log_int(rng, 1, 65536), x)
    if kind == "thin":
        return _case("", "infer", D, wide, rng.randint(12, 15), rng.randint(1, 2), act, "bf16", _log_int(rng, 256, 16384), "normal")
    if kind == "small_f32":
        return _case("", "infer", rng.randint(50, 1000), rng.randint(2, 40), rng.randint(1, 6), rng.randint(4, 32), act, "f32",
                     _log_int(rng, 16, 8192), "normal")
    if kind == "layer_f32":
        return _case("", "infer", D, wide, rng.randint(4, 9), rng.randint(8, 32), act, "f32", _log_int(rng, 16, 6304), x)
    D = 128 * rng.randint(2, 8)                    # (8-bit weights exist for multiples of 128, the training forward of 64)
    if kind == "w8":
        return _case("", "infer", D, D, rng.randint(6, 11), rng.randint(8, 32), act, "w8", _log_int(rng, 2048, 65536), x)
    if kind == "host":
        return _case("", "host", min(D, 768), min(D, 768), rng.randint(4, 8), rng.randint(8, 32), act, "bf16", _log_int(rng, 512, 50432), x)
    if kind == "train":
        return _case("", "train", min(D, 768), min(D, 768), rng.randint(3, 8), rng.randint(4, 12), act, "bf16", _log_int(rng, 256, 50432), x)
    return _case("", "stack", min(D, 768), min(D, 768), rng.randint(4, 8), rng.randint(8, 16), act, "bf16", _log_int(rng, 256, 12608),
                 x if x != "clusters" else "normal", layers=rng.randint(2, 4))


# ---------------------------------------------------------------------------------------------------- inputs
def _tdtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _weights(case, gen):
    """Tensors of one layer in the layouts of fff_create, with the variances of workloads.py."""
    D, O, l, nl = case["D"], case["O"], case["l"], 1 << case["depth"]
    td = _tdtype(case)

    def normal(std, *shape):
        return (torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32) * std).to(td)
    return dict(node_w=normal(D ** -0.5, nl - 1, D), node_b=torch.zeros((nl - 1,), dtype=td, device="cuda"),
                w1=normal(D ** -0.5, nl, l, D), b1=normal(wl.LEAF_BIAS_STD, nl, l),
                w2=normal(l ** -0.5, nl, O, l), b2=normal(wl.LEAF_BIAS_STD, nl, O))


def _e4m3(w):
    """8-bit codes and one scale per leaf, as workloads.quantize_e4m3 makes them."""
    amax = w.float().flatten(1).abs().amax(dim=1)
    scale = torch.where(amax > 0, amax / wl.E4M3_MAX, torch.ones_like(amax))
    codes = (w.float() / scale.view(-1, 1, 1)).to(torch.float8_e4m3fn).view(torch.uint8)
    return codes.contiguous(), scale.contiguous()


def _layer(case, w):
    args = (case["D"], case["O"], case["depth"], case["l"], case["act"])
    if case["dtype"] == "w8":
        c1, s1 = _e4m3(w["w1"])
        c2, s2 = _e4m3(w["w2"])
        layer = binding.FFFLayer(*args, "bf16", w["node_w"], w["node_b"], c1, w["b1"], c2, w["b2"], w1_scale=s1, w2_scale=s2)
    else:
        layer = binding.FFFLayer(*args, case["dtype"], **w)
    layer.reserve(case["B"])
    return layer


class _Tokens:
    """Rows of the case's kind; `rows(which)` draws rows again for the tokens `which`."""

    def __init__(self, case, gen):
        self.case, self.gen = case, gen
        if case["x"] == "clusters":
            self.centres = torch.randn((wl.N_CLUSTERS, case["D"]), generator=gen, device="cuda")
            p = torch.from_numpy(np.asarray(wl.zipf_weights())).cuda()
            self.cluster = torch.multinomial(p, case["B"], replacement=True, generator=gen)

    def rows(self, which):
        x = torch.randn((which.numel(), self.case["D"]), generator=self.gen, device="cuda")
        if self.case["x"] == "layernorm":
            x = (x - x.mean(1, keepdim=True)) / x.std(1, unbiased=False, keepdim=True)
        elif self.case["x"] == "clusters":
            x = self.centres[self.cluster[which]] + wl.CLUSTER_SIGMA * x
        return x.to(_tdtype(self.case))


def _path_margin(x, node_w, depth, want_leaf=False):
    """The smallest routing logit, in magnitude, that each row meets on its way (the biases are zero)."""
    pos = torch.zeros((x.shape[0],), dtype=torch.int64, device=x.device)
    least = torch.full((x.shape[0],), math.inf, device=x.device)
    for m in range(depth):
        logit = (node_w[(1 << m) - 1 + pos].float() * x.float()).sum(1)
        least = torch.minimum(least, logit.abs())
        pos = 2 * pos + (logit >= 0).long()
    return (least, pos) if want_leaf else least


def _redrawn(case, gen, margin_of, margin):
    """Tokens of the case's kind, redrawn where margin_of(rows) is below `margin`."""
    src = _Tokens(case, gen)
    todo = torch.arange(case["B"], device="cuda")
    x = src.rows(todo)
    for _ in range(60):
        todo = torch.cat([t[margin_of(x[t]) < margin] for t in todo.split(4096 if case["path"] == "stack" else 65536)])
        if todo.numel() == 0:
            break
        x[todo] = src.rows(todo)
    return x


def _activation(name, v):
    f = torch.nn.functional
    return {"relu": f.relu, "gelu": f.gelu, "silu": f.silu, "gelu_tanh": lambda u: f.gelu(u, approximate="tanh")}[name](v)


def _stack_margin(case, ws, gammas, betas, x):
    """_path_margin over all layers of a residual stack with layer norm, the rows in between rounded as they are stored."""
    td, least = _tdtype(case), torch.full((x.shape[0],), math.inf, device=x.device)
    for w, g, b in zip(ws, gammas, betas):
        z = torch.nn.functional.layer_norm(x.float(), (case["D"],), g.float(), b.float(), LN_EPS).to(td)
        margin, leaf = _path_margin(z, w["node_w"], case["depth"], True)
        least = torch.minimum(least, margin)
        h = torch.einsum("bd,bld->bl", z.float(), w["w1"][leaf].float()) + w["b1"][leaf].float()
        h = _activation(case["act"], h).to(td).float()
        y = torch.einsum("bl,bol->bo", h, w["w2"][leaf].float()) + w["b2"][leaf].float()
        x = x + y.to(td)
    return least


def prepare(case, seed):
    """What a program holds before the call: the layer (or stack) with its workspace, and the tokens."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["path"] == "stack":
        ws = [_weights(case, gen) for _ in range(case["layers"])]
        layers = [_layer(case, w) for w in ws]
        td, D = _tdtype(case), case["D"]
        gammas = [(1 + 0.1 * torch.randn((D,), generator=gen, device="cuda")).to(td) for _ in layers]
        betas = [(0.1 * torch.randn((D,), generator=gen, device="cuda")).to(td) for _ in layers]
        stack = binding.FFFStack(layers, layer_norm=True, gammas=gammas, betas=betas, eps=LN_EPS, residual=True)
        x = _redrawn(case, gen, lambda rows: _stack_margin(case, ws, gammas, betas, rows), STACK_MARGIN)
        stack.forward(x)                           # the first call of a size allocates the buffers between the layers
        return dict(path="stack", stack=stack, x=x)
    w = _weights(case, gen)
    layer = _layer(case, w)
    # (the training forward takes no decision)
    x = _redrawn(case, gen, lambda rows: _path_margin(rows, w["node_w"], case["depth"]), 0.0 if case["path"] == "train" else MARGIN)
    state = dict(path=case["path"], layer=layer, x=x)
    if case["path"] == "host":
        state["x"] = x.cpu().pin_memory()
        state["y"] = torch.empty((case["B"], case["O"]), dtype=x.dtype).pin_memory()
        state["leaf"] = torch.empty((case["B"],), dtype=torch.int32).pin_memory()
        layer.forward_infer_host(state["x"], state["y"], state["leaf"])        # allocates the staging buffers
    elif case["path"] == "train":
        layer.forward_train(x)                     # the first call of a size allocates its workspace
    return state


def run(state):
    if state["path"] == "infer":
        return state["layer"].forward_infer(state["x"])
    if state["path"] == "host":
        state["layer"].forward_infer_host(state["x"], state["y"], state["leaf"])
        return state["y"], state["leaf"]
    if state["path"] == "train":
        return state["layer"].forward_train(state["x"])
    return state["stack"].forward(state["x"])


# ---------------------------------------------------------------------------------------------------- cost and tolerance
def _touched(n, B):
    """Expected number of distinct leaves (or nodes of one level) that B spread-out tokens reach."""
    return n * -math.expm1(B * math.log1p(-1.0 / n)) if n > 1 else 1.0


def work(case):
    B, D, O, d, l, nl = case["B"], case["D"], case["O"], case["depth"], case["l"], 1 << case["depth"]
    e = 4 if case["dtype"] == "f32" else 2
    ew = 1 if case["dtype"] == "w8" else e
    if case["path"] == "train":
        # every node and every leaf for every token; y, the mixture weights and the entropies come out
        flops = 2.0 * B * ((nl - 1) * D + nl * l * D + nl * (l + 1) * O)
        params = (nl - 1) * (D + 1) * e + nl * (l * (D + 1) + O * (l + 1)) * e
        return {"bytes": B * (D + O) * e + params + 4.0 * B * nl + 4.0 * (nl - 1), "flops": flops}
    B_eff = min(B, 8 * wl.N_CLUSTERS) if case["x"] == "clusters" else B     # (a cluster's tokens share a few leaves)
    leaves = _touched(nl, B_eff)
    nodes = sum(_touched(1 << m, B_eff) for m in range(d))
    params = nodes * (D + 1) * e + leaves * ((l * D + O * l) * ew + (l + O) * e + (8 if case["dtype"] == "w8" else 0))
    layers = case.get("layers", 1)
    flops = 2.0 * B * (d * D + l * D + l * O) * layers
    return {"bytes": B * (D + O) * e + (params + 4.0 * B) * layers, "flops": flops}


def tolerance(case):
    """About four times what the outputs differ by from the same path in 64 bits."""
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 6e-6}
    # sums of exact bf16 products in float32, hidden values and outputs rounded to bf16; no token changes its leaf
    return {"rel": 1e-2, "max": 7e-2}
