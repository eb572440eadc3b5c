"""The work that users of this library have it do, as cases that can be timed.

Four kinds, all through the public binding:

  product   Y = act(W_hybrid X + bias) of one pruned layer (HybridLayer.spmm): inference of linear and pointwise
            layers, and of convolutions that the caller has lowered to a matrix
  conv      one or more 3x3 / 1x1 convolutions in a row on NHWC activations (HybridLayer.spmm_conv), bias and ReLU
            fused, each layer's output being the next one's input
  compress  one layer is pruned and handed back: mask projection, encoding, decoded pruned weights
  prune     one pruning iteration over a whole network (PruningNetwork.step: saliency from the gradients, masks, global
            selection, encodings), and the decoded pruned weights that training goes on with

Shapes are those of the layers in workloads.py (a 256x1024 linear layer, ResNet-50 / VGG-16 / MobileNetV2 layers, the
4096x4096x8192 sweep); only shapes are used, weights and activations are drawn.
"""
import math

import numpy as np
import torch

from paper_2311_14272_b200 import binding as B
from paper_2311_14272_b200 import workloads as wl

NETWORKS = {"vgg16": wl.config3, "mobilenetv2": wl.config4}


def _product(name, rows, k, ncols, nm, block, keep, f32=False, bias=False, relu=False):
    return {"name": name, "kind": "product", "rows": rows, "k": k, "ncols": ncols, "n": nm[0], "m": nm[1],
            "block_rows": block[0], "block_k": block[1], "keep": keep, "f32": f32, "bias": bias, "relu": relu}


def _conv(name, channels, rows, side, batch, kernel, layers, nm, block, keep, nhwc_out=True):
    return {"name": name, "kind": "conv", "channels": channels, "rows": rows, "side": side, "batch": batch, "kernel": kernel,
            "layers": layers, "n": nm[0], "m": nm[1], "block_rows": block[0], "block_k": block[1], "keep": keep,
            "nhwc_out": nhwc_out}


def _compress(name, rows, k, nm, block, keep):
    return {"name": name, "kind": "compress", "rows": rows, "k": k, "n": nm[0], "m": nm[1], "block_rows": block[0],
            "block_k": block[1], "keep": keep}


def _prune(name, network, nm, block, samples, kappa):
    return {"name": name, "kind": "prune", "network": network, "n": nm[0], "m": nm[1], "block_rows": block[0],
            "block_k": block[1], "samples": samples, "kappa": kappa}


def listed():
    return [
        # the smallest call of a service: one linear layer on 512 tokens, where launch latency is the time
        _product("linear_256x1024x512", 256, 1024, 512, (2, 4), (32, 64), 0.5),
        # one image through a 7x7 pointwise layer: 49 columns, so rows of X and Y start at odd addresses
        _product("pointwise_one_image_7x7", 160, 960, 49, (2, 8), (32, 32), 0.5, bias=True),
        # the widest pointwise layer of a mobile network at batch 64, bound by its 180 MB of activations
        _product("pointwise_expand_112x112_b64", 96, 16, 64 * 112 * 112, (2, 8), (32, 32), 0.5, bias=True, relu=True),
        # the last, incomplete batch of an evaluation set: a lowered 14x14 convolution with 31 images, 6076 columns
        _product("resnet50_3x3_last_batch", 256, 2304, 31 * 14 * 14, (1, 4), (64, 64), 0.25, bias=True, relu=True),
        # the same layer as a convolution, full batch
        _conv("resnet50_3x3_conv_b32", 256, 256, 14, 32, 3, 1, (1, 4), (64, 64), 0.25),
        # the widest convolution of VGG-16: 64 channels at 224x224
        _conv("vgg16_conv1_2_b16", 64, 64, 224, 16, 3, 1, (2, 4), (64, 64), 0.4),
        # a stage of three convolutions in a row, 128 -> 256 -> 256 -> 256 channels at 56x56
        _conv("vgg16_stage3_b16", 128, 256, 56, 16, 3, 3, (2, 4), (64, 64), 0.3),
        # a large linear layer on many tokens, 2:4
        _product("linear_4096x4096x8192_2of4", 4096, 4096, 8192, (2, 4), (128, 64), 0.5),
        # the same with a pattern beyond 2:4 and fp32 results
        _product("linear_4096x4096x8192_4of8_f32", 4096, 4096, 8192, (4, 8), (128, 64), 0.25, f32=True),
        # that layer's weights pruned: mask, encoding, pruned weights back
        _compress("compress_4096x4096_2of4", 4096, 4096, (2, 4), (128, 64), 0.5),
        # one pruning iteration of a network of few large layers, and of one of many small layers
        _prune("prune_vgg16", "vgg16", (2, 4), (64, 64), 4, 0.8),
        _prune("prune_mobilenetv2", "mobilenetv2", (2, 8), (32, 32), 4, 0.86),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges that listed() stands for."""
    kind = rng.choice(["product", "product", "product", "conv", "conv", "compress", "prune"])
    nm = rng.choice([(2, 4), (2, 4), (1, 4), (3, 4), (1, 8), (2, 8), (2, 8), (4, 8)])
    block = (rng.choice([32, 64, 128]), rng.choice([32, 64, 64, 128]))
    keep = round(rng.uniform(0.1, 1.0), 2)
    if kind == "product":
        rows, k = _log(rng, 16, 4096), _log(rng, 32, 4096)
        opts = dict(f32=rng.random() < 0.25, bias=rng.random() < 0.5, relu=rng.random() < 0.5)
        flops_per_col = 2.0 * rows * k * max(keep, 0.2) * nm[0] / nm[1]
        if rng.random() < 0.4:
            # pixels of a 7x7 or 14x14 layer, any number of images: any number of columns, odd ones among them
            pixels = rng.choice([49, 196])
            ncols = pixels * max(1, min(_log(rng, 1, 64), int(1e9 / flops_per_col / pixels)))
        else:
            ncols = 8 * max(4, _log(rng, 32, min(800000, 6e10 / flops_per_col, 9e7 / (rows + k))) // 8)
        c = _product("", rows, k, ncols, nm, block, keep, **opts)
    elif kind == "conv":
        channels = 64 * rng.choice([1, 1, 2, 2, 4, 4, 8])
        rows = 64 * _log(rng, 1, 8) if rng.random() < 0.7 else _log(rng, 24, 512)
        side = rng.choice([224, 112, 56, 56, 28, 28, 14, 14, 7])
        kernel = rng.choice([3, 3, 3, 1])
        most = max(1, int(min(1.6e10 / (2.0 * kernel * kernel * channels * rows * keep * nm[0] / nm[1]),
                              5.2e7 / (channels + rows)) / side ** 2))
        layers = 1 if rows % 64 or rng.random() < 0.7 else 2
        # output as the next convolution's activation, or as a [channels, pixels] matrix
        c = _conv("", channels, rows, side, min(_log(rng, 1, 64), most), kernel, layers, nm, (block[0], 64), keep,
                  layers > 1 or rng.random() < 0.7)
    elif kind == "compress":
        c = _compress("", _log(rng, 16, 4096), _log(rng, 32, 4096), nm, block, keep)
    else:
        c = _prune("", rng.choice(sorted(NETWORKS)), nm, block, rng.randint(1, 4), 0.0)
        density = nm[0] / nm[1]
        c["kappa"] = round(1.0 - density * rng.uniform(0.3, 0.95), 3)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs and state

def _normal(g, shape, std):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).mul_(std)


def _weight(g, rows, k):
    return _normal(g, (rows, k), math.sqrt(2.0 / k)).to(torch.bfloat16)


def _saliency(g, w):
    return w.float().abs() * (torch.rand(w.shape, generator=g, device="cuda") + 0.5)


def _activation(g, shape):
    """max(0, N(0, 1)) in bf16, drawn in pieces: the widest activations have 10^8 elements."""
    out = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    flat = out.view(-1)
    for at in range(0, flat.numel(), 1 << 24):
        part = flat[at:at + (1 << 24)]
        part.copy_(torch.randn(part.shape, generator=g, device="cuda").clamp_(min=0))
    return out


def _keep(case, k):
    """The case's keep ratio, or 1 where it would leave a layer of few blocks without any."""
    return case["keep"] if case["keep"] * math.ceil(k / case["block_k"]) >= 0.5 else 1.0


def _layer(case, g, rows, k):
    L = B.HybridLayer(rows, k, case["n"], case["m"], case["block_rows"], case["block_k"], _keep(case, k))
    w = _weight(g, rows, k)
    L.build_mask(_saliency(g, w)).encode(w)
    return L


def prepare(case, seed):
    B.load()
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    if kind == "product":
        rows, k, ncols = case["rows"], case["k"], case["ncols"]
        L = _layer(case, g, rows, k)
        if case["bias"] or case["relu"]:
            L.set_epilogue(_normal(g, (rows,), 0.1) if case["bias"] else None, case["relu"])
        y = torch.empty((rows, ncols), dtype=torch.float32 if case["f32"] else torch.bfloat16, device="cuda")
        return {"kind": kind, "layer": L, "x": _activation(g, (k, ncols)), "y": y, "y_dtype": 1 if case["f32"] else 0}
    if kind == "conv":
        b, side, kn = case["batch"], case["side"], case["kernel"]
        layers, outs, c = [], [], case["channels"]
        for _ in range(case["layers"]):
            L = _layer(case, g, case["rows"], kn * kn * c)
            L.set_epilogue(_normal(g, (case["rows"],), 0.1), True)
            shape = (b, side, side, case["rows"]) if case["nhwc_out"] else (case["rows"], b * side * side)
            outs.append(torch.empty(shape, dtype=torch.bfloat16, device="cuda"))
            layers.append(L)
            c = case["rows"]
        return {"kind": kind, "layers": layers, "x": _activation(g, (b, side, side, case["channels"])), "outs": outs,
                "kernel": kn, "nhwc_out": case["nhwc_out"]}
    if kind == "compress":
        w = _weight(g, case["rows"], case["k"])
        L = B.HybridLayer(case["rows"], case["k"], case["n"], case["m"], case["block_rows"], case["block_k"],
                          _keep(case, case["k"]))
        s = _saliency(g, w)
        L.build_mask(s).encode(w)                  # the layer's buffers, as every later iteration finds them
        return {"kind": kind, "layer": L, "w": w, "s": s}
    shapes = _shapes(case)
    weights = [_weight(g, r, k) for r, k in shapes]
    grads = [[_normal(g, s, 1e-2).to(torch.bfloat16) for _ in range(case["samples"])] for s in shapes]
    net = B.PruningNetwork(shapes, case["n"], case["m"], case["block_rows"], case["block_k"])
    net.step(weights, grads, case["kappa"])        # the network's buffers, as every later iteration finds them
    return {"kind": kind, "net": net, "weights": weights, "grads": grads, "kappa": case["kappa"]}


def run(state):
    kind = state["kind"]
    if kind == "product":
        return state["layer"].spmm(state["x"], y=state["y"], y_dtype=state["y_dtype"])
    if kind == "conv":
        x, kn = state["x"], state["kernel"]
        for L, y in zip(state["layers"], state["outs"]):
            x = L.spmm_conv(x, kn, kn, kn // 2, y=y, nhwc_out=state["nhwc_out"])
        return state["outs"]
    if kind == "compress":
        L = state["layer"]
        L.build_mask(state["s"]).encode(state["w"])
        return L.decode()
    net = state["net"]
    kept = net.step(state["weights"], state["grads"], state["kappa"])
    return [np.array(kept, dtype=np.int64)] + [L.decode() for L in net.layers]


# ------------------------------------------------------------------------------------------------ the results in 64 bits

def _pruned64(case, g, rows, k):
    """The pruned weight matrix of _layer(case, g, rows, k), from the definition of the pattern, as float64 [rows, k]."""
    w = _weight(g, rows, k)
    s = _saliency(g, w).double()
    bm, bk, n, m = case["block_rows"], case["block_k"], case["n"], case["m"]
    nrt, nblk, kkeep = _blocks(case, rows, k)
    s = torch.nn.functional.pad(s, (0, nblk * bk - k, 0, nrt * bm - rows))
    # the n largest of every m consecutive elements, the lower index first among equals
    groups = s.view(-1, m)
    order = torch.sort(groups, dim=1, descending=True, stable=True).indices[:, :n]
    kept = torch.zeros_like(groups).scatter_(1, order, 1.0)
    # the kkeep blocks of every row tile with the largest sums of what is left
    score = (groups * kept).view(nrt, bm, nblk, bk).sum(dim=(1, 3))
    best = torch.sort(score, dim=1, descending=True, stable=True).indices[:, :kkeep]
    blocks = torch.zeros_like(score).scatter_(1, best, 1.0)
    kept = kept.view(nrt, bm, nblk, bk) * blocks[:, None, :, None]
    return w.double() * kept.view(nrt * bm, nblk * bk)[:rows, :k]


def exact(case, seed):
    """What run returns for these inputs in float64; None where the outputs are bytes and integers."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["kind"] == "product":
        w = _pruned64(case, g, case["rows"], case["k"])
        bias = _normal(g, (case["rows"],), 0.1).double() if case["bias"] else None
        y = w @ _activation(g, (case["k"], case["ncols"])).double()
        if bias is not None:
            y += bias[:, None]
        return y.clamp_(min=0) if case["relu"] else y
    if case["kind"] == "conv":
        kn, rows, c, layers = case["kernel"], case["rows"], case["channels"], []
        for _ in range(case["layers"]):
            w = _pruned64(case, g, rows, kn * kn * c)
            layers.append((w.view(rows, kn, kn, c), _normal(g, (rows,), 0.1).double()))
            c = rows
        x, outs = _activation(g, (case["batch"], case["side"], case["side"], case["channels"])), []
        for w, bias in layers:
            out = torch.empty(x.shape[:3] + (rows,), dtype=torch.float64, device="cuda")
            for b in range(x.shape[0]):                       # one image at a time, filter tap by filter tap
                p = torch.nn.functional.pad(x[b].double(), (0, 0, kn // 2, kn // 2, kn // 2, kn // 2))
                acc = bias.expand(x.shape[1], x.shape[2], rows).clone()
                for i in range(kn):
                    for j in range(kn):
                        acc += p[i:i + x.shape[1], j:j + x.shape[2]] @ w[:, i, j].t()
                out[b] = acc.clamp_(min=0)
            outs.append(out)
            x = out
        return outs if case["nhwc_out"] else [o.reshape(-1, rows).t().contiguous() for o in outs]
    return None


# ------------------------------------------------------------------------------------------------ work and tolerance

def _shapes(case):
    return [(layer.rows, layer.k) for layer in NETWORKS[case["network"]]()]


def _blocks(case, rows, k):
    """-> (row tiles, blocks per row tile, kept blocks per row tile)"""
    nrt, nblk = math.ceil(rows / case["block_rows"]), math.ceil(k / case["block_k"])
    kkeep = min(nblk, math.floor(_keep(case, k) * nblk + 0.5))
    return nrt, nblk, kkeep


def _encoding_bytes(case, rows, k, kkeep):
    nrt = math.ceil(rows / case["block_rows"])
    nnz = nrt * kkeep * case["block_rows"] * case["block_k"] * case["n"] // case["m"]
    return 2 * nnz + nnz * (2 if case["m"] == 4 else 3) // 8 + 4 * nrt * kkeep, nnz


def work(case):
    if case["kind"] in ("product", "conv"):
        total_bytes, flops = 0, 0
        k, layers = case.get("k"), case.get("layers", 1)
        for i in range(layers):
            if case["kind"] == "conv":
                c = case["channels"] if i == 0 else case["rows"]
                k, ncols = case["kernel"] ** 2 * c, case["batch"] * case["side"] ** 2
            else:
                c, ncols = k, case["ncols"]
            nrt, nblk, kkeep = _blocks(case, case["rows"], k)
            enc, nnz = _encoding_bytes(case, case["rows"], k, kkeep)
            touched = 1.0 - (1.0 - kkeep / nblk) ** nrt           # share of the blocks that some row tile keeps
            x_rows = c if case["kind"] == "conv" else c * touched
            total_bytes += enc + 2 * ncols * x_rows + (4 if case.get("f32") else 2) * case["rows"] * ncols
            flops += 2.0 * nnz * ncols
        return {"bytes": total_bytes, "flops": flops}
    if case["kind"] == "compress":
        rows, k = case["rows"], case["k"]
        _, nblk, kkeep = _blocks(case, rows, k)
        # saliency and the kept half of W in; bits, encoding and pruned weights out
        return {"bytes": rows * k * (4 + 2.0 * kkeep / nblk + 1 / 8 + 2) + _encoding_bytes(case, rows, k, kkeep)[0],
                "flops": 2.0 * rows * k}
    params = sum(r * k for r, k in _shapes(case))
    density = 1.0 - case["kappa"]
    # gradients and weights in; bits, values with their offsets and pruned weights out
    return {"bytes": params * (2.0 * case["samples"] + 2 + 1 / 8 + 2 + density * 2.4), "flops": params * (case["samples"] + 4.0)}


def tolerance(case):
    if case["kind"] in ("compress", "prune"):
        return "exact"
    # Against the product in 64 bits: bf16 results differ by 1.7e-3 (their rounding), by 2.4e-3 after three layers in a
    # row, fp32 results by up to 4e-7 for sums of 2048 terms; about four times that, and twice as much for the longest sums.
    if case.get("f32"):
        return {"rel": 4e-6}
    return {"rel": 7e-3 if case.get("layers", 1) == 1 else 1e-2}
