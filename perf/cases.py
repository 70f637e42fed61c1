"""The work that is timed: whole networks, single layers in their three input codings, the bare contraction, the coding
of weight matrices and the training-side step, each through the package's public calls.

listed() are fixed sizes, draw() others of the same ranges.  Sizes are those of dab_synth.configs and
dab_synth.networks or generic ones; inputs have the distributions those workloads have (post-ReLU activations with 60 %
exact zeros, N(0, 1) activations with both signs behind a normalisation layer, Laplace or normal weight rows, sparse
stroke images).  Filters are coded in prepare(): a program that runs inference codes them once and keeps them.
"""
import functools
import math

import torch

import paper_1804_02941_b200 as dab
from dab_synth import networks

NETWORKS = {"sketch_a_net": networks.sketch_a_net, "alexnet_like": networks.alexnet_like,
            "resnet18_like": networks.resnet18_like}
MAX_VALUES = 4.6e8   # patch values (patches x row length) of a drawn layer: those of the largest listed one
MAX_MACS = 3.0e10    # multiply-accumulates of a drawn layer: those of the largest listed one


def _conv(name, coding, N, C, H, Cout, k, stride=1, pad=0, zeros=0.6, W=None):
    return {"name": name, "kind": "conv", "coding": coding, "N": N, "C": C, "H": H, "W": H if W is None else W,
            "Cout": Cout, "k": k, "stride": stride, "pad": pad, "zeros": zeros}


def listed():
    return [
        # a sketch classified as it is drawn: one image through the Sketch-A-Net-shaped network, where latency counts
        {"name": "net_sketch_b1", "kind": "net", "net": "sketch_a_net", "batch": 1},
        # batched inference through the two larger network shapes (layers before and behind the binarized ones included)
        {"name": "net_alexnet_b32", "kind": "net", "net": "alexnet_like", "batch": 32},
        {"name": "net_resnet18_b32", "kind": "net", "net": "resnet18_like", "batch": 32},
        # one small layer at batch 1: 64 -> 64 channels on 32 x 32
        _conv("conv_64x32_b1", "dab", 1, 64, 32, 64, 3, 1, 1),
        # the layer that a ResNet-18-shaped stack at batch 256 spends most of its time in
        _conv("conv_64x56_b256", "dab", 256, 64, 56, 64, 3, 1, 1),
        # a deeper layer behind a normalisation layer (both signs, no zeros), the last and odd batch of an epoch
        _conv("conv_256x14_b61_signed", "dab", 61, 256, 14, 256, 3, 1, 1, zeros=0.0),
        # a 5 x 5 layer of an AlexNet-shaped network, odd sizes throughout
        _conv("conv5x5_96x27_b37", "dab", 37, 96, 27, 256, 5, 1, 2),
        # the paper's fully binarized layers with XNOR-style inputs
        _conv("conv_sign_128x28_b256", "sign", 256, 128, 28, 128, 3, 1, 1),
        # the paper's weights-only binarized layers: full-precision activations
        _conv("conv_wbin_256x14_b256", "wbin", 256, 256, 14, 256, 3, 1, 1),
        # the bare contraction of two coded matrices, the largest of the sweep
        {"name": "gemm_8192x8192x4608", "kind": "gemm", "M": 8192, "N": 8192, "n": 4608},
        # coding the weights of a fully connected layer (9216 -> 4096): loading a model, or a step of its training
        {"name": "rows_4096x9216", "kind": "rows", "rows": 4096, "n": 9216, "dist": "normal"},
        # forward and backward of the weight binarization of a 512 -> 512 3 x 3 layer in one training step
        {"name": "train_512x4608", "kind": "train", "rows": 512, "n": 4608},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_conv(rng):
    while True:
        k = rng.choice((1, 3, 3, 3, 5))
        c = {"kind": "conv", "coding": rng.choice(("dab", "dab", "dab", "sign", "wbin")), "N": _log(rng, 1, 256),
             "C": _log(rng, 16, 512), "H": _log(rng, 6, 60), "W": 0, "Cout": _log(rng, 16, 512), "k": k,
             "stride": rng.choice((1, 1, 1, 2)), "pad": rng.choice((0, k // 2)), "zeros": rng.choice((0.6, 0.6, 0.0))}
        c["W"] = max(k, c["H"] + rng.choice((0, 0, -1, 3)))
        if c["C"] * k * k > 8192:
            continue
        n, patches, _, _ = _conv_sizes(c)
        if patches * n <= MAX_VALUES and patches * n * c["Cout"] <= MAX_MACS:
            return c


def draw(rng):
    kind = rng.choice(("conv", "conv", "conv", "conv", "net", "gemm", "rows", "train"))
    if kind == "conv":
        return _draw_conv(rng)
    if kind == "net":
        return {"kind": "net", "net": rng.choice(sorted(NETWORKS)), "batch": _log(rng, 1, 32)}
    if kind == "gemm":
        return {"kind": "gemm", "M": _log(rng, 64, 8192), "N": _log(rng, 64, 8192), "n": _log(rng, 256, 4608)}
    if kind == "rows":
        return {"kind": "rows", "rows": _log(rng, 64, 4096), "n": _log(rng, 256, 9216),
                "dist": rng.choice(("normal", "laplace"))}
    return {"kind": "train", "rows": _log(rng, 64, 1024), "n": _log(rng, 128, 4608)}


def _conv_sizes(c):
    """Row length, patches, Ho, Wo."""
    ho = (c["H"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1
    wo = (c["W"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1
    return c["C"] * c["k"] * c["k"], c["N"] * ho * wo, ho, wo


@functools.lru_cache(maxsize=None)
def _network(name):
    return NETWORKS[name]()


def _laplace(shape, b, g):
    u = torch.rand(shape, device="cuda", generator=g) - 0.5
    return -b * torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp(max=0.4999999))


def _coded(rows, n, g):
    return dab.dab_binarize(_laplace((rows, n), 0.05, g))


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    if kind == "net":
        layers, shape = _network(case["net"])
        x = torch.from_numpy(networks.network_input(shape, case["batch"], seed)).cuda()
        return {"case": case, "net": dab.Network(layers), "x": x}
    if kind == "conv":
        x = torch.randn((case["N"], case["C"], case["H"], case["W"]), device="cuda", generator=g)
        if case["zeros"] > 0:
            x = x.abs() * (torch.rand(x.shape, device="cuda", generator=g) >= case["zeros"])
        n = case["C"] * case["k"] * case["k"]
        w = torch.randn((case["Cout"], n), device="cuda", generator=g) * math.sqrt(2.0 / n)
        return {"case": case, "x": x, "w": dab.dab_binarize(w)}
    if kind == "gemm":
        return {"case": case, "a": _coded(case["M"], case["n"], g), "b": _coded(case["N"], case["n"], g)}
    if kind == "rows":
        shape = (case["rows"], case["n"])
        values = _laplace(shape, 0.05, g) if case["dist"] == "laplace" else torch.randn(shape, device="cuda", generator=g) * 0.01
        return {"case": case, "values": values}
    shape = (case["rows"], case["n"])
    return {"case": case, "W": torch.randn(shape, device="cuda", generator=g) * 0.02,
            "grad": torch.randn(shape, device="cuda", generator=g)}


def _codes(c):
    return {"mask": c.mask, "K": c.K, "alpha": c.alpha, "beta": c.beta, "flags": c.flags}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "net":
        return dab.dab_network_forward(state["net"], state["x"])
    if kind == "conv":
        geometry = (case["k"], case["k"], (case["stride"], case["stride"]), (case["pad"], case["pad"]))
        if case["coding"] == "wbin":
            return dab.dab_wbin_conv(state["x"], state["w"], *geometry)
        return dab.dab_binary_conv(state["x"], state["w"], *geometry, sign_inputs=case["coding"] == "sign")
    if kind == "gemm":
        return dab.dab_binary_gemm(state["a"], state["b"])
    if kind == "rows":
        return _codes(dab.dab_binarize(state["values"]))
    Wc, coded, Wt = dab.dab_binarize_train(state["W"])
    return {"Wc": Wc, "Wt": Wt, "grad_W": dab.dab_binarize_backward(Wc, coded, state["grad"]), **_codes(coded)}


def _code_bytes(rows, n):
    return rows * (4 * dab.dab_default_ld(n) + 16)


def _net_work(name, batch):
    """Multiply-accumulates of every convolution; weights (full-precision or coded), the images and the logits once."""
    layers, (c, h, w) = _network(name)
    flops, size = 0, 4 * batch * c * h * w
    saved = None
    for l in layers:
        if l["kind"] == "save":
            saved = (c, h, w)
        if "kh" not in l:
            continue
        ci, hi, wi = saved if l.get("on_saved") else (c, h, w)
        ho = (hi + 2 * l["pad"][0] - l["kh"]) // l["stride"][0] + 1
        wo = (wi + 2 * l["pad"][1] - l["kw"]) // l["stride"][1] + 1
        co = l.get("Cout", ci)
        if l["kind"] != "maxpool":
            n = ci * l["kh"] * l["kw"]
            flops += 2 * batch * ho * wo * co * n
            size += _code_bytes(co, n) if l["kind"] == "conv_binary" else 4 * co * n
        if l.get("on_saved"):
            saved = (co, ho, wo)
        else:
            c, h, w = co, ho, wo
    return {"bytes": size + 4 * batch * c * h * w, "flops": flops}


def work(case):
    """A multiply-accumulate on two coded values counts as two operations.  The search for the best split of a row has
    no agreed operation count and is left out."""
    kind = case["kind"]
    if kind == "net":
        return _net_work(case["net"], case["batch"])
    if kind == "conv":
        n, patches, _, _ = _conv_sizes(case)
        x = 4 * case["N"] * case["C"] * case["H"] * case["W"]
        return {"bytes": x + _code_bytes(case["Cout"], n) + 4 * patches * case["Cout"], "flops": 2 * patches * n * case["Cout"]}
    if kind == "gemm":
        M, N, n = case["M"], case["N"], case["n"]
        return {"bytes": _code_bytes(M, n) + _code_bytes(N, n) + 4 * M * N, "flops": 2 * M * N * n}
    rows, n = case["rows"], case["n"]
    if kind == "rows":
        return {"bytes": 4 * rows * n + _code_bytes(rows, n), "flops": 0}
    # W read, W_real and the dense filters written; W_real and the upstream gradient read, the gradient written
    return {"bytes": 4 * rows * n * 5 + _code_bytes(rows, n), "flops": 0}


def tolerance(case):
    """Codes are whole numbers and equal (K, masks and flags differ in nothing).  Scales and outputs are sums in fp64,
    or exact integer sums, rounded once to fp32: another order of the terms moves the last bit of one output in about
    1e8, which leaves most networks as they are.  Where such a bit moves a value across a threshold, or a split between
    two near-ties, the layers behind it see another code: with the first layer's weights moved by one last bit each,
    the logits of 32 images differed by 0 to 6 % (measured), nearly all of it in one image."""
    if case["kind"] == "net":
        return {"rel": 0.02, "max": 0.3}
    return {"rel": 1e-6}
