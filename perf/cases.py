"""The work a user of this package has it do, as measurable cases.

Families and the public entry points they go through (paper_2512_14090_b200.binding):

  linear    aiq_qlinear: y = x * dequant(W)^T with packed weights, the memory-bound layer the method targets
  quantize  aiq_quantize_layer (and its per-tensor variant): one weight matrix to codes and scales
  forward   Model.aiq_forward: one scheme, one image batch, logits
  eval      Model.aiq_eval_schemes: many candidate schemes on an evaluation set (what both searches call)
  load      Model(...) and the first batch: fold and quantize a checkpoint, then serve

Every array is drawn on the GPU from the case's seed; network parameters come from aiq_workloads.gen_model.
"""
import math

import numpy as np
import torch

from paper_2512_14090_b200 import binding as aiq
from aiq_workloads import (resnet20, heavy_early_resnet20, plain_convnet20, mobilenet_v2, gen_model,
                           gen_random_scheme, mixed_int4_int8_scheme, one_layer_lowered_schemes,
                           coordinate_step_schemes, conv_layer_indices)

NETS = {
    "resnet20": resnet20,
    "heavy_early_resnet20": heavy_early_resnet20,
    "plain_convnet20": plain_convnet20,
    "mobilenet_v2_cifar": lambda: mobilenet_v2("cifar"),
    "mobilenet_v2_imagenet": lambda: mobilenet_v2("imagenet"),
}


def listed():
    return [
        # the classifier-sized layer of MobileNetV2's head, one row: nothing but latency
        dict(name="linear_head_i8_m1", family="linear", n=1280, k=320, bits=8, m=1, bias=True),
        # single-row inference on a large layer at 4 bits: the weight stream
        dict(name="linear_8192_i4_m1", family="linear", n=8192, k=8192, bits=4, m=1, bias=False),
        # a small batch on a 16-bit layer, between the weight stream and the tensor cores
        dict(name="linear_4096_f16_m16", family="linear", n=4096, k=4096, bits=16, m=16, bias=False),
        # the largest batch of the linear sweep
        dict(name="linear_8192_i8_m256", family="linear", n=8192, k=8192, bits=8, m=256, bias=False),
        # packing a large layer
        dict(name="quantize_8192_i4", family="quantize", n=8192, k=8192, bits=4, per_tensor=False),
        # CIFAR ResNet-20 under a scheme that mixes all four bit-widths, one ordinary batch
        dict(name="forward_resnet20_b64", family="forward", net="resnet20", batch=64, scheme="mixed"),
        # MobileNetV2 on CIFAR shapes, ten layers at 4 bits: a single image, and a large batch
        dict(name="forward_mbv2_cifar_b1", family="forward", net="mobilenet_v2_cifar", batch=1, scheme="int4_int8"),
        dict(name="forward_mbv2_cifar_b256", family="forward", net="mobilenet_v2_cifar", batch=256, scheme="int4_int8"),
        # MobileNetV2 on ImageNet shapes, uniform 8 bits, a serving batch
        dict(name="forward_mbv2_imagenet_b32", family="forward", net="mobilenet_v2_imagenet", batch=32, scheme="int8"),
        # a step of the greedy search: 21 candidates, one layer of an all-8 scheme lowered to 4, 10,000 images
        dict(name="eval_resnet20_greedy", family="eval", net="resnet20", images=10000, schemes="greedy", base=8,
             low=4, count=21, chunk=5008),
        # a coordinate-descent step: 52 candidates that move one layer of an all-8 MobileNetV2 to 32, 16 or 4 bits
        dict(name="eval_mbv2_imagenet_cd", family="eval", net="mobilenet_v2_imagenet", images=512,
             schemes="coordinate", base=8, low=4, count=52, chunk=32),
        # loading a checkpoint: fold, quantize at every bit-width, first single-image answer
        dict(name="load_mbv2_imagenet", family="load", net="mobilenet_v2_imagenet", batch=1, scheme="int8"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    family = rng.choice(["linear", "linear", "linear", "quantize", "forward", "forward", "forward", "eval", "eval", "load"])
    if family == "linear":
        # half of them rows a multiple of 32 long, as layers usually are; the rest of any length
        n, k = _log_int(rng, 64, 8192), _log_int(rng, 64, 8192)
        if rng.random() < 0.5:
            k = max(64, k // 32 * 32)
        return dict(family="linear", n=n, k=k, bits=rng.choice([4, 8, 16, 32]), m=_log_int(rng, 1, 256),
                    bias=rng.random() < 0.5)
    if family == "quantize":
        n, k = _log_int(rng, 64, 8192), _log_int(rng, 64, 8192)
        if rng.random() < 0.5:
            k = max(64, k // 32 * 32)
        return dict(family="quantize", n=n, k=k, bits=rng.choice([4, 8, 16, 32]), per_tensor=rng.random() < 0.25)
    if family in ("forward", "load"):
        return dict(family=family, net=rng.choice(sorted(NETS)), batch=_log_int(rng, 1, 256 if family == "forward" else 16),
                    scheme=rng.choice(["mixed", "int4_int8", "int8", "int8", "float32"]))
    net = rng.choice(["resnet20", "resnet20", "heavy_early_resnet20", "plain_convnet20", "mobilenet_v2_cifar",
                      "mobilenet_v2_imagenet"])
    most = {"resnet20": 10000, "heavy_early_resnet20": 2500, "plain_convnet20": 1000, "mobilenet_v2_cifar": 1000,
            "mobilenet_v2_imagenet": 256}[net]
    chunk = {"resnet20": 5008, "heavy_early_resnet20": 1024, "plain_convnet20": 1024, "mobilenet_v2_cifar": 256,
             "mobilenet_v2_imagenet": 32}[net]
    base = rng.choice([8, 8, 32])
    return dict(family="eval", net=net, images=_log_int(rng, 96, most), schemes=rng.choice(["greedy", "coordinate"]),
                base=base, low=4 if base == 8 else rng.choice([8, 4]), count=rng.randint(4, 20), chunk=chunk)


def _scheme(arch, kind):
    L = len(arch["layers"])
    if kind == "mixed":
        return gen_random_scheme(L, 42)
    if kind == "int4_int8":
        return mixed_int4_int8_scheme(L, conv_layer_indices(arch), 10, 43)
    return np.full(L, {"int8": 8, "float32": 32}[kind], np.uint8)


def _schemes(arch, case):
    cand = conv_layer_indices(arch)
    # `count` candidates spread evenly over the network's depth
    pick = [cand[i * len(cand) // case["count"]] for i in range(case["count"])] if case["count"] < len(cand) else cand
    L = len(arch["layers"])
    if case["schemes"] == "greedy":
        return one_layer_lowered_schemes(L, pick, base=case["base"], low=case["low"])
    return coordinate_step_schemes(L, pick, base=case["base"], alternatives=(16, 8, 4) if case["base"] == 32 else (32, 16, 4))


def _randn(shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda")


def prepare(case, seed):
    family = case["family"]
    if family == "linear":
        n, k, bits, m = case["n"], case["k"], case["bits"], case["m"]
        w = _randn((n, k), 3 * seed) * 0.02
        packed = torch.empty(n * aiq.aiq_packed_row_bytes(k, bits), dtype=torch.uint8, device="cuda")
        scales = torch.empty(n, device="cuda")
        aiq.aiq_quantize_layer(w, bits, packed, scales)
        ws = aiq.aiq_qlinear_workspace_bytes(n, k, bits, m)
        return dict(case=case, packed=packed, scales=scales, bias=_randn((n,), 3 * seed + 2) * 0.1 if case["bias"] else None,
                    x=_randn((m, k), 3 * seed + 1), y=torch.empty((m, n), device="cuda"),
                    ws=torch.empty(ws, dtype=torch.uint8, device="cuda") if ws else None)
    if family == "quantize":
        n, k, bits = case["n"], case["k"], case["bits"]
        return dict(case=case, w=_randn((n, k), seed) * 0.02,
                    packed=torch.empty(n * aiq.aiq_packed_row_bytes(k, bits), dtype=torch.uint8, device="cuda"),
                    scales=torch.empty(n, device="cuda"), flag=torch.zeros(1, dtype=torch.int32, device="cuda"),
                    scratch=torch.zeros(1, dtype=torch.int32, device="cuda"))
    arch = NETS[case["net"]]()
    params = gen_model(arch, seed)
    image = (arch["in_c"], arch["in_h"], arch["in_w"])
    model = aiq.Model(arch, params)
    if family in ("forward", "load"):
        batch = case["batch"]
        return dict(case=case, model=model, arch=arch, params=params, scheme=_scheme(arch, case["scheme"]),
                    x=_randn((batch,) + image, seed + 1), logits=torch.empty((batch, model.n_classes), device="cuda"),
                    ws=torch.empty(model.aiq_workspace_bytes(batch, 1), dtype=torch.uint8, device="cuda"))
    images, schemes = case["images"], _schemes(arch, case)
    x = _randn((images,) + image, seed + 1)
    # A trained network spreads its answers over the classes; one with random weights puts nearly every image into
    # one.  Taking most of the mean logits (to three decimals) out of the classifier's bias gives it such answers.
    mean = model.aiq_forward(np.full(model.n_layers, 32, np.uint8), x[:64]).mean(0).cpu().numpy()
    params[-1]["bias"] = params[-1]["bias"] - np.round(np.float32(0.9) * mean, 3)
    model = aiq.Model(arch, params)
    chunk = min(case["chunk"], images)
    aiq.aiq_set_eval_options(chunk, True)
    ws = torch.empty(model.aiq_workspace_bytes(chunk, len(schemes)), dtype=torch.uint8, device="cuda")
    # labels: what the full-precision model answers
    labels = torch.empty((1, images), dtype=torch.int32, device="cuda")
    model.aiq_eval_schemes(np.full((1, model.n_layers), 32, np.uint8), x, torch.zeros(images, dtype=torch.int32, device="cuda"),
                           preds=labels, workspace=ws)
    return dict(case=case, model=model, params=params, x=x, labels=labels[0], schemes=schemes, ws=ws, chunk=chunk,
                preds=torch.empty((len(schemes), images), dtype=torch.int32, device="cuda"))


def run(s):
    case = s["case"]
    family = case["family"]
    if family == "linear":
        aiq.aiq_qlinear(s["packed"], s["scales"], s["bias"], case["n"], case["k"], case["bits"], s["x"], s["y"], workspace=s["ws"])
        return s["y"]
    if family == "quantize":
        if case["per_tensor"]:
            aiq.aiq_quantize_layer_per_tensor(s["w"], case["bits"], s["packed"], s["scales"], s["scratch"], nonfinite_flag=s["flag"])
        else:
            aiq.aiq_quantize_layer(s["w"], case["bits"], s["packed"], s["scales"], nonfinite_flag=s["flag"])
        return s["packed"], s["scales"], s["flag"]
    if family == "forward":
        return s["model"].aiq_forward(s["scheme"], s["x"], logits=s["logits"], workspace=s["ws"])
    if family == "load":
        model = aiq.Model(s["arch"], s["params"], mem=s["model"].mem)
        logits = model.aiq_forward(s["scheme"], s["x"], logits=s["logits"], workspace=s["ws"])
        # the packed weights the scheme serves from, one view per layer
        packed = [model.layer_packed(i, int(b))[0] for i, b in enumerate(s["scheme"])]
        return logits, packed
    aiq.aiq_set_eval_options(s["chunk"], True)
    acc, _ = s["model"].aiq_eval_schemes(s["schemes"], s["x"], s["labels"], preds=s["preds"], workspace=s["ws"])
    return acc, s["preds"]


def _shapes(arch):
    """Per layer (weights, output pixels)."""
    out = []
    done = {-1: (arch["in_h"], arch["in_w"])}
    todo = list(range(len(arch["layers"])))
    while todo:
        for i in list(todo):
            l = arch["layers"][i]
            if l["input"] in done:
                h, w = done[l["input"]]
                done[i] = (1, 1) if l["kind"] == "fc" else ((h + 2 * l["pad"] - l["k"]) // l["stride"] + 1,
                                                            (w + 2 * l["pad"] - l["k"]) // l["stride"] + 1)
                todo.remove(i)
    for i, l in enumerate(arch["layers"]):
        cin = 1 if l["kind"] == "dw" else l["cin"]
        out.append((l["cout"] * cin * l["k"] * l["k"], done[i][0] * done[i][1]))
    return out


def _versions(arch, schemes):
    """Distinct evaluations of every layer: candidates that agree on all of a layer's ancestors share its output."""
    layers, ver, count = arch["layers"], {-1: [0] * len(schemes)}, {}
    todo = list(range(len(layers)))
    while todo:
        for i in list(todo):
            l = layers[i]
            if l["input"] in ver and l["residual"] in ver:
                keys = [(int(s[i]), a, b) for s, a, b in zip(schemes, ver[l["input"]], ver[l["residual"]])]
                ids = {k: j for j, k in enumerate(dict.fromkeys(keys))}
                ver[i], count[i] = [ids[k] for k in keys], len(ids)
                todo.remove(i)
    return [count[i] for i in range(len(layers))]


def work(case):
    family = case["family"]
    if family == "linear":
        n, k, m = case["n"], case["k"], case["m"]
        return dict(bytes=n * k * case["bits"] / 8 + 4 * n + 4 * m * (k + n), flops=2 * m * n * k)
    if family == "quantize":
        n, k = case["n"], case["k"]
        return dict(bytes=n * k * (4 + case["bits"] / 8) + 4 * n, flops=2 * n * k)
    arch = NETS[case["net"]]()
    shapes = _shapes(arch)
    image = 4 * arch["in_c"] * arch["in_h"] * arch["in_w"]
    weights = sum(w for w, _ in shapes)
    if family in ("forward", "load"):
        scheme = _scheme(arch, case["scheme"])
        out = case["batch"] * (image + 4 * arch["n_classes"])
        flops = 2 * case["batch"] * sum(w * p for w, p in shapes)
        if family == "load":        # float32 parameters in; folded weights and the four widths out
            return dict(bytes=weights * (4 + 4 + 7.5) + out, flops=flops)
        return dict(bytes=sum(w * int(b) / 8 for (w, _), b in zip(shapes, scheme)) + out, flops=flops)
    schemes = _schemes(arch, case)
    versions = _versions(arch, schemes)
    used = sum(w * int(b) / 8 for i, (w, _) in enumerate(shapes) for b in {int(s[i]) for s in schemes})
    return dict(bytes=case["images"] * (image + 4 + 4 * len(schemes)) + used,
                flops=2 * case["images"] * sum(w * p * v for (w, p), v in zip(shapes, versions)))


def tolerance(case):
    """Four times what the package's own compute paths (float32 kernels, two tensor-core formulations, layer by
    layer or fused) were seen to differ by from one another, or a layer's result from its float64 value."""
    if case["family"] == "quantize":
        return "exact"
    if case["family"] == "linear":
        return {"rel": 3e-5, "max": 2e-4}
    mobilenet = case["net"].startswith("mobilenet")
    if case["family"] in ("forward", "load"):       # the packed weights of "load" are bytes: none may differ
        return {"rel": 1e-3, "max": 4e-3} if mobilenet else {"rel": 1.6e-4, "max": 4e-4}
    # Predictions change where an image's two largest logits are closer than the logits' own error (seen: 2e-4 of
    # them on the residual networks, 1e-3 on the plain and the MobileNet ones); an accuracy moves by 1 / images for
    # each, against accuracies of 0.1 and more.
    differ = {"resnet20": 8e-4, "heavy_early_resnet20": 8e-4}.get(case["net"], 5e-3)
    total = case["images"] * case["count"]
    differ = max(differ, 3 / total)
    return {"rel": min(0.03, math.sqrt(differ / total) / 0.1), "differ": differ}
