"""The work that programs on this library spend their time in, as measurable cases.

Three kinds, all through the public Python entry points:

``model``   one pass of a whole pruned network (``PrunedNetwork``): selection, slicing, planning and packing belong to the
            preparation, the pass takes float32 images to float32 logits.  ``mode`` says how the program calls it:
            "graph" (device buffers, the launch sequence replayed as a CUDA graph: a serving loop), "eager" (device
            buffers, every launch enqueued by the call: the default of ``run``) or "host" (pinned host images in, host
            logits out).  ``keep`` is the percentage of filters every prunable layer keeps; 0 takes the layer table's
            own counts.
``task``    one fused conv task (conv + bias + activation, optionally + residual) with the buffers the caller keeps: the
            unit that a pruning loop times and a program with its own executor calls.
``select``  L1-norm selection of one layer's filters and the slicing of the layer and of its consumer.

Inputs are standard normal, weights Kaiming-normal on the full layer, biases N(0, 0.01^2), as everywhere in this
repository.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as wl
import paper_2207_01260_b200 as cp
from paper_2207_01260_b200.pipeline import PrunedNetwork


def _model(name, model, batch, mode="graph", keep=0):
    return {"name": name, "kind": "model", "model": model, "batch": batch, "mode": mode, "keep": keep}


def _task(name, batch, C, hw, K, R, stride, act, groups=1, residual=False):
    return {"name": name, "kind": "task", "batch": batch, "C": C, "hw": hw, "K": K, "R": R, "stride": stride, "act": act,
            "groups": groups, "residual": residual}


def listed():
    return [
        # throughput serving and the repository's benchmark: a full batch of ImageNet-sized images
        _model("resnet18 batch 64", "resnet18", 64),
        _model("mobilenet_v2 batch 64", "mobilenet_v2", 64),
        # the same for the CIFAR-sized network
        _model("vgg16 batch 128", "vgg16_cifar", 128),
        # latency serving: one image at a time
        _model("resnet18 batch 1", "resnet18", 1),
        _model("mobilenet_v2 batch 1", "mobilenet_v2", 1),
        _model("vgg16 batch 1", "vgg16_cifar", 1),
        # a ragged batch of the network with 5x5 depthwise layers, through the plain (eager) call
        _model("mnasnet batch 20 eager", "mnasnet1_0", 20, mode="eager", keep=60),
        # shortcut-aware pruning (block outputs pruned too), images and logits in host memory
        _model("resnet18 shared batch 6 host", "resnet18_shared", 6, mode="host"),
        # a step of the sweep over the kept filters that a pruning loop walks: odd channel counts, full batch
        _task("conv 3x3 131 to 203 batch 64", 64, 131, 28, 203, 3, 1, "relu"),
        # a depthwise layer of a pruned inverted-residual block
        _task("depthwise 3x3 108 batch 64", 64, 108, 56, 108, 3, 1, "relu6", groups=108),
        # the smallest call: one pruned layer on one small image (64 filters of which 48 are kept, 32x32)
        _task("conv 3x3 64 to 48 batch 1", 1, 64, 32, 48, 3, 1, "relu"),
        # pruning one of the widest layers together with its consumer
        {"name": "select 358 of 512", "kind": "select", "K": 512, "C": 512, "R": 3, "keep": 358, "K2": 512, "R2": 3, "depthwise": False},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    u = rng.random()
    if u < 0.5:
        model = rng.choice(["resnet18", "resnet18_shared", "mobilenet_v2", "mnasnet1_0", "vgg16_cifar"])
        batch = _log_int(rng, 1, 112 if model == "vgg16_cifar" else 48)
        return {"kind": "model", "model": model, "batch": batch, "mode": rng.choice(["graph", "graph", "graph", "eager", "host"]),
                "keep": rng.randint(40, 80)}
    if u < 0.85:
        s = rng.choice(wl.sweep_shapes())
        depthwise = s["groups"] > 1
        C = s["C"] if s["C"] < 16 else rng.randint(s["C"] // 2, s["C"])
        K = C if depthwise else rng.randint(max(1, s["K"] // 4), s["K"])
        return {"kind": "task", "batch": _log_int(rng, 1, 64), "C": C, "hw": s["H"], "K": K, "R": s["R"], "stride": s["stride"],
                "act": s["act"], "groups": C if depthwise else 1, "residual": not depthwise and s["stride"] == 1 and rng.random() < 0.25}
    K, R, depthwise = _log_int(rng, 24, 1280), rng.choice([1, 3]), rng.random() < 0.3
    return {"kind": "select", "K": K, "C": _log_int(rng, 16, 512), "R": R, "keep": rng.randint(K // 4, K),
            "K2": _log_int(rng, 16, 512), "R2": 3 if depthwise else rng.choice([1, 3]), "depthwise": depthwise}


# ------------------------------------------------------------------------------------------------ models

def _table(case):
    k, name = case["keep"], case["model"]
    if k == 0:
        return wl.MODELS[name]()
    if name == "vgg16_cifar":
        return wl.vgg16_cifar([max(1, w * k // 100) for w in wl.VGG16_WIDTHS])
    if name == "resnet18":
        return wl.resnet18(k, 100)
    if name == "resnet18_shared":
        return wl.resnet18(k, 100, k, 100)
    return {"mobilenet_v2": wl.mobilenet_v2, "mnasnet1_0": wl.mnasnet1_0}[name](k, 100)


def _weights(table, rng):
    out = {}
    for l in table["layers"]:
        if l["kind"] == "conv":
            shape = (l["K"], l["C"] // l["groups"], l["R"], l["S"])
        elif l["kind"] == "fc":
            shape = (l["out_features"], l["in_features"])
        else:
            continue
        fan_in = int(np.prod(shape[1:]))
        w = rng.standard_normal(shape, dtype=np.float32) * np.float32(math.sqrt(2.0 / fan_in))
        out[l["name"]] = (w, rng.standard_normal(shape[0], dtype=np.float32) * np.float32(0.01))
    return out


def _model_work(case):
    """Images, parameters and logits once each; the multiply-adds of the pruned layers."""
    m = wl.pruned_shapes(_table(case))
    size = wl.spatial_sizes(m)
    n, (H, W, C) = case["batch"], m["input"]
    bytes_, flops = 4.0 * n * H * W * C, 0.0
    for l in m["layers"]:
        if l["kind"] == "conv":
            h, w = size[l["in"]]
            p, q = (h + 2 * l["pad"] - l["R"]) // l["stride"] + 1, (w + 2 * l["pad"] - l["S"]) // l["stride"] + 1
            per_pixel = l["K"] * (l["C"] // l["groups"]) * l["R"] * l["S"]
            flops += 2.0 * n * p * q * per_pixel
            bytes_ += 2.0 * per_pixel + 4.0 * l["K"]
        elif l["kind"] == "fc":
            flops += 2.0 * n * l["in_features"] * l["out_features"]
            bytes_ += 2.0 * l["in_features"] * l["out_features"] + 4.0 * l["out_features"]
    return {"bytes": bytes_ + 4.0 * n * m["layers"][-1]["out_features"], "flops": flops}


# ------------------------------------------------------------------------------------------------ the interface

def _normal(gen, shape, std=1.0):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32) * std


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": case}
    if case["kind"] == "model":
        table = _table(case)
        s["net"] = net = PrunedNetwork(table, _weights(table, np.random.default_rng(seed)), case["batch"])
        x = _normal(gen, (case["batch"],) + tuple(table["input"]))
        logits = torch.zeros((case["batch"], net.model.classes), dtype=torch.float32, device="cuda")
        if case["mode"] == "host":
            x, logits = x.cpu().pin_memory(), logits.cpu().pin_memory()
        s["x"], s["logits"] = x, logits
    elif case["kind"] == "task":
        n, C, hw, K, R, g = case["batch"], case["C"], case["hw"], case["K"], case["R"], case["groups"]
        s["plan"] = plan = cp.cprune_task_plan(n, C, hw, hw, K, R, R, case["stride"], R // 2, g, case["act"], case["residual"])
        w = _normal(gen, (K, C // g, R, R), math.sqrt(2.0 / (C // g * R * R)))
        s["w"], s["b"] = cp.cprune_pack_weights(plan, w, _normal(gen, (K,), 0.01))
        s["x"] = cp.cprune_cast_input(_normal(gen, (n, hw, hw, C)))
        s["res"] = cp.cprune_cast_input(_normal(gen, (n, plan.P, plan.Q, K))) if case["residual"] else None
        s["y"] = torch.zeros((n, plan.out_h, plan.out_w, plan.k_pad), dtype=torch.bfloat16, device="cuda")
        s["ws"] = torch.empty(max(16, plan.workspace_bytes), dtype=torch.uint8, device="cuda")
    else:
        K, C, R, K2, R2 = case["K"], case["C"], case["R"], case["K2"], case["R2"]
        s["w"] = _normal(gen, (K, C, R, R), math.sqrt(2.0 / (C * R * R)))
        s["b"] = _normal(gen, (K,), 0.01)
        s["w_next"] = _normal(gen, (K, 1, R2, R2) if case["depthwise"] else (K2, K, R2, R2), math.sqrt(2.0 / (K * R2 * R2)))
        s["ws"] = torch.empty(cp.cprune_select_workspace_bytes(K), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "model":
        if case["mode"] == "host":
            return s["net"].run_host(s["x"], s["logits"])
        return s["net"].run(s["x"], s["logits"], use_graph=case["mode"] == "graph")
    if case["kind"] == "task":
        return cp.cprune_task_run(s["plan"], s["x"], s["w"], s["b"], s["res"], s["y"], s["ws"])
    return cp.cprune_select_filters(s["w"], case["keep"], s["b"], s["w_next"], case["depthwise"], s["ws"])


def work(case):
    if case["kind"] == "model":
        return _model_work(case)
    if case["kind"] == "task":
        n, C, hw, K, R, g = case["batch"], case["C"], case["hw"], case["K"], case["R"], case["groups"]
        p = (hw + 2 * (R // 2) - R) // case["stride"] + 1
        values = n * hw * hw * C + n * p * p * K * (2 if case["residual"] else 1) + K * (C // g) * R * R
        return {"bytes": 2.0 * values + 4.0 * K, "flops": 2.0 * n * p * p * K * (C // g) * R * R}
    K, C, R, keep, K2, R2 = case["K"], case["C"], case["R"], case["keep"], case["K2"], case["R2"]
    row, nxt = C * R * R, (1 if case["depthwise"] else K2) * R2 * R2
    # every filter is read for its norm, the kept ones are written; of the consumer the kept part is read and written
    return {"bytes": 4.0 * (K * row + keep * row + 2 * keep * nxt + 3 * keep), "flops": 2.0 * K * row}


def tolerance(case):
    """About four times what the tensor-core kernels and the CUDA-core family (other order of the float32 sums, same bf16
    roundings between layers) were measured to differ by on the listed cases and on drawn ones."""
    if case["kind"] == "select":
        return "exact"                                  # indices and copies
    if case["kind"] == "task":
        return {"rel": 4e-4, "max": 0.032}              # measured up to 7.5e-5 and 7.8e-3: single bf16 results rounded the other way
    # logits behind up to 54 layers that each store bf16: measured up to 2.8e-3, 5.4e-3 and 6.5e-3
    rel = {"resnet18": 1.2e-2, "resnet18_shared": 1.2e-2, "vgg16_cifar": 2e-2, "mobilenet_v2": 2.5e-2, "mnasnet1_0": 2.5e-2}[case["model"]]
    return {"rel": rel, "max": 5 * rel}
