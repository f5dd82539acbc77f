"""Performance cases of the FedOptima server-side hot path, through its public
entry points (`paper_2504_13850_gb300.api`).

Three kinds of work make up the path:

  step       one training iteration of the server as its loop runs it: a
             device's activation batch is uploaded, the scheduled batch is
             trained on (forward, softmax cross-entropy, backward,
             SGD-momentum update) and the loss of the step is read.  The
             server step is one sequential SGD chain, so the next step of a
             server cannot begin before this one has ended.
  aggregate  one FedAsync update of a device-side model (device-resident, or
             arriving in page-locked host memory).
  colsum     the standalone deterministic column sums.

A step returns the loss, the logits and the updated parameters (the server's
own buffers).
"""
import math

import numpy as np
import torch

from paper_2504_13850_gb300 import api
from paper_2504_13850_gb300 import workloads as W

LR, MOMENTUM = 0.01, 0.9
DEVICES, OMEGA, DEPTH = 2, 4, 2      # a small queue: the step does not depend on it


# ------------------------------------------------------------------- cases

def listed():
    return [
        # the fp32 path and the smallest call: the repository's tiny CNN
        {"name": "tiny_f32", "kind": "step", "net": "tiny", "batch": 16, "hw": 16, "dtype": "f32"},
        # VGG-style server part at its configured batch
        {"name": "vgg", "kind": "step", "net": "vgg", "batch": 64, "hw": 16, "dtype": "bf16"},
        # the same network at a batch that is no multiple of a tile
        {"name": "vgg_odd_batch", "kind": "step", "net": "vgg", "batch": 37, "hw": 16, "dtype": "bf16"},
        # ResNet-18 stages 3-4 at the configured batch and map
        {"name": "resnet", "kind": "step", "net": "resnet", "batch": 128, "hw": 16, "dtype": "bf16", "classes": 100},
        # the same stages on the 28 x 28 maps that 224-pixel images give
        {"name": "resnet_224", "kind": "step", "net": "resnet", "batch": 24, "hw": 28, "dtype": "bf16",
         "classes": 1000},
        # MobileNetV3-Large server part: many small layers, launches and latency
        {"name": "mobilenet", "kind": "step", "net": "mobilenet", "batch": 64, "hw": 4, "dtype": "bf16",
         "classes": 200},
        # a device's own trainer (its first layer has 3 input channels)
        {"name": "device", "kind": "step", "net": "device", "batch": 64, "hw": 32, "dtype": "bf16"},
        # transformer encoder server part, the benchmark's headline
        {"name": "transformer", "kind": "step", "net": "encoder", "batch": 32, "len": 128, "d": 512, "heads": 8,
         "blocks": 4, "classes": 2, "dtype": "bf16"},
        # one encoder block of small width: ragged length and batch, heads of 32
        {"name": "encoder_ragged", "kind": "step", "net": "encoder", "batch": 19, "len": 77, "d": 256, "heads": 8,
         "blocks": 1, "classes": 5, "dtype": "bf16"},
        # FedAsync of the transformer workload's device model
        {"name": "aggregate", "kind": "aggregate", "n": 30522 * 512 + 2 * 3_152_384, "host": False},
        # FedAsync of a small device model that arrives in host memory
        {"name": "aggregate_host", "kind": "aggregate", "n": 700_003, "host": True},
        # bias-gradient reduction of a large odd matrix
        {"name": "column_sums", "kind": "colsum", "rows": 65_500, "cols": 1000, "dtype": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.choice(["tiny", "vgg", "vgg", "resnet", "resnet", "resnet", "mobilenet", "mobilenet", "device",
                       "encoder", "encoder", "encoder", "aggregate", "colsum"])
    if pick == "tiny":
        return {"kind": "step", "net": "tiny", "batch": _log(rng, 1, 256), "hw": 16,
                "dtype": rng.choice(["f32", "f32", "bf16"])}
    if pick == "vgg":
        return {"kind": "step", "net": "vgg", "batch": _log(rng, 1, 64), "hw": 16, "dtype": "bf16"}
    if pick == "resnet":
        hw = rng.choice([7, 8, 12, 14, 16, 20, 24, 28])
        return {"kind": "step", "net": "resnet", "batch": _log(rng, 1, 24 * 28 * 28 // hw ** 2) if hw > 12 else
                _log(rng, 1, 128), "hw": hw, "dtype": "bf16", "classes": rng.choice([10, 100, 200, 1000])}
    if pick == "mobilenet":
        hw = rng.choice([4, 7, 14])
        return {"kind": "step", "net": "mobilenet", "batch": _log(rng, 1, 96 if hw == 4 else 64), "hw": hw,
                "dtype": "bf16", "classes": rng.choice([10, 100, 200, 1000])}
    if pick == "device":
        return {"kind": "step", "net": "device", "batch": _log(rng, 1, 64), "hw": 32, "dtype": "bf16"}
    if pick == "encoder":
        d = rng.choice([128, 256, 384, 512, 768])
        blocks = rng.choice([1, 2])
        length = rng.randint(8, 128)
        most = min(64, 4 * 32 * 128 * 512 ** 2 // (blocks * length * d * d))
        return {"kind": "step", "net": "encoder", "batch": _log(rng, 1, most), "len": length, "d": d,
                "heads": d // rng.choice([32, 64, 64]), "blocks": blocks, "classes": rng.choice([2, 5, 20]),
                "dtype": "bf16"}
    if pick == "aggregate":
        return {"kind": "aggregate", "n": _log(rng, 20_000, 40_000_000), "host": rng.random() < 0.25}
    return {"kind": "colsum", "rows": _log(rng, 64, 100_000), "cols": _log(rng, 10, 1500),
            "dtype": rng.choice(["bf16", "bf16", "f32"])}


# ---------------------------------------------------------------- networks

def _net(case):
    """(op list, input [H, W, C], classes) of a step case."""
    net, hw = case["net"], case.get("hw", 0)
    if net == "tiny":
        return W.tiny_cnn_ops(), (hw, hw, 32), 10
    if net == "vgg":
        return W.vgg_ops(), (hw, hw, 128), 10
    if net == "resnet":
        return W.resnet_ops(case["classes"]), (hw, hw, 128), case["classes"]
    if net == "mobilenet":
        return W.mobilenet_ops(case["classes"]), (hw, hw, 112), case["classes"]
    if net == "device":
        return W.vgg_device_ops(), (hw, hw, 3), 10
    d = case["d"]
    ops = W.transformer_ops(d=d, heads=case["heads"], ffn=4 * d, blocks=case["blocks"], classes=case["classes"])
    return ops, (case["len"], 1, d), case["classes"]


class _Buffer:
    """A device buffer of a server as an array that torch can view; keeps the server alive."""

    def __init__(self, owner, ptr, shape):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f4", "data": (ptr, False), "version": 3}


def _inputs(case, seed):
    """(activations, labels, lengths or None, list of parameter tensors), on the GPU.

    Values as in the repository's workloads: rectified normal maps for the
    convolutional parts, normal hidden states for the encoder; He-normal
    weights, unit scales, zero shifts and biases.
    """
    ops, hwc, classes = _net(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    B = case["batch"]
    x = torch.randn((B, *hwc), generator=g, device="cuda")
    lengths = None
    if case["net"] == "encoder":
        lengths = torch.randint(max(1, hwc[0] // 4), hwc[0] + 1, (B,), generator=g, device="cuda", dtype=torch.int32)
    elif case["net"] != "device":
        x = x.relu_()
    x = x.to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)
    labels = torch.randint(0, classes, (B,), generator=g, device="cuda", dtype=torch.int32)
    params = []
    for name, shape in W.param_shapes(ops):
        n = int(np.prod(shape))
        if name == "W":
            p = torch.randn(n, generator=g, device="cuda") * math.sqrt(2.0 / int(np.prod(shape[1:])))
        else:
            p = torch.full((n,), 1.0 if name in ("scale", "gamma") else 0.0, device="cuda")
        params.append(p.reshape(shape))
    return x, labels, lengths, params


def _padded(params):
    """The server's parameter vector: every tensor starts at a multiple of 64 floats."""
    out = torch.zeros(sum((p.numel() + 63) // 64 * 64 for p in params), device=params[0].device,
                      dtype=params[0].dtype)
    at = 0
    for p in params:
        out[at:at + p.numel()] = p.reshape(-1)
        at += (p.numel() + 63) // 64 * 64
    return out


# --------------------------------------------------------------- the passes

def prepare(case, seed):
    if case["kind"] == "step":
        ops, hwc, classes = _net(case)
        x, labels, lengths, params = _inputs(case, seed)
        s = api.Server(ops, DEVICES, OMEGA, DEPTH, case["batch"], hwc, classes, case["dtype"], LR, MOMENTUM,
                       seq=lengths is not None)
        theta = _padded(params)
        ptr, n = s.params_device()
        assert n == theta.numel()
        torch.cuda.synchronize()
        s.load_params_device(theta.data_ptr(), n)
        s.synchronize()
        logits, dims, _ = s.tensor(len(ops))
        return {"kind": "step", "server": s, "x": x, "labels": labels, "lengths": lengths, "steps": 0,
                "logits": torch.as_tensor(_Buffer(s, logits, (dims[0], dims[3])), device="cuda"),
                "theta": torch.as_tensor(_Buffer(s, ptr, (n,)), device="cuda")}
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "aggregate":
        n = case["n"]
        glob = torch.randn(n, generator=g, device="cuda") * 0.05
        local = torch.randn(n, generator=g, device="cuda") * 0.05
        if case["host"]:
            local = local.cpu().pin_memory()
        # the smallest server that takes uploads of device models
        b = W.tiny_cnn_ops()
        s = api.Server(b, DEVICES, 1, 1, 1, (16, 16, 32), 10, "f32", LR, MOMENTUM)
        small = torch.zeros(2, 64, device="cuda")
        torch.cuda.synchronize()
        for t in range(3):      # the global version is a few models ahead of the one that arrives
            s.aggregate(small[0], small[1], 0, t)
        s.synchronize()
        return {"kind": "aggregate", "server": s, "global": glob, "local": local, "t": 3}
    x = torch.randn((case["rows"], case["cols"]), generator=g, device="cuda")
    return {"kind": "colsum", "x": x.to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float32),
            "out": torch.empty(case["cols"], device="cuda")}


def run(st):
    if st["kind"] == "step":
        s, i = st["server"], st["steps"]
        s.enqueue_activations(i % DEVICES, st["x"], st["labels"], st["lengths"])
        s.server_step()
        st["steps"] = i + 1
        return {"loss": s.read_losses(i, 1), "logits": st["logits"], "theta": st["theta"]}
    if st["kind"] == "aggregate":
        _, st["t"] = st["server"].aggregate(st["global"], st["local"], 0, st["t"] - 2)
        return st["global"]
    api.column_sums(st["x"], st["out"])
    return st["out"]


# ---------------------------------------------------------------- yardsticks

def work(case):
    """Bytes: the uploaded batch, parameters and momentum read and written once, the logits.
    Operations: two per multiplication of the forward, the weight gradients
    and the input gradients that a layer's input needs."""
    if case["kind"] == "aggregate":
        return {"bytes": 12.0 * case["n"], "flops": 2.0 * case["n"]}
    if case["kind"] == "colsum":
        return {"bytes": float(case["rows"] * case["cols"] * (2 if case["dtype"] == "bf16" else 4) + 4 * case["cols"]),
                "flops": float(case["rows"] * case["cols"])}
    ops, hwc, classes = _net(case)
    B = case["batch"]
    shapes = [(hwc[0], hwc[1], hwc[2])]
    flops = 0.0
    for op in ops:
        h, w, c = shapes[op["in0"]]
        k, st = op.get("k", 1), op.get("stride", 1)
        kind = op["kind"]
        passes = 2 if op["in0"] == 0 else 3
        if kind in ("conv", "dwconv"):
            h, w = (h - 1) // st + 1, (w - 1) // st + 1
            per = k * k * (c if kind == "conv" else 1)
            c = op.get("cout", c)
            flops += passes * 2.0 * B * h * w * c * per
        elif kind == "linear":
            flops += passes * 2.0 * B * h * w * c * op["cout"]
            c = op["cout"]
        elif kind == "attention":
            c = op["c"]
            flops += 7 * 2.0 * B * h * h * c        # S and O; dV, dP, dQ, dK and S again
        elif kind == "maxpool2":
            h, w = h // 2, w // 2
        elif kind == "avgpool":
            h = w = 1
        elif kind == "meanpool":
            h = 1
        elif kind == "flatten":
            h, w, c = 1, 1, h * w * c
        shapes.append((h, w, c))
    esz = 2 if case["dtype"] == "bf16" else 4
    nbytes = B * hwc[0] * hwc[1] * hwc[2] * esz + 16.0 * W.num_params(ops) + 4.0 * B * classes
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "aggregate":
        return {"rel": 1e-6}
    if case["kind"] == "colsum" or case["dtype"] == "f32":
        return {"rel": 1e-5}
    return {"rel": 2e-2}


# -------------------------------------------------- the same in 64-bit torch

def _conv(x, w, stride):
    """NHWC convolution, padding k // 2, as a sum of shifted matrix products."""
    co, k, _, ci = w.shape
    p = k // 2
    B, H, Wd, _ = x.shape
    ho, wo = (H - 1) // stride + 1, (Wd - 1) // stride + 1
    x = torch.nn.functional.pad(x, (0, 0, p, p, p, p))
    y = 0
    for r in range(k):
        for s in range(k):
            win = x[:, r:r + (ho - 1) * stride + 1:stride, s:s + (wo - 1) * stride + 1:stride]
            y = y + win @ w[:, r, s].T
    return y


def _dwconv(x, w, stride):
    c, k, _ = w.shape
    p = k // 2
    ho, wo = (x.shape[1] - 1) // stride + 1, (x.shape[2] - 1) // stride + 1
    x = torch.nn.functional.pad(x, (0, 0, p, p, p, p))
    return sum(x[:, r:r + (ho - 1) * stride + 1:stride, s:s + (wo - 1) * stride + 1:stride] * w[:, r, s]
               for r in range(k) for s in range(k))


def _attention(qkv, heads, lengths):
    B, L, _, c3 = qkv.shape
    q, k, v = qkv.reshape(B, L, 3, heads, c3 // 3 // heads).permute(2, 0, 3, 1, 4)
    s = q @ k.transpose(-1, -2) / math.sqrt(q.shape[-1])
    s = s.masked_fill(torch.arange(L, device=qkv.device) >= lengths.view(B, 1, 1, 1), -math.inf)
    return (s.softmax(-1) @ v).permute(0, 2, 1, 3).reshape(B, L, 1, c3 // 3)


def _forward(ops, x, lengths, params):
    at, t = iter(params), [x]
    for op in ops:
        a, kind = t[op["in0"]], op["kind"]
        if kind == "conv":
            y = _conv(a, next(at), op["stride"])
            y = y + next(at) if op["bias"] else y
        elif kind == "dwconv":
            y = _dwconv(a, next(at), op["stride"])
            y = y + next(at) if op["bias"] else y
        elif kind == "linear":
            y = a @ next(at).T
            y = y + next(at) if op["bias"] else y
        elif kind == "affine":
            y = a * next(at) + next(at)
        elif kind == "layernorm":
            y = torch.nn.functional.layer_norm(a, a.shape[-1:], next(at), next(at), 1e-5)
        elif kind == "relu":
            y = a.relu()
        elif kind == "gelu":
            y = torch.nn.functional.gelu(a)
        elif kind == "hswish":
            y = a * (a + 3).clamp(0, 6) / 6
        elif kind == "hsigmoid":
            y = (a + 3).clamp(0, 6) / 6
        elif kind == "maxpool2":
            y = torch.nn.functional.max_pool2d(a.permute(0, 3, 1, 2), 2).permute(0, 2, 3, 1)
        elif kind == "add":
            y = a + t[op["in1"]]
        elif kind == "chmul":
            y = a * t[op["in1"]]
        elif kind == "avgpool":
            y = a.mean((1, 2), keepdim=True)
        elif kind == "meanpool":
            m = (torch.arange(a.shape[1], device=a.device) < lengths.view(-1, 1)).to(a.dtype)
            y = ((a[:, :, 0] * m[..., None]).sum(1) / lengths.view(-1, 1).to(a.dtype))[:, None, None]
        elif kind == "flatten":
            y = a.reshape(a.shape[0], 1, 1, -1)
        elif kind == "attention":
            y = _attention(a, op["heads"], lengths)
        else:
            raise ValueError(kind)
        t.append(y)
    return t[-1].reshape(x.shape[0], -1)


def exact(case, seed):
    if case["kind"] == "step":
        ops, _, _ = _net(case)
        x, labels, lengths, params = _inputs(case, seed)
        params = [p.double().requires_grad_() for p in params]
        logits = _forward(ops, x.double(), lengths, params)
        torch.nn.functional.cross_entropy(logits, labels.long()).backward()
        theta = _padded([(p - LR * p.grad).detach() for p in params])
        # no value for the loss: one number's rounding error is a draw, not a measure of precision
        return {"loss": None, "logits": logits.detach(), "theta": theta}
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "aggregate":
        glob = (torch.randn(case["n"], generator=g, device="cuda") * 0.05).double()
        local = (torch.randn(case["n"], generator=g, device="cuda") * 0.05).double()
        return glob + (local - glob) / 3
    x = torch.randn((case["rows"], case["cols"]), generator=g, device="cuda")
    return x.to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float32).double().sum(0)
