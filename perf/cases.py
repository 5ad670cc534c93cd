"""Performance cases of libmembrane: the calls that a user of the library makes, over their range.

A case is a dict of plain values. ``listed()`` holds the named ones, ``draw(rng)`` gives more of the
same ranges, ``prepare`` makes what a program has in hand before the call (device buffers, a net with
its weights), ``run`` makes one pass through the public calls, ``work`` counts what a pass cannot do
without, and ``exact`` computes the same outputs in 64 bits with plain torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch
import torch.nn.functional as F

from paper_1612_02120_gb300 import membrane as m

# (kind, ksize, cin, cout, relu[, dilation[, max-out groups]])
CONV, MAXF, SIGMOID, SOFTMAX2, SOFTMAX = (m.MB_CONV, m.MB_MAXFILTER, m.MB_HEAD_SIGMOID, m.MB_HEAD_SOFTMAX2,
                                          m.MB_HEAD_SOFTMAX)


def _maxout_stack(cin, features):
    layers, d = [], 1
    for f in features:
        layers += [(CONV, 4, cin, f, 0, d, 2), (MAXF, 2, f, f, 0, d, 1)]
        cin, d = f, 2 * d
    return layers, d


def _nets():
    teacher = [(CONV, 5, 1, 32, 1), (MAXF, 2, 32, 32, 0), (CONV, 5, 32, 32, 1), (MAXF, 2, 32, 32, 0),
               (CONV, 5, 32, 32, 1), (SIGMOID, 1, 32, 1, 0)]
    student = [(CONV, 3, 1, 16, 1), (CONV, 3, 16, 16, 1), (SIGMOID, 1, 16, 1, 0)]
    fm, d = _maxout_stack(1, (32, 32, 32))
    fm3, d3 = _maxout_stack(1, (32, 32, 32, 32))
    me, _ = _maxout_stack(12, (32, 40, 48, 56, 64))
    return {"teacher": teacher, "student": student, "fastmemb": fm + [(SOFTMAX2, 4, 32, 2, 0, d, 1)],
            "fastmemb_3nm": fm3 + [(SOFTMAX2, 4, 32, 2, 0, d3, 1)],
            "maskextend": me[:-1] + [(SOFTMAX, 1, 64, 3, 0, 1, 1)]}


NETS = _nets()
PRECS = {"fp32": m.MB_PREC_FP32, "bf16": m.MB_PREC_BF16, "fp8": m.MB_PREC_FP8, "fp16": m.MB_PREC_FP16}
RADIUS = {"teacher": 7, "student": 2, "fastmemb": 26, "fastmemb_3nm": 54, "maskextend": 54}
MIN_SIDE = {"teacher": 8, "student": 8, "fastmemb": 27, "fastmemb_3nm": 55, "maskextend": 55}


def listed():
    return [
        # one tile under a cursor: the smallest call, where launch and pipeline fill count
        {"name": "teacher_bf16_tile", "kind": "volume", "net": "teacher", "prec": "bf16", "z": 1, "h": 256, "w": 256},
        # the benchmark's volume, with the tuning choice that its autotuner records for it
        {"name": "teacher_bf16_volume", "kind": "volume", "net": "teacher", "prec": "bf16", "z": 32, "h": 1024,
         "w": 1024, "tuned": True},
        # blocks of a stack cut unevenly, mapped in one call
        {"name": "teacher_bf16_blocks", "kind": "batch", "blocks": 16, "lo": 256, "hi": 1024, "deep": 8},
        # a stack whose slices are no multiple of anything, at the lowest precision
        {"name": "teacher_fp8_ragged", "kind": "volume", "net": "teacher", "prec": "fp8", "z": 8, "h": 1000,
         "w": 1333},
        # reference maps: the targets that a student is trained on
        {"name": "teacher_fp32_targets", "kind": "volume", "net": "teacher", "prec": "fp32", "z": 16, "h": 512,
         "w": 512},
        # the fast pass over whole planes
        {"name": "student_bf16_planes", "kind": "volume", "net": "student", "prec": "bf16", "z": 8, "h": 4096,
         "w": 4096},
        # optimiser steps of the training configuration (batch 32 of 512 x 512)
        {"name": "student_train_steps", "kind": "train", "prec": "bf16", "n": 64, "h": 512, "w": 512, "batch": 32,
         "steps": 4},
        # one gradient of a small odd batch, as an outside optimiser asks for it
        {"name": "student_grad_small", "kind": "grad", "prec": "fp32", "n": 3, "h": 131, "w": 257},
        # the paper's network over a volume, in the type that the benchmark lists first
        {"name": "fastmemb_bf16_volume", "kind": "volume", "net": "fastmemb", "prec": "bf16", "z": 8, "h": 1024,
         "w": 1024},
        # the deeper variant on large 3 nm planes
        {"name": "fastmemb_3nm_fp16_planes", "kind": "volume", "net": "fastmemb_3nm", "prec": "fp16", "z": 2,
         "h": 2048, "w": 2048},
        # the FP32 network on a part of one slice, at an odd origin and size
        {"name": "fastmemb_fp32_region", "kind": "region", "net": "fastmemb", "prec": "fp32", "z": 1, "h": 1024,
         "w": 1024, "y0": 101, "x0": 37, "rows": 611, "cols": 803},
        # an object followed through 16 sections
        {"name": "maskextend_fp16_sections", "kind": "mask", "prec": "fp16", "h": 512, "w": 512, "steps": 16,
         "direction": 1},
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _volume_dims(rng, net, voxels, hi):
    """z, h, w with at most `voxels` voxels; sides spread over the logarithm of [lo, hi]."""
    lo = max(48, MIN_SIDE[net] + 1)
    h, w = _side(rng, lo, hi), _side(rng, lo, hi)
    while h * w > voxels:
        h, w = max(lo, h // 2), max(lo, w // 2)
    z = max(1, min(int(round(math.exp(rng.uniform(0.0, math.log(40.0))))), voxels // (h * w)))
    return z, h, w


def draw(rng: random.Random):
    kind = rng.choice(["volume"] * 7 + ["batch", "train", "grad", "region", "mask"])
    if kind == "volume":
        net, prec, voxels, hi = rng.choice([
            ("teacher", "bf16", 30_000_000, 4096), ("teacher", "fp8", 30_000_000, 4096),
            ("teacher", "fp32", 4_000_000, 2048), ("student", "bf16", 120_000_000, 4096),
            ("student", "fp32", 30_000_000, 4096), ("fastmemb", "bf16", 8_000_000, 2048),
            ("fastmemb", "fp16", 8_000_000, 2048), ("fastmemb_3nm", "fp16", 8_000_000, 2560),
            ("fastmemb_3nm", "bf16", 8_000_000, 2560)])
        z, h, w = _volume_dims(rng, net, voxels, hi)
        case = {"kind": kind, "net": net, "prec": prec, "z": z, "h": h, "w": w}
        if net.startswith("fastmemb") and rng.random() < 0.3:
            case["subsample"] = 2
        return case
    if kind == "batch":
        return {"kind": kind, "blocks": rng.randint(2, 24), "lo": rng.randint(64, 256), "hi": rng.randint(300, 900),
                "deep": rng.randint(1, 6)}
    if kind == "region":
        net, prec = rng.choice([("fastmemb", "fp32"), ("fastmemb", "bf16"), ("teacher", "bf16"), ("teacher", "fp32"),
                                ("student", "bf16")])
        h, w = rng.randint(200, 1200), rng.randint(200, 1200)
        rows, cols = rng.randint(33, min(h, 700)), rng.randint(33, min(w, 700))
        return {"kind": kind, "net": net, "prec": prec, "z": rng.randint(1, 2), "h": h, "w": w,
                "y0": rng.randint(0, h - rows), "x0": rng.randint(0, w - cols), "rows": rows, "cols": cols}
    if kind == "mask":
        return {"kind": kind, "prec": rng.choice(["fp16", "fp16", "fp32"]), "h": rng.randint(64, 400),
                "w": rng.randint(64, 400), "steps": rng.randint(1, 8), "direction": rng.choice([1, -1])}
    h, w = _side(rng, 40, 640), _side(rng, 40, 640)
    if kind == "grad":
        return {"kind": kind, "prec": rng.choice(["fp32", "bf16"]), "n": rng.randint(1, 16), "h": h, "w": w}
    return {"kind": kind, "prec": rng.choice(["fp32", "bf16"]), "n": rng.randint(4, 48), "h": h, "w": w,
            "batch": rng.randint(2, 24), "steps": rng.randint(1, 4)}


# --- inputs ---------------------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _em_slices(g, z, h, w):
    """uint8 EM-like slices [z][h][w]: bright cells, dark membranes along the zero lines of a smooth
    random field, sensor noise, a 3x3 blur."""
    out = torch.empty((z, h, w), dtype=torch.uint8, device="cuda")
    for i in range(z):
        coarse = torch.randn((1, 1, h // 12 + 3, w // 12 + 3), device="cuda", generator=g)
        field = F.interpolate(coarse, size=(h, w), mode="bilinear", align_corners=True)
        v = 0.67 - 0.43 * torch.exp(-(field / 0.18) ** 2)
        v += 0.07 * torch.randn((1, 1, h, w), device="cuda", generator=g)
        v = F.avg_pool2d(F.pad(v, (1, 1, 1, 1), mode="reflect"), 3, stride=1)
        out[i] = (v[0, 0] * 255.0).round().clamp(0, 255).to(torch.uint8)
    return out


def _params(net, seed):
    """He-normal FP32 parameters, W then b per layer. The student's first layer is drawn for the input
    x - 1/2; the last layer of the deep max-out stacks has zero mean over its input channels, which
    keeps their maps away from saturation."""
    rng = np.random.default_rng([int(seed), len(net)])
    layers = [t for t in NETS[net] if t[0] != MAXF]
    parts = []
    for i, t in enumerate(layers):
        k, cin, co = t[1], t[2], t[3] * (t[6] if len(t) > 6 else 1)
        w = rng.standard_normal((co, cin, k * k)) * math.sqrt(2.0 / (cin * k * k))
        b = rng.standard_normal(co) * (0.0 if net == "student" else 0.01)
        if net == "student" and i == 0:
            b = b - 0.5 * w.sum(axis=(1, 2))
        if net.startswith("fastmemb") and i == len(layers) - 1:
            w = w - w.mean(axis=1, keepdims=True)
        parts += [w.reshape(-1), b]
    return np.concatenate(parts).astype(np.float32)


def _block_shapes(case, seed):
    rng = random.Random(case["blocks"] * 7919 + case["hi"])  # the cut of the stack is the case's own
    return [(rng.randint(1, case["deep"]), rng.randint(case["lo"], case["hi"]), rng.randint(case["lo"], case["hi"]))
            for _ in range(case["blocks"])]


def _disks(n, h, w):
    yy, xx = torch.meshgrid(torch.arange(h, device="cuda"), torch.arange(w, device="cuda"), indexing="ij")
    return torch.stack([((yy - h / 2 - 2 * i) ** 2 + (xx - w / 2 + i) ** 2 <= (min(h, w) / 5) ** 2).to(torch.uint8)
                        for i in range(n)])


def _inputs(case, seed):
    """The tensors of a case: what exact() needs too."""
    g, kind = _generator(seed), case["kind"]
    if kind in ("volume", "region"):
        return {"x": _em_slices(g, case["z"], case["h"], case["w"])}
    if kind == "batch":
        return {"xs": [_em_slices(g, d, h, w) for d, h, w in _block_shapes(case, seed)]}
    if kind in ("train", "grad"):
        x = _em_slices(g, case["n"], case["h"], case["w"])
        smooth = F.avg_pool2d(x.float()[:, None] / 255.0, 5, stride=1, padding=2, count_include_pad=False)[:, 0]
        return {"x": x, "t": torch.sigmoid(14.0 * (0.52 - smooth)).contiguous()}
    z = case["steps"] + 4  # the sections that the recursion reads
    em = _em_slices(g, z, case["h"], case["w"])
    return {"em": em, "memb": (1.0 - em.float() / 255.0).contiguous(), "seeds": _disks(4, case["h"], case["w"])}


def prepare(case, seed):
    state = dict(case, **_inputs(case, seed))
    kind = case["kind"]
    if kind in ("volume", "region"):
        net = m.Net(NETS[case["net"]], PRECS[case["prec"]], 0, _params(case["net"], seed))
        if case["prec"] == "fp8":
            n = min(4, case["z"])
            m.mb_calibrate_fp8(net.handle, state["x"][:n], n, case["h"], case["w"])
        if case.get("tuned"):
            m.mb_set_tuning(net.handle, 0, 4)
        h, w = (case["h"], case["w"]) if kind == "volume" else (case["rows"], case["cols"])
        s = case.get("subsample", 1)
        state["out"] = torch.empty((case["z"], -(-h // s), -(-w // s)), device="cuda")
    elif kind == "batch":
        net = m.Net(NETS["teacher"], m.MB_PREC_BF16, 0, _params("teacher", seed))
        state["outs"] = [torch.empty(x.shape, device="cuda") for x in state["xs"]]
        state["list"] = [(x, *x.shape, x.shape[2], x.shape[1] * x.shape[2], o, x.shape[2], x.shape[1] * x.shape[2])
                         for x, o in zip(state["xs"], state["outs"])]
    elif kind in ("train", "grad"):
        state["params"] = _params("student", seed)
        net = m.Net(NETS["student"], PRECS[case["prec"]], 0, state["params"])
        state["grad"] = torch.empty(net.n_params, device="cuda")
    else:
        net = m.Net(NETS["maskextend"], PRECS[case["prec"]], 0, _params("maskextend", seed))
        n, h, w = case["steps"], case["h"], case["w"]
        state["masks"] = torch.empty((n, h, w), dtype=torch.uint8, device="cuda")
        state["probs"] = torch.empty((n, 3, h, w), device="cuda")
    state["net"] = net
    return state


def run(s):
    net, kind, stream = s["net"].handle, s["kind"], torch.cuda.current_stream()
    if kind == "volume":
        if s.get("subsample"):
            m.mb_infer_volume_subsampled(net, s["x"], s["z"], s["h"], s["w"], 2, s["out"], stream=stream)
        else:
            m.mb_infer_volume(net, s["x"], s["z"], s["h"], s["w"], s["out"], stream=stream)
        return s["out"]
    if kind == "region":
        m.mb_infer_region(net, s["x"], s["z"], s["h"], s["w"], s["y0"], s["x0"], s["rows"], s["cols"], s["out"],
                          stream=stream)
        return s["out"]
    if kind == "batch":
        m.mb_infer_batch(net, s["list"], stream=stream)
        return s["outs"]
    if kind == "grad":
        loss = m.mb_student_loss_grad(net, s["x"], s["t"], s["n"], s["h"], s["w"], s["grad"], stream)
        return {"loss": loss, "grad": s["grad"]}
    if kind == "train":
        curve, weights = np.zeros(s["steps"], np.float32), np.empty_like(s["params"])
        m.mb_load_weights(net, s["params"])
        m.mb_student_train(net, s["x"], s["t"], s["n"], s["h"], s["w"],
                           m.train_cfg(batch=s["batch"], steps=s["steps"], seed=7), None, curve, stream)
        m.mb_get_weights(net, weights)
        return {"curve": curve, "weights": weights}
    z0 = 2 if s["direction"] > 0 else s["steps"] + 1
    m.mb_mask_extend_dir(net, s["em"], s["memb"], s["steps"] + 4, s["h"], s["w"], s["seeds"], z0, s["steps"],
                         s["direction"], s["masks"], s["probs"], stream=stream)
    return {"masks": s["masks"], "probs": s["probs"]}


# --- work -----------------------------------------------------------------------------------------

def _flop_per_pixel(net):
    """FLOPs of one output pixel of the dense map: 2 per weight of every convolution."""
    return sum(2.0 * t[1] ** 2 * t[2] * t[3] * (t[6] if len(t) > 6 else 1) for t in NETS[net] if t[0] != MAXF)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        px = sum(d * h * w for d, h, w in _block_shapes(case, 0))
        return {"bytes": 5.0 * px, "flops": px * _flop_per_pixel("teacher")}
    if kind in ("volume", "region"):
        px_in = case["z"] * case["h"] * case["w"]
        px = px_in if kind == "volume" else case["z"] * case["rows"] * case["cols"]
        flops = px * _flop_per_pixel(case["net"])
        if kind == "region":
            px_in = px
        if case.get("subsample"):  # the first layer at full resolution, the others on a quarter of the pixels
            first = 2.0 * 16 * 64
            flops, px = px * (first + (_flop_per_pixel(case["net"]) - first) / 4), px / 4
        return {"bytes": 1.0 * px_in + 4.0 * px, "flops": flops}
    if kind in ("train", "grad"):  # forward, data gradient and weight gradient
        px = case["h"] * case["w"] * (case["n"] if kind == "grad" else case["batch"] * case["steps"])
        return {"bytes": 5.0 * px, "flops": 3.0 * px * _flop_per_pixel("student")}
    px = case["h"] * case["w"]
    return {"bytes": px * (5.0 * (case["steps"] + 4) + 4.0 + 13.0 * case["steps"]),
            "flops": case["steps"] * px * _flop_per_pixel("maskextend")}


# --- the same outputs in 64 bits ------------------------------------------------------------------

def _conv64(x, w, b, d):
    """Valid dilated cross-correlation of x [cin][H][W]; one matrix product per tap over the flattened
    rows, where a tap is a shift."""
    k, cols = w.shape[2], x.shape[2]
    ho, wo = x.shape[1] - (k - 1) * d, cols - (k - 1) * d
    flat = x.contiguous().view(x.shape[0], -1)
    n = (ho - 1) * cols + wo
    y = torch.zeros((w.shape[0], ho * cols), dtype=torch.float64, device=x.device)
    part = y[:, :n]
    for ky in range(k):
        for kx in range(k):
            o = (ky * cols + kx) * d
            part.addmm_(w[:, :, ky, kx], flat[:, o:o + n])
    return y.view(-1, ho, cols)[:, :, :wo] + b[:, None, None]


def _forward64(net, params, x):
    """Layers of `net` on a padded input x [c][H][W] (float64): its map [h][w] or class maps [3][h][w]."""
    p, o = torch.from_numpy(params).cuda().double(), 0
    for t in NETS[net]:
        kind, k, cin, cout = t[:4]
        d, groups = (t[5] if len(t) > 5 else 1), (t[6] if len(t) > 6 else 1)
        if kind == MAXF:
            a = torch.maximum(x[:, :, :-d], x[:, :, d:])
            x = torch.maximum(a[:, :-d], a[:, d:])
            continue
        co = cout * groups
        w = p[o:o + co * cin * k * k].view(co, cin, k, k)
        b = p[o + w.numel():o + w.numel() + co]
        o += w.numel() + co
        x = _conv64(x, w, b, d)
        if kind == CONV:
            x = x.clamp_min(0) if t[4] else x.view(cout, groups, *x.shape[1:]).amax(1)
        elif kind == SIGMOID:
            x = torch.sigmoid(x[0])
        elif kind == SOFTMAX2:
            x = torch.sigmoid(x[1] - x[0])
        else:
            x = torch.softmax(x, 0)
    return x


def _pad64(maps, r):
    return F.pad(maps.double()[None], (r, r, r, r), mode="reflect")[0]


def _map64(net, params, slices, box=None):
    r, out = RADIUS[net], []
    for s in slices:
        x = _pad64(s[None], r) / 255.0
        if box:
            y0, x0, rows, cols = box
            x = x[:, y0:y0 + rows + 2 * r, x0:x0 + cols + 2 * r]
        out.append(_forward64(net, params, x).float())
    return torch.stack(out)


def _grad64(case, params, x, t):
    q = torch.from_numpy(params).cuda()
    if case["prec"] == "bf16":  # the forward copy of a BF16 student is its rounded weights
        q = q.bfloat16()
    q = q.double().requires_grad_(True)
    w1, b1, w2, b2, wh, bh = (q[0:144].view(16, 1, 3, 3), q[144:160], q[160:2464].view(16, 16, 3, 3), q[2464:2480],
                              q[2480:2496], q[2496])
    total, loss = x.numel(), 0.0
    for s, target in zip(x, t):
        a = (_pad64(s[None], 2) / 255.0)[None]
        a = F.relu(F.conv2d(F.relu(F.conv2d(a, w1, b1)), w2, b2))[0]
        p = torch.sigmoid((a * wh[:, None, None]).sum(0) + bh)
        part = ((p - target.double()) ** 2).sum() / total
        part.backward(retain_graph=True)
        loss += float(part.detach())
    return {"loss": loss, "grad": q.grad}


def _masks64(case, params, em, memb, seeds):
    s, n, r = case["direction"], case["steps"], RADIUS["maskextend"]
    z0 = 2 if s > 0 else n + 1
    masks = {z0 + s * (i - 4): seeds[i].double() for i in range(4)}
    probs = []
    for step in range(n):
        z = z0 + s * step
        maps = [em[z + s * k].double() / 255.0 for k in (-1, 0, 1)]
        maps += [masks[z + s * k] for k in (-4, -3, -2, -1)]
        maps += [memb[z + s * k].double() for k in (-2, -1, 0, 1, 2)]
        p = _forward64("maskextend", params, _pad64(torch.stack(maps), r))
        mean = F.avg_pool2d(_pad64(p[:1], 1)[None], 3, stride=1)[0, 0]
        masks[z] = (mean >= 0.5).double()
        probs.append(p.float())
    return {"masks": None, "probs": torch.stack(probs)}  # a mask is a decision, not a computed number


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":  # which slices a step draws is the library's own
        return None
    i = _inputs(case, seed)
    if kind == "batch":
        return [_map64("teacher", _params("teacher", seed), x) for x in i["xs"]]
    if kind == "grad":
        return _grad64(case, _params("student", seed), i["x"], i["t"])
    if kind == "mask":
        return _masks64(case, _params("maskextend", seed), i["em"], i["memb"], i["seeds"])
    box = (case["y0"], case["x0"], case["rows"], case["cols"]) if kind == "region" else None
    out = _map64(case["net"], _params(case["net"], seed), i["x"], box)
    return out[:, ::2, ::2].contiguous() if case.get("subsample") else out
