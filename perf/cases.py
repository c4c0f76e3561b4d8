"""The work a user of the library has it do, as cases that can be timed: the
segmentation chain on lone tiles, batches and whole slides, its single
operations, the per-object steps after it, and a training step of the
schedule picker. Everything goes through the public Python entry points.

Inputs are the seeded nuclei tiles of the library's own generator (the GPU
twin of synth/), at the sizes and nuclei densities of the benchmark
configurations; the single operations get what the step before them in the
chain produces.
"""
from __future__ import annotations

import math
import os
import random

import numpy as np
import torch

import paper_1405_7958_gb300 as rt
from paper_1405_7958_gb300 import picker as picker_mod

WEIGHTS = os.path.join(os.path.dirname(rt.__file__), "data", "picker_config4.npz")
BYTES_CHAIN, BYTES_RF = 9, 2                   # per pixel: image 1, labels 4, distances 4; R and F 1 each
MAX_BATCH_PX = 8 * 4096 * 4096


def listed():
    return [
        # the 512 x 512 reconstruction on its own: the smallest call, where latency counts
        {"name": "recon_512", "op": "recon", "H": 512, "W": 512, "density": 229.0, "flat": True, "conn": 8,
         "given_marker": False},
        # a lightly loaded server: one ragged tile, the trained picker attached
        {"name": "lone_1k_learned", "op": "chain", "tiles": 1, "H": 1021, "W": 1153, "density": 178.8,
         "learned": True, "extra": False},
        # one 4K tile at a time, the plain schedule
        {"name": "lone_4k", "op": "chain", "tiles": 1, "H": 4096, "W": 4096, "density": 178.8, "learned": False,
         "extra": False},
        # the throughput form: 8 4K tiles a call, R and F returned too
        {"name": "batch_8x4k", "op": "chain", "tiles": 8, "H": 4096, "W": 4096, "density": 178.8, "learned": True,
         "extra": True},
        # a call of uneven tiles: sides 1024..4096 in steps of 256, 50..400 nuclei per megapixel
        {"name": "uneven_16", "op": "uneven", "tiles": 16, "lo": 1024, "hi": 4096, "step": 256, "learned": False},
        # a whole slide as one image: the largest call
        {"name": "slide_16k", "op": "chain", "tiles": 1, "H": 16384, "W": 16384, "density": 178.8, "learned": False,
         "extra": False},
        # the chain's operations called one by one on a 4K tile (one of them ragged)
        {"name": "fill_4k", "op": "fill", "H": 4096, "W": 4096, "density": 178.8, "conn": 4},
        {"name": "label_4k", "op": "label", "H": 4096, "W": 4096, "density": 178.8, "conn": 8},
        {"name": "edt_4k_ragged", "op": "edt", "H": 4001, "W": 3907, "density": 178.8},
        # the per-object steps after the chain
        {"name": "watershed_4k", "op": "watershed", "H": 4096, "W": 4096, "density": 178.8, "h": 2},
        {"name": "object_features_4k", "op": "features", "H": 4096, "W": 4096, "density": 250.0},
        # one training step of the picker: forward, backward, update
        {"name": "picker_step_256", "op": "train", "batch": 256},
    ]


def _log(rng: random.Random, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _side(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(_log(rng, lo, hi)))


def draw(rng):
    op = rng.choice(["recon", "chain", "chain", "batch", "uneven", "slide", "fill", "label", "edt", "watershed",
                     "features", "train"])
    density = round(rng.uniform(50.0, 400.0), 1)
    if op == "train":
        return {"op": "train", "batch": _side(rng, 64, 2048)}
    if op == "recon":
        return {"op": "recon", "H": _side(rng, 256, 4096), "W": _side(rng, 256, 4096), "density": density,
                "flat": rng.random() < 0.5, "conn": rng.choice([8, 8, 8, 4]), "given_marker": rng.random() < 0.3}
    if op == "chain":
        return {"op": "chain", "tiles": 1, "H": _side(rng, 512, 4096), "W": _side(rng, 512, 4096),
                "density": density, "learned": rng.random() < 0.5, "extra": rng.random() < 0.5}
    if op == "batch":
        H, W = _side(rng, 512, 4096), _side(rng, 512, 4096)
        return {"op": "chain", "tiles": max(2, min(rng.randint(2, 10), MAX_BATCH_PX // (H * W))), "H": H, "W": W,
                "density": density, "learned": rng.random() < 0.5, "extra": rng.random() < 0.5}
    if op == "uneven":
        lo, hi = rng.choice([(512, 2048), (1024, 4096), (700, 3000)])
        return {"op": "uneven", "tiles": rng.randint(3, 16), "lo": lo, "hi": hi, "step": rng.choice([256, 173, 1]),
                "learned": rng.random() < 0.5}
    if op == "slide":
        return {"op": "chain", "tiles": 1, "H": _side(rng, 5000, 14000), "W": _side(rng, 5000, 14000),
                "density": density, "learned": False, "extra": False}
    H, W = _side(rng, 700, 8192), _side(rng, 700, 8192)
    case = {"op": op, "H": H, "W": W, "density": density}
    if op == "fill":
        case["conn"] = rng.choice([4, 4, 8])
    elif op == "label":
        case["conn"] = rng.choice([8, 8, 4])
    elif op == "watershed":
        case["h"] = rng.choice([0, 2, 2, 8])
    return case


# ------------------------------------------------------------------- inputs
def _shapes(case, seed):
    """(H, W, nuclei, tile seed) of every tile of a chain case."""
    if case["op"] != "uneven":
        n = int(round(case["density"] * case["H"] * case["W"] / 1e6))
        return [(case["H"], case["W"], n, 1000 * seed + i) for i in range(case.get("tiles", 1))]
    # the sides belong to the case (a server's tiles), the contents to the seed
    rng = random.Random("%(tiles)d %(lo)d %(hi)d %(step)d" % case)
    out = []
    for i in range(case["tiles"]):
        H = case["lo"] + case["step"] * rng.randint(0, (case["hi"] - case["lo"]) // case["step"])
        W = case["lo"] + case["step"] * rng.randint(0, (case["hi"] - case["lo"]) // case["step"])
        out.append((H, W, int(round(rng.uniform(50.0, 400.0) * H * W / 1e6)), 1000 * seed + i))
    return out


def _tile(case, seed):
    H, W, n, s = _shapes(case, seed)[0]
    if case.get("flat"):
        return rt.synth_tile(H, W, s, n, kind="disk", vlo=40, vhi=90, rmin=4, rmax=12, background="flat")
    return rt.synth_tile(H, W, s, n)


def _int(n=1):
    return torch.zeros(n, dtype=torch.int32, device="cuda")


def _some_objects(labels, k, seed):
    """The label image with k of its objects (about two thirds of them), so
    that the number of feature rows belongs to the case, not to the seed."""
    own = torch.arange(labels.numel(), dtype=torch.int32, device=labels.device).reshape(labels.shape)
    ids = labels[labels == own].cpu()
    k = max(1, min(k, ids.numel()))
    keep = torch.zeros(labels.numel() + 1, dtype=torch.bool, device=labels.device)
    pick = torch.randperm(ids.numel(), generator=torch.Generator().manual_seed(seed))[:k]
    keep[ids[pick].to(labels.device).to(torch.int64)] = True
    return torch.where(keep[labels.to(torch.int64)], labels, torch.full_like(labels, -1)), k


def _train_batch(case, seed):
    g = torch.Generator().manual_seed(seed)
    B = case["batch"]
    scale = torch.rand(24, generator=g) * 100 + 0.1
    x = (torch.randn(B, 24, generator=g) + torch.randn(24, generator=g)) * scale
    return x, torch.randint(0, 3, (B,), generator=g, dtype=torch.int32)


def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "case": case}
    if op == "train":
        x, y = _train_batch(case, seed)
        s["x"], s["y"] = x.cuda(), y.cuda()
        s["picker"] = rt.Picker(seed=seed)
        s["picker"].set_norm(s["x"])
        s["status"] = _int()
        return s
    if op in ("chain", "uneven"):
        shapes = _shapes(case, seed)
        s["images"] = [rt.synth_tile(H, W, sd, n) for H, W, n, sd in shapes]
        s["params"] = rt.SegParams(policy=1, pick_min_prob=600) if case["learned"] else rt.SegParams()
        s["ctx"] = rt.Context(workspace_bytes=rt.segment_workspace_bytes([t[:2] for t in shapes], s["params"]))
        if case["learned"]:
            s["picker"] = picker_mod.load(WEIGHTS)
            s["picker"].attach(s["ctx"])
        s["outputs"] = []
        for H, W, _, _ in shapes:
            o = {"L": torch.empty((H, W), dtype=torch.int32, device="cuda"),
                 "D": torch.empty((H, W), dtype=torch.int32, device="cuda"), "n_kept": _int(), "status": _int()}
            if case.get("extra"):
                o["R"] = torch.empty((H, W), dtype=torch.uint8, device="cuda")
                o["F"] = torch.empty((H, W), dtype=torch.uint8, device="cuda")
            s["outputs"].append(o)
        return s
    s["image"] = _tile(case, seed)
    s["status"], s["count"] = _int(), _int()
    if op == "recon":
        if case["given_marker"]:
            s["marker"] = rt.marker(s["image"], 30)
        s["out"] = torch.empty_like(s["image"])
        return s
    # what the chain's step before this one hands over
    if op == "fill":
        s["binary"] = (rt.reconstruct(s["image"]) < 80).to(torch.uint8)
        s["out"] = torch.empty_like(s["binary"])
        return s
    o = rt.segment_batch([s["image"]])[0]
    s["out"] = torch.empty_like(o["L"])
    if op == "label":
        s["binary"] = o["F"]
    elif op == "edt":
        s["binary"] = (o["L"] >= 0).to(torch.uint8)
    elif op == "watershed":
        s["labels"], s["d2"] = o["L"], o["D"]
    elif op == "features":
        s["labels"], s["cap"] = _some_objects(o["L"], _shapes(case, seed)[0][2] // 2, seed)
    return s


# --------------------------------------------------------------------- pass
def run(s):
    op, case = s["op"], s["case"]
    if op in ("chain", "uneven"):
        return rt.segment_batch(s["images"], s["params"], outputs=s["outputs"], ctx=s["ctx"])
    if op == "recon":
        R = rt.reconstruct(s["image"], s.get("marker"), conn=case["conn"], out=s["out"], status=s["status"])
        return {"R": R, "status": s["status"]}
    if op == "fill":
        return {"F": rt.fill_holes(s["binary"], conn=case["conn"], out=s["out"], status=s["status"]),
                "status": s["status"]}
    if op == "label":
        L = rt.label_area(s["binary"], conn=case["conn"], out=s["out"], n_kept=s["count"], status=s["status"])
        return {"L": L, "n_kept": s["count"], "status": s["status"]}
    if op == "edt":
        return {"D": rt.edt(s["binary"], out=s["out"], status=s["status"]), "status": s["status"]}
    if op == "watershed":
        B = rt.watershed(s["labels"], s["d2"], case["h"], out=s["out"], n_basins=s["count"], status=s["status"])
        return {"B": B, "n_basins": s["count"], "status": s["status"]}
    if op == "features":
        labels, feat = rt.object_features(s["labels"], s["image"], s["cap"], n_obj=s["count"], status=s["status"])
        return {"labels": labels, "features": feat, "n_obj": s["count"], "status": s["status"]}
    pk = s["picker"]
    logits, act, _ = pk.forward(s["x"], with_act=True, tensor_cores=True, status=s["status"])
    grad, loss = pk.backward(s["x"], act, logits, s["y"], tensor_cores=True, status=s["status"])
    pk.step()
    return {"logits": logits, "grad": grad, "loss": loss, "master": pk.master, "m": pk.m, "v": pk.v}


# --------------------------------------------------------------------- work
def work(case):
    op = case["op"]
    if op == "train":
        B, P = case["batch"], rt.Picker.NPARAM
        # input and labels in; parameters and moments in and out, gradient and logits out
        return {"bytes": B * (24 * 4 + 4 + 12) + P * (4 * 7 + 2), "flops": 6 * B * (24 * 64 + 64 * 64 + 64 * 3)}
    if op in ("chain", "uneven"):
        px = sum(H * W for H, W, _, _ in _shapes(case, 0))
        return {"bytes": px * (BYTES_CHAIN + (BYTES_RF if case.get("extra") else 0)), "flops": 0}
    per = {"recon": 3 if case.get("given_marker") else 2, "fill": 2, "label": 5, "edt": 5, "watershed": 12,
           "features": 5}[op]
    return {"bytes": case["H"] * case["W"] * per, "flops": 0}


# -------------------------------------------------------------------- exact
def exact(case, seed):
    """Only the object features and the picker's training step are computed
    in floating point; every other output is a whole number."""
    if case["op"] == "features":
        return _exact_features(case, seed)
    if case["op"] == "train":
        return _exact_train(case, seed)
    return None


def _exact_features(case, seed):
    s = prepare(case, seed)
    dev = s["image"].device
    L, img = s["labels"].to(torch.int64), s["image"].to(torch.int64)
    H, W = L.shape
    r, c = torch.nonzero(L >= 0, as_tuple=True)
    ids, k = torch.unique(L[r, c], return_inverse=True)
    n, v = ids.numel(), img[r, c]
    if n == 0:
        return None

    def total(x):
        return torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, k, x.to(torch.float64))

    def extreme(x, how, start):
        return torch.full((n,), start, dtype=torch.int64, device=dev).scatter_reduce_(0, k, x, how)

    pad = torch.full((H + 2, W + 2), -1, dtype=torch.int64, device=dev)
    pad[1:-1, 1:-1] = L
    same = [pad[r + 1 + dr, c + 1 + dc] == L[r, c] for dr, dc in ((-1, 0), (1, 0), (0, -1), (0, 1))]
    area = total(torch.ones_like(v))
    per = total(4 - sum(x.to(torch.int64) for x in same))
    r0, r1, c0, c1 = extreme(r, "amin", H), extreme(r, "amax", -1), extreme(c, "amin", W), extreme(c, "amax", -1)
    y, x = (r - r0[k]), (c - c0[k])
    sy, sx = total(y), total(x)
    vrr, vcc = (area * total(y * y) - sy * sy) / area ** 2, (area * total(x * x) - sx * sx) / area ** 2
    vrc = (area * total(y * x) - sy * sx) / area ** 2
    half, disc = (vrr + vcc) / 2, torch.sqrt(((vrr - vcc) / 2) ** 2 + vrc ** 2)
    l1, l2 = half + disc, torch.clamp(half - disc, min=0)
    ecc = torch.where(l1 > 0, torch.sqrt(1 - l2 / torch.where(l1 > 0, l1, torch.ones_like(l1))), torch.zeros_like(l1))
    si = total(v)
    hist = torch.bincount(k * 256 + v, minlength=n * 256).reshape(n, 256).to(torch.float64)
    p = hist / area[:, None]
    entropy = -torch.where(p > 0, p * torch.log2(torch.where(p > 0, p, torch.ones_like(p))), torch.zeros_like(p)).sum(1)
    median = (2 * hist.cumsum(1) < area[:, None]).sum(1)
    right = same[3]
    a, b = v[right] >> 5, img[r[right], c[right] + 1] >> 5
    g = torch.bincount(k[right] * 64 + a * 8 + b, minlength=n * 64).reshape(n, 64).to(torch.float64)
    d = (torch.arange(64, device=dev) // 8 - torch.arange(64, device=dev) % 8).to(torch.float64)
    n2 = g.sum(1)
    div = torch.where(n2 > 0, n2, torch.ones_like(n2))
    cols = [area, per, r1 - r0 + 1, c1 - c0 + 1, r0 + sy / area, c0 + sx / area, 4 * torch.sqrt(l1),
            4 * torch.sqrt(l2), ecc, 4 * math.pi * area / per ** 2, si / area,
            torch.sqrt((area * total(v * v) - si * si) / area ** 2), extreme(v, "amin", 256), extreme(v, "amax", -1),
            median, entropy, n2, (g * d ** 2).sum(1) / div, (g * g).sum(1) / div ** 2,
            (g / (1 + d.abs())).sum(1) / div]
    return {"labels": None, "features": torch.stack([q.to(torch.float64) for q in cols], 1), "n_obj": None,
            "status": None}


def _exact_train(case, seed):
    x, y = (t.numpy() for t in _train_batch(case, seed))
    x, B = x.astype(np.float64), len(x)
    pk = rt.Picker(seed=seed)
    master = pk.master.cpu().numpy().astype(np.float64)
    w = pk.wb.view(torch.bfloat16).to(torch.float64).cpu().numpy()   # the weights the forward works on
    sizes = (("W1", (64, 24)), ("b1", (64,)), ("W2", (64, 64)), ("b2", (64,)), ("W3", (3, 64)), ("b3", (3,)))
    q, at = {}, 0
    for name, shape in sizes:
        q[name] = w[at:at + math.prod(shape)].reshape(shape)
        at += math.prod(shape)
    sd = x.std(0, ddof=1) if B > 1 else np.zeros(24)
    xn = (x - x.mean(0)) / np.maximum(sd, 1e-6)
    h1 = np.maximum(xn @ q["W1"].T + q["b1"], 0)
    h2 = np.maximum(h1 @ q["W2"].T + q["b2"], 0)
    z = h2 @ q["W3"].T + q["b3"]
    top = z.max(1, keepdims=True)
    e = np.exp(z - top)
    loss = np.mean(np.log(e.sum(1)) + top[:, 0] - z[np.arange(B), y])
    dz = e / e.sum(1, keepdims=True)
    dz[np.arange(B), y] -= 1
    dz /= B
    dh2 = (dz @ q["W3"]) * (h2 > 0)
    dh1 = (dh2 @ q["W2"]) * (h1 > 0)
    g = {"W1": dh1.T @ xn, "b1": dh1.sum(0), "W2": dh2.T @ h1, "b2": dh2.sum(0), "W3": dz.T @ h2, "b3": dz.sum(0)}
    grad = np.concatenate([g[name].ravel() for name, _ in sizes])
    m, v = 0.1 * grad, 0.001 * grad * grad
    master = master - 3e-3 * (grad / (np.abs(grad) + 1e-8) + 1e-4 * master)
    return {"logits": z, "grad": grad, "loss": np.array([loss]), "master": master, "m": m, "v": v}
