"""The workloads that the library's speed is judged on.

Each case is one call (or one short sequence of calls) that a program using
the library makes, with the sizes of the repository's benchmark and tests:
single images of every pixel type, batches in one persistent launch, the main
problem (smoothed rows and a bend angle), the queries of Sec. 3, the
standalone FHT / DP / read-back layers, and the network of the learned window
proposal, forward and training.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_1912_01884_gb300 as fd
from paper_1912_01884_gb300 import learned

DEV = "cuda"
C = 32                        # channels of the proposal network
RESUMED, SECOND = 1000, 1e-6  # Adam steps before the measured one, second moments then
TYPES = {"u8": torch.uint8, "i32": torch.int32, "f32": torch.float32}


def listed():
    return [
        # One small image, one call: latency (the benchmark's 256 x 256 workload).
        {"name": "detect_u8_256", "kind": "detect", "type": "u8", "h": 256, "w": 256, "n": 64, "B": 8},
        # One large image, one call: a document photo or a camera frame.
        {"name": "detect_u8_2048", "kind": "detect", "type": "u8", "h": 2048, "w": 2048, "n": 128, "B": 16},
        # One very large float response map.
        {"name": "detect_f32_8192", "kind": "detect", "type": "f32", "h": 8192, "w": 8192, "n": 128, "B": 24},
        # A data set of images of many sizes, kept in one tuned plan and run again
        # and again (the benchmark's headline workload).
        {"name": "batch_u8_mixed", "kind": "batch", "type": "u8", "count": 256, "hlo": 512, "hhi": 4096,
         "wlo": 512, "whi": 3072, "step": 256, "nlo": 32, "nhi": 256, "bend": 8, "tune": True},
        # A short batch of int32 images of ragged sizes (filter responses), run as planned.
        {"name": "batch_i32_ragged", "kind": "batch", "type": "i32", "count": 24, "hlo": 200, "hhi": 1200,
         "wlo": 201, "whi": 1500, "step": 1, "nlo": 16, "nhi": 128, "bend": 6, "tune": False},
        # The paper's main problem on one image: smoothed rows, bend angle of 10 degrees.
        {"name": "main_u8_2048", "kind": "main", "type": "u8", "h": 2048, "w": 2048, "n": 128, "r": 2,
         "gamma": 0.1745},
        # The main problem on a batch: the rows of every image smoothed, then one launch.
        {"name": "main_batch_u8_2048", "kind": "main_batch", "type": "u8", "count": 16, "h": 2048, "w": 2048,
         "n": 128, "r": 2, "gamma": 0.1745},
        # Two different curves of one image (the two page borders of Sec. 3).
        {"name": "two_u8_2048", "kind": "query", "query": "two", "type": "u8", "h": 2048, "w": 2048,
         "n": 128, "B": 16},
        # The three layers by themselves, as a program uses that wants the Hough
        # images or DP values: a ragged float image.
        {"name": "layers_f32_1531", "kind": "layers", "type": "f32", "h": 1024, "w": 1531, "n": 64, "B": 12},
        # The proposal network on a batch of camera frames.
        {"name": "propose_1024", "kind": "propose", "count": 64, "h": 1024, "w": 1024, "bands": 16},
        # One convolution layer of that network, forward and both gradients.
        {"name": "conv_layer_256", "kind": "conv", "count": 32, "h": 256, "w": 256, "dil": 4},
        # One training step of that network, in the middle of its training.
        {"name": "train_step_1024", "kind": "train", "count": 32, "h": 1024, "w": 1024, "bands": 16},
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], evenly spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _rows(rng, lo, hi, n):
    return max(1, _spread(rng, lo, hi) // n) * n


def draw(rng):
    kind = rng.choice(["detect", "detect", "detect", "batch", "batch", "main", "main_batch", "query", "query",
                       "layers", "propose", "conv", "train"])
    n = rng.choice([16, 32, 64, 128, 128, 256])
    typ = rng.choice(["u8", "u8", "i32", "f32"])
    if kind == "detect":
        return {"kind": kind, "type": typ, "h": _rows(rng, 256, 8192, n), "w": _spread(rng, 200, 8192), "n": n,
                "B": rng.choice([max(1, n // 8), n // 5 + 1, n // 4])}
    if kind == "batch":
        nlo, nhi = rng.choice([(16, 128), (32, 256), (64, 64), (32, 128)])
        hlo, wlo = _spread(rng, 256, 1024), _spread(rng, 200, 1024)
        return {"kind": kind, "type": typ, "count": _spread(rng, 4, 64), "hlo": hlo, "hhi": 2 * hlo, "wlo": wlo,
                "whi": 2 * wlo, "step": rng.choice([1, 16, 256]), "nlo": nlo, "nhi": nhi,
                "bend": rng.choice([4, 6, 8]), "tune": False}
    r = rng.choice([0, 1, 2, 3])
    gamma = round(rng.uniform(0.08, 0.35), 4)
    if kind == "main":
        return {"kind": kind, "type": typ, "h": _rows(rng, 256, 4096, n), "w": _spread(rng, 200, 4096), "n": n,
                "r": r, "gamma": gamma}
    if kind == "main_batch":
        n = min(n, 128)
        return {"kind": kind, "type": typ, "count": _spread(rng, 2, 16), "h": _rows(rng, 256, 2048, n),
                "w": _spread(rng, 200, 2048), "n": n, "r": max(1, r), "gamma": gamma}
    if kind == "query":
        return {"kind": kind, "query": rng.choice(["two", "padded", "through", "horizontal"]), "type": typ,
                "h": _rows(rng, 256, 4096, 256), "w": 256 * _spread(rng, 1, 16) if rng.random() < 0.5
                else 256 * _spread(rng, 1, 15) + 64, "n": min(n, 64), "B": max(1, min(n, 64) // 8)}
    if kind == "layers":
        return {"kind": kind, "type": typ, "h": _rows(rng, 128, 4096, n), "w": _spread(rng, 150, 4096), "n": n,
                "B": max(1, n // 6)}
    bands = rng.choice([8, 16])
    if kind == "conv":
        return {"kind": kind, "count": _spread(rng, 1, 32), "h": _spread(rng, 64, 256), "w": 64 * _spread(rng, 1, 5),
                "dil": rng.choice([1, 2, 4, 8])}
    return {"kind": kind, "count": _spread(rng, 1, 32), "h": 4 * bands * _spread(rng, 4, 16),
            "w": 256 * _spread(rng, 1, 4), "bands": bands}


# ---------------------------------------------------------------------------
# Inputs.

def _polyline(rng, h, w, n, B):
    """Columns [h] of one rasterised polyline of links with bends within B."""
    k = h // n
    most = min(n - 1, max(1, w // (2 * k) if k * n > w else n - 1))
    d = [int(rng.integers(-most, most + 1))]
    for _ in range(1, k):
        d.append(int(np.clip(d[-1] + rng.integers(-B, B + 1), -(n - 1), n - 1)))
    offs = np.concatenate([[0], np.cumsum(d)])
    lo, hi = -int(offs.min()), w - 1 - int(offs.max())
    x = (int(rng.integers(lo, hi + 1)) if hi >= lo else w // 2) + offs[:-1]
    y = np.arange(n)
    cols = x[:, None] + np.round(np.asarray(d)[:, None] * y[None, :] / max(1, n - 1)).astype(np.int64)
    return np.clip(cols.reshape(-1), 0, w - 1)


def _image(rng, gen, typ, h, w, n, B, lines=2):
    """One image of `typ`: noise and bright polylines (float images: |N(0, 1)|
    and ridges of height 3 and Gaussian width 1.5)."""
    if typ == "f32":
        img = torch.randn(h, w, generator=gen, device=DEV).abs_()
    else:
        img = torch.randint(0, 41 if typ == "u8" else 1000, (h, w), generator=gen, device=DEV, dtype=TYPES[typ])
    y = torch.arange(h, device=DEV)
    for _ in range(lines):
        x = torch.from_numpy(_polyline(rng, h, w, n, B)).to(DEV)
        if typ == "f32":
            for dx in range(-3, 4):
                xx = x + dx
                ok = (xx >= 0) & (xx < w)
                img[y[ok], xx[ok]] += 3.0 * math.exp(-dx * dx / 4.5)
        else:
            img[y, x] = int(rng.integers(120, 201)) * (1 if typ == "u8" else 25)
    return img


def _gens(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    return np.random.default_rng(int(seed)), gen


def _heights(lo, hi):
    return [n for n in (1, 2, 4, 8, 16, 32, 64, 128, 256) if lo <= n <= hi]


def _batch_shapes(case):
    """(h, w, n, B) of every image of a batch: the same for every seed, as a
    data set's sizes are."""
    rng = np.random.default_rng(12345 + case["count"])
    got = []
    for _ in range(case["count"]):
        n = int(rng.choice(_heights(case["nlo"], case["nhi"])))
        h = int(rng.integers(case["hlo"] // case["step"], case["hhi"] // case["step"] + 1)) * case["step"]
        w = int(rng.integers(case["wlo"] // case["step"], case["whi"] // case["step"] + 1)) * case["step"]
        got.append((max(1, h // n) * n, max(w, 64), n, max(1, n // case["bend"])))
    return got


def _query_shape(case):
    """(h, w, k): horizontal curves take bands of columns."""
    return case["h"], case["w"], (case["w"] if case["query"] == "horizontal" else case["h"]) // case["n"]


def prepare(case, seed):
    rng, gen = _gens(seed)
    kind = case["kind"]
    s = {"case": case}
    if kind in ("detect", "main", "layers", "query"):
        s["img"] = _image(rng, gen, case["type"], case["h"], case["w"], case["n"], case.get("B", case["n"] // 8))
    if kind == "layers":
        # a program that uses the layers keeps their arrays
        h, w, k = case["h"], case["w"], case["h"] // case["n"]
        s["hough"] = torch.empty(k, 2, case["n"], w + case["n"], device=DEV,
                                 dtype=torch.float32 if case["type"] == "f32" else torch.int32)
        code = fd._dtype_code(s["img"])
        s["ws"] = torch.empty(max(1, fd.fht_workspace_bytes(code, h, w, k)), dtype=torch.uint8, device=DEV)
    elif kind == "batch":
        shapes = _batch_shapes(case)
        imgs = [_image(rng, gen, case["type"], h, w, n, B, 1) for h, w, n, B in shapes]
        s["plan"] = fd.BatchPlan(imgs, [h // n for h, w, n, B in shapes], [B for h, w, n, B in shapes])
        if case["tune"]:
            s["plan"].autotune()
    elif kind == "main_batch":
        h, w, n = case["h"], case["w"], case["n"]
        s["imgs"] = [_image(rng, gen, case["type"], h, w, n, n // 8) for _ in range(case["count"])]
        s["rows"] = [fd.gauss_rows(im, case["r"]) for im in s["imgs"]]
        s["plan"] = fd.BatchPlan(s["rows"], [h // n] * case["count"], [2 * n - 2] * case["count"])
        s["plan"].angle(case["gamma"])
    elif kind in ("propose", "train"):
        N, h, w, bands = case["count"], case["h"], case["w"], case["bands"]
        s["model"] = learned.LaneProposer(seed=seed % 1000, device=DEV)
        s["imgs"] = torch.cat([learned.lane_images(seed + i, min(16, N - i), h, w, bands, max(1, h // bands // 6), DEV)
                               for i in range(0, N, 16)])
        s["labels"] = torch.randint(4, 28, (N, bands), generator=gen, device=DEV, dtype=torch.int32)
        if kind == "train":
            # training resumed after RESUMED steps: second moments of the size
            # that the gradients have had (from zero ones the first step moves
            # every parameter by the learning rate, whatever its gradient is)
            s["model"].step_count = RESUMED
            for part in _params(s["model"]):
                part["vw"].fill_(SECOND)
                part["vb"].fill_(SECOND)
    elif kind == "conv":
        N, h, w = case["count"], case["h"], case["w"]
        x = torch.randn(N, h, w, C, generator=gen, device=DEV).clamp_(min=0).to(torch.bfloat16)
        s.update(x=x, dz=(torch.randn(N, h, w, C, generator=gen, device=DEV) * 0.01).to(torch.bfloat16),
                 wt=(torch.randn(9, C, C, generator=gen, device=DEV) * math.sqrt(2 / 288)).to(torch.bfloat16),
                 bias=torch.randn(C, generator=gen, device=DEV) * 0.1,
                 y=torch.empty_like(x), dx=torch.empty_like(x),
                 wflip=torch.empty(9, C, C, device=DEV, dtype=torch.bfloat16),
                 dw=torch.empty(9, C, C, device=DEV), db=torch.empty(C, device=DEV))
    return s


# ---------------------------------------------------------------------------
# One pass.

def _ok(code):
    if code:
        raise fd.FhtdpError(code, fd.lib().fhtdp_last_error().decode())


def _plan_outputs(plan):
    """Every image's polyline and score: vertices, displacements and scores of
    the images one after the other."""
    return torch.cat(plan.x), torch.cat(plan.d), torch.cat(plan.score)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "detect":
        return fd.detect_polyline(s["img"], case["h"] // case["n"], case["B"])
    if kind == "main":
        return fd.detect_polyline_angle(s["img"], case["h"] // case["n"], case["r"], case["gamma"])
    if kind == "query":
        h, w, k = _query_shape(case)
        if case["query"] == "two":
            return fd.detect_two_polylines(s["img"], k, case["B"], max(1, w // 32))
        if case["query"] == "padded":
            return fd.detect_polyline_padded(s["img"], k, case["B"])
        if case["query"] == "through":
            return fd.detect_through_point(s["img"], k, case["B"], k // 2, w // 2)
        return fd.detect_polyline_horizontal(s["img"], k, case["B"])
    if kind == "layers":
        h, w, k, B = case["h"], case["w"], case["h"] // case["n"], case["B"]
        V = fd.fht_bands(s["img"], k, out=s["hough"], ws=s["ws"])
        fd.polyline_dp(V, h, w, k, B)
        return (V,) + tuple(fd.backtrack(V, h, w, k, B))
    if kind == "batch":
        s["plan"].run()
        return _plan_outputs(s["plan"])
    if kind == "main_batch":
        for im, rows in zip(s["imgs"], s["rows"]):
            fd.gauss_rows(im, case["r"], out=rows)
        s["plan"].run()
        return _plan_outputs(s["plan"])
    if kind == "propose":
        pred, conf = s["model"].forward(s["imgs"], case["bands"])
        return {"pred": pred, "conf": conf, "logits": _logits(s["model"], case)}
    if kind == "train":
        loss = s["model"].train_step(s["imgs"], s["labels"], case["bands"])
        return {"loss": loss, "state": _training_state(s["model"])}
    L, st = fd.lib(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    N, h, w, dil = case["count"], case["h"], case["w"], case["dil"]
    p = {a: v.data_ptr() for a, v in s.items() if isinstance(v, torch.Tensor)}
    _ok(L.fhtdp_cnn_conv3x3(p["x"], C, N, h, w, dil, p["wt"], p["bias"], 1, p["y"], st))
    _ok(L.fhtdp_cnn_conv3x3_dgrad(p["dz"], N, h, w, dil, p["wt"], p["wflip"], p["dx"], st))
    s["dw"].zero_()
    s["db"].zero_()
    _ok(L.fhtdp_cnn_conv3x3_wgrad(p["x"], C, N, h, w, dil, p["dz"], p["dw"], p["db"], st))
    return {"y": s["y"], "dx": s["dx"], "dw": s["dw"], "db": s["db"]}


def _training_state(model):
    """What a training step updates: weights, biases and first moments (which
    hold the gradients)."""
    return [{a: v for a, v in part.items() if a[0] != "v"} for part in _params(model)]


def _up(v):
    return (v + 255) // 256 * 256


def _logits(model, case):
    """The last layer's output, which a forward pass leaves in the workspace
    (after the pooled input and the other three layers' outputs)."""
    N, H, W = case["count"], case["h"] // 4, case["w"] // 4
    px = N * H * W
    at = _up(2 * px) + 3 * _up(2 * px * C)
    return model._ws[at:at + 2 * px * C].view(torch.bfloat16).view(N, H, W, C)


def _params(model):
    """Per layer, views of the documented parameter block: FP32 weights, bias
    and their Adam moments (first, second)."""
    got, o = [], 0
    for layer in range(4):
        rows = 16 if layer == 0 else 9 * C
        part = {}
        for name, count, size in (("w", rows * C, 4), ("b", C, 4), ("mw", rows * C, 4), ("vw", rows * C, 4),
                                  ("mb", C, 4), ("vb", C, 4), ("w16", rows * C, 2)):
            if size == 4:
                part[name] = model.params[o:o + 4 * count].view(torch.float32)
            o = _up(o + size * count)
        got.append(part)
    return got


# ---------------------------------------------------------------------------
# What one pass cannot do without.

def _method(h, w, n, size):
    """Bytes and additions / comparisons of the method on one image: the image
    read once, the polyline written; the FHT's additions over both slope signs
    and one addition and two comparisons per DP state."""
    k = h // n
    states = k * 2 * n * (w + n)
    return h * w * size + 4 * (2 * k + 2), states * (math.log2(n) + 3)


def work(case):
    kind = case["kind"]
    size = {"u8": 1}.get(case.get("type"), 4)
    if kind == "batch":
        every = [_method(h, w, n, size) for h, w, n, B in _batch_shapes(case)]
        return {"bytes": sum(b for b, f in every), "flops": sum(f for b, f in every)}
    if kind in ("detect", "main", "main_batch", "layers", "query"):
        h, w, n = case["h"], case["w"], case["n"]
        if kind == "query" and case["query"] == "horizontal":
            h, w = w, h
        b, f = _method(h, w, n, size)
        if kind in ("main", "main_batch"):
            f += h * w * 2 * (2 * case["r"] + 1)
        if kind == "main_batch":   # the smoothed rows are written and read
            b, f = (b + 8 * h * w) * case["count"], f * case["count"]
        if kind == "layers":
            b += 4 * (h // n) * 2 * n * (w + n)
        return {"bytes": b, "flops": f}
    N, h, w = case["count"], case["h"], case["w"]
    if kind == "conv":
        px = N * h * w
        return {"bytes": px * C * 2 * 4, "flops": 3 * px * 2 * 9 * C * C}
    px = N * h * w // 16
    layers = 2 * 9 * C * px * (1 + 3 * C)
    act = 2 * px * C
    if kind == "propose":   # the images read, the four layers' outputs written
        return {"bytes": N * h * w + 4 * act, "flops": layers}
    # ... and read once more by the backward pass, which writes nothing so large
    return {"bytes": N * h * w + 8 * act, "flops": 3 * layers - 2 * 9 * C * px}


# ---------------------------------------------------------------------------
# The results in 64 bits.

def _bands64(img, n, r):
    """float64 Hough values [k][2n - 1][W] (row d + n - 1) of the smoothed,
    zero-padded bands; columns modulo W."""
    h, w = img.shape
    x = img.double()
    if r:
        sm = torch.zeros_like(x)
        for t in range(-r, r + 1):
            lo, hi = max(0, -t), min(w, w - t)
            sm[:, lo:hi] += math.comb(2 * r, r + t) * x[:, lo + t:hi + t]
        x = sm
    x = torch.cat([x, torch.zeros(h, n, dtype=torch.float64, device=img.device)], 1)
    halves = []
    for sign in (1, -1):
        cur = x.view(h, 1, -1)   # [sub-bands][shift][W]
        m = 1
        while m < n:
            m *= 2
            a, b = cur[0::2], cur[1::2]
            cur = torch.stack([a[:, q >> 1] + torch.roll(b[:, q >> 1], -sign * (q - (q >> 1)), -1)
                               for q in range(m)], 1)
        halves.append(cur)
    return halves


def _tables(case, n):
    if "gamma" in case:
        t = np.arctan(np.arange(-(n - 1), n) / n)
        ok = np.abs(t[:, None] - t[None, :]) <= case["gamma"]
    else:
        d = np.arange(2 * n - 1)
        ok = np.abs(d[:, None] - d[None, :]) <= case["B"]
    return [(int(np.flatnonzero(row)[0]), int(np.flatnonzero(row)[-1])) for row in ok]


def _dp64(img, case, keep=False, padded=False):
    """The optimum's score in 64 bits, and with `keep` every DP value in the
    layout of polyline_dp."""
    n = case["n"]
    h, w = img.shape
    k, D, W = h // n, 2 * n - 1, w + n
    vw = W if padded else w
    plus, minus = _bands64(img, n, case.get("r", 0))
    win = _tables(case, n)
    dead = float("-inf")
    x = torch.arange(W, device=img.device)
    d = torch.arange(D, device=img.device) - (n - 1)
    end = x[None, :] + d[:, None]
    dies = (end < 0) | (end >= vw) | (x[None, :] >= vw)
    V, kept = None, []
    for b in range(k - 1, -1, -1):
        H = torch.cat([torch.flip(minus[b][1:], [0]), plus[b]], 0)
        if V is not None:
            M = torch.stack([V[lo:hi + 1].max(0).values for lo, hi in win])   # at the end column
            H = H + torch.gather(M, 1, end.clamp(0, W - 1))
        V = torch.where(dies, torch.full_like(H, dead), H)
        if keep:
            kept.append(torch.stack([V[n - 1:], torch.flip(V[:n], [0])]))
    score = V.max().reshape(1)
    return score, torch.stack(kept[::-1]) if keep else None


def _conv64(x, wt, dil):
    """float64 3x3 dilated convolution, NHWC, weights [9][ci][co]."""
    N, H, W, ci = x.shape
    p = torch.nn.functional.pad(x, (0, 0, dil, dil, dil, dil))
    y = torch.zeros(N, H, W, wt.shape[2], dtype=torch.float64, device=x.device)
    for t in range(9):
        oy, ox = (t // 3) * dil, (t % 3) * dil
        y += p[:, oy:oy + H, ox:ox + W] @ wt[t]
    return y


def _wgrad64(x, dz, dil):
    N, H, W, ci = x.shape
    p = torch.nn.functional.pad(x, (0, 0, dil, dil, dil, dil))
    z = dz.reshape(-1, dz.shape[3])
    return torch.stack([p[:, (t // 3) * dil:(t // 3) * dil + H, (t % 3) * dil:(t % 3) * dil + W]
                        .reshape(-1, ci).T @ z for t in range(9)])


def _net64(model, imgs):
    """Activations of the four layers (the input first) in 64 bits, from the
    bf16 weights; and the layers' weights."""
    N, h, w = imgs.shape
    x = imgs.view(N, h // 4, 4, w // 4, 4).double().mean((2, 4)).unsqueeze(3) / 255.0
    state = _training_state(model)
    acts, ws = [x], []
    for layer, dil in enumerate((1, 2, 4, 8)):
        wt = state[layer]["w"].to(torch.bfloat16).double()
        wt = wt.view(16, C)[:9].reshape(9, 1, C) if layer == 0 else wt.view(9, C, C)
        y = _conv64(acts[-1], wt, dil) + state[layer]["b"].double()
        acts.append(y.clamp(min=0) if layer < 3 else y)
        ws.append(wt)
    return acts, ws


def _head64(logits, bands):
    N, H, W, _ = logits.shape
    return torch.logsumexp(logits.view(N, bands, H // bands * W, C), 2)


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("conv", "propose", "train"):
        # whole numbers have no nearer value; plans and queries of several
        # images are the same method as the single calls
        if case["type"] != "f32" or kind in ("batch", "main_batch") or case.get("query") in ("two", "through"):
            return None
        img = prepare(case, seed)["img"]
        if case.get("query") == "horizontal":
            img = img.T.contiguous()
        score, V = _dp64(img, case, keep=kind == "layers", padded=case.get("query") == "padded")
        if kind == "layers":
            return V, None, None, score
        return None, None, score
    s = prepare(case, seed)
    if kind == "conv":
        x, dz, wt, dil = s["x"].double(), s["dz"].double(), s["wt"].double(), case["dil"]
        return {"y": (_conv64(x, wt, dil) + s["bias"].double()).clamp(min=0),
                "dx": _conv64(dz, torch.flip(wt, [0]).transpose(1, 2), dil),
                "dw": _wgrad64(x, dz, dil), "db": dz.sum((0, 1, 2))}
    acts, ws = _net64(s["model"], s["imgs"])
    bands = case["bands"]
    if kind == "propose":
        return {"pred": None, "conf": torch.softmax(_head64(acts[4], bands), 2).max(2).values, "logits": acts[4]}
    N, H, W, _ = acts[4].shape
    pooled = _head64(acts[4], bands)
    lse = torch.logsumexp(pooled, 2, keepdim=True)
    hot = torch.nn.functional.one_hot(s["labels"].long(), C).double()
    loss = ((lse.squeeze(2) - (pooled * hot).sum(2)).sum() / (N * bands)).reshape(1)
    g = (torch.exp(pooled - lse) - hot) / (N * bands)
    per = acts[4].view(N, bands, H // bands * W, C)
    dz = (g.unsqueeze(2) * torch.exp(per - pooled.unsqueeze(2))).view(N, H, W, C)
    state = _training_state(s["model"])
    out = [None] * 4
    for layer in (3, 2, 1, 0):
        dil = (1, 2, 4, 8)[layer]
        gw, gb = _wgrad64(acts[layer], dz, dil).reshape(-1), dz.sum((0, 1, 2))
        if layer:
            dz = _conv64(dz, torch.flip(ws[layer], [0]).transpose(1, 2), dil) * (acts[layer] > 0)
        else:   # the first layer's block has 16 rows, nine of them taps
            gw = torch.cat([gw, torch.zeros(7 * C, dtype=torch.float64, device=DEV)])
        c1, c2 = 1 / (1 - 0.9 ** (RESUMED + 1)), 1 / (1 - 0.999 ** (RESUMED + 1))
        v = lambda g: (0.999 * SECOND + 0.001 * g * g) * c2          # noqa: E731
        step = lambda p, g: p.double() - s["model"].lr * 0.1 * g * c1 / (v(g).sqrt() + 1e-8)   # noqa: E731
        out[layer] = {"w": step(state[layer]["w"], gw), "b": step(state[layer]["b"], gb),
                      "mw": 0.1 * gw, "mb": 0.1 * gb}
    return {"loss": loss, "state": out}
