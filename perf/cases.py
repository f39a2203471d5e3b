"""Performance cases of the per-frame hot path: what a program that tracks tools in K video streams calls.

A tick case is one `submit` + `sync` of a context (the newest frame of every stream goes through resize, encoder,
ConvLSTM, heads and, where switched on, the overlay), with the arguments marshalled once as a frame loop does.  A clip
case takes several ticks through one context with three submits in flight.  The stage cases call the stage-level entry
points on buffers of the caller.  Frames follow the recipe of the synthetic endoscopy video (drifting gradients,
elliptical blobs, noise of +-8); weights are fan-in scaled, so that logits spread over a few units and masks are real.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2402_04466_b200 import binding

RING = 2          # device frames per stream that a tick case goes round
IN_FLIGHT = 3     # submits a clip keeps in flight

_PALETTE = ((255, 0, 0), (0, 255, 0), (0, 0, 255), (255, 255, 0), (255, 0, 255), (0, 255, 255), (255, 128, 0), (128, 128, 128))

_RESULT = np.dtype({"names": ["conf", "cx", "cy", "count", "masks", "probs", "overlay"],
                    "formats": [("<f4", 8), ("<f4", 8), ("<f4", 8), ("<i4", 8), "<u8", "<u8", "<u8"],
                    "offsets": [16, 48, 80, 112, 144, 152, 160], "itemsize": ctypes.sizeof(binding.tt_result)})


def _tick(name, src, net, enc, stride, hidden, tools, streams, precision="bf16", conf="gap_linear", overlay=False,
          host=False, recurrent=True, ticks=1):
    c = {"kind": "tick", "src_w": src[0], "src_h": src[1], "net_w": net[0], "net_h": net[1], "enc": enc, "stride": stride,
         "hidden": hidden, "tools": tools, "streams": streams, "precision": precision, "conf": conf, "overlay": overlay,
         "host": host, "recurrent": recurrent, "ticks": ticks}
    if name:
        c["name"] = name
    return c


def listed():
    vga, hd = ((854, 480), (640, 480), "32,64,128", "2,2,2", 128, 7), ((1920, 1080), (1280, 720), "64,128,256", "2,2,2", 256, 7)
    return [
        # the smallest call: one 128x128 stream on the fp32 path, a latency check of a few small launches
        _tick("tick_tiny_fp32", (128, 128), (64, 64), "16", "1", 16, 4, 1, precision="fp32", conf="mean_sigmoid"),
        # fp32 path with a strided encoder and several streams
        _tick("tick_fp32_k3", (428, 240), (320, 240), "16,32", "2,2", 32, 5, 3, precision="fp32", conf="mean_sigmoid"),
        # one endoscopy stream by itself: the latency of a frame when nothing else runs
        _tick("tick_480p_k1", *vga, 1),
        # the headline: five concurrent endoscopy streams, frames already on the device
        _tick("tick_480p_k5", *vga, 5),
        # six streams with the overlay drawn for the display, frames arriving in pinned host memory
        _tick("tick_480p_k6_overlay_host", *vga, 6, overlay=True, host=True),
        # a feed-forward segmentation model on three streams (no recurrent cell)
        _tick("tick_480p_k3_feedforward", *vga, 3, recurrent=False),
        # a camera and a network whose sizes fit no tile, smaller model, other tool count and confidence
        _tick("tick_ragged_k3", (799, 601), (500, 374), "32,64", "2,2", 64, 5, 3, conf="mean_sigmoid"),
        # a full-HD stream by itself
        _tick("tick_1080p_k1", *hd, 1),
        # the largest: eight full-HD streams
        _tick("tick_1080p_k8", *hd, 8),
        # a recorded clip of five streams, six frames each, from pinned host memory, three submits in flight
        _tick("clip_480p_k5_host", *vga, 5, host=True, ticks=6),
        # format conversion alone, for a program with a model of its own: full-HD frames with padded rows
        {"name": "preprocess_1080p_k4", "kind": "preprocess", "src_w": 1920, "src_h": 1080, "net_w": 1280, "net_h": 720,
         "pad": 64, "streams": 4},
        # post-processing alone, on the fp32 channels-last state of a program's own recurrent cell
        {"name": "postprocess_160x90_k8", "kind": "postprocess", "hm": 90, "wm": 160, "hidden": 256, "tools": 7, "streams": 8,
         "channels_last": True, "conf": "gap_linear"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    cap = work(listed()[8])
    while True:
        kind = rng.choice(["tick"] * 7 + ["preprocess", "preprocess", "postprocess"])
        if kind == "postprocess":
            return {"kind": kind, "hm": _log(rng, 15, 120), "wm": _log(rng, 20, 200), "hidden": rng.choice([16, 24, 64, 128, 256, 512]),
                    "tools": rng.randint(1, 8), "streams": rng.randint(1, 8), "channels_last": rng.random() < 0.75,
                    "conf": rng.choice(["gap_linear", "mean_sigmoid"])}
        net_w, aspect, scale = _log(rng, 96, 1280), rng.choice([4 / 3, 16 / 9, 1.0]), math.exp(rng.uniform(math.log(0.75), math.log(2.5)))
        if rng.random() < 0.7:
            net_w = (net_w + 3) // 4 * 4
        net_h = max(64, int(net_w / aspect))
        src_w, src_h = min(1920, int(net_w * scale)), max(64, min(1080, int(net_h * scale * rng.choice([1.0, 0.8]))))
        streams = rng.randint(1, 8)
        if kind == "preprocess":
            return {"kind": kind, "src_w": src_w, "src_h": src_h, "net_w": net_w, "net_h": net_h, "pad": rng.choice([0, 0, 5, 64]), "streams": streams}
        fp32 = rng.random() < 0.25
        if fp32:
            enc, stride = rng.choice([("16", "1"), ("16", "2"), ("8,24", "2,2"), ("16,32", "2,2")])
            hidden = rng.choice([16, 24, 32])
        else:
            enc, stride = rng.choice([("32,64,128", "2,2,2"), ("64,128,256", "2,2,2"), ("32,64", "2,2"), ("32,64,64", "1,2,2"), ("64,128", "2,1")])
            hidden = rng.choice([64, 128, 256])
        recurrent = rng.random() < 0.8
        if not recurrent:
            hidden = int(enc.split(",")[-1])
        c = _tick(None, (src_w, src_h), (net_w, net_h), enc, stride, hidden, rng.randint(1, 8), streams, "fp32" if fp32 else "bf16",
                  rng.choice(["gap_linear", "mean_sigmoid"]), rng.random() < 0.25, rng.random() < 0.25, recurrent, rng.choice([1, 1, 1, 1, 4]))
        w = work(c)
        # a drawn case costs no more than the largest listed one; the fp32 path has no tensor cores and takes smaller models
        if w["bytes"] <= cap["bytes"] and w["flops"] <= (3e9 if fp32 else cap["flops"]):
            return c


# ------------------------------------------------------------------------------------------------ shapes and work
def _ints(text):
    return [int(v) for v in text.split(",")]


def _layers(c):
    """[(cin, cout, stride, h_out, w_out)] of the encoder."""
    out, cin, h, w = [], 3, c["net_h"], c["net_w"]
    for co, s in zip(_ints(c["enc"]), _ints(c["stride"])):
        h, w = (h - 1) // s + 1, (w - 1) // s + 1
        out.append((cin, co, s, h, w))
        cin = co
    return out


def work(case):
    c, k = case, case["streams"]
    if c["kind"] == "preprocess":
        n = c["net_w"] * c["net_h"] * 3
        return {"bytes": k * (3 * c["src_w"] * c["src_h"] + 4 * n), "flops": k * 8 * n}
    if c["kind"] == "postprocess":
        p = c["hm"] * c["wm"]
        return {"bytes": k * p * (4 * c["hidden"] + 9 * c["tools"]), "flops": k * p * 2 * c["hidden"] * c["tools"]}
    lay = _layers(c)
    p, hid, half = lay[-1][3] * lay[-1][4], c["hidden"], 2 if c["precision"] == "bf16" else 4
    flops = sum(18 * ci * co * h * w for ci, co, _, h, w in lay) + 2 * p * hid * c["tools"]
    weights = sum(9 * ci * co for ci, co, *_ in lay)
    nbytes = 3 * c["src_w"] * c["src_h"] + 5 * c["tools"] * p + (4 * c["src_w"] * c["src_h"] if c["overlay"] else 0)
    if c["recurrent"]:
        flops += 18 * (lay[-1][1] + hid) * 4 * hid * p
        weights += 9 * (lay[-1][1] + hid) * 4 * hid
        nbytes += p * hid * 2 * (4 + half)          # cell state and hidden state, read and written
    return {"bytes": c["ticks"] * (k * nbytes + half * weights), "flops": c["ticks"] * k * flops}


def tolerance(case):
    if case["kind"] == "preprocess":
        return {"rel": 1e-6, "max": 1e-5}             # fp32 arithmetic on bytes: measured 1.3e-7 against 64 bits
    # fp32 sums: measured 2e-7 against 64 bits for probabilities, logits and confidences.  The rest is room for one pixel
    # at the threshold that changes sides: it moves a size by 1 and a centroid by a fraction of a pixel.
    if case["kind"] == "postprocess":
        return {"rel": 1e-4, "max": 1e-2, "differ": 1e-4}
    if case["precision"] == "fp32":
        return {"rel": 4e-4, "max": 1e-2, "differ": 1e-3}
    # bf16 operands: measured up to 1.9e-3 against 64 bits for the probabilities; pixels whose logit lies within that of
    # the threshold change sides (0.04 % of the mask)
    return {"rel": 8e-3, "max": 1e-1, "differ": 4e-3}


# ------------------------------------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _frames(seed, streams, n, w, h):
    """uint8 [n][streams][h][w][3]: gradients that drift, 1..7 grey elliptical blobs, noise of +-8."""
    g, dev = _gen(seed), _device()
    yy = torch.arange(h, device=dev, dtype=torch.float32).view(h, 1)
    xx = torch.arange(w, device=dev, dtype=torch.float32).view(1, w)
    out = torch.empty((n, streams, h, w, 3), dtype=torch.uint8, device=dev)
    for s in range(streams):
        blobs = torch.rand((1 + (seed + s) % 7, 8), generator=g, device=dev).tolist()
        for t in range(n):
            img = torch.stack([96 + 64 * xx / w + 0 * yy + t, 56 + 48 * yy / h + 0 * xx - t, 48 + 40 * (xx + yy) / (w + h)], dim=-1)
            for b in blobs:
                a, bb = w / 20 + b[0] * w * 0.075, h / 30 + b[1] * h / 15
                cx, cy = w * (0.12 + 0.76 * b[2]) + 2 * t, h * (0.12 + 0.76 * b[3]) - t
                ct, st = math.cos(6.283 * b[4]), math.sin(6.283 * b[4])
                u, v = (xx - cx) * ct + (yy - cy) * st, -(xx - cx) * st + (yy - cy) * ct
                img = torch.where(((u / a) ** 2 + (v / bb) ** 2 <= 1).unsqueeze(-1), 200 + 40 * b[5], img)
            img = img.floor() + torch.randint(-8, 9, img.shape, generator=g, device=dev)
            out[t, s] = img.clamp(0, 255).to(torch.uint8)
    return out


def _weights(c, seed):
    """fp32 host arrays; on the bf16 path every weight (not the biases) is a bf16 value already."""
    g, dev = _gen(seed + 77), _device()

    def normal(shape, sigma, shift=0.0, rounded=True):
        v = torch.randn(shape, generator=g, device=dev) * sigma + shift
        if rounded and c["precision"] == "bf16":
            v = v.bfloat16().float()
        return v.cpu().numpy()

    out, ch, t = {}, c["hidden"], c["tools"]
    for l, (ci, co, *_) in enumerate(_layers(c)):
        out[f"enc_w{l}"] = normal((co, ci, 3, 3), math.sqrt(2 / (9 * ci)))
        out[f"enc_b{l}"] = normal((co,), 0.05, rounded=False)
        last = co
    if c["recurrent"]:
        out["lstm_w"] = normal((4 * ch, last + ch, 3, 3), math.sqrt(1 / (9 * (last + ch))))
        out["lstm_b"] = normal((4 * ch,), 0.05, rounded=False)
    sigma = (8.0 if c["recurrent"] else 1.0) * math.sqrt(1 / ch)
    out["head_w"] = normal((t, ch), sigma)
    out["head_b"] = normal((t,), 0.05, -0.5, rounded=False)
    if c["conf"] == "gap_linear":
        out["conf_w"] = normal((t, ch), sigma)
        out["conf_b"] = normal((t,), 0.05, rounded=False)
    return out


def _hidden_state(c, seed):
    """Channels-last state with the spread of o * tanh(c'), and head weights."""
    g, dev, t = _gen(seed), _device(), c["tools"]
    h = 0.4 * torch.tanh(torch.randn((c["streams"], c["hm"], c["wm"], c["hidden"]), generator=g, device=dev))
    sigma = 8.0 * math.sqrt(1 / c["hidden"])
    w = [torch.randn((t, c["hidden"]), generator=g, device=dev) * sigma for _ in range(2)]
    b = [torch.randn((t,), generator=g, device=dev) * 0.05 - 0.5 for _ in range(2)]
    return h if c["channels_last"] else h.permute(0, 3, 1, 2).contiguous(), w, b


def _source(c, seed):
    """Frames with padded rows, [streams][src_h * pitch]."""
    k, h, w, pitch = c["streams"], c["src_h"], c["src_w"], 3 * c["src_w"] + c["pad"]
    buf = torch.full((k, h, pitch), 201, dtype=torch.uint8, device=_device())
    buf[:, :, :3 * w] = _frames(seed, k, 1, w, h)[0].reshape(k, h, 3 * w)
    return buf.reshape(k, h * pitch)


# ------------------------------------------------------------------------------------------------ prepare and run
class _Model:
    """The attributes that binding.make_config reads."""
    norm_div, norm_mean, norm_std, threshold, palette = 255.0, 0.5, 0.25, 0.5, _PALETTE

    def __init__(self, c):
        self.src_w, self.src_h, self.net_w, self.net_h = c["src_w"], c["src_h"], c["net_w"], c["net_h"]
        self.enc_cout, self.enc_stride = _ints(c["enc"]), _ints(c["stride"])
        self.hidden, self.n_tools, self.precision, self.conf_mode = c["hidden"], c["tools"], c["precision"], c["conf"]
        self.overlay, self.recurrent = c["overlay"], c["recurrent"]


def _ring(c):
    return c["ticks"] if c["ticks"] > 1 else RING


def prepare(case, seed):
    c = case
    if c["kind"] == "preprocess":
        return {"case": c, "src": _source(c, seed)}
    if c["kind"] == "postprocess":
        h, w, b = _hidden_state(c, seed)
        return {"case": c, "h": h, "w": w, "b": b}
    k = c["streams"]
    frames = _frames(seed, k, _ring(c), c["src_w"], c["src_h"])
    if c["host"]:
        frames = frames.cpu().pin_memory()
    ctx = binding.Context(binding.make_config(_Model(c), max_streams=k), _weights(c, seed))
    states = (ctypes.c_void_p * k)(*[ctx.state_create().value for _ in range(k)])
    calls = []
    for ring in frames:
        call = (binding.tt_frame * k)()
        for s in range(k):
            call[s].data, call[s].on_device, call[s].frame_index = ring[s].data_ptr(), 0 if c["host"] else 1, len(calls)
        calls.append(call)
    results = (binding.tt_result * binding.TT_MAX_STREAMS)()
    torch.cuda.synchronize()
    return {"case": c, "frames": frames, "ctx": ctx, "states": states, "calls": calls, "results": results,
            "records": np.frombuffer(results, dtype=_RESULT)[:k], "views": {}, "next": 0}


def _view(state, ptr, shape, dtype):
    """The library's output buffers recur from tick to tick: a program wraps each of them once."""
    v = state["views"].get(ptr)
    if v is None:
        v = state["views"][ptr] = binding.device_tensor(ptr, shape, dtype)
        v.owner = state["ctx"]      # the memory is the context's: it lives as long as a view of it
    return v


def _collect(state, out):
    c, ctx, rec, t = state["case"], state["ctx"], state["records"], state["case"]["tools"]
    status = ctx.sync_raw(state["results"])
    if status:
        raise RuntimeError(f"tt_sync: status {status}")
    out["conf"].append(rec["conf"][:, :t].copy())
    out["centroid"].append(np.stack([rec["cx"][:, :t], rec["cy"][:, :t]]))
    out["count"].append(rec["count"][:, :t].astype(np.float32))   # sizes in pixels: a pixel at the threshold moves one by 1
    shape = (t, ctx.hm, ctx.wm)
    out["probs"].append([_view(state, int(p), shape, np.float32) for p in rec["probs"]])
    out["masks"].append([_view(state, int(p), shape, np.uint8) for p in rec["masks"]])
    if c["overlay"]:
        out["overlay"].append([_view(state, int(p), (c["src_h"], c["src_w"], 4), np.uint8) for p in rec["overlay"]])


def run(state):
    c = state["case"]
    if c["kind"] == "preprocess":
        return binding.preprocess(state["src"], c["src_w"], c["src_h"], 3 * c["src_w"] + c["pad"], c["net_w"], c["net_h"])
    if c["kind"] == "postprocess":
        w, b = state["w"], state["b"]
        out = binding.postprocess(state["h"], c["channels_last"], w[0], b[0], w[1], b[1], conf_mode=c["conf"])
        rec = out.pop("results")
        out["conf"] = np.stack([r["conf"] for r in rec])
        out["centroid"] = np.stack([[r["cx"], r["cy"]] for r in rec])
        out["count"] = np.stack([r["count"] for r in rec]).astype(np.float32)
        return out
    ctx, k = state["ctx"], c["streams"]
    out = {n: [] for n in ("conf", "centroid", "count", "probs", "masks", "overlay")}
    flying = 0
    for _ in range(c["ticks"]):
        if flying == IN_FLIGHT:
            _collect(state, out)
            flying -= 1
        status = ctx.submit_raw(k, state["calls"][state["next"]], state["states"])
        if status:
            raise RuntimeError(f"tt_submit_frames: status {status}")
        state["next"] = (state["next"] + 1) % len(state["calls"])
        flying += 1
    while flying:
        _collect(state, out)
        flying -= 1
    # maps stay readable until the third submit after theirs: a clip hands on the last one's, and every tick's records
    for n in ("probs", "masks", "overlay"):
        out[n] = out[n][-1] if out[n] else []
    return out


# ------------------------------------------------------------------------------------------------ the same in 64 bits
def _taps(n_in, n_out, dev):
    s = ((torch.arange(n_out, device=dev, dtype=torch.float64) * 2 + 1) * n_in - n_out).clamp(0, (n_in - 1) * 2 * n_out)
    i0 = torch.div(s, 2 * n_out, rounding_mode="floor")
    f = (s - i0 * 2 * n_out) / (2 * n_out)
    i0 = i0.long()
    return i0, (i0 + 1).clamp(max=n_in - 1), f


def _resize(img, w, h):
    """uint8 [H][W][3] -> normalised float64 [3][h][w]."""
    x = img.double().permute(2, 0, 1)
    x0, x1, fx = _taps(img.shape[1], w, img.device)
    y0, y1, fy = _taps(img.shape[0], h, img.device)
    x = x[:, :, x0] + fx * (x[:, :, x1] - x[:, :, x0])
    x = x[:, y0] + fy.view(-1, 1) * (x[:, y1] - x[:, y0])
    return (x / 255.0 - 0.5) / 0.25


def exact(case, seed):
    c = case
    if c["kind"] == "preprocess":
        f = _source(c, seed).view(c["streams"], c["src_h"], -1)[:, :, :3 * c["src_w"]].reshape(c["streams"], c["src_h"], c["src_w"], 3)
        return torch.stack([_resize(x, c["net_w"], c["net_h"]) for x in f])
    if c["kind"] == "postprocess":
        h, w, b = _hidden_state(c, seed)
        h = (h if c["channels_last"] else h.permute(0, 2, 3, 1)).double()
        z = (h @ w[0].double().T + b[0].double()).permute(0, 3, 1, 2)
        p = z.sigmoid()
        conf = (h.mean((1, 2)) @ w[1].double().T + b[1].double()).sigmoid() if c["conf"] == "gap_linear" else p.mean((2, 3))
        return {"logits": z, "probs": p, "masks": None, "conf": conf, "centroid": None, "count": None}
    dev, k = _device(), c["streams"]
    wt = {n: torch.from_numpy(v).to(dev).double() for n, v in _weights(c, seed).items()}
    frames, strides = _frames(seed, k, _ring(c), c["src_w"], c["src_h"]), _ints(c["stride"])
    conf, probs = torch.empty((c["ticks"], k, c["tools"]), dtype=torch.float64), []
    for s in range(k):
        h = cell = None
        for t in range(c["ticks"]):
            x = _resize(frames[t, s], c["net_w"], c["net_h"]).unsqueeze(0)
            for l, st in enumerate(strides):
                x = F.conv2d(x, wt[f"enc_w{l}"], wt[f"enc_b{l}"], stride=st, padding=1).relu()
            if c["recurrent"]:
                if h is None:
                    h = cell = torch.zeros((1, c["hidden"], *x.shape[2:]), dtype=torch.float64, device=dev)
                i, f, g, o = F.conv2d(torch.cat([x, h], 1), wt["lstm_w"], wt["lstm_b"], padding=1).chunk(4, 1)
                cell = f.sigmoid() * cell + i.sigmoid() * g.tanh()
                x = h = o.sigmoid() * cell.tanh()
            p = (torch.einsum("tc,chw->thw", wt["head_w"], x[0]) + wt["head_b"].view(-1, 1, 1)).sigmoid()
            conf[t, s] = ((wt["conf_w"] @ x[0].mean((1, 2)) + wt["conf_b"]).sigmoid() if c["conf"] == "gap_linear" else p.mean((1, 2))).cpu()
        probs.append(p)
    # masks, sizes and centroids hang on pixels whose logit lies within rounding of the threshold, and the overlay on the masks
    none = [None] * c["ticks"]
    return {"conf": [v for v in conf], "centroid": none, "count": none, "probs": probs, "masks": [None] * k,
            "overlay": [None] * k if c["overlay"] else []}
