"""Performance cases of the lane-detection library: what its users have it do, through its public entry points.

A case is a dict of plain values.  Its "kind" names the call:

  detect    Detector.detect: lanes of n frames of one size from disparity and image in device memory
  host      Detector.detect_host_ptr: the same from page-locked host buffers, results on the host
  groups    Detector.detect_groups: frames of several sizes in one call
  learned   Net.detect: the network-ranked form, with the shipped weights
  stereo    Stereo.run: disparity of n rectified pairs
  pairs     Stereo.detect: lanes of n rectified pairs (disparity, then the whole path)
  grad      Net.grad: forward and backward of one training step of the proposal network

Frames are rendered on the GPU after the recipes of paper_1807_02752_gb300/scenes.py (road profile, lane
field lines, textured obstacles, sensor noise, outlier and invalid disparities), every value drawn from the
seed.  All calls of a process go to one stream of its own, as a program with one camera pipeline issues
them, so captured calls replay as CUDA graphs and passes follow one another.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_1807_02752_gb300 import ld, scenes

TOP_K = 96                 # coarse starts the learned form evaluates (99 % agreement with the full search)
POS_WEIGHT = 10.0          # weight of the lane cells in the training loss
CHANNELS = (1, 16, 32, 32, 16)
MAX_PIXELS = 64 * 1242 * 375

_stream = None


def listed():
    return [
        # the smallest frame the repository's recipes render: launches and serial stages are everything
        {"name": "frame_320x120", "kind": "detect", "w": 320, "h": 120, "n": 1, "n_disp": 48},
        # one camera frame at the paper's size, already on the device: the latency of a live pipeline
        {"name": "frame_1242x375", "kind": "detect", "w": 1242, "h": 375, "n": 1, "n_disp": 128},
        # the same frame from the capture software's pinned buffers, result read back
        {"name": "host_frame_1242x375", "kind": "host", "w": 1242, "h": 375, "n": 1, "n_disp": 128},
        # a few cameras of the odd size of another recording, too few frames to be split into two halves
        {"name": "batch8_1241x376", "kind": "detect", "w": 1241, "h": 376, "n": 8, "n_disp": 128},
        # the throughput workload: offline processing of recorded drives
        {"name": "batch64_1242x375", "kind": "detect", "w": 1242, "h": 375, "n": 64, "n_disp": 128},
        # the largest frames: full HD with shadows, dashes and 30 % outliers
        {"name": "batch16_1920x1080", "kind": "detect", "w": 1920, "h": 1080, "n": 16, "n_disp": 256},
        # cameras of three sizes in one call
        {"name": "groups_three_sizes", "kind": "groups", "sizes": "16x1242x375+8x1280x720+8x1920x1080", "n_disp": 256},
        # the network-ranked search on the throughput workload
        {"name": "learned_batch64_1242x375", "kind": "learned", "w": 1242, "h": 375, "n": 64, "n_disp": 128},
        # the disparity of one live stereo pair
        {"name": "stereo_pair_1242x375", "kind": "stereo", "w": 1242, "h": 375, "n": 1, "n_disp": 128},
        # lanes from recorded stereo pairs, the whole system
        {"name": "pairs_batch64_1242x375", "kind": "pairs", "w": 1242, "h": 375, "n": 64, "n_disp": 128},
        # forward and backward of the proposal network at its training batch
        {"name": "grad_batch64_1242x375", "kind": "grad", "w": 1242, "h": 375, "n": 64, "n_disp": 128},
    ]


def _n_disp(h):
    return 48 if h <= 140 else 128 if h <= 480 else 256


def _draw_size(rng):
    """A frame size between the smallest and the largest recipe: height over its logarithm, a camera's aspect."""
    h = round(math.exp(rng.uniform(math.log(120), math.log(1080))))
    w = round(h * rng.uniform(1.7, 3.3))
    return min(max(w, 320), 1920), h


def draw(rng):
    kind = rng.choice(["detect", "detect", "detect", "detect", "host", "groups", "learned", "stereo", "pairs", "grad"])
    if kind == "groups":
        sizes, left = [], MAX_PIXELS
        for _ in range(rng.randint(2, 4)):
            w, h = _draw_size(rng)
            most = max(1, min(16, left // (w * h)))
            n = round(math.exp(rng.uniform(0.0, math.log(most))))
            sizes.append("%dx%dx%d" % (n, w, h))
            left = max(0, left - n * w * h)
        return {"kind": kind, "sizes": "+".join(sizes), "n_disp": 256}
    w, h = _draw_size(rng)
    if kind == "host":
        return {"kind": kind, "w": w, "h": h, "n": rng.choice([1, 1, 2, 3]), "n_disp": _n_disp(h)}
    if kind in ("learned", "grad"):   # the proposal serves and is trained on frames of about the paper's size
        h = rng.randint(200, 480)
        w = min(1920, round(h * rng.uniform(2.5, 3.5)))
    most = min(64, MAX_PIXELS // (w * h))
    if kind in ("stereo", "pairs"):   # the cost of a pair follows its rows, not its pixels alone
        h = min(h, 480)
        w = min(max(w, 320), 1600)
        most = min(64, MAX_PIXELS // (w * h))
        n = round(math.exp(rng.uniform(0.0, math.log(most))))
    else:
        n = round(math.exp(rng.uniform(0.0, math.log(most))))
    return {"kind": kind, "w": w, "h": h, "n": max(1, n), "n_disp": _n_disp(h)}


# ---- inputs -------------------------------------------------------------------------------------------


def _recipe(w, h, n, n_disp):
    """The scene recipe of a size: small frames, the paper's size (cleaner for a single frame), full HD."""
    if h <= 140:
        base = scenes.SMALL_320x120
    elif h <= 480:
        base = scenes.SINGLE_1242x375 if n == 1 else scenes.BATCH64_1242x375
    else:
        base = scenes.HD_1920x1080
    scale = w / base.width
    stripe = (max(3.0, base.stripe_px[0] * scale), max(6.0, base.stripe_px[1] * scale))
    # the disparity of the bottom row stays below the bins of the recipe's own height, not of a larger handle
    return scenes.with_size(base, width=w, height=h, n_disp=min(n_disp, _n_disp(h)), stripe_px=stripe)


def _geometry(cfg, r):
    """Road profile and lane field lines of one frame (scenes' own sampling, drawn again until both exist)."""
    v = np.arange(cfg.height, dtype=np.float64)
    for _ in range(100):
        try:
            vh, _, _, beta = scenes._road(cfg, r)
            road = v > vh
            f = beta[0] + beta[1] * v + beta[2] * v * v
            fp = beta[1] + 2.0 * beta[2] * v
            alpha, s = scenes._lanes(cfg, r, f, fp, road)
            return vh, beta, alpha, s
        except RuntimeError:
            continue
    raise RuntimeError("no road and lanes found for this size")


def _render_frame(cfg, r, gen, dev):
    """One frame on the GPU: (disparity before outliers float32, image uint8, lane mask), all [h][w]."""
    W, H = cfg.width, cfg.height
    vh, beta, alpha, s = _geometry(cfg, r)
    rand = lambda *shape: torch.rand(*shape, generator=gen, device=dev)  # noqa: E731
    v = torch.arange(H, device=dev, dtype=torch.float32)
    road = v > vh
    f = torch.from_numpy(np.polyval(beta[::-1], np.arange(H, dtype=np.float64))).to(dev)
    fm = float(f[-1])
    sky = torch.where(rand(H, W) < 0.5, torch.zeros((), device=dev), 0.5 + 2.5 * rand(H, W))
    disp = torch.where(road[:, None], f.float()[:, None], sky)
    level = torch.where(road, torch.full_like(v, r.uniform(90, 120)), torch.full_like(v, r.uniform(140, 190)))
    shade = np.zeros(H, bool)
    if cfg.shadow_frac > 0:
        first = int(math.floor(vh)) + 1
        while shade.sum() < cfg.shadow_frac * (H - first):
            v0 = int(r.integers(first, H - 1))
            shade[v0:v0 + int(r.integers(5, 40))] = True
    shade = torch.from_numpy(shade).to(dev)
    level = torch.where(shade, level * r.uniform(0.5, 0.7), level)
    img = level[:, None].expand(H, W).clone()
    u = torch.arange(W, device=dev, dtype=torch.float32)
    sub = (torch.arange(4, device=dev, dtype=torch.float64) + 0.5) / 4 - 0.5
    vs = v.double()[:, None] + sub
    fs = beta[0] + beta[1] * vs + beta[2] * vs * vs                                   # [H][4]
    lanes = torch.zeros((H, W), dtype=torch.bool, device=dev)
    phase = r.uniform(0, 1)
    for si in s:
        half = torch.clamp(r.uniform(*cfg.stripe_px) * fs / fm, min=1.0).float()[:, None] / 2
        c = (alpha[0] + (alpha[1] + si) * fs + alpha[2] * fs * fs).float()[:, None]   # [H][1][4]
        lo = torch.maximum((u - 0.5)[None, :, None], c - half)
        hi = torch.minimum((u + 0.5)[None, :, None], c + half)
        cov = (torch.clamp(hi - lo, 0.0, 1.0) * (vs > vh)[:, None]).mean(dim=2)
        if cfg.dashed:
            cov = cov * (torch.remainder(65.0 / f.clamp(min=1e-3) + phase, 1.0) < 0.5)[:, None]
        cov = cov * road[:, None]
        lum = r.uniform(200, 240)
        row_lum = torch.where(shade, torch.full_like(v, 0.6 * lum), torch.full_like(v, lum))[:, None]
        img = img + cov * (row_lum - img)
        lanes |= cov > 0.5
    v_lo, v_hi = int(math.ceil(vh)) + 20, H - 41
    for _ in range(int(r.integers(cfg.obstacles[0], cfg.obstacles[1] + 1))):
        if v_hi <= v_lo:
            break
        vb = int(r.integers(v_lo, v_hi + 1))
        fb = float(np.polyval(beta[::-1], vb))
        hgt = int(r.integers(40, 151) * H / 375.0)
        wid = min(int(r.uniform(60, 250) * (W / 1242.0) * fb / fm + 20), W - 1)
        u0, v0 = int(r.integers(0, W - wid + 1)), max(0, vb - hgt + 1)
        disp[v0:vb + 1, u0:u0 + wid] = fb
        img[v0:vb + 1, u0:u0 + wid] = 30 + 190 * rand(vb + 1 - v0, wid)
        lanes[v0:vb + 1, u0:u0 + wid] = False
    img = img + 6.0 * torch.randn((H, W), generator=gen, device=dev)
    return disp, img.round().clamp(0, 255).to(torch.uint8), lanes


def _frames(w, h, n, n_disp, seed, what="frames"):
    """n frames on the GPU: "frames" (disparity, image), "pairs" (left, right), "maps" (block sums, labels)."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed * 1000003 + w * 1009 + h * 31 + n)
    cfg = _recipe(w, h, n, n_disp)
    first, second = [], []
    for k in range(n):
        disp, img, lanes = _render_frame(cfg, np.random.default_rng([seed, w, h, k]), gen, dev)
        if what == "frames":
            p = torch.rand((h, w), generator=gen, device=dev)
            any_d = (cfg.n_disp - 1) * torch.rand((h, w), generator=gen, device=dev)
            disp = torch.where(p < cfg.outlier_frac, any_d, disp)
            disp = torch.where(torch.rand((h, w), generator=gen, device=dev) < cfg.invalid_frac, torch.zeros_like(disp), disp)
            first.append(disp)
            second.append(img)
        elif what == "pairs":
            first.append(img)
            second.append(_right_image(img, disp, gen))
        else:
            x, y = _proposal_maps(img, lanes)
            first.append(x)
            second.append(y)
    return torch.stack(first).contiguous(), torch.stack(second).contiguous()


def _right_image(left, disp, gen):
    """The right image of a pair: each left pixel lands at round(u - d), the nearest surface wins, columns
    nothing lands on take the next landed value to their right (or left of them at the edge), sigma 2 noise."""
    h, w = left.shape
    col = torch.arange(w, device=left.device).expand(h, w)
    x = torch.round(col - disp).long()
    key = (disp * 4096.0).long() * 256 + left.long() + 1
    key = torch.where((x >= 0) & (x < w), key, torch.zeros_like(key))
    hit = torch.zeros((h, w), dtype=torch.int64, device=left.device)
    hit.scatter_reduce_(1, x.clamp(0, w - 1), key, reduce="amax")
    filled = hit > 0
    nxt = torch.where(filled, col, torch.full_like(col, w)).flip(1).cummin(1).values.flip(1)
    prv = torch.where(filled, col, torch.full_like(col, -1)).cummax(1).values
    take = torch.where(nxt < w, nxt, prv).clamp(0, w - 1)
    val = ((hit - 1) % 256).gather(1, take).float()
    noise = 2.0 * torch.randn((h, w), generator=gen, device=left.device)
    return (val + noise).round().clamp(0, 255).to(torch.uint8)


def _proposal_maps(img, lanes):
    """The network's input and labels from a rendered frame: sums over 4 x 4 blocks of the horizontal gradient
    of strong edges in Q12 (int32), and the blocks that a lane marking covers (uint8)."""
    h, w = img.shape
    g = torch.nn.functional.pad(img.float()[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    dx = g[:, 2:] - g[:, :-2]
    gx = dx[:-2] + 2 * dx[1:-1] + dx[2:]
    gx = torch.where(gx.abs() > 100, gx.abs() * 3072, torch.zeros_like(gx))
    pad = (0, -w % 4, 0, -h % 4)
    block = lambda t: torch.nn.functional.pad(t, pad).reshape((h + 3) // 4, 4, (w + 3) // 4, 4)  # noqa: E731
    return block(gx).sum(dim=(1, 3)).int(), (block(lanes.float()).sum(dim=(1, 3)) > 0).to(torch.uint8)


def _initial_weights(seed):
    """He-initialised weights of the proposal network, flat in the library's order (float32, host)."""
    r = np.random.default_rng([seed, 77])
    parts = []
    for ci, co in zip(CHANNELS[:-1], CHANNELS[1:]):
        parts += [r.normal(0, math.sqrt(2 / (9 * ci)), co * ci * 9), r.normal(0, 0.01, co)]
    parts += [r.normal(0, math.sqrt(1 / 16), 16), np.array([-2.0])]
    return np.concatenate(parts).astype(np.float32)


# ---- the calls ----------------------------------------------------------------------------------------


def _sizes(case):
    if case["kind"] == "groups":
        return [tuple(int(x) for x in part.split("x")) for part in case["sizes"].split("+")]
    return [(case["n"], case["w"], case["h"])]


def _the_stream():
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    kind, sizes = case["kind"], _sizes(case)
    what = "pairs" if kind in ("stereo", "pairs") else "maps" if kind == "grad" else "frames"
    data = [_frames(w, h, n, case["n_disp"], seed + 17 * k, what) for k, (n, w, h) in enumerate(sizes)]
    stream = _the_stream()
    max_w, max_h = max(w for _, w, _ in sizes), max(h for _, _, h in sizes)
    det = ld.Detector(max_w, max_h, sum(n for n, _, _ in sizes), ld.default_params(n_disp=case["n_disp"]), stream=stream)
    n, w, h = sizes[0]
    s = {"kind": kind, "w": w, "h": h, "n": n, "det": det, "data": data}
    if kind == "host":
        d, i = data[0]
        s["data"] = [(d.cpu().pin_memory(), i.cpu().pin_memory())]
        s["out"] = np.zeros(n, ld.LANES_DTYPE)
    elif kind == "stereo":
        s["stereo"] = ld.Stereo(det)
        s["out"] = torch.empty((n, h, w), dtype=torch.float32, device="cuda")
    elif kind == "grad":
        s["net"] = ld.Net(det, training=True)
        s["net"].set_params(torch.from_numpy(_initial_weights(seed)).cuda())
    else:
        s["out"] = [det.alloc_lanes(n) for n, _, _ in sizes]
        if kind == "pairs":
            s["stereo"] = ld.Stereo(det)
        if kind == "learned":
            s["net"] = ld.Net(det)
            theta = np.load(os.path.join(os.path.dirname(ld.__file__), "proposal_weights.npy"))
            s["net"].set_params(torch.from_numpy(theta.astype(np.float32)).cuda())
    torch.cuda.synchronize()
    return s


def run(s):
    kind, (a, b) = s["kind"], s["data"][0]
    if kind == "detect":
        return s["det"].detect(a, b, out=s["out"][0])
    if kind == "host":
        s["det"].detect_host_ptr(a.data_ptr(), b.data_ptr(), s["w"], s["h"], s["n"], s["out"])
        return s["out"].view(np.uint8)
    if kind == "groups":
        return s["det"].detect_groups(s["data"], outs=s["out"])
    if kind == "learned":
        return s["net"].detect(a, b, top_k=TOP_K, out=s["out"][0])
    if kind == "stereo":
        return s["stereo"].run(a, b, out=s["out"])
    if kind == "pairs":
        return s["stereo"].detect(a, b, out=s["out"][0])
    return s["net"].grad(a, b, s["w"], s["h"])


def work(case):
    """Inputs read once and results written once; floating-point work only where the call is a contraction
    (the plain path's work is integer histograms, dynamic programming and RANSAC)."""
    px = sum(n * w * h for n, w, h in _sizes(case))
    n = sum(n for n, _, _ in _sizes(case))
    lanes = n * ld.LANES_DTYPE.itemsize
    macs = sum(9 * ci * co for ci, co in zip(CHANNELS[:-1], CHANNELS[1:])) + 16      # per cell, forward
    kind = case["kind"]
    if kind in ("detect", "host", "groups"):
        return {"bytes": 5 * px + lanes, "flops": 0}
    if kind == "learned":
        cells = case["n"] * ((case["h"] + 3) // 4) * ((case["w"] + 3) // 4)
        return {"bytes": 5 * px + lanes + 4 * ld.NET_PARAMS, "flops": 2 * macs * cells}
    if kind == "stereo":
        return {"bytes": 2 * px + 4 * px, "flops": 0}
    if kind == "pairs":
        return {"bytes": 2 * px + lanes, "flops": 0}
    cells = case["n"] * ((case["h"] + 3) // 4) * ((case["w"] + 3) // 4)
    backward = 2 * macs - 9 * CHANNELS[0] * CHANNELS[1]     # no gradient of the input is needed
    return {"bytes": 5 * cells + 8 * ld.NET_PARAMS + 4, "flops": 2 * (macs + backward) * cells}


def exact(case, seed):
    """Gradient and loss of the training case in float64 (the other calls return whole-number decisions)."""
    if case["kind"] != "grad":
        return None
    xs, labels = _frames(case["w"], case["h"], case["n"], case["n_disp"], seed, "maps")
    theta = torch.from_numpy(_initial_weights(seed)).cuda().double().requires_grad_()
    total = xs.numel()
    grad = torch.zeros_like(theta)
    loss = 0.0
    for x, y in zip(xs.split(8), labels.split(8)):
        at, a = 0, (x.double() * 2.0 ** -22)[:, None]
        for ci, co in zip(CHANNELS[:-1], CHANNELS[1:]):
            k = theta[at:at + co * ci * 9].reshape(co, ci, 3, 3)
            bias = theta[at + co * ci * 9:at + co * ci * 9 + co]
            at += co * ci * 9 + co
            rows = torch.nn.functional.unfold(a, 3, padding=1)                        # [n][9 ci][cells]
            a = torch.relu(k.reshape(co, -1) @ rows + bias[:, None]).reshape(a.shape[0], co, *a.shape[2:])
        z = (a * theta[at:at + 16, None, None]).sum(dim=1) + theta[at + 16]
        y = y.double()
        softplus = torch.nn.functional.softplus
        part = (POS_WEIGHT * y * softplus(-z) + (1 - y) * softplus(z)).sum() / total
        grad += torch.autograd.grad(part, theta)[0]
        loss += float(part)
    return grad.detach(), torch.tensor([loss], dtype=torch.float64)
