"""Workloads of the object-removal framework, each one call sequence that a user's program makes.

A case is a dict of plain values.  `kind` is the entry point it goes through:

  removal   an `api.Inpainter` kept for its image size: new photo in (`reset`), whole removal (`run` with
            its trace), photo and mask out (`result`)
  oneshot   `api.remove_object`: a context made, run and freed for one photo
  steps     a kept `api.Inpainter` driven one iteration at a time (`step`), as an interactive editor does
  batch     an `api.Batch` of independent photos: `reset`, `run`, every `result`
  serve     an `api.Server` that is handed all its requests at once and polled for every result

Photos are Voronoi regions with gratings and noise, masks are ellipses, random-walk blobs, rectangles or
strips: the mobile-camera workloads of the method (Table 3 of the paper), drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_1403_4238_gb300 import api

DEFAULTS = {"kind": "removal", "mask": "ellipses", "frac": 0.08, "form": "plain", "alpha": -1.0, "overlap": False,
            "input": "host", "steps": 0, "n": 1, "regions": 12, "amp": 30.0}


def listed():
    return [
        # the smallest job: a 20x16 object in a thumbnail; launches, copies and the few iterations count alike
        {"name": "thumbnail", "W": 128, "H": 96, "r": 4, "mask": "rect", "frac": 320 / (128 * 96), "regions": 6},
        # an editor that shows every fill as it happens, the first 24 of a mid-size photo
        {"name": "steps_photo", "kind": "steps", "W": 512, "H": 384, "r": 4, "steps": 24},
        # the paper's main photo size with three objects, 9x9 patches, exhaustive search
        {"name": "photo", "W": 512, "H": 384, "r": 4},
        # a portrait photo of odd height, 13x13 patches, tensor-core form, input on the device
        {"name": "portrait_tc", "W": 480, "H": 639, "r": 6, "form": "tc", "frac": 0.05, "regions": 16, "amp": 40.0,
         "input": "device"},
        # one photo through the convenience call: create, run, result, free; a large ragged object, the paper's
        # largest patch (17x17)
        {"name": "oneshot_photo", "kind": "oneshot", "W": 576, "H": 384, "r": 8, "mask": "blob", "frac": 0.1,
         "regions": 8, "amp": 40.0},
        # restricted search area (factor 0.25 around the object), the paper's fast setting
        {"name": "portrait_area", "W": 480, "H": 639, "r": 4, "mask": "ellipse", "frac": 0.03, "alpha": 0.25,
         "regions": 16, "amp": 40.0},
        # a thin horizontal strip (a wire, a pole) with the partial-overlap search, which alone can fill close to it
        {"name": "strip_overlap", "W": 1024, "H": 550, "r": 4, "mask": "strip", "frac": 10 / 550, "overlap": True},
        # patches above the engine's largest radius: coarse texture, 25x25
        {"name": "large_patch", "W": 512, "H": 384, "r": 12},
        # full-HD photo, 13x13 patches, exhaustive search, tensor-core form
        {"name": "hd_tc", "W": 1920, "H": 1080, "r": 6, "form": "tc", "mask": "blob", "frac": 0.045, "regions": 40,
         "amp": 40.0, "input": "device"},
        # the same job in the default form
        {"name": "hd_plain", "W": 1920, "H": 1080, "r": 6, "mask": "blob", "frac": 0.045, "regions": 40, "amp": 40.0},
        # an album: mixed sizes 256..1280 x 256..720, 9x9 and 11x11 patches, 3-10 % masks, one launch
        {"name": "album", "kind": "batch", "n": 60, "W": 1280, "H": 720, "r": 5},
        # a burst of requests to the server: mixed sizes 320..1920 x 240..1080, 2-12 % masks
        {"name": "burst", "kind": "serve", "n": 24, "W": 1920, "H": 1080, "r": 5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["plain"] * 4 + ["tc"] * 3 + ["oneshot", "steps", "area", "overlap", "large", "batch", "serve"])
    c = {"W": _log(rng, 128, 1920), "H": _log(rng, 96, 1080), "r": rng.randint(3, 8),
         "frac": round(rng.uniform(0.02, 0.1), 4), "mask": rng.choice(["ellipses", "blob", "ellipse"]),
         "regions": rng.randint(6, 40), "amp": round(rng.uniform(20, 45), 1), "input": rng.choice(["host", "device"])}
    if what == "tc":
        c |= {"form": "tc", "r": rng.randint(3, 6)}
    elif what == "oneshot":
        c |= {"kind": "oneshot", "W": _log(rng, 128, 1024), "H": _log(rng, 96, 768)}
    elif what == "steps":
        c |= {"kind": "steps", "steps": rng.randint(8, 64), "W": _log(rng, 256, 1024), "H": _log(rng, 192, 768)}
    elif what == "area":
        c |= {"alpha": round(rng.uniform(0.25, 1.0), 2), "mask": "ellipse", "W": _log(rng, 400, 1280),
              "H": _log(rng, 400, 1080), "frac": round(rng.uniform(0.03, 0.08), 4)}
    elif what == "overlap":
        c |= {"overlap": True, "mask": rng.choice(["strip", "ellipse"]), "W": _log(rng, 160, 1024),
              "H": _log(rng, 160, 600), "frac": round(rng.uniform(0.02, 0.05), 4)}
    elif what == "large":
        c |= {"r": rng.randint(9, 16), "W": _log(rng, 200, 640), "H": _log(rng, 160, 480),
              "frac": round(rng.uniform(0.03, 0.08), 4)}
    elif what == "batch":
        c = {"kind": "batch", "n": _log(rng, 4, 60), "W": rng.randint(400, 1280), "H": rng.randint(300, 720), "r": 5}
    elif what == "serve":
        c = {"kind": "serve", "n": _log(rng, 2, 24), "W": rng.randint(400, 1920), "H": rng.randint(300, 1080), "r": 5}
    if "frac" in c:  # small patches go with objects that take them at most some 4000 iterations
        c["frac"] = round(min(c["frac"], 2000 * (2 * c["r"] + 1) ** 2 / (c["W"] * c["H"])), 4)
    return c


# ---------------------------------------------------------------- inputs

def _image(g, W, H, regions, amp):
    """(H, W, 3) uint8 on the GPU: flat Voronoi regions + three gratings + noise, tones 40..215 (neither crushed
    blacks nor clipped whites); `g` a numpy Generator."""
    dev = torch.device("cuda")
    ys = torch.arange(H, device=dev, dtype=torch.float32)[:, None]
    xs = torch.arange(W, device=dev, dtype=torch.float32)[None, :]
    sx, sy = g.uniform(0, W, regions), g.uniform(0, H, regions)
    colours = torch.from_numpy(g.integers(40, 216, (regions, 3)).astype(np.float32)).to(dev)
    best = torch.full((H, W), float("inf"), device=dev)
    label = torch.zeros((H, W), dtype=torch.int64, device=dev)
    for k in range(regions):
        d = (xs - float(sx[k])) ** 2 + (ys - float(sy[k])) ** 2
        closer = d < best
        best = torch.where(closer, d, best)
        label.masked_fill_(closer, k)
    out = colours[label]
    for _ in range(3):
        th, lam, ph = g.uniform(0, math.pi), g.uniform(8.0, 48.0), g.uniform(0, 2 * math.pi)
        wave = torch.sin(2 * math.pi / lam * (xs * math.cos(th) + ys * math.sin(th)) + ph)
        out += (float(amp) * wave)[..., None]
    gen = torch.Generator(device=dev).manual_seed(int(g.integers(0, 2**31)))
    out += 4.0 * torch.randn((H, W, 3), generator=gen, device=dev)
    return out.add_(0.5).floor_().clamp_(40, 215).to(torch.uint8).contiguous()


def _mask(g, W, H, kind, frac):
    """(H, W) uint8 on the GPU, nonzero = remove, covering close to `frac` of the image."""
    dev = torch.device("cuda")
    if kind in ("rect", "strip"):
        if kind == "strip":
            w, h = W, max(1, round(frac * H))
        else:
            h = max(1, round(math.sqrt(frac * W * H * 0.8)))
            w = max(1, round(frac * W * H / h))
        x0, y0 = int(g.integers(0, W - w + 1)), int(g.integers(H // 8, max(H // 8 + 1, H - h - H // 8)))
        m = torch.zeros((H, W), dtype=torch.uint8, device=dev)
        m[y0:y0 + h, x0:x0 + w] = 1
        return m
    n = {"ellipses": 3, "ellipse": 1, "blob": 24}[kind]
    if kind == "blob":  # discs along a random walk
        px, py = g.uniform(0.35, 0.65) * W, g.uniform(0.35, 0.65) * H
        cx, cy, base = [], [], 0.45 * math.sqrt(frac * W * H / math.pi)
        for _ in range(n):
            cx.append(px)
            cy.append(py)
            t = g.uniform(0, 2 * math.pi)
            px = min(max(px + base * math.cos(t), 0.2 * W), 0.8 * W)
            py = min(max(py + base * math.sin(t), 0.2 * H), 0.8 * H)
        ax = ay = g.uniform(0.6, 1.4, n)
    else:
        spread = 0.3 if kind == "ellipses" else 0.1
        cx, cy = W * g.uniform(0.5 - spread, 0.5 + spread, n), H * g.uniform(0.5 - spread, 0.5 + spread, n)
        ax, ay = g.uniform(0.7, 1.4, n), g.uniform(0.7, 1.4, n)
    rot = g.uniform(0, math.pi, n)
    ys = torch.arange(H, device=dev, dtype=torch.float32)[:, None]
    xs = torch.arange(W, device=dev, dtype=torch.float32)[None, :]
    least = torch.full((H, W), float("inf"), device=dev)  # the scale at which a pixel enters the union
    for k in range(n):
        dx, dy = xs - float(cx[k]), ys - float(cy[k])
        u = (dx * math.cos(rot[k]) + dy * math.sin(rot[k])) / float(ax[k])
        v = (dy * math.cos(rot[k]) - dx * math.sin(rot[k])) / float(ay[k])
        least = torch.minimum(least, u * u + v * v)
    keep = max(1, int(frac * W * H))
    return (least <= torch.kthvalue(least.flatten(), keep).values).to(torch.uint8).contiguous()


def _members(c, g):
    """The photos of a batch or of a burst: (W, H, r, mask fraction) each, up to the case's size."""
    lo_w, lo_h = (256, 256) if c["kind"] == "batch" else (320, 240)
    top = 0.1 if c["kind"] == "batch" else 0.12
    return [(int(g.integers(lo_w, c["W"] + 1)), int(g.integers(lo_h, c["H"] + 1)), int(g.integers(4, 6)),
             float(g.uniform(0.03, top))) for _ in range(c["n"])]


def _photo(c, seed):
    g = np.random.Generator(np.random.PCG64(int(seed)))
    return _image(g, c["W"], c["H"], c["regions"], c["amp"]), _mask(g, c["W"], c["H"], c["mask"], c["frac"])


def prepare(case, seed):
    c = {**DEFAULTS, **case}
    if c["kind"] in ("batch", "serve"):
        g = np.random.Generator(np.random.PCG64(int(seed)))
        photos = []
        for W, H, r, frac in _members(c, np.random.Generator(np.random.PCG64(c["n"]))):  # sizes belong to the case
            photos.append((_image(g, W, H, 12, 30.0).cpu().numpy(), _mask(g, W, H, "ellipses", frac).cpu().numpy(), r))
        if c["kind"] == "batch":
            return {"case": c, "batch": api.Batch(photos)}
        return {"case": c, "server": api.Server(hbm_budget_bytes=40 << 30), "photos": photos}
    rgb, mask = _photo(c, seed)
    host = (rgb.cpu().numpy(), mask.cpu().numpy())
    options = dict(form=c["form"], alpha=c["alpha"], overlap=c["overlap"])
    state = {"case": c, "rgb": rgb if c["input"] == "device" else host[0],
             "mask": mask if c["input"] == "device" else host[1], "options": options}
    if c["kind"] != "oneshot":
        state["job"] = api.Inpainter(*host, c["r"], **options)
    else:
        state |= {"rgb": host[0], "mask": host[1]}
    return state


FIELDS = ("px", "py", "qx", "qy", "ssd", "priority", "confidence")


def _cap(c):
    """Records that a removal keeps: a few times the iterations it usually takes (their number depends on the photo)."""
    return c["steps"] or int(8 * c["frac"] * c["W"] * c["H"] / (2 * c["r"] + 1) ** 2) + 32


def _records(c, trace):
    out = np.zeros(_cap(c), trace.dtype)
    out[: min(len(trace), len(out))] = trace[: len(out)]
    return {"iterations": len(trace), **{f: np.ascontiguousarray(out[f]) for f in FIELDS}}


def run(state):
    c = state["case"]
    if c["kind"] == "batch":
        b = state["batch"]
        b.reset()
        status = b.run()
        got = [b.result(i) for i in range(b.n)]
        return {"rgb": [g[0] for g in got], "status": np.array(status), "iterations": np.array([g[1] for g in got]),
                "evals": np.array([g[2] for g in got], np.int64)}
    if c["kind"] == "serve":
        s = state["server"]
        ids = [s.submit(*p) for p in state["photos"]]
        s.wait_idle()
        got = [s.poll(i) for i in ids]
        return {"rgb": [g[0] for g in got], "status": np.array([g[1]["status"] for g in got]),
                "iterations": np.array([g[1]["iterations"] for g in got])}
    if c["kind"] == "oneshot":
        out, trace = api.remove_object(state["rgb"], state["mask"], c["r"], **state["options"])
        return {"rgb": out, **_records(c, trace)}
    job = state["job"]
    job.reset(state["rgb"], state["mask"])
    if c["kind"] == "steps":
        steps = []
        while len(steps) < c["steps"]:
            rec = job.step()
            if rec is None:
                break
            steps.append(rec)
        trace = np.array(steps)
    else:
        _, _, trace = job.run(trace=True)
    out, left = job.result(with_mask=True)
    return {"rgb": out, "mask": left, **_records(c, trace)}


def _size(c, W, H, r, frac):
    """(bytes, operations) of one removal: photo and mask in, photo out; about 2 |Omega| / P^2 iterations of
    P^2 / 2 known pixels x 6 operations (3 channels) at every candidate centre."""
    todo = frac * W * H
    if c["steps"]:
        todo = min(todo, c["steps"] * (2 * r + 1) ** 2 / 2)
    cand = max(1, W - 2 * r) * max(1, H - 2 * r)
    if c["alpha"] >= 0:
        cand = min(cand, todo * 4 / math.pi * (1 + 2 * c["alpha"]) ** 2)
    return 8.0 * W * H, 6.0 * todo * cand


def work(case):
    c = {**DEFAULTS, **case}
    if c["kind"] in ("batch", "serve"):
        each = [_size(c, *m) for m in _members(c, np.random.Generator(np.random.PCG64(c["n"])))]
    else:
        each = [_size(c, c["W"], c["H"], c["r"], c["frac"])]
    return {"bytes": sum(e[0] for e in each), "flops": sum(e[1] for e in each)}


# ---------------------------------------------------------------- plain evaluation in 64 bits

def _priorities(unknown, conf, gray, r):
    """{(y, x): (priority, confidence)} of the fill front (Eq. 1-2)."""
    H, W = unknown.shape
    e = np.pad(unknown, 1, mode="edge").astype(np.int64)
    s = np.pad(unknown, 1, constant_values=True)
    front = unknown & ~(s[:-2, 1:-1] & s[2:, 1:-1] & s[1:-1, :-2] & s[1:-1, 2:])
    nx = (e[:-2, 2:] + 2 * e[1:-1, 2:] + e[2:, 2:]) - (e[:-2, :-2] + 2 * e[1:-1, :-2] + e[2:, :-2])
    ny = (e[2:, :-2] + 2 * e[2:, 1:-1] + e[2:, 2:]) - (e[:-2, :-2] + 2 * e[:-2, 1:-1] + e[:-2, 2:])
    gx, gy, ok = np.zeros((H, W), np.int64), np.zeros((H, W), np.int64), np.zeros((H, W), bool)
    gx[1:-1, 1:-1] = gray[1:-1, 2:] - gray[1:-1, :-2]
    gy[1:-1, 1:-1] = gray[2:, 1:-1] - gray[:-2, 1:-1]
    ok[1:-1, 1:-1] = ~(unknown[1:-1, 1:-1] | unknown[:-2, 1:-1] | unknown[2:, 1:-1] | unknown[1:-1, :-2]
                       | unknown[1:-1, 2:])
    mag = np.where(ok, gx * gx + gy * gy, -1)
    got = {}
    for y, x in np.argwhere(front):
        y0, y1, x0, x1 = max(0, y - r), min(H, y + r + 1), max(0, x - r), min(W, x + r + 1)
        c = np.cumsum(np.where(unknown, 0.0, conf)[y0:y1, x0:x1].ravel())[-1] / ((y1 - y0) * (x1 - x0))
        m = mag[y0:y1, x0:x1]
        k = np.unravel_index(np.argmax(m), m.shape)
        d = 0.0
        if m[k] >= 0 and (nx[y, x] or ny[y, x]):
            n = math.sqrt(float(nx[y, x] ** 2 + ny[y, x] ** 2))
            d = abs(float(-gy[y0:y1, x0:x1][k] * nx[y, x] + gx[y0:y1, x0:x1][k] * ny[y, x])) / n / 510.0
        got[(int(y), int(x))] = (c * d, float(c))
    return got


def exact(case, seed):
    c = {**DEFAULTS, **case}
    if c["kind"] not in ("removal", "steps") or c["overlap"] or c["alpha"] >= 0 or c["r"] > 8 or work(case)["flops"] > 1.2e9:
        return None
    rgb, mask = (t.cpu().numpy() for t in _photo(c, seed))
    (H, W), r = mask.shape, c["r"]
    img, unknown = rgb.astype(np.int64), mask != 0
    conf = np.where(unknown, 0.0, 1.0)
    trace = {f: [] for f in FIELDS}
    while unknown.any() and not (c["kind"] == "steps" and len(trace["px"]) == c["steps"]):
        gray = np.where(unknown, 0, (299 * img[..., 0] + 587 * img[..., 1] + 114 * img[..., 2] + 500) // 1000)
        pri = _priorities(unknown, conf, gray, r)
        py, px = max(pri, key=lambda k: (pri[k][0], -k[0], -k[1]))
        bad = np.zeros((H - 2 * r, W - 2 * r), np.int64)
        ssd = np.zeros((H - 2 * r, W - 2 * r), np.int64)
        fill = []
        for dy in range(-r, r + 1):
            for dx in range(-r, r + 1):
                part = (slice(r + dy, H - r + dy), slice(r + dx, W - r + dx))
                bad += unknown[part]
                y, x = py + dy, px + dx
                if not (0 <= y < H and 0 <= x < W):
                    continue
                if unknown[y, x]:
                    fill.append((dy, dx))
                else:
                    ssd += ((img[part] - img[y, x]) ** 2).sum(-1)
        q = int(np.argmin(np.where(bad == 0, ssd, np.iinfo(np.int64).max)))
        qy, qx = q // (W - 2 * r) + r, q % (W - 2 * r) + r
        p, cp = pri[(py, px)]
        for dy, dx in fill:
            img[py + dy, px + dx] = img[qy + dy, qx + dx]
            unknown[py + dy, px + dx] = False
            conf[py + dy, px + dx] = cp
        for f, v in zip(FIELDS, (px, py, qx, qy, int(ssd.flat[q]), p, cp)):
            trace[f].append(v)
    out = {"rgb": img.astype(np.uint8), "mask": unknown.astype(np.uint8), "iterations": len(trace["px"])}
    for f in FIELDS:
        out[f] = np.zeros(_cap(c), np.float64 if f in ("priority", "confidence") else np.int64)
        out[f][: min(len(trace[f]), _cap(c))] = trace[f][: _cap(c)]
    return out
