"""The calls whose speed this library is judged by, from the smallest to the largest.

A case names a family (the public entry point), its geometry and its inputs. Frames are
drawn on the GPU from the seed alone, with the forward model of ``synth`` (objects seen by
p x p views through a circular aperture, Poisson photons, 2 DN read noise, 100 DN offset):
Gaussian beads, textured cells with a bright membrane, and a vessel tree with moving spots.
"""
import math

import numpy as np
import torch

from paper_2310_09467_gb300 import lfc

FRAME_BYTES_MAX = 12 * 2 * 2040 * 2040  # the largest call: the benchmark's 12 frames


def listed():
    return [
        # a cropped preview while a sample is focused: one small frame scored over the default candidates
        {"name": "judge_1x195", "family": "judge", "frames": "195x195p13", "kinds": "beads2000"},
        # the same crop stored: latency and launches of one small call
        {"name": "compress_1x195", "family": "compress", "frames": "195x195p13", "kinds": "beads2000"},
        # one frame of the smaller camera format, stored as it arrives
        {"name": "compress_1x1300", "family": "compress", "frames": "1300x1300p13", "kinds": "beads2000"},
        # the benchmark's step: 12 full frames of beads and cells on the device
        {"name": "compress_12x2040", "family": "compress", "frames": "12*2040x2040p15", "kinds": "beads20,beads2000,cells500"},
        # a camera stream's micro-batch of three formats, one graph replay each
        {"name": "stream_3_mixed", "family": "batch", "frames": "1300x1300p13,2040x2040p15,2550x2160p15",
         "kinds": "beads2000,cells500,vessel300"},
        # frames in pinned host memory to containers in pinned host memory
        {"name": "host_3x2550", "family": "host", "frames": "3*2550x2160p15", "kinds": "cells500,vessel300,beads2000"},
        # a time series: spatial and temporal candidates (52) on every frame after the key frame
        {"name": "series_6x2040", "family": "series", "frames": "6*2040x2040p15", "kinds": "vessel300"},
        # the criterion alone over both byte layouts (52 candidates)
        {"name": "judge_layouts_2x2040", "family": "judge_layouts", "frames": "2*2040x2040p15", "kinds": "beads200,cells500"},
        # one stored frame read back
        {"name": "decompress_1x1300", "family": "decompress", "frames": "1300x1300p13", "kinds": "beads2000"},
        # a stored batch read back
        {"name": "decompress_12x2040", "family": "decompress", "frames": "12*2040x2040p15", "kinds": "beads20,beads2000,cells500"},
        # the coder alone on blocks of ragged sizes (1 byte to the largest block)
        {"name": "bzip2_24_ragged", "family": "bzip2", "blocks": 24, "largest": 720000, "data": "frame"},
        # one training step of the proposal network at its batch of 32
        {"name": "train_32", "family": "train", "batch": 32, "classes": 26},
    ]


def draw(rng):
    family = rng.choice(["judge", "compress", "compress", "batch", "host", "series", "judge_layouts", "decompress",
                         "decompress", "bzip2", "train"])
    if family == "train":
        return {"family": family, "batch": _log(rng, 1, 32), "classes": rng.randint(2, 64)}
    if family == "bzip2":
        return {"family": family, "blocks": _log(rng, 1, 100), "largest": _log(rng, 1000, 720000),
                "data": rng.choice(["frame", "sparse", "words"])}
    share = {"series": 2, "judge_layouts": 2}.get(family, 1)  # twice the candidates a frame
    room = FRAME_BYTES_MAX // share
    groups, n, kinds = [], _log(rng, 1, 12), []
    mixed = family in ("batch", "compress") and rng.random() < 0.5
    while n > 0 and len(groups) < 4:
        p = rng.randint(7, 19)
        w, h = (p * max(2, round(_log(rng, 150, 2550) / p)) for _ in range(2))
        k = rng.randint(1, n) if mixed else n
        k = min(k, room // (2 * w * h))
        if k < 1:
            break
        groups.append("%d*%dx%dp%d" % (k, w, h, p))
        room -= k * 2 * w * h
        n -= k
        if not mixed:
            break
    for _ in range(rng.randint(1, 3)):
        kinds.append(rng.choice(["beads20", "beads200", "beads2000", "cells500", "vessel300"]))
    if family == "series":
        kinds = ["vessel%d" % rng.choice([100, 300, 1000])]
    return {"family": family, "frames": ",".join(groups), "kinds": ",".join(kinds)}


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _geometry(case):
    """[(width, height, pitch)] of the case's frames."""
    out = []
    for g in case["frames"].split(","):
        count, size = g.split("*") if "*" in g else ("1", g)
        size, p = size.split("p")
        w, h = size.split("x")
        out += [(int(w), int(h), int(p))] * int(count)
    return out


# ------------------------------------------------------------------ frames
def _gen(*seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(np.random.SeedSequence([int(s) for s in seed]).generate_state(1, np.uint64)[0] >> np.uint64(1)))
    return g


def _axes(w, h, p):
    """Per pixel column and row: lenslet index and view offset, on the GPU; the aperture."""
    c = (p - 1) / 2.0
    x, y = (torch.arange(n, device="cuda") for n in (w, h))
    du, dv = (((a % p) - c) / (p - 1) for a in (x, y))
    open_ = ((x % p - c)[None, :] ** 2 + (y % p - c)[:, None] ** 2) <= (p / 2.0) ** 2
    return (x // p).float(), (y // p).float(), du.float(), dv.float(), open_


def _spots(s, t, du, dv, cx, cy, d, sigma, amp):
    """A sum of Gaussians, each shifted by its disparity in every view: separable, so one product."""
    gx = torch.exp(-((s[None, :] - (cx[:, None] + d[:, None] * du[None, :])) ** 2) / (2 * sigma ** 2))
    gy = torch.exp(-((t[None, :] - (cy[:, None] + d[:, None] * dv[None, :])) ** 2) / (2 * sigma ** 2))
    return (gy * amp).t() @ gx


def _uniform(rng, lo, hi, n):
    return torch.as_tensor(rng.uniform(lo, hi, n), dtype=torch.float32, device="cuda")


def _field(kind, w, h, p, rng, step=0):
    """Expected photons of a unit-level field, height x width."""
    s, t, du, dv, open_ = _axes(w, h, p)
    nx, ny = w // p, h // p
    scale = min(1.0, min(nx, ny) / 136.0)
    if kind == "beads":
        n = 200
        f = _spots(s, t, du, dv, _uniform(rng, 0, nx, n), _uniform(rng, 0, ny, n), _uniform(rng, -3, 3, n), 1.5, 1.0)
    elif kind == "cells":
        f = torch.zeros((h, w), device="cuda")
        tex = torch.as_tensor(rng.uniform(0, 1, (256, 256)), dtype=torch.float32, device="cuda")
        for _ in range(50):
            a, b = rng.uniform(10, 40, 2) * scale
            th, cx, cy, d = rng.uniform(0, math.pi), rng.uniform(0, nx), rng.uniform(0, ny), rng.uniform(-3, 3)
            r = max(a, b) + 4.5 + abs(d)
            xa, xb = (p * min(nx, max(0, int(v))) for v in (cx - r, cx + r + 2))
            ya, yb = (p * min(ny, max(0, int(v))) for v in (cy - r, cy + r + 2))
            if xa >= xb or ya >= yb:
                continue
            X = (s[xa:xb] - (cx + d * du[xa:xb]))[None, :]
            Y = (t[ya:yb] - (cy + d * dv[ya:yb]))[:, None]
            xr, yr = X * math.cos(th) + Y * math.sin(th), Y * math.cos(th) - X * math.sin(th)
            q = torch.sqrt((xr / float(a)) ** 2 + (yr / float(b)) ** 2)
            ring = torch.exp(-(((q - 1.0) * float(min(a, b))) ** 2) / 4.5)
            ix, iy = ((v / 4.0 + 100.0) for v in (xr, yr))
            x0, y0 = ix.floor(), iy.floor()
            fx, fy = (v * v * (3 - 2 * v) for v in (ix - x0, iy - y0))
            x0, y0 = x0.long() & 255, y0.long() & 255
            x1, y1 = (x0 + 1) & 255, (y0 + 1) & 255
            noise = (tex[y0, x0] * (1 - fx) + tex[y0, x1] * fx) * (1 - fy) + (tex[y1, x0] * (1 - fx) + tex[y1, x1] * fx) * fy
            f[ya:yb, xa:xb] += (ring + 0.3 * (q < 1.0)) * noise
    else:
        segs, front = [], [(rng.uniform(0.3, 0.7) * nx, 0.0, math.pi / 2 + rng.uniform(-0.3, 0.3), 0.45 * ny)]
        for _ in range(3):
            nxt = []
            for xa, ya, an, ln in front:
                xb, yb = xa + ln * math.cos(an), ya + ln * math.sin(an)
                segs.append((xa, ya, xb, yb, rng.uniform(3, 8) * scale, rng.uniform(-3, 3)))
                nxt += [(xb, yb, an + sg * rng.uniform(0.3, 0.8), ln * 0.65) for sg in (-1, 1)]
            front = nxt
        f = torch.zeros((h, w), device="cuda")
        for xa, ya, xb, yb, rad, d in segs:
            X, Y = (s - d * du)[None, :] - xa, (t - d * dv)[:, None] - ya
            vx, vy = xb - xa, yb - ya
            par = torch.clamp((X * vx + Y * vy) / (vx * vx + vy * vy + 1e-12), 0, 1)
            f += torch.exp(-((X - par * vx) ** 2 + (Y - par * vy) ** 2) / (2 * (rad / 2.0) ** 2))
        f = 0.5 * (0.2 + 0.8 * torch.clamp(f, max=1.0))
        which, pos, speed = rng.integers(0, len(segs), 40), rng.uniform(0, 1, 40), rng.uniform(0.5, 2.5, 40) * scale
        cx, cy, dd = [], [], []
        for i in range(40):
            xa, ya, xb, yb, _, d = segs[which[i]]
            fr = (pos[i] + step * speed[i] / (math.hypot(xb - xa, yb - ya) + 1e-9)) % 1.0
            cx.append(xa + fr * (xb - xa))
            cy.append(ya + fr * (yb - ya))
            dd.append(d)
        cx, cy, dd = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in (cx, cy, dd))
        f += _spots(s, t, du, dv, cx, cy, dd, 1.0, 1.0)
    return f * open_


def _frame(kind, geometry, seed, step=0):
    """One raw frame as an int16 tensor of the uint16 counts: the field from ``seed``, the noise from it and ``step``."""
    name, level = kind.rstrip("0123456789"), float(kind[len(kind.rstrip("0123456789")):])
    w, h, p = geometry
    lam = _field(name, w, h, p, np.random.default_rng(seed), step) * level
    g = _gen(*seed, step)
    dn = torch.poisson(lam, generator=g) + 2.0 * torch.randn((h, w), generator=g, device="cuda") + 100.0
    dn = torch.clamp(torch.round(dn), 0, 65535).to(torch.int32)
    return torch.where(dn >= 32768, dn - 65536, dn).to(torch.int16).contiguous()


def _frames(case, seed):
    kinds = case["kinds"].split(",")
    return [_frame(kinds[i % len(kinds)], g, (seed, i)) for i, g in enumerate(_geometry(case))]


# --------------------------------------------------------------- the network
SHAPES = [(3, 3, 2, 32), (32,), (3, 3, 32, 32), (32,), (3, 3, 32, 32), (32,), (3, 3, 32, 32), (32,)]


def _train_inputs(case, seed):
    """Thumbnails (n x 2 x 256 x 256), labels and He-normal parameters."""
    n, k = case["batch"], case["classes"]
    kinds = ["%s%d" % (a, b) for b in (20, 200, 2000) for a in ("beads", "cells", "vessel")]
    thumbs = torch.zeros((n, 2, 256, 256), device="cuda")
    for i in range(n):
        raw = (_frame(kinds[i % 9], (2040, 2040, 15), (seed, i)).to(torch.int32) & 0xFFFF).float()
        mosaic = raw.view(136, 15, 136, 15).permute(1, 0, 3, 2).reshape(2040, 2040)
        for c, img in enumerate((raw, mosaic)):
            mean = img.view(255, 8, 255, 8).mean(dim=(1, 3))
            thumbs[i, c, :255, :255] = torch.log1p(torch.clamp(mean - 100.0, min=0.0)) / 8.0
    rng = np.random.default_rng((seed, 77))
    labels = torch.as_tensor(rng.integers(0, k, n), dtype=torch.int32, device="cuda")
    flat = []
    for shape in SHAPES + [(32, k), (k,)]:
        fan = math.prod(shape[:-1]) if len(shape) > 1 else 0
        std = math.sqrt((2.0 if len(shape) == 4 else 1.0) / fan) if fan else 0.05
        flat.append((rng.standard_normal(math.prod(shape)) * std).astype(np.float32))
    return thumbs, labels, np.concatenate(flat)


# ------------------------------------------------------------------ the coder
def _block_sizes(case):
    """Sizes spread over their logarithm from 1 byte to the largest, the largest ones repeated."""
    n, top = case["blocks"], case["largest"]
    return [max(1, int(round(top ** min(1.0, (i + 1) / max(1.0, 0.6 * n))))) - (i % 3 if i else 0) * (top > 1000 and i > n // 2)
            for i in range(n)]


def _block_bytes(case, seed, total):
    rng = np.random.default_rng((seed, 5))
    if case["data"] == "frame":  # raw frames as their bytes
        side = 15 * max(2, min(136, math.isqrt(max(1, total // 2)) // 15 + 1))
        parts, got = [], 0
        while got < total:
            f = _frame(["cells500", "beads2000"][len(parts) % 2], (side, side, 15), (seed, len(parts)))
            parts.append(f.view(torch.uint8).reshape(-1))
            got += parts[-1].numel()
        return torch.cat(parts)[:total].contiguous()
    if case["data"] == "sparse":  # a high-byte plane: zeros with a few small values
        b = np.where(rng.random(total) < 0.02, rng.integers(1, 9, total), 0).astype(np.uint8)
    else:  # text-like: words of a small vocabulary
        vocab = [bytes(rng.integers(97, 123, rng.integers(2, 10)).astype(np.uint8)) + b" " for _ in range(2000)]
        picks = rng.zipf(1.3, total // 4 + 8) % 2000
        b = np.frombuffer(b"".join(vocab[i] for i in picks), dtype=np.uint8)
        b = np.resize(b, total)
    return torch.as_tensor(b, device="cuda")


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    family = case["family"]
    st = {"family": family}
    if family == "train":
        st["thumbs"], st["labels"], flat = _train_inputs(case, seed)
        st["net"] = lfc.Cnn(case["classes"], case["batch"], seed=0)
        st["net"].set_params(flat)
        return st
    if family == "bzip2":
        sizes = _block_sizes(case)
        st["offsets"], st["sizes"] = [int(v) for v in np.cumsum([0] + sizes[:-1])], sizes
        st["data"] = _block_bytes(case, seed, sum(sizes))
        st["plan"] = lfc.Plan(2040, 2040, 15, max_frames=-(-case["blocks"] // 12))
        st["stride"] = lfc.max_stream_bytes(max(sizes))
        st["out"] = torch.zeros(len(sizes) * st["stride"], dtype=torch.uint8, device="cuda")
        return st
    geo = _geometry(case)
    st["pitch"] = [g[2] for g in geo]
    w, h, p = max(g[0] for g in geo), 0, 1
    area = max(g[0] * g[1] for g in geo)
    p = next(g[2] for g in geo if g[0] == w)
    h = p * -(-area // (w * p))  # the plan serves frames up to this width and area
    ids = sorted(lfc.default_ids() + [c | 8 for c in lfc.default_ids()]) if family == "judge_layouts" else None
    plan = st["plan"] = lfc.Plan(w, h, p, max_frames=len(geo), candidate_ids=ids, temporal=family == "series")
    if family == "series":
        kind = case["kinds"].split(",")[0]
        frames = [_frame(kind, geo[0], (seed, 0), step=i) for i in range(len(geo))]
        st["prevs"] = [None] + frames[:-1]
    else:
        frames, st["prevs"] = _frames(case, seed), None
    st["frames"] = frames
    n = len(frames)
    if family in ("judge", "judge_layouts"):
        return st
    if family == "host":
        st["frames"] = [f.cpu().pin_memory() for f in frames]
        st["out"] = torch.zeros(plan.slots(frames)[1], dtype=torch.uint8).pin_memory()
        st["sizes"] = np.zeros(n, dtype=np.uint64)
        return st
    st["out"] = torch.zeros(plan.slots(frames)[1], dtype=torch.uint8, device="cuda")
    st["sizes"] = torch.zeros(n, dtype=torch.int64, device="cuda")
    if family == "batch":
        st["batch"] = plan.batch(frames, st["pitch"], out=st["out"], sizes=st["sizes"])
    if family == "decompress":
        plan.compress(frames, st["pitch"], out=st["out"], sizes=st["sizes"])
        size = st["sizes"].cpu().tolist()
        st["blobs"] = [st["out"][o:o + k].clone() for o, k in zip(plan.slots(frames)[0], size)]
        st["restored"] = [torch.zeros_like(f) for f in frames]
        del st["out"], st["sizes"], st["frames"]
    return st


def run(st):
    family = st["family"]
    if family in ("judge", "judge_layouts"):
        return st["plan"].judge(st["frames"], st["pitch"])
    if family in ("compress", "series"):
        out, sizes, _ = st["plan"].compress(st["frames"], st["pitch"], prevs=st["prevs"], out=st["out"], sizes=st["sizes"])
        return out, sizes
    if family == "host":
        out, sizes, _ = st["plan"].compress_host(st["frames"], st["pitch"], out=st["out"], sizes=st["sizes"])
        return out, sizes
    if family == "batch":
        st["batch"].launch()
        return st["batch"].out, st["batch"].sizes
    if family == "decompress":
        return st["plan"].decompress(st["blobs"], st["restored"])
    if family == "bzip2":
        out, sizes, _ = st["plan"].bzip2_encode(st["data"], st["offsets"], st["sizes"], out=st["out"], stride=st["stride"])
        return out, sizes
    st["net"].set_thumbnails(st["thumbs"])
    loss = st["net"].backward(st["labels"])
    return loss, st["net"].get_params(grads=True)[1]


def work(case):
    """Bytes: every frame (or block) and its container once, at the ratio of 2.7 such frames code to. The codec has no
    floating operations; a training step has its convolutions' (forward, input gradient, weight gradient)."""
    family = case["family"]
    if family == "train":
        n, k = case["batch"], case["classes"]
        params = sum(math.prod(s) for s in SHAPES) + 33 * k
        conv = 2 * 9 * 65536 * 32 * n
        return {"bytes": 4.0 * (n * 2 * 65536 + 2 * params + 2 * n), "flops": float(conv * (2 * 2 + 3 * 3 * 32))}
    if family == "bzip2":
        return {"bytes": sum(_block_sizes(case)) * (1 + 1 / 2.7), "flops": 0.0}
    raw = float(sum(2 * w * h for w, h, _ in _geometry(case)))
    n = len(_geometry(case))
    if family in ("judge", "judge_layouts"):
        return {"bytes": raw + n * (1 + 256 * 8), "flops": 0.0}
    return {"bytes": raw * (1 + 1 / 2.7), "flops": 0.0}


def exact(case, seed):
    """Loss and gradients of the training step in 64 bits; everything else is whole numbers and bytes."""
    if case["family"] != "train":
        return None
    thumbs, labels, flat = _train_inputs(case, seed)
    k, at, par = case["classes"], 0, []
    for shape in SHAPES + [(32, k), (k,)]:
        size = math.prod(shape)
        par.append(torch.as_tensor(flat[at:at + size], dtype=torch.float64, device="cuda").reshape(shape).requires_grad_())
        at += size
    losses, n = [], case["batch"]
    for i in range(n):  # frame by frame: one image's convolutions as products
        x = thumbs[i].double()
        for layer in range(4):
            wt, bias = par[2 * layer], par[2 * layer + 1]
            pad = torch.nn.functional.pad(x, (1, 1, 1, 1))
            cols = torch.cat([pad[:, a:a + 256, b:b + 256] for a in range(3) for b in range(3)]).reshape(-1, 65536)
            x = torch.relu(wt.reshape(-1, 32).t() @ cols + bias[:, None]).reshape(32, 256, 256)
        logits = x.mean(dim=(1, 2)) @ par[8] + par[9]
        loss = torch.logsumexp(logits, 0) - logits[labels[i].long()]
        (loss / n).backward()
        losses.append(loss.detach())
    return torch.stack(losses), torch.cat([q.grad.reshape(-1) for q in par])
