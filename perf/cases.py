"""The filter's work as its users have it done, for timing and for comparing outputs.

Images follow the three content types the library is used on: 16-bit and 8-bit photographs
(smooth fields, polygon step edges, salt-and-pepper impulses), 8-bit sensor noise, and float
fields with heavy-tailed outliers. Kernels are disks (radius 2 to 128), hexagons and ellipses.
Sizes run from a thumbnail (one partly filled wave of the GPU) to a 67-megapixel scan, with odd
widths (rows that are not a multiple of 16 bytes) among them. Every image tensor is allocated
densely, as ``torch.empty`` gives it, and the outputs are new tensors on every call.
"""
import math

import numpy as np
import torch

import paper_2505_22938_gb300 as fim

_TORCH = {"u8": torch.uint8, "u16": torch.uint16, "f32": torch.float32}
_BYTES = {"u8": 1, "u16": 2, "f32": 4}
_QUARTILES = (25.0, 50.0, 75.0)


def listed():
    return [
        # a thumbnail or a single detector window, smallest kernel of the 8-bit workload: one call's latency
        _case("u8_256_r4", "u8", 256, 256, 4, content="noise"),
        # a web-sized photograph with an odd width, denoised
        _case("u8_1021x763_r10", "u8", 1021, 763, 10),
        # a small image under a large kernel (background estimation of a microscope field)
        _case("u16_512_r48", "u16", 512, 512, 48),
        # 16-megapixel 16-bit photograph: impulse removal, edge-preserving smoothing
        _case("u16_4096_r8", "u16", 4096, 4096, 8),
        _case("u16_4096_r32", "u16", 4096, 4096, 32),
        # one plane of a 24-megapixel camera image, the large radius of the 16-bit workload
        _case("u16_6000x4000_r48", "u16", 6000, 4000, 48),
        # ragged mid-size image at the radius where a tile's footprint outgrows shared memory
        _case("u16_2999x2003_r96", "u16", 2999, 2003, 96),
        # ragged float image (a depth or height map), middle radius
        _case("f32_1537x1021_r24", "f32", 1537, 1021, 24),
        # 67-megapixel float scan, the first radius of the float workload
        _case("f32_8192_r64", "f32", 8192, 8192, 64),
        # convex polygon kernel on float data
        _case("f32_4096_hex64", "f32", 4096, 4096, 64, shape="hexagon"),
        # the three quartiles of one image from one call
        _case("u16_4096_r16_quartiles", "u16", 4096, 4096, 16, op="quartiles"),
        # a batch of images of uneven sizes, types and radii in one prepared run
        {"name": "batch_16_mixed", "op": "batch", "jobs": 16, "mix": 5, "lo": 512, "hi": 2560},
    ]


def _case(name, dtype, w, h, r, op="median", shape="circle", content="photo", pct=50.0):
    c = {"op": op, "dtype": dtype, "w": w, "h": h, "r": r, "shape": shape, "content": content, "pct": pct}
    return c if name is None else {"name": name, **c}


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    if rng.random() < 0.08:
        return {"op": "batch", "jobs": rng.randint(3, 20), "mix": rng.randint(10, 1 << 20), "lo": rng.randint(200, 600),
                "hi": rng.randint(1000, 2400)}
    dtype = rng.choice(("u8", "u16", "f32"))
    op = rng.choices(("median", "percentile", "quartiles", "map", "radii"), (60, 14, 12, 7, 7))[0]
    shape = rng.choices(("circle", "hexagon", "ellipse"), (80, 10, 10))[0] if op == "median" else "circle"
    r = int(round(_log_uniform(rng, 2, 128)))
    # the largest images only for the kernels users run them with; large kernels cost more per pixel
    most = 24e6 * min(1.0, (48.0 / r) ** 2) / (3 if op in ("quartiles", "radii") else 1)
    px = _log_uniform(rng, 6e4, most)
    aspect = _log_uniform(rng, 0.5, 2.0)
    w, h = int(math.sqrt(px * aspect)), int(math.sqrt(px / aspect))
    if rng.random() < 0.4:  # many images have rows of whole 16-byte words
        w = max(32, w // 16 * 16)
    content = "noise" if dtype == "u8" and rng.random() < 0.3 else "photo"
    return _case(None, dtype, w, h, r, op=op, shape=shape, content=content, pct=rng.choice((5.0, 25.0, 60.0, 90.0)))


# ---- inputs ----------------------------------------------------------------------------------

def _fields(gen, h, w):
    """Unit-variance sum of white noise smoothed by Gaussians of 2, 16 and 64 pixels."""
    hh, ww = -(-h // 64) * 64, -(-w // 64) * 64
    f = torch.zeros((hh, ww), device="cuda")
    fy = torch.fft.fftfreq(hh, device="cuda")[:, None]
    fx = torch.fft.rfftfreq(ww, device="cuda")[None, :]
    d2 = fy * fy + fx * fx
    for sigma in (2.0, 16.0, 64.0):
        noise = torch.randn((hh, ww), generator=gen, device="cuda")
        g = torch.fft.irfft2(torch.fft.rfft2(noise) * torch.exp(-2.0 * math.pi ** 2 * sigma ** 2 * d2), s=(hh, ww))
        f += g / (g.std() * math.sqrt(3.0) + 1e-12)
    return f[:h, :w]


def _photo(gen, rng, h, w):
    """16-bit photograph in float: fields, 32 polygon steps whose size follows the image, impulses."""
    img = 32768.0 + 8192.0 * _fields(gen, h, w)
    scale = math.sqrt(h * w) / 4096.0
    for _ in range(32):
        nv = int(rng.integers(3, 9))
        rad = float(rng.uniform(64, 1024)) * scale
        cx, cy = float(rng.uniform(0, w)), float(rng.uniform(0, h))
        ang = np.sort(rng.uniform(0, 2 * math.pi, nv))
        vx, vy = cx + rad * np.cos(ang), cy + rad * np.sin(ang)
        step = float(rng.uniform(-12000, 12000))
        x0, x1 = max(0, int(vx.min())), min(w - 1, int(vx.max()) + 1)
        y0, y1 = max(0, int(vy.min())), min(h - 1, int(vy.max()) + 1)
        if x1 < x0 or y1 < y0:
            continue
        yy = torch.arange(y0, y1 + 1, device="cuda", dtype=torch.float32)[:, None]
        xx = torch.arange(x0, x1 + 1, device="cuda", dtype=torch.float32)[None, :]
        inside = torch.ones((y1 - y0 + 1, x1 - x0 + 1), dtype=torch.bool, device="cuda")
        for i in range(nv):
            ax, ay = float(vx[i]), float(vy[i])
            bx, by = float(vx[(i + 1) % nv]), float(vy[(i + 1) % nv])
            inside &= (bx - ax) * (yy - ay) - (by - ay) * (xx - ax) >= 0
        img[y0:y1 + 1, x0:x1 + 1] += inside * step
    u = torch.rand((h, w), generator=gen, device="cuda")
    img = torch.where(u < 0.025, torch.zeros_like(img), torch.where(u > 0.975, torch.full_like(img, 65535.0), img))
    return img.round_().clamp_(0, 65535)


def _image(dtype, content, h, w, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if dtype == "f32":
        f = _fields(gen, h, w)
        u = torch.rand((h, w), generator=gen, device="cuda")
        t = torch.rand((h, w), generator=gen, device="cuda", dtype=torch.float64)
        cauchy = (10.0 * torch.tan(math.pi * (t - 0.5))).clamp_(-1e30, 1e30).float()
        return (torch.where(u < 0.01, f + cauchy, f) + 0.0).contiguous()
    if content == "noise":
        top = 256 if dtype == "u8" else 65536
        return torch.randint(0, top, (h, w), generator=gen, device="cuda", dtype=torch.int32).to(_TORCH[dtype])
    img = _photo(gen, np.random.Generator(np.random.PCG64(seed)), h, w).to(torch.int32)
    return (img >> 8).to(torch.uint8) if dtype == "u8" else img.to(torch.uint16)


def _hexagon(r):
    return [(r * math.cos(k * math.pi / 3), r * math.sin(k * math.pi / 3)) for k in range(6)]


def _kernel(shape, r):
    if shape == "hexagon":
        return fim.fim_create_kernel_polygon(_hexagon(float(r)))
    if shape == "ellipse":
        return fim.fim_create_kernel_ellipse(r, max(1, r // 2))
    return fim.fim_create_kernel_circle(r)


def _radii(r):
    return sorted({max(1, r // 2), r})


def _jobs(case):
    """(w, h, dtype, r) of a batch's images: sides uniform, types uniform, radii log-uniform in [2, 128]."""
    rng = np.random.Generator(np.random.PCG64(case["mix"]))
    jobs = []
    for _ in range(case["jobs"]):
        w, h = (int(v) for v in rng.integers(case["lo"], case["hi"] + 1, 2))
        dtype = ("u8", "u16", "f32")[int(rng.integers(0, 3))]
        jobs.append((w, h, dtype, int(round(math.exp(rng.uniform(math.log(2.0), math.log(128.0)))))))
    return jobs


def prepare(case, seed):
    if case["op"] == "batch":
        imgs, outs, kernels, jobs = [], [], [], []
        for i, (w, h, dtype, r) in enumerate(_jobs(case)):
            img = _image(dtype, "photo", h, w, 1000 * seed + i)
            out = torch.empty_like(img)
            k = fim.fim_create_kernel_circle(r)
            jobs.append(fim.make_job(img.data_ptr(), out.data_ptr(), w, h, w * _BYTES[dtype], fim.DTYPES[dtype], k))
            imgs.append(img)
            outs.append(out)
            kernels.append(k)
        torch.cuda.synchronize()
        return {"op": "batch", "imgs": imgs, "outs": outs, "batch": fim.fim_batch_create(jobs, kernels)}
    img = _image(case["dtype"], case["content"], case["h"], case["w"], seed)
    s = {"op": case["op"], "img": img, "pct": case["pct"]}
    if case["op"] == "radii":
        s["kernels"] = [_kernel("circle", r) for r in _radii(case["r"])]
    else:
        s["kernel"] = _kernel(case["shape"], case["r"])
    if case["op"] == "map":  # a percentile that rises across the image from left to right
        s["map"] = torch.linspace(0.0, 100.0, case["w"], device="cuda").repeat(case["h"], 1).contiguous()
    return s


def _plain(t):
    """uint16 tensors as the same bits in int16, which every torch operation takes."""
    return t.view(torch.int16) if t.dtype == torch.uint16 else t


def run(state):
    op = state["op"]
    if op == "median":
        return _plain(fim.median(state["img"], state["kernel"]))
    if op == "percentile":
        return _plain(fim.percentile(state["img"], state["kernel"], state["pct"]))
    if op == "quartiles":
        return [_plain(t) for t in fim.percentiles(state["img"], state["kernel"], _QUARTILES)]
    if op == "map":
        return _plain(fim.percentile_map(state["img"], state["kernel"], state["map"]))
    if op == "radii":
        return [_plain(t) for t in fim.median_radii(state["img"], state["kernels"])]
    state["batch"].run(torch.cuda.current_stream().cuda_stream)
    return [_plain(t) for t in state["outs"]]


def work(case):
    """Each input read once and each output written once (and a percentile map read once)."""
    if case["op"] == "batch":
        return {"bytes": float(sum(2 * w * h * _BYTES[d] for w, h, d, _ in _jobs(case))), "flops": 0.0}
    px, es = case["w"] * case["h"], _BYTES[case["dtype"]]
    outs = {"quartiles": 3, "radii": len(_radii(case["r"]))}.get(case["op"], 1)
    return {"bytes": float(px * es * (1 + outs) + (4 * px if case["op"] == "map" else 0)), "flops": 0.0}


def exact(case, seed):
    """The window of every pixel gathered and its middle value selected, in 64 bits, where that is quick."""
    if case["op"] not in ("median", "percentile") or case["shape"] != "circle":
        return None
    h, w, r = case["h"], case["w"], case["r"]
    offs = [(dx, dy) for dy in range(-r, r + 1) for dx in range(-r, r + 1) if dx * dx + dy * dy <= r * r]
    n = len(offs)
    if w * h * n > 3e9:
        return None
    rank = (n - 1) // 2 if case["op"] == "median" else min(n - 1, math.floor(case["pct"] / 100.0 * (n - 1) + 0.5))
    img = _image(case["dtype"], case["content"], h, w, seed).to(torch.float64)
    dx = torch.tensor([o[0] for o in offs], device="cuda")
    dy = torch.tensor([o[1] for o in offs], device="cuda")
    out = torch.empty((h, w), dtype=torch.float64, device="cuda")
    step = max(1, int(1e8 / n))
    for a in range(0, h * w, step):
        p = torch.arange(a, min(h * w, a + step), device="cuda")
        ys = ((p // w)[:, None] + dy).clamp_(0, h - 1)
        xs = ((p % w)[:, None] + dx).clamp_(0, w - 1)
        out.view(-1)[a:a + p.numel()] = torch.kthvalue(img[ys, xs], rank + 1, dim=1).values
    return out
