"""What the framework is timed on: the work its users have it do, through its public entry points.

Five kinds of call:
  pair    the whole method on one frame pair (gpm.Context.run): ingest, dense match field, planes of every level,
          restricted matching, fill, flow and occlusion
  field   the dense match field alone (no plane levels): gpm.Context.match and flow_and_occlusion
  planes  planes, assignment and occlusion from match fields the caller already has (gpm_import of its offsets, then
          the levels without PatchMatch iterations)
  batch   several pairs of different sizes per step, replayed from CUDA graphs (batch.BatchRunner)
  ingest  frames to normalised RGBX texels in the caller's own buffers (gpm_ingest_noalloc)

The frames are synthetic piecewise-planar scenes like the framework's own (scene.py): fractal value noise, textured
layers under random homographies, a global gain and Gaussian noise on frame 2; rendered here on the GPU, because they
are made many times.
"""
import ctypes
import math
import random

import torch
import torch.nn.functional as F

from paper_1804_03787_gb300 import batch, gpm

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
STORAGE = {"f32": gpm.GPM_F32, "f16": gpm.GPM_F16, "bf16": gpm.GPM_BF16}

# A case's values where it does not say otherwise.
DEFAULTS = {"cells": "64/32/16/8", "radius": 4, "iters": 8, "hyp": 512, "storage": "f32", "frames": "f32",
            "equalize": 0, "census": 0, "interp": 0}


def listed():
    return [
        # a caller that owns its buffers readies one 1280x720 pair, HSV equalisation on: microseconds of memory traffic
        {"name": "ingest_1280x720", "kind": "ingest", "sizes": "1280x720", "equalize": 1},
        # the smallest whole calls: thumbnails and region crops, bound by launches and latency
        {"name": "pair_128x96", "kind": "pair", "sizes": "128x96", "cells": "32/16/8", "radius": 3, "iters": 4,
         "hyp": 256},
        # an odd-sized crop, BF16 frames as a network hands them over, the benchmark's parameters
        {"name": "pair_253x187_bf16", "kind": "pair", "sizes": "253x187", "storage": "bf16", "frames": "bf16"},
        # a dense match field alone (7x7 patches), to be consumed by the caller's own stages
        {"name": "field_511x383", "kind": "field", "sizes": "511x383", "radius": 3, "iters": 4},
        # planes and occlusion from another matcher's offsets
        {"name": "planes_512x384", "kind": "planes", "sizes": "512x384"},
        # MPI-Sintel's frame size, plain FP32: the benchmark configuration
        {"name": "pair_1024x436", "kind": "pair", "sizes": "1024x436"},
        # the paper's preset: 7x7 patches, two levels of 80/40 px windows
        {"name": "preset_1024x436", "kind": "pair", "sizes": "1024x436", "cells": "80/40", "radius": 3},
        # the illumination-robust data term, FP16 texels
        {"name": "census_512x384_f16", "kind": "pair", "sizes": "512x384", "storage": "f16", "census": 1},
        # equalised frames and a flow without holes (edge-aware fill), BF16 texels
        {"name": "fill_1280x720_bf16", "kind": "pair", "sizes": "1280x720", "storage": "bf16", "equalize": 1,
         "interp": 1},
        # throughput: one step over a mixed-size batch, FP16 texels, CUDA graphs
        {"name": "batch_mixed_f16", "kind": "batch", "sizes": "256x192,512x384,1024x436,1280x720", "storage": "f16"},
        # the largest frames that are served, FP16 texels and frames
        {"name": "pair_1920x1080_f16", "kind": "pair", "sizes": "1920x1080", "storage": "f16", "frames": "f16"},
    ]


def _size(rng, lo, hi):
    """A frame size whose pixel count is log-uniform in [lo, hi], aspect 4:3 to 2.35:1, odd sides among them."""
    px = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a = rng.uniform(1.33, 2.35)
    return max(96, int(math.sqrt(px * a))), max(96, int(math.sqrt(px / a)))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "field", "planes", "batch", "ingest"])
    c = {"kind": kind, "storage": rng.choice(["f32", "f32", "f16", "bf16"])}
    if kind == "ingest":
        c["sizes"] = "%dx%d" % _size(rng, 128 * 96, 1920 * 1080)
        c["equalize"] = rng.randrange(2)
        return c
    if kind == "batch":
        c["sizes"] = ",".join("%dx%d" % _size(rng, 128 * 96, 1024 * 436) for _ in range(rng.randint(2, 6)))
    else:
        c["sizes"] = "%dx%d" % _size(rng, 128 * 96, 1280 * 720)
        c["frames"] = rng.choice(["f32", c["storage"]])
    c["radius"] = rng.choice([3, 4])
    c["iters"] = rng.choice([4, 6, 8])
    if kind != "field":
        c["cells"] = rng.choice(["64/32/16/8", "64/32/16", "32/16/8", "80/40", "64/32"])
        c["hyp"] = rng.choice([128, 256, 512])
    if kind == "pair":
        option = rng.choice(["", "", "", "equalize", "interp", "census"])
        if option:
            c[option] = 1
    return c


# ------------------------------------------------------------------ scenes
def _homography(src, dst):
    """The 3x3 homography (float64, last entry 1) through four point pairs."""
    A, b = torch.zeros(8, 8, dtype=torch.float64), torch.zeros(8, dtype=torch.float64)
    for i, ((x, y), (u, v)) in enumerate(zip(src, dst)):
        A[2 * i] = torch.tensor([x, y, 1, 0, 0, 0, -u * x, -u * y], dtype=torch.float64)
        A[2 * i + 1] = torch.tensor([0, 0, 0, x, y, 1, -v * x, -v * y], dtype=torch.float64)
        b[2 * i], b[2 * i + 1] = u, v
    return torch.cat([torch.linalg.solve(A, b), torch.ones(1, dtype=torch.float64)]).reshape(3, 3)


def _map(Hm, x, y):
    h = [float(v) for v in Hm.reshape(-1)]
    w = h[6] * x + h[7] * y + h[8]
    return (h[0] * x + h[1] * y + h[2]) / w, (h[3] * x + h[4] * y + h[5]) / w


def _inside(quad, x, y):
    ok = torch.ones_like(x, dtype=torch.bool)
    for (ax, ay), (bx, by) in zip(quad, quad[1:] + quad[:1]):
        ok &= (bx - ax) * (y - ay) - (by - ay) * (x - ax) >= 0
    return ok


def _texture(g, rng, W, H, margin):
    """Fractal value noise over the frame grown by margin: five octaves from a period of 32 px, each half as strong."""
    cw, ch = W + 2 * margin, H + 2 * margin
    out, amp, norm, period = torch.zeros(1, 3, ch, cw, device="cuda"), 1.0, 0.0, 32
    for _ in range(5):
        lat = torch.rand(1, 3, ch // period + 3, cw // period + 3, generator=g, device="cuda")
        up = F.interpolate(lat, scale_factor=period, mode="bicubic", align_corners=False)
        out += amp * up[..., :ch, :cw]
        norm, amp, period = norm + amp, amp / 2, period // 2
    base = torch.tensor([rng.uniform(0.2, 0.8) for _ in range(3)], device="cuda").view(1, 3, 1, 1)
    return base + 0.9 * (out / norm - 0.5)


def _sample(tex, margin, x, y):
    """The texture at frame coordinates (bilinear): 3 x H x W."""
    h, w = tex.shape[2], tex.shape[3]
    grid = torch.stack([(x + margin) * (2.0 / (w - 1)) - 1, (y + margin) * (2.0 / (h - 1)) - 1], -1)
    return F.grid_sample(tex, grid[None].float(), mode="bilinear", padding_mode="border", align_corners=True)[0]


def _scene(W, H, seed):
    """Frames 1 and 2 (H x W x 3, float32 in [0, 1]) and the true flows of both directions (H x W x 2, float64)."""
    rng = random.Random(seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    disp = min(64.0, W / 13.0)
    margin = int(disp) + 8
    frame = [(0.0, 0.0), (W - 1.0, 0.0), (W - 1.0, H - 1.0), (0.0, H - 1.0)]
    quads, motions = [frame], []
    for _ in range(rng.randint(4, 7)):
        area, aspect, th = rng.uniform(0.02, 0.08) * W * H, rng.uniform(0.5, 2.0), rng.uniform(0, math.pi)
        hw, hh = min(0.5 * math.sqrt(area * aspect), 0.45 * W), min(0.5 * math.sqrt(area / aspect), 0.45 * H)
        cx, cy = rng.uniform(0.1, 0.9) * W, rng.uniform(0.1, 0.9) * H
        quads.append([(cx + math.cos(th) * a - math.sin(th) * b, cy + math.sin(th) * a + math.cos(th) * b)
                      for a, b in ((-hw, -hh), (hw, -hh), (hw, hh), (-hw, hh))])
    for k, q in enumerate(quads):
        # a common translation, and corners that move a little apart: moderate zoom and perspective
        d = disp / 8 if k == 0 else disp
        side = min(math.dist(q[0], q[1]), math.dist(q[1], q[2]))
        tx, ty, j = rng.uniform(-0.6, 0.6) * d, rng.uniform(-0.6, 0.6) * d, min(0.3 * d, 0.1 * side)
        motions.append(_homography(q, [(x + tx + rng.uniform(-j, j), y + ty + rng.uniform(-j, j)) for x, y in q]))
    y, x = torch.meshgrid(torch.arange(H, dtype=torch.float64, device="cuda"),
                          torch.arange(W, dtype=torch.float64, device="cuda"), indexing="ij")
    f1, f2 = torch.empty(3, H, W, device="cuda"), torch.empty(3, H, W, device="cuda")
    fwd, bwd = torch.empty(2, H, W, dtype=torch.float64, device="cuda"), torch.empty(2, H, W, dtype=torch.float64,
                                                                                  device="cuda")
    for k, (q, M) in enumerate(zip(quads, motions)):  # painter's order, the background first
        tex = _texture(g, rng, W, H, margin)
        px, py = _map(torch.linalg.inv(M), x, y)
        in1 = _inside(q, x, y) if k else torch.ones_like(x, dtype=torch.bool)
        in2 = _inside(q, px, py) if k else torch.ones_like(x, dtype=torch.bool)
        f1 = torch.where(in1, _sample(tex, margin, x, y), f1)
        f2 = torch.where(in2, _sample(tex, margin, px, py), f2)
        qx, qy = _map(M, x, y)
        fwd = torch.where(in1, torch.stack([qx - x, qy - y]), fwd)
        bwd = torch.where(in2, torch.stack([px - x, py - y]), bwd)
    f2 = f2 * rng.uniform(0.8, 1.2)
    noise = 2.0 / 255.0
    f1 = (f1 + noise * torch.randn(3, H, W, generator=g, device="cuda")).clamp(0, 1)
    f2 = (f2 + noise * torch.randn(3, H, W, generator=g, device="cuda")).clamp(0, 1)
    hwc = lambda t: t.permute(1, 2, 0).contiguous()  # noqa: E731
    return hwc(f1), hwc(f2), hwc(fwd), hwc(bwd), g


def _matches(fwd, bwd, g):
    """Another matcher's offsets, int32 [2][n][2]: the true flows rounded, one in seven a random pixel of the frame."""
    H, W, _ = fwd.shape
    y, x = torch.meshgrid(torch.arange(H, device="cuda"), torch.arange(W, device="cuda"), indexing="ij")
    top = torch.tensor([W - 1, H - 1], device="cuda")
    p, out = torch.stack([x, y], -1), []
    for flow in (fwd, bwd):
        t = (p + flow.round().long()).clamp(min=0).minimum(top)
        far = (torch.rand(H, W, 2, generator=g, device="cuda") * (top + 1)).long().minimum(top)
        t = torch.where(torch.rand(H, W, 1, generator=g, device="cuda") < 1 / 7, far, t)
        out.append((t - p).reshape(-1, 2).int())
    return torch.stack(out).contiguous()


# ------------------------------------------------------------------ a case's state and its pass
def _full(case):
    return {**DEFAULTS, **case}


def _sizes(c):
    return [tuple(int(v) for v in s.split("x")) for s in c["sizes"].split(",")]


def _cells(c):
    return () if c["kind"] == "field" else tuple(int(v) for v in c["cells"].split("/"))


def prepare(case, seed):
    c = _full(case)
    sizes = _sizes(c)
    scenes = [_scene(w, h, 1000 * seed + k) for k, (w, h) in enumerate(sizes)]
    if c["kind"] == "ingest":
        (w, h), (f1, f2) = sizes[0], scenes[0][:2]
        texel = torch.float32 if c["storage"] == "f32" else DTYPES[c["storage"]]
        outs = [torch.empty(h, w, 4, dtype=texel, device="cuda") for _ in range(2)]
        return {"c": c, "lib": gpm.load(), "frames": (f1, f2), "outs": outs}
    params = gpm.default_params(patch_radius=c["radius"], cells=_cells(c), num_hyp=c["hyp"],
                                pm_iters=0 if c["kind"] == "planes" else c["iters"], storage=STORAGE[c["storage"]],
                                equalize=c["equalize"], census=c["census"], interp=c["interp"])
    if c["kind"] == "batch":
        host = [(s[0].cpu().numpy(), s[1].cpu().numpy()) for s in scenes]
        return {"c": c, "runner": batch.BatchRunner(params, host, list(range(len(host))), streams=2)}
    frames = [(scenes[0][0].to(DTYPES[c["frames"]]), scenes[0][1].to(DTYPES[c["frames"]]))]
    state = {"c": c, "frames": frames, "ctx": gpm.Context(params, *sizes[0])}
    if c["kind"] == "planes":
        state["matches"] = _matches(*scenes[0][2:])
    return state


def run(state):
    kind = state["c"]["kind"]
    if kind == "ingest":
        f1, f2 = state["frames"]
        h, w, _ = f1.shape
        o1, o2 = state["outs"]
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        status = state["lib"].gpm_ingest_noalloc(ptr(f1), ptr(f2), w, h, 3 * w, 1, state["c"]["equalize"],
                                                 STORAGE[state["c"]["storage"]], ptr(o1), ptr(o2),
                                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if status != gpm.GPM_OK:
            raise gpm.GpmError(status, "gpm_ingest_noalloc")
        return {"frame1": o1, "frame2": o2}
    if kind == "batch":
        runner = state["runner"]
        runner.run()
        return {"flow": [f for g in runner.groups for f in g["flows"]], "occ": [o for g in runner.groups for o in g["occs"]]}
    ctx = state["ctx"]
    if kind == "planes":
        ctx.match(state["frames"], 0)
        status = ctx.lib.gpm_import(ctx.h, 0, gpm.NNF, ctypes.c_void_p(state["matches"].data_ptr()), 0)
        if status != gpm.GPM_OK:
            raise gpm.GpmError(status, "gpm_import")
        for level in range(1, ctx.params.num_scales + 1):
            ctx.fit_planes(level)
            ctx.match(None, level)
        flows, occs = ctx.flow_and_occlusion()
    else:
        flows, occs = ctx.run(state["frames"])
    return {"flow": flows[0], "occ": occs[0]}


def work(case):
    """What the method cannot do without, whatever the kernels skip: frames in and flow and occlusion out; one full
    patch cost per pixel, direction and half of the iterations' visits (an incumbent changes or is confirmed by one),
    six operations per square tap and 24 per warped one on the twentieth of the pixels that stay without a plane; and
    for each window, direction and stage the hypotheses' solves (200 operations) and tests of a quarter of the matches
    (14 operations)."""
    c = _full(case)
    nbytes = flops = 0.0
    for w, h in _sizes(c):
        n = w * h
        if c["kind"] == "ingest":
            nbytes += 2 * n * (12 + (16 if c["storage"] == "f32" else 8))
            flops += 2 * n * 6
            continue
        elem = 4 if c["frames"] == "f32" else 2
        nbytes += n * (2 * 3 * elem + 8 + 1)
        taps = (2 * c["radius"] + 1) ** 2
        if c["kind"] != "planes":
            flops += 2 * n * taps * 6 * (1 + c["iters"] / 2)
        else:
            nbytes += 2 * n * 8
        for s in _cells(c):
            windows = (2 * w / s) * (2 * h / s)
            flops += 2 * windows * c["hyp"] * (200 + 14 * s * s / 4)
            if c["kind"] != "planes":
                flops += 2 * 0.05 * n * taps * 24 * c["iters"]
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    """The ingest's texels in 64 bits.  The other kinds have none: their outputs follow from some 10^8 comparisons in
    sequence (which candidate, which hypothesis, which plane), not from a formula, and take minutes on the host."""
    c = _full(case)
    if c["kind"] != "ingest":
        return None
    f = [t.double() for t in prepare(case, seed)["frames"]]
    if c["equalize"]:
        out = []
        for t in f:
            v = t.max(-1).values
            b = (v * 256).floor().clamp(0, 255).long()
            cdf = torch.bincount(b.reshape(-1), minlength=256).cumsum(0).double()
            low, n = cdf[cdf > 0][0], v.numel()
            if low == n:
                out.append(t)
                continue
            lut = ((cdf - low) / (n - low))[b]
            out.append(torch.where((v > 0)[..., None], t * (lut / v.clamp(min=1e-300))[..., None], lut[..., None].expand_as(t)))
        f = out
    f[1] = f[1] * (f[0].sum() / f[1].sum())
    return {k: F.pad(t, (0, 1)) for k, t in zip(("frame1", "frame2"), f)}
