"""Performance cases of the framework: what its users have it do, over the
sizes of its own scenes, tests and benchmark.

Every case goes through the public entry points (``amh.Context``,
``amh.Batch``, ``amh.Net``, ``amh.median4``, ``amh.fuse`` and, where the
Python binding only returns host arrays, the C-ABI calls of ``include/amh.h``
with the caller's own buffers).

    listed()            the named cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs and the handles a program keeps
    run(state)          one pass, its outputs whole
    work(case)          bytes and operations the pass cannot do without
    exact(case, seed)   the outputs in 64 bits, where they have such a value

Inputs are ray-cast on the GPU from a seeded scene (a ground plane, a back
wall, slanted panels and spheres with a 3-D noise albedo, about a tenth of
the surface without texture, per-view gain and bias), the structure of the
scenes in ``paper_1805_07920_gb300/synth``.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1805_07920_gb300 import amh, learned, synth

PLANES, DEPTH_MIN, DEPTH_MAX = 4, 2.0, 14.0
LARGEST = 3200 * 2112 * 6 * (8 * 10 + 8)      # cost of the largest listed case, in (hypothesis, view) pairs
NET = [("e1", 16, 32), ("e2", 32, 64), ("e3", 64, 96), ("e4", 96, 128),
       ("d3", 128, 96), ("d2", 96, 64), ("d1", 64, 32), ("out", 32, 16)]
LEARNING_RATE = 1e-4


def listed():
    return [
        # the smallest call: one small reference with two sources, every launch and wait counts
        {"name": "iterate_160x120_2src", "kind": "iterate", "width": 160, "height": 120, "sources": 2, "iters": 3, "form": "uint8"},
        # few pixels, the most sources a context takes
        {"name": "iterate_97x73_32src", "kind": "iterate", "width": 97, "height": 73, "sources": 32, "iters": 2, "form": "uint8"},
        # an ordinary preview-size reconstruction
        {"name": "iterate_640x480_5src", "kind": "iterate", "width": 640, "height": 480, "sources": 5, "iters": 5, "form": "uint8"},
        # ragged size, FP16 images
        {"name": "iterate_1365x911_8src_f16", "kind": "iterate", "width": 1365, "height": 911, "sources": 8, "iters": 4, "form": "f16"},
        # a video frame less a row and a column, samples through the texture unit's filter
        {"name": "iterate_1919x1079_6src_filter", "kind": "iterate", "width": 1919, "height": 1079, "sources": 6, "iters": 6, "form": "filter"},
        # the headline workload: full-size reference, ten sources, six iterations
        {"name": "iterate_3200x2112_10src", "kind": "iterate", "width": 3200, "height": 2112, "sources": 10, "iters": 6, "form": "uint8"},
        # every view of a small scene in turn the reference, uneven sizes, the graph-replayed batch
        {"name": "batch_6refs_960x540_1280x720", "kind": "batch", "width": 1280, "height": 720, "refs": 6, "sources": 4, "iters": 6, "form": "uint8"},
        # the learned form: the network's proposal after two iterations, five iterations in all
        {"name": "learned_1600x1056_10src", "kind": "learned", "width": 1600, "height": 1056, "sources": 10, "iters": 5},
        # the network alone on the grid of a 1600x1056 reference, its output to the caller's pinned buffer
        {"name": "infer_800x528", "kind": "infer", "width2": 800, "height2": 528},
        # one training step on the same grid: example, forward, backward, Adam, gradients read
        {"name": "train_800x528", "kind": "train", "width2": 800, "height2": 528},
        # the 4x4 median of a full-size depth map
        {"name": "median_3200x2112", "kind": "median", "width": 3200, "height": 2112},
        # consistency fusion of ten views' maps
        {"name": "fuse_10views_1600x1056", "kind": "fuse", "width": 1600, "height": 1056, "views": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    w = _log(rng, lo, hi)
    h = max(16, int(w * rng.uniform(0.55, 0.8)))
    return (w, h) if rng.random() < 0.8 else (h, w)


def draw(rng):
    kind = rng.choice(["iterate"] * 5 + ["batch", "learned", "infer", "train", "median", "fuse"])
    while True:
        if kind == "iterate":
            w, h = _size(rng, 72, 3200)
            c = {"kind": kind, "width": w, "height": h, "sources": _log(rng, 1, 32), "iters": rng.randint(1, 6),
                 "form": rng.choice(["uint8", "uint8", "f16", "filter"])}
            cost = w * h * c["iters"] * (8 * c["sources"] + 8)
        elif kind == "batch":
            w, h = _size(rng, 128, 1920)
            c = {"kind": kind, "width": w, "height": h, "refs": rng.randint(3, 12), "sources": rng.randint(2, 10),
                 "iters": rng.randint(1, 6), "form": rng.choice(["uint8", "uint8", "f16", "filter"])}
            c["sources"] = min(c["sources"], c["refs"] - 1)
            cost = w * h * c["refs"] * c["iters"] * (8 * c["sources"] + 8)
        elif kind == "learned":
            w, h = _size(rng, 160, 1920)
            c = {"kind": kind, "width": w, "height": h, "sources": rng.randint(2, 10), "iters": rng.randint(3, 6)}
            cost = w * h * c["iters"] * (8 * c["sources"] + 8)
        elif kind in ("infer", "train"):
            w, h = _size(rng, 64, 1600)
            c = {"kind": kind, "width2": (w + 7) // 8 * 8, "height2": (h + 7) // 8 * 8}
            cost = 0
        elif kind == "median":
            w, h = _size(rng, 64, 3200)
            c = {"kind": kind, "width": w, "height": h}
            cost = 0
        else:
            w, h = _size(rng, 120, 1920)
            c = {"kind": kind, "width": w, "height": h, "views": rng.randint(2, 20)}
            cost = w * h * c["views"] * c["views"] * 3
        if cost <= LARGEST:
            return c


# ---------------------------------------------------------------------------
# seeded scenes, ray-cast on the GPU
# ---------------------------------------------------------------------------
def _cameras(n, sizes, arc_deg, radius=7.0, height=-1.0):
    cams = []
    for i in range(n):
        a = math.radians(-arc_deg / 2 + arc_deg * i / max(1, n - 1))
        R, t = synth.look_at((radius * math.sin(a), height, -radius * math.cos(a)), (0.0, 0.0, 0.0))
        w, h = sizes[i % len(sizes)]
        cams.append(synth.Camera(synth.intrinsics(w, h, 0.875 * max(w, h)), R, t, w, h))
    return cams


def _noise(p, seed):
    """Value noise in [0, 1] at p (3, n): hashed lattice values, trilinear."""
    i = torch.floor(p)
    f = p - i
    f = f * f * (3.0 - 2.0 * f)
    i = i.to(torch.int32)
    out = 0.0
    for k in range(8):
        d = [(k >> a) & 1 for a in range(3)]
        h = (i[0] + d[0]) * 374761393 + (i[1] + d[1]) * 668265263 + (i[2] + d[2]) * 1274126177 + seed
        h = (h ^ (h >> 13)) * 1274126177
        h = ((h ^ (h >> 16)) & 0xFFFF).to(torch.float32) * (1.0 / 65535.0)
        for a in range(3):
            h = h * (f[a] if d[a] else 1.0 - f[a])
        out = out + h
    return out


def _render(cam, rng_seed, gain, bias, want_normals=False):
    """uint8 image, depth and (optional) camera-frame normals of one view."""
    rng = np.random.default_rng(rng_seed)
    dev = torch.device("cuda")
    W, H = cam.width, cam.height
    x = torch.arange(W, device=dev, dtype=torch.float32).repeat(H)
    y = torch.arange(H, device=dev, dtype=torch.float32).repeat_interleave(W)
    K, R = cam.K, cam.R
    o = cam.centre
    rc = torch.stack([(x - K[0, 2]) / K[0, 0], (y - K[1, 2]) / K[1, 1], torch.ones_like(x)])
    d = torch.stack([sum(float(R[r, k]) * rc[r] for r in range(3)) for k in range(3)])    # R^T ray: depth 1 along the axis
    best = torch.full_like(x, 60.0)
    nrm = torch.zeros_like(d)
    off = torch.zeros_like(x)

    def hit(t, ok, n, tex):
        nonlocal best, nrm, off
        m = ok & (t > 0.1) & (t < best)
        best = torch.where(m, t, best)
        nrm = torch.where(m[None], n, nrm)
        off = torch.where(m, torch.full_like(off, tex), off)

    def plane(point, normal, tex, extent=None):
        n = np.asarray(normal, float)
        n = n / np.linalg.norm(n)
        den = sum(float(n[k]) * d[k] for k in range(3))
        t = float(n @ (np.asarray(point) - o)) / torch.where(den.abs() < 1e-6, torch.full_like(den, 1e-6), den)
        ok = torch.ones_like(x, dtype=torch.bool)
        if extent is not None:
            q = [float(o[k]) + t * d[k] - float(point[k]) for k in range(3)]
            ok = q[0] * q[0] + q[1] * q[1] + q[2] * q[2] < extent * extent
        nn = torch.tensor(n, device=dev, dtype=torch.float32)[:, None].expand_as(d)
        hit(t, ok, torch.where(den[None] > 0, -nn, nn), tex)

    plane((0, 1.5, 0), (0, -1, 0), 2.0)
    plane((0, 0, 4.0), (0, 0, -1), 5.0)
    for k in range(4):
        c = (rng.uniform(-2.5, 2.5), rng.uniform(-0.3, 1.0), rng.uniform(-1.0, 2.5))
        plane(c, (rng.uniform(-0.7, 0.7), rng.uniform(-0.4, 0.4), -1.0), 9.0 + k, rng.uniform(0.4, 0.9))
    for k in range(5):
        r = rng.uniform(0.35, 0.8)
        c = np.array([rng.uniform(-2.5, 2.5), 1.5 - r, rng.uniform(-1.5, 2.0)])
        oc = o - c
        A = (d * d).sum(0)
        B = sum(float(oc[i]) * d[i] for i in range(3))
        disc = B * B - A * float(oc @ oc - r * r)
        t = (-B - torch.sqrt(disc.clamp_min(0))) / A
        p = torch.stack([float(oc[i]) + t * d[i] for i in range(3)]) / r
        hit(t, disc > 0, p, 21.0 + k)
    P = torch.stack([float(o[i]) + best * d[i] for i in range(3)])
    base = K[0, 0] / 7.0 / 24.0                    # a noise period of about 24 pixels at the scene's depth
    val = torch.zeros_like(x)
    for octave in range(3):
        q = P * (base * 2.0 ** octave) + off[None] * 3.7
        val = val + _noise(q, int(rng_seed) * 17 + octave) * 0.5 ** octave
    val = val / 1.75
    flat = _noise(P * 0.9 + 31.0, int(rng_seed) * 17 + 7) > 0.68
    albedo = torch.where(flat, torch.full_like(val, 0.55), 0.05 + 0.9 * val)
    img = (255.0 * gain * albedo + bias).clamp(0, 255).round().to(torch.uint8).reshape(H, W)
    depth = best.reshape(H, W)
    if not want_normals:
        return img, depth, None
    n = torch.stack([sum(float(R[r, k]) * nrm[k] for k in range(3)) for r in range(3)], -1)
    return img, depth, n.reshape(H, W, 3).contiguous()


def _views(n, sizes, seed, arc_deg, normals=False):
    cams = _cameras(n, sizes, arc_deg)
    rng = np.random.default_rng(seed + 1)
    out = [_render(c, seed, rng.uniform(0.8, 1.2), rng.uniform(-25, 25), normals) for c in cams]
    return cams, [v[0] for v in out], [v[1] for v in out], [v[2] for v in out]


def _nearest(ref, n, n_src):
    return sorted([v for v in range(n) if v != ref], key=lambda v: (abs(v - ref), v))[:n_src]


def _flags(form):
    return amh.AMH_FLAG_TEXTURE_BILINEAR if form == "filter" else 0


def _context(case, seed, form):
    n = case["sources"] + 1
    cams, imgs, _, _ = _views(n, [(case["width"], case["height"])], seed, min(60.0, 3.0 * n))
    if form == "f16":
        imgs = [im.to(torch.float16) for im in imgs]
    p = amh.default_params(depth_min=DEPTH_MIN, depth_max=DEPTH_MAX, seed=seed, flags=_flags(form))
    ctx = amh.Context(cams, imgs, n // 2, _nearest(n // 2, n, case["sources"]), p)
    H, W = case["height"], case["width"]
    maps = dict(depth=torch.empty(H, W, device="cuda"), normal=torch.empty(H, W, 3, device="cuda"),
                cost=torch.empty(H, W, device="cuda"), selected=torch.empty(H, W, dtype=torch.int32, device="cuda"))
    return ctx, maps


# ---------------------------------------------------------------------------
# network inputs
# ---------------------------------------------------------------------------
def _fields(w2, h2, seed):
    """Features (h2, w2, 6), targets (h2, w2, 4) and mask (h2, w2) like those
    of a state after two iterations: smooth depth and normals with outliers."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def smooth(ch, cells):
        z = torch.randn(1, ch, max(2, h2 // cells), max(2, w2 // cells), device="cuda", generator=g)
        return torch.nn.functional.interpolate(z, (h2, w2), mode="bilinear", align_corners=False)[0]

    def noise(ch):
        return torch.randn(ch, h2, w2, device="cuda", generator=g)

    bad = (torch.rand(h2, w2, device="cuda", generator=g) < 0.15).float()
    x = torch.zeros(6, h2, w2, device="cuda")
    x[0] = (0.2 * smooth(1, 8)[0] + 0.1 * noise(1)[0]).clamp(-0.5, 0.5)
    x[1] = (0.4 * smooth(1, 40)[0] + (0.01 + 0.4 * bad) * noise(1)[0]).clamp(-1, 1)
    n = 0.4 * smooth(3, 30) + (0.05 + 0.5 * bad) * noise(3)
    n[2] = -1.0 - n[2].abs()
    x[2:5] = n / n.norm(dim=0, keepdim=True)
    x[5] = (0.05 + 0.1 * noise(1)[0].abs() + 0.4 * bad).clamp(0, 1)
    t = 0.02 * noise(4) + bad * (0.3 * smooth(4, 20) + 0.1 * noise(4))
    mask = (torch.rand(h2, w2, device="cuda", generator=g) < 0.85).to(torch.uint8)
    hwc = lambda a: a.permute(1, 2, 0).contiguous()
    return hwc(x), hwc(t) * mask[..., None], mask


def _initial_weights(seed):
    rng = np.random.default_rng(seed)
    out = {}
    for name, cin, cout in NET:
        sd = math.sqrt(2.0 / (9 * cin)) * (0.1 if name == "out" else 1.0)
        out[name] = (rng.normal(0, sd, (9, cout, cin)).astype(np.float32), rng.normal(0, 0.02, cout).astype(np.float32))
    return out


def _trained_weights():
    z = np.load(learned.WEIGHTS)
    return {name: (z[name + "_w"].reshape(9, cout, cin), z[name + "_b"]) for name, cin, cout in NET}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "iterate":
        ctx, maps = _context(case, seed, case["form"])
        return dict(kind=kind, ctx=ctx, iters=case["iters"], maps=maps)
    if kind == "learned":
        ctx, maps = _context(case, seed, "uint8")
        net = amh.Net(*amh.net_size_for(case["width"], case["height"]))
        net.load(learned.WEIGHTS)
        return dict(kind=kind, ctx=ctx, net=net, iters=case["iters"], maps=maps)
    if kind == "batch":
        n = case["refs"]
        sizes = [(case["width"], case["height"]), (case["width"] * 3 // 4, case["height"] * 3 // 4)]
        cams, imgs, _, _ = _views(n, sizes, seed, min(60.0, 6.0 * n))
        if case["form"] == "f16":
            imgs = [im.to(torch.float16) for im in imgs]
        p = amh.default_params(depth_min=DEPTH_MIN, depth_max=DEPTH_MAX, seed=seed, flags=_flags(case["form"]))
        stream = torch.cuda.Stream()      # graphs cannot be captured on the default stream
        b = amh.Batch(cams, [im.cpu().numpy() for im in imgs], list(range(n)),
                      [_nearest(r, n, case["sources"]) for r in range(n)], p, stream=ctypes.c_void_p(stream.cuda_stream))
        out = [dict(plane=torch.empty(c.height, c.width, 4, device="cuda"), cost=torch.empty(c.height, c.width, device="cuda"),
                    wmask=torch.empty(c.height, c.width, dtype=torch.int32, device="cuda"),
                    choice=torch.empty(c.height, c.width, dtype=torch.uint8, device="cuda")) for c in cams]
        torch.cuda.synchronize()
        return dict(kind=kind, batch=b, iters=case["iters"], out=out, stream=stream)
    if kind == "infer":
        w2, h2 = case["width2"], case["height2"]
        net = amh.Net(w2, h2)
        net.load(learned.WEIGHTS)
        x = np.zeros((h2, w2, 16), np.float32)
        x[..., :6] = _fields(w2, h2, seed)[0].cpu().numpy()
        net.set_input(x)
        return dict(kind=kind, net=net, out=torch.empty(h2, w2, 16, pin_memory=True))
    if kind == "train":
        w2, h2 = case["width2"], case["height2"]
        net = amh.Net(w2, h2)
        net.set_params(_initial_weights(seed))
        grads = [(torch.empty(9, cout, cin, pin_memory=True), torch.empty(cout, pin_memory=True)) for _, cin, cout in NET]
        return dict(kind=kind, net=net, example=_fields(w2, h2, seed), mirror=(bool(seed & 1), bool(seed & 2)), grads=grads)
    if kind == "median":
        _, _, depth, _ = _views(1, [(case["width"], case["height"])], seed, 0.0)
        g = torch.Generator(device="cuda").manual_seed(seed)
        d = depth[0]
        d = d * (1.0 + 0.002 * torch.randn(d.shape, device="cuda", generator=g))
        out = torch.rand(d.shape, device="cuda", generator=g)
        d = torch.where(out < 0.08, DEPTH_MIN + (DEPTH_MAX - DEPTH_MIN) * out / 0.08, d)
        return dict(kind=kind, depth=d.contiguous())
    n = case["views"]
    cams, depth, normal = _fusion_maps(case, seed)
    return dict(kind=kind, cams=cams, depth=depth, normal=normal)


def _fusion_maps(case, seed):
    """Depth and normal maps as the method leaves them: the surface with small
    errors, a tenth of the pixels wrong, a few without depth."""
    n = case["views"]
    cams, _, depth, normal = _views(n, [(case["width"], case["height"])], seed, min(90.0, 5.0 * n), normals=True)
    g = torch.Generator(device="cuda").manual_seed(seed)
    for v in range(n):
        d = depth[v] * (1.0 + 0.0003 * torch.randn(depth[v].shape, device="cuda", generator=g))
        u = torch.rand(d.shape, device="cuda", generator=g)
        d = torch.where(u < 0.1, DEPTH_MIN + (DEPTH_MAX - DEPTH_MIN) * u / 0.1, d)
        depth[v] = torch.where(u > 0.98, torch.zeros_like(d), d).contiguous()
        m = normal[v] + 0.1 * torch.randn(normal[v].shape, device="cuda", generator=g)
        normal[v] = (m / m.norm(dim=-1, keepdim=True)).contiguous()
    return cams, depth, normal


def run(state):
    kind = state["kind"]
    if kind == "iterate":
        ctx = state["ctx"]
        ctx.init_random()
        ctx.iterate(state["iters"])
        ctx.read_maps_device(**state["maps"])
        return state["maps"]
    if kind == "learned":
        ctx, net = state["ctx"], state["net"]
        ctx.init_random()
        ctx.iterate(2)
        net.features(ctx)
        net.forward()
        net.propose(ctx)
        ctx.iterate(1)
        amh.clear_proposal(ctx)
        ctx.iterate(state["iters"] - 3)
        ctx.read_maps_device(**state["maps"])
        return state["maps"]
    if kind == "batch":
        b = state["batch"]
        b.run(state["iters"])
        for r, o in enumerate(state["out"]):
            s = amh.State(plane=o["plane"].data_ptr(), cost=o["cost"].data_ptr(), wmask=o["wmask"].data_ptr(),
                          choice=o["choice"].data_ptr())
            b._check(amh.lib().amh_batch_get_state(b.ctx, r, ctypes.byref(s), amh.AMH_MEM_DEVICE))
        return state["out"]
    if kind == "infer":
        net = state["net"]
        net._check(amh.lib().amh_net_forward(net.ctx, ctypes.c_void_p(state["out"].data_ptr())))
        return state["out"]
    if kind == "train":
        net = state["net"]
        net.set_example(*state["example"], *state["mirror"])
        net.forward()
        loss = net.backward()
        net.adam(LEARNING_RATE)
        for layer, (gw, gb) in enumerate(state["grads"]):
            net._check(amh.lib().amh_net_grads(net.ctx, layer, ctypes.c_void_p(gw.data_ptr()), ctypes.c_void_p(gb.data_ptr())))
        return dict(loss=loss, grads=state["grads"])
    if kind == "median":
        return amh.median4(state["depth"])
    points, count = amh.fuse(state["cams"], state["depth"], state["normal"])
    return dict(points=points, count=count)


# ---------------------------------------------------------------------------
# work and 64-bit values
# ---------------------------------------------------------------------------
def _net_flops(w2, h2):
    px = w2 * h2
    level = dict(e1=0, e2=1, e3=2, e4=3, d3=2, d2=1, d1=0, out=0)
    return sum(18 * cin * cout * (px >> (2 * level[name])) for name, cin, cout in NET)


def _update_work(px, sources, iters, es, views_px):
    # 8 hypotheses x sources, the own plane and at least one candidate on four
    # views, the initialisation; 36 samples of 22 operations and 80 a pair.
    # Images read once, 24 bytes of maps written a pixel.
    pairs = px * (iters * (8 * sources + 2 * min(4, sources)) + sources)
    return {"bytes": views_px * es + 24 * px, "flops": 872 * pairs}


def work(case):
    kind = case["kind"]
    if kind in ("iterate", "learned"):
        px = case["width"] * case["height"]
        es = 2 if case.get("form") == "f16" else 1
        w = _update_work(px, case["sources"], case["iters"], es, px * (case["sources"] + 1))
        if kind == "learned":
            w2, h2 = amh.net_size_for(case["width"], case["height"])
            w["flops"] += _net_flops(w2, h2)
        return w
    if kind == "batch":
        w, h, n = case["width"], case["height"], case["refs"]
        px = ((n + 1) // 2) * w * h + (n // 2) * (w * 3 // 4) * (h * 3 // 4)
        return _update_work(px, case["sources"], case["iters"], 2 if case["form"] == "f16" else 1, px)
    if kind in ("infer", "train"):
        px = case["width2"] * case["height2"]
        weights = sum(9 * cin * cout for _, cin, cout in NET)
        if kind == "infer":     # input features, weights, 16 output channels
            return {"bytes": px * (32 + 64) + 4 * weights, "flops": _net_flops(case["width2"], case["height2"])}
        # features, targets, mask; weights and two moments read and written, gradients
        return {"bytes": px * (24 + 16 + 1) + 28 * weights, "flops": 3 * _net_flops(case["width2"], case["height2"])}
    px = case["width"] * case["height"]
    if kind == "median":
        return {"bytes": 8 * px, "flops": 60 * px}
    n = case["views"]
    return {"bytes": n * px * (4 + 12 + 24 + 1), "flops": n * (n - 1) * px * 40}


def _network64(x, params):
    """The network in 64 bits on (1, 16, h, w) features, by library operators."""
    F = torch.nn.functional

    def conv(t, name):
        w, b = params[name]
        cout, cin = w.shape[1], w.shape[2]
        return F.conv2d(t, w.reshape(3, 3, cout, cin).permute(2, 3, 0, 1), b, padding=1)

    up = lambda t: F.interpolate(t, scale_factor=2, mode="nearest")
    e1 = torch.relu(conv(x, "e1"))
    e2 = torch.relu(conv(F.avg_pool2d(e1, 2), "e2"))
    e3 = torch.relu(conv(F.avg_pool2d(e2, 2), "e3"))
    e4 = torch.relu(conv(F.avg_pool2d(e3, 2), "e4"))
    d3 = torch.relu(conv(up(e4), "d3")) + e3
    d2 = torch.relu(conv(up(d3), "d2")) + e2
    d1 = torch.relu(conv(up(d2), "d1")) + e1
    return conv(d1, "out")


def _params64(params, grad=False):
    return {k: tuple(torch.tensor(a, dtype=torch.float64, device="cuda", requires_grad=grad) for a in v) for k, v in params.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "infer":
        x = _fields(case["width2"], case["height2"], seed)[0].double()
        x = torch.nn.functional.pad(x, (0, 10)).permute(2, 0, 1)[None]
        with torch.no_grad():
            return _network64(x, _params64(_trained_weights()))[0].permute(1, 2, 0).contiguous()
    if kind == "train":
        x, t, m = (a.double() for a in _fields(case["width2"], case["height2"], seed))
        dims = ([1] if seed & 1 else []) + ([0] if seed & 2 else [])
        x, t, m = (torch.flip(a, dims) for a in (x, t, m))
        if seed & 1:      # a mirror negates that component of the normals
            x[..., 2] *= -1
            t[..., 1] *= -1
        if seed & 2:
            x[..., 3] *= -1
            t[..., 2] *= -1
        params = _params64(_initial_weights(seed), grad=True)
        out = _network64(torch.nn.functional.pad(x, (0, 10)).permute(2, 0, 1)[None], params)[0].permute(1, 2, 0)
        loss = ((out[..., :4] - t).abs() * m[..., None]).sum() / m.sum().clamp_min(1)
        loss.backward()
        return dict(loss=float(loss.detach()), grads=[tuple(p.grad for p in params[name]) for name, _, _ in NET])
    if kind == "median":
        d = prepare(case, seed)["depth"].double()
        H, W = d.shape
        ys, xs = torch.arange(H, device="cuda"), torch.arange(W, device="cuda")
        v = torch.stack([d[(ys + dy).clamp(0, H - 1)][:, (xs + dx).clamp(0, W - 1)] for dy in (-2, -1, 0, 1) for dx in (-2, -1, 0, 1)])
        v = torch.sort(v, 0).values
        return 0.5 * (v[7] + v[8])
    if kind == "fuse":
        return dict(points=_fuse64(*_fusion_maps(case, seed)), count=None)
    # the checkerboard update chooses among hypotheses at every step: a
    # rounding at a tie takes another branch, so 64 bits give another run
    return None


def _fuse64(cams, depths, normals, f_eps=0.3, f_ang=30.0, f_con=2):
    """The consistency fusion's points in 64 bits."""
    T = lambda a: torch.tensor(np.asarray(a, np.float64), device="cuda")
    cam = [(T(c.K), T(c.R), T(c.t), T(c.centre)) for c in cams]
    cos_ang = math.cos(math.radians(f_ang))

    def pixel_rays(c, K):
        y, x = torch.meshgrid(torch.arange(c.height, device="cuda", dtype=torch.float64),
                              torch.arange(c.width, device="cuda", dtype=torch.float64), indexing="ij")
        return torch.stack([x, y, torch.ones_like(x)], -1) @ torch.linalg.inv(K).T

    world = []
    for c, (K, R, t, _), D, N in zip(cams, cam, depths, normals):
        world.append((((D.double()[..., None] * pixel_rays(c, K)) - t) @ R, N.double() @ R))
    out = []
    for i in range(len(cams)):
        X, n = world[i]
        sx, sn, cnt = X.clone(), n.clone(), torch.zeros(X.shape[:2], dtype=torch.int64, device="cuda")
        has = depths[i] > 0
        for j in range(len(cams)):
            if j == i:
                continue
            K, R, t, C = cam[j]
            Xc = X @ R.T + t
            z = Xc[..., 2]
            uv = Xc @ K.T
            ok = has & (z > 0)
            zs = torch.where(ok, z, torch.ones_like(z))
            ui, vi = torch.floor(uv[..., 0] / zs + 0.5), torch.floor(uv[..., 1] / zs + 0.5)
            ok &= (ui >= 0) & (ui < cams[j].width) & (vi >= 0) & (vi < cams[j].height)
            ui, vi = torch.where(ok, ui, 0).long(), torch.where(ok, vi, 0).long()
            Dj = depths[j].double()[vi, ui]
            ok &= Dj > 0
            base = torch.linalg.norm(cam[i][3] - C)
            ok &= K[0, 0] * base * (1 / zs - 1 / torch.where(ok, Dj, torch.ones_like(Dj))).abs() <= f_eps
            nj = world[j][1][vi, ui]
            ok &= (n * nj).sum(-1) / (n.norm(dim=-1) * nj.norm(dim=-1)).clamp_min(1e-300) >= cos_ang
            sx += torch.where(ok[..., None], world[j][0][vi, ui], 0)
            sn += torch.where(ok[..., None], nj, 0)
            cnt += ok
        pts = torch.cat([sx / (1 + cnt)[..., None], sn / sn.norm(dim=-1, keepdim=True).clamp_min(1e-300)], -1)
        out.append(torch.where((has & (cnt >= f_con))[..., None], pts, 0))
    return out
