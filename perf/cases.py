"""Performance cases of the rasterizer: what a program that uses the library has it do, over the
sizes it is used at.

    view      one frame, or a stereo pair, of a scene: camera and gaze of the frame, then a
              foveated or a full-resolution render (launched directly or as CUDA graphs)
    rounds    one frame rendered incrementally while a tracker's predictions come in
    train     one step of 3DGS training: differentiable full render, then the gradients of all
              scene parameters
    net_train gradients of the learned periphery's loss on a batch of crops
    net_fill  the learned fill of a foveated frame, alone or after the render it belongs to
    sort      the stable pair sort by (tile, depth) keys

A case is a dict of plain values.  Inputs are drawn on the GPU from the seed; ``exact`` restates
each path in plain float64 PyTorch.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2507_04147_gb300 as a3fr
from paper_2507_04147_gb300 import autograd, periphery, synth

DEV = "cuda"
THETA = (18.0, 36.0)
LEVELS = {1: (4,), 2: (4, 2), 3: (4, 2, 1), 4: (4, 3, 2, 1)}
THETAS = {1: (), 2: (18.0,), 3: THETA, 4: (10.0, 18.0, 36.0)}
EXPECTED_PX = (120.0, 0.0)      # expected distance to the final prediction per exit (rounds)
LABELS = {(0, 0): 1, (1, 1): 2, (1, 0): 3, (0, 1): 4}    # (dx, dy) in a 2x2 block -> label


def _view(name, n, width, height, eyes=2, sh=3, scene="uniform", mode="foveated", tile=32, batch=1,
          graph=True, layers=3, fill=0, count_frac=0.0):
    return {"name": name, "kind": "view", "n": n, "width": width, "height": height, "eyes": eyes, "sh": sh,
            "scene": scene, "mode": mode, "tile": tile, "batch": batch, "graph": graph, "layers": layers,
            "fill": fill, "count_frac": count_frac}


def listed():
    return [
        # a thumbnail or a small scene with the library's defaults: latency and launches
        _view("view_20k_256", 20_000, 256, 256, eyes=1, sh=0, tile=16, graph=False),
        # every option of the foveation on a ragged stereo pair
        _view("stereo_60k_options", 60_000, 1003, 717, sh=1, tile=16, graph=False, layers=4, fill=1,
              count_frac=0.1),
        # the headset frame of the benchmark, as the autotuner runs it
        _view("stereo_500k_1280", 500_000, 1280, 1280),
        # the largest headset frame: clustered scene at the headset's full resolution
        _view("stereo_3m_2064", 3_000_000, 2064, 2208, scene="clustered", batch=2),
        # a desktop view of a large scene, no foveation, default tile, direct launches
        _view("full_1m_1080p", 1_000_000, 1920, 1080, eyes=1, mode="full", tile=16, graph=False),
        # incremental rendering: periphery first, then a round per prediction
        {"name": "rounds_300k_1280", "kind": "rounds", "n": 300_000, "width": 1280, "height": 1280, "eyes": 2,
         "sh": 3, "scene": "uniform", "tile": 32},
        # training: a full-size step and a small ragged one
        {"name": "train_1m_1024", "kind": "train", "n": 1_000_000, "width": 1024, "height": 1024, "sh": 3,
         "scene": "uniform"},
        {"name": "train_50k_ragged", "kind": "train", "n": 50_001, "width": 517, "height": 389, "sh": 1,
         "scene": "uniform"},
        # the learned periphery: a training batch, the fill of a headset frame, a whole compact frame
        {"name": "net_train_16x256", "kind": "net_train", "arch": 0, "batch": 16, "width": 256, "height": 256},
        {"name": "net_fill_2064", "kind": "net_fill", "arch": 0, "n": 200_000, "width": 2064, "height": 2208,
         "eyes": 2, "sh": 0, "scene": "uniform", "tile": 32, "render": False},
        {"name": "net_compact_frame_1280", "kind": "net_fill", "arch": 1, "n": 500_000, "width": 1280,
         "height": 1280, "eyes": 2, "sh": 3, "scene": "uniform", "tile": 32, "render": True},
        # the pair sort on one frame's worth of (tile << 32 | depth) keys
        {"name": "sort_4m_45", "kind": "sort", "n": 4_000_000, "bits": 45},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["view", "view", "view", "train", "train", "net_train", "net_fill", "rounds", "sort"])
    if kind == "view":
        eyes = rng.choice([1, 2])
        c = _view("", log(5_000, 1_500_000), log(120, 1920), log(120, 1280), eyes=eyes, sh=rng.randint(0, 3),
                  scene=rng.choice(["uniform", "clustered"]), mode=rng.choice(["foveated", "foveated", "full"]),
                  tile=rng.choice([16, 32]), batch=rng.choice([1, 2]), graph=rng.random() < 0.5,
                  layers=rng.randint(2, 4), fill=rng.choice([0, 0, 1]), count_frac=rng.choice([0.0, 0.0, 0.2]))
        del c["name"]
        return c
    if kind == "rounds":
        return {"kind": kind, "n": log(10_000, 500_000), "width": log(200, 1280), "height": log(200, 1280),
                "eyes": rng.choice([1, 2]), "sh": rng.randint(0, 3), "scene": rng.choice(["uniform", "clustered"]),
                "tile": rng.choice([16, 32])}
    if kind == "train":
        return {"kind": kind, "n": log(4_000, 800_000), "width": log(96, 1024), "height": log(96, 1024),
                "sh": rng.randint(0, 3), "scene": rng.choice(["uniform", "clustered"])}
    if kind == "net_train":
        return {"kind": kind, "arch": rng.choice([0, 1]), "batch": rng.randint(1, 16),
                "width": rng.randint(33, 256), "height": rng.randint(33, 256)}
    if kind == "net_fill":
        return {"kind": kind, "arch": rng.choice([0, 1]), "n": log(20_000, 300_000), "width": log(200, 1920),
                "height": log(200, 1280), "eyes": rng.choice([1, 2]), "sh": rng.randint(0, 3),
                "scene": rng.choice(["uniform", "clustered"]), "tile": rng.choice([16, 32]),
                "render": rng.random() < 0.5}
    return {"kind": "sort", "n": log(1_000, 4_000_000), "bits": rng.randint(24, 64)}


# ---------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def _scene(case, seed):
    """(means, log_scales, quats, opacity_logits, sh) CUDA float32 of the synthetic recipes: a
    uniform cube in front of the eyes, or 64 Gaussian clusters."""
    g, n, k = _gen(seed), case["n"], (case["sh"] + 1) ** 2

    def u(*s):
        return torch.rand(*s, device=DEV, generator=g)

    def z(*s):
        return torch.randn(*s, device=DEV, generator=g)

    if case["scene"] == "uniform":
        a = 2.0 * u(n, 3) - 1.0
        means = torch.stack([a[:, 0], a[:, 1], 4.0 + 2.0 * a[:, 2]], 1)
        log_scales, logits = -4.0 + 0.5 * z(n, 3), 1.5 * z(n)
    else:
        centres = torch.cat([2.0 * u(64, 2) - 1.0, 2.0 + 4.0 * u(64, 1)], 1)
        sigma, which = 0.05 + 0.25 * u(64), torch.randint(64, (n,), device=DEV, generator=g)
        means = centres[which] + z(n, 3) * sigma[which, None]
        # opacities Beta(1/2, 1/2) = sin^2 of a uniform angle
        op = torch.sin(0.5 * math.pi * u(n)).square().clamp(1e-6, 1.0 - 1e-6)
        log_scales, logits = -4.5 + 0.5 * z(n, 3), torch.log(op / (1.0 - op))
    quats = torch.nn.functional.normalize(z(n, 4), dim=1)
    sh = 0.2 * z(n, k, 3)
    sh[:, 0] = (u(n, 3) - 0.5) * (2.0 * math.sqrt(math.pi))
    return [t.float().contiguous() for t in (means, log_scales, quats, logits, sh)]


def _head(case, seed):
    """(cameras, gaze pixels) of the frame: 90 degree field of view, eyes 63 mm apart."""
    r = np.random.default_rng(1000 + int(seed))
    yaw, eyes, w, h = r.uniform(-5.0, 5.0), case.get("eyes", 1), case["width"], case["height"]
    cams = synth.stereo_cameras(w, h, yaw) if eyes == 2 else [synth.pinhole_camera(w, h, 90.0, yaw)]
    ax, ay = np.radians(r.uniform(-15.0, 15.0, 2))
    gaze = np.array([[0.5 * (w - 1) + 0.5 * w * math.tan(ax), 0.5 * (h - 1) + 0.5 * w * math.tan(ay)]] * eyes,
                    dtype=np.float32)
    return cams, gaze


def _net_params(case, seed):
    """Parameters in mid-training: the initial layers with the zero-initialised last layer moved."""
    ws, bs = periphery.unpack(periphery.init_params(int(seed), case["arch"]), case["arch"])
    r = np.random.default_rng(2000 + int(seed))
    ws = [w.copy() for w in ws]
    ws[-1][:] = r.normal(0.0, 1e-3, ws[-1].shape)
    bs = [r.normal(0.0, 1e-2, b.shape).astype(np.float32) for b in bs]
    bs[-1] *= 0.1
    return periphery.pack(ws, bs)


def _crops(case, seed):
    """Smooth images in [0, 1], depths of 2..6 and the targets (here: the images themselves)."""
    g, b, h, w = _gen(seed), case["batch"], case["height"], case["width"]
    x = torch.zeros(b, 4, h, w, device=DEV)
    for cells, amp in ((8, 0.5), (32, 0.3), (128, 0.2)):
        a = torch.rand(b, 4, min(h, cells), min(w, cells), device=DEV, generator=g)
        x += amp * torch.nn.functional.interpolate(a, (h, w), mode="bilinear", align_corners=False)
    img = x[:, :3].permute(0, 2, 3, 1).contiguous()
    return img, (2.0 + 4.0 * x[:, 3]).contiguous()


def _fovea(case):
    layers = case.get("layers", 3)
    return a3fr.Fovea(THETAS[layers], 0.0, LEVELS[layers], case.get("fill", 0), case.get("count_frac", 0.0))


def prepare(case, seed):
    kind = case["kind"]
    st = SimpleNamespace(case=case, kind=kind)
    if kind == "sort":
        g, n, bits = _gen(seed), case["n"], case["bits"]
        # depth bits of 0.5..6 below, tile indices above, cut to the key width
        depth = (0.5 + 5.5 * torch.rand(n, device=DEV, generator=g)).view(torch.int32).long()
        tile = torch.randint(1 << max(1, min(bits, 63) - 32), (n,), device=DEV, generator=g)
        key = (tile << 32) | depth
        st.keys = key if bits >= 63 else key & ((1 << bits) - 1)
        st.vals = torch.arange(n, dtype=torch.int32, device=DEV)
        st.keys_alt, st.vals_alt = torch.empty_like(st.keys), torch.empty_like(st.vals)
        st.ws = torch.empty(a3fr.sort_pairs_workspace_bytes(n), dtype=torch.uint8, device=DEV)
        return st
    if kind == "net_train":
        st.img, st.depth = _crops(case, seed)
        st.net = periphery.Periphery(_net_params(case, seed), arch=case["arch"])
        return st
    st.cams, st.gaze = _head(case, seed)
    st.params = _scene(case, seed)
    if kind == "train":
        st.params = [p.requires_grad_() for p in st.params]
        st.rast = autograd.GaussianRasterizer(*st.params)
        st.dl = torch.randn(1, case["height"], case["width"], 3, device=DEV, generator=_gen(seed + 1))
        return st
    st.scene = a3fr.Scene(*st.params, tile=case["tile"])
    st.scene.set_batch(case.get("batch", 1))
    st.scene.graph_mode(case.get("graph", False))
    st.fovea, st.side = _fovea(case), torch.cuda.Stream()
    st.out = torch.zeros(case["eyes"], case["height"], case["width"], 3, device=DEV)
    if kind == "rounds":
        st.rounds = a3fr.Rounds(EXPECTED_PX, sir=False)
        st.early = (st.gaze + np.float32(0.06 * case["width"])).astype(np.float32)
    if kind == "net_fill":
        st.scene.keep_aux(True)
        st.net = periphery.Periphery(_net_params(case, seed), arch=case["arch"])
        if not case["render"]:
            _frame(st)
    return st


# ---------------------------------------------------------------------------- one pass
def _frame(st):
    for eye, cam in enumerate(st.cams):
        st.scene.set_camera(eye, cam)
    st.scene.set_gaze(st.gaze, st.side)
    return st.scene.render_foveated(st.fovea, out=st.out)


def run(st):
    case, kind = st.case, st.kind
    if kind == "view":
        if case["mode"] == "foveated":
            return _frame(st)
        for eye, cam in enumerate(st.cams):
            st.scene.set_camera(eye, cam)
        return st.scene.render_full(out=st.out)
    if kind == "rounds":
        # the host waits for each round, as a driver does that has to know which prediction it used
        stream = torch.cuda.current_stream()
        for eye, cam in enumerate(st.cams):
            st.scene.set_camera(eye, cam)
        st.scene.begin_frame(st.fovea, st.rounds, out=st.out)
        for k, gaze in enumerate((st.early, st.gaze)):
            st.scene.post_prediction(k + 1, gaze)
            st.scene.render_round(st.out)
            stream.synchronize()
        return [st.out, int(st.scene.round_status()["complete"])]
    if kind == "train":
        st.rast.set_camera(0, st.cams[0])
        img = autograd.render(st.rast)
        return [img.detach(), *torch.autograd.grad(img, st.params, st.dl)]
    if kind == "net_train":
        g, loss = st.net.grads(st.img, st.depth, st.img)
        return [g, loss]
    if kind == "net_fill":
        if case["render"]:
            _frame(st)
        st.net.fill(st.scene, st.out)
        return st.out
    keys, vals = st.keys.clone(), st.vals.clone()
    a3fr.sort_pairs(keys, vals, st.keys_alt, st.vals_alt, case["bits"], st.ws)
    return [keys, vals]


def _net_macs(arch):
    return sum(i * o * k * k for i, o, k in periphery.ARCH_LAYERS[arch])


def work(case):
    kind = case["kind"]
    if kind == "sort":
        return {"bytes": 2 * 12 * case["n"], "flops": 0}
    px = case.get("eyes", 1) * case["width"] * case["height"]
    if kind == "net_train":
        px *= case["batch"]
        blocks = case["batch"] * ((case["width"] + 1) // 2) * ((case["height"] + 1) // 2)
        return {"bytes": 12 * px + 16 * blocks, "flops": 3 * 2 * blocks * _net_macs(case["arch"])}
    k = (case["sh"] + 1) ** 2
    n, eyes = case["n"], case.get("eyes", 1)
    scene = {"bytes": 4 * n * (11 + 3 * k) + 12 * px, "flops": n * eyes * (250 + 6 * k)}
    if kind == "train":
        return {"bytes": 2 * scene["bytes"], "flops": 3 * scene["flops"]}
    if kind == "net_fill":
        blocks = eyes * ((case["width"] + 1) // 2) * ((case["height"] + 1) // 2)
        net = {"bytes": 16 * blocks + 9 * px, "flops": 2 * blocks * _net_macs(case["arch"])}
        return {f: net[f] + (scene[f] if case["render"] else 0) for f in net}
    return scene


# ---------------------------------------------------------------------------- in 64 bits
def _sh(d, coef):
    """Colour of the real SH coefficients coef [n, k, 3] along unit directions d [n, 3]."""
    x, y, z = d.unbind(1)
    pi, k = math.pi, coef.shape[1]
    b = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if k > 1:
        c = math.sqrt(3 / (4 * pi))
        b += [-c * y, c * z, -c * x]
    if k > 4:
        a, e, f = 0.5 * math.sqrt(15 / pi), 0.25 * math.sqrt(5 / pi), 0.25 * math.sqrt(15 / pi)
        b += [a * x * y, -a * y * z, e * (2 * z * z - x * x - y * y), -a * x * z, f * (x * x - y * y)]
    if k > 9:
        a, e, f = 0.25 * math.sqrt(35 / (2 * pi)), 0.5 * math.sqrt(105 / pi), 0.25 * math.sqrt(21 / (2 * pi))
        g, h = 0.25 * math.sqrt(7 / pi), 0.25 * math.sqrt(105 / pi)
        q = 4 * z * z - x * x - y * y
        b += [-a * y * (3 * x * x - y * y), e * x * y * z, -f * y * q, g * z * (2 * z * z - 3 * x * x - 3 * y * y),
              -f * x * q, h * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return (torch.stack(b, 1)[:, :, None] * coef).sum(1)


def _project(params, cam, tile):
    """Records [n, 10] (u, v, conic, opacity, colour, depth), tile rectangles and visibility."""
    means, log_scales, quats, logits, coef = params
    w2c = torch.tensor(cam.world_to_cam, dtype=torch.float64, device=DEV)
    rot, shift = w2c[:, :3], w2c[:, 3]
    t = means @ rot.T + shift
    z = t[:, 2]
    seen = z > cam.znear
    z = torch.where(seen, z, torch.ones_like(z))
    q = torch.nn.functional.normalize(quats, dim=1)
    w, x, y, zq = q.unbind(1)
    r = torch.stack([1 - 2 * (y * y + zq * zq), 2 * (x * y - w * zq), 2 * (x * zq + w * y),
                     2 * (x * y + w * zq), 1 - 2 * (x * x + zq * zq), 2 * (y * zq - w * x),
                     2 * (x * zq - w * y), 2 * (y * zq + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    m = r * torch.exp(log_scales)[:, None, :]
    fx, fy = float(cam.fx), float(cam.fy)
    lx, ly = 1.3 * 0.5 * cam.width / fx, 1.3 * 0.5 * cam.height / fy
    xc, yc = (t[:, 0] / z).clamp(-lx, lx), (t[:, 1] / z).clamp(-ly, ly)
    o = torch.zeros_like(z)
    jac = torch.stack([fx / z, o, -fx * xc / z, o, fy / z, -fy * yc / z], 1).view(-1, 2, 3)
    a = jac @ rot @ m
    cov = a @ a.transpose(1, 2)
    ca, cb, cc = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = ca * cc - cb * cb
    mid = 0.5 * (ca + cc)
    radius = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1)))).detach()
    u, v = fx * t[:, 0] / z + cam.cx, fy * t[:, 1] / z + cam.cy
    tx, ty = -(-cam.width // tile), -(-cam.height // tile)

    def cells(c, lim):
        lo = torch.floor((c.detach() - radius) / tile).clamp(0, lim)
        hi = (torch.floor((c.detach() + radius) / tile) + 1).clamp(0, lim)
        return lo.long(), hi.long()

    (x0, x1), (y0, y1) = cells(u, tx), cells(v, ty)
    seen = seen & (x0 < x1) & (y0 < y1)
    d = torch.nn.functional.normalize(means + rot.T @ shift, dim=1)
    rgb = torch.relu(_sh(d, coef) + 0.5)
    rec = torch.stack([u, v, cc / det, -cb / det, ca / det, torch.sigmoid(logits), *rgb.unbind(1), z], 1)
    return rec, (x0, y0, x1, y1), seen


def _lists(rec, rect, seen, tx, ty):
    """Per tile the Gaussians in depth order: (indices, first of each tile, counts)."""
    idx = seen.nonzero()[:, 0]
    idx = idx[torch.argsort(rec[idx, 9], stable=True)]
    x0, y0, x1, y1 = (r[idx] for r in rect)
    cnt = (x1 - x0) * (y1 - y0)
    rep = torch.repeat_interleave(torch.arange(len(idx), device=DEV), cnt)
    k = torch.arange(len(rep), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[rep]
    w = (x1 - x0)[rep]
    tile = (y0[rep] + k // w) * tx + x0[rep] + k % w
    order = torch.argsort(tile, stable=True)
    counts = torch.bincount(tile, minlength=tx * ty)
    return idx[rep[order]], torch.cumsum(counts, 0) - counts, counts


def _composite(rec, gid, first, counts, cam, tile, dl=None, budget=1 << 24):
    """(colour [H, W, 3], depth [H, W]); with dl (gradient of the image), rec.grad receives the
    gradient of sum(dl * image)."""
    tx, ty = -(-cam.width // tile), -(-cam.height // tile)
    px = torch.arange(tile * tile, device=DEV)
    out = torch.zeros(tx * ty, tile * tile, 4, dtype=torch.float64, device=DEV)

    def split(img):     # [H, W, c] -> [tiles, pixels, c], zero past the edge
        pad = torch.zeros(ty * tile, tx * tile, img.shape[2], dtype=torch.float64, device=DEV)
        pad[:cam.height, :cam.width] = img
        return pad.view(ty, tile, tx, tile, -1).permute(0, 2, 1, 3, 4).reshape(tx * ty, tile * tile, -1)

    dl = None if dl is None else split(dl.double())
    order = torch.argsort(counts, descending=True).tolist()
    n_of = counts.tolist()
    k = 0
    while k < len(order) and n_of[order[k]] > 0:
        length = n_of[order[k]]
        t = torch.tensor(order[k:k + max(1, budget // (length * tile * tile))], device=DEV)
        k += len(t)
        at = torch.arange(length, device=DEV)
        valid = at < counts[t][:, None]
        r = rec[gid[(first[t][:, None] + at).clamp(max=len(gid) - 1)]]
        x = ((t % tx) * tile)[:, None] + px % tile
        y = ((t // tx) * tile)[:, None] + px // tile
        dx, dy = r[:, :, 0:1] - x[:, None, :], r[:, :, 1:2] - y[:, None, :]
        power = -0.5 * (r[:, :, 2:3] * dx * dx + r[:, :, 4:5] * dy * dy) - r[:, :, 3:4] * dx * dy
        alpha = (r[:, :, 5:6] * torch.exp(power)).clamp(max=0.99)
        alpha = torch.where(valid[:, :, None] & (power <= 0) & (alpha >= 1 / 255), alpha, 0.0)
        log_t = torch.cumsum(torch.log1p(-alpha), 1)
        w = alpha * torch.exp(log_t - torch.log1p(-alpha)) * (log_t >= math.log(1e-4))
        c = w.transpose(1, 2) @ r[:, :, 6:10]
        if dl is not None:
            (c[:, :, :3] * dl[t]).sum().backward()
        out[t] = c.detach()
    img = out.view(ty, tx, tile, tile, 4).permute(0, 2, 1, 3, 4).reshape(ty * tile, tx * tile, 4)
    img = img[:cam.height, :cam.width]
    return img[:, :, :3], img[:, :, 3]


def _tile_levels(cam, tile, gaze, radii, levels):
    tx, ty = -(-cam.width // tile), -(-cam.height // tile)
    x0 = torch.arange(tx, dtype=torch.float64, device=DEV) * tile
    y0 = torch.arange(ty, dtype=torch.float64, device=DEV) * tile
    dx = torch.maximum(x0 - gaze[0], gaze[0] - (x0 + tile - 1).clamp(max=cam.width - 1)).clamp(min=0)
    dy = torch.maximum(y0 - gaze[1], gaze[1] - (y0 + tile - 1).clamp(max=cam.height - 1)).clamp(min=0)
    d2 = dx[None, :] ** 2 + dy[:, None] ** 2
    lv = torch.full_like(d2, levels[-1])
    for r, level in reversed(list(zip(radii, levels))):
        lv[d2 <= r * r] = level
    return lv


def _shifted(a, dy, dx):
    """a[y + dy, x + dx], zero outside."""
    h, w = a.shape[:2]
    p = torch.zeros(h + 2, w + 2, *a.shape[2:], dtype=a.dtype, device=DEV)
    p[1:-1, 1:-1] = a
    return p[1 + dy:1 + dy + h, 1 + dx:1 + dx + w]


def _foveate(img, lv, tile, fill):
    """(image with the skipped pixels inherited or interpolated, which pixels are rendered)."""
    h, w = img.shape[:2]
    y, x = torch.arange(h, device=DEV), torch.arange(w, device=DEV)
    label = torch.tensor([[LABELS[dx, dy] for dx in (0, 1)] for dy in (0, 1)], device=DEV)
    live = lv[(y // tile)[:, None], x // tile] >= label[(y % 2)[:, None], x % 2]
    out = torch.where(live[:, :, None], img, img[(y - y % 2)[:, None], x - x % 2])
    if fill:
        seen = live[:, :, None].double()
        for steps in (((-1, -1), (-1, 1), (1, -1), (1, 1)), ((-1, 0), (1, 0), (0, -1), (0, 1))):
            total = sum(_shifted(img * seen, *s) for s in steps)
            count = sum(_shifted(seen, *s) for s in steps)
            out = torch.where((seen > 0) | (count == 0), out, total / count.clamp(min=1))
    return out, live


def _net(ws, bs, x, arch):
    """Corrections [b, 16, h, w] of the block inputs x [b, 4, h, w]."""
    def conv(i, v):
        return torch.nn.functional.conv2d(v, ws[i], bs[i], padding=ws[i].shape[-1] // 2)

    h = torch.relu(torch.nn.functional.conv2d(x, ws[0][:, :4], bs[0], padding=1))
    if arch == periphery.COMPACT:
        return conv(2, torch.relu(conv(1, h)))
    for b in range(4):
        h = h + conv(2 + 2 * b, torch.relu(conv(1 + 2 * b, h)))
    return conv(9, h)


def _predict(img, depth, ws, bs, arch):
    """Bilinear base plus correction of every pixel, [b, h, w, 3]."""
    b, h, w = img.shape[:3]
    tl = img[:, ::2, ::2]
    right = torch.cat([tl[:, :, 1:], tl[:, :, -1:]], 2)
    down, diag = (torch.cat([a[:, 1:], a[:, -1:]], 1) for a in (tl, right))
    base = torch.stack([tl, (tl + right) / 2, (tl + down) / 2, (tl + right + down + diag) / 4], -1)
    x = torch.cat([tl, depth[:, ::2, ::2, None] / 8], 3).permute(0, 3, 1, 2)
    r = torch.cat([_net(ws, bs, x[i:i + 1], arch) for i in range(b)]).permute(0, 2, 3, 1)
    p = base + r[..., :12].reshape(*base.shape)
    bh, bw = tl.shape[1:3]
    p = p.view(b, bh, bw, 3, 2, 2).permute(0, 1, 4, 2, 5, 3).reshape(b, 2 * bh, 2 * bw, 3)
    return p[:, :h, :w]


def _net_doubles(case, seed):
    ws, bs = periphery.unpack(_net_params(case, seed), case["arch"])
    return [[torch.tensor(a, dtype=torch.float64, device=DEV) for a in g] for g in (ws, bs)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "sort":
        return None
    if kind == "net_train":
        ws, bs = _net_doubles(case, seed)
        leaves = [t.requires_grad_() for t in ws + bs]
        img, depth = (t.double() for t in _crops(case, seed))
        total, count = 0.0, img.numel()
        for i in range(case["batch"]):
            e = _predict(img[i:i + 1], depth[i:i + 1], ws, bs, case["arch"]) - img[i:i + 1]
            loss = e.square().sum() / count
            loss.backward()
            total += float(loss.detach())
        return [torch.cat([t.grad.reshape(-1) for t in leaves]), total]
    cams, gazes = _head(case, seed)
    params = [p.double() for p in _scene(case, seed)]
    if kind == "train":
        leaves = [p.requires_grad_() for p in params]
        dl = torch.randn(1, case["height"], case["width"], 3, device=DEV, generator=_gen(seed + 1))
        rec, rect, seen = _project(leaves, cams[0], 16)
        leaf = rec.detach().requires_grad_()
        lists = _lists(rec.detach(), rect, seen, -(-case["width"] // 16), -(-case["height"] // 16))
        img, _ = _composite(leaf, *lists, cams[0], 16, dl=dl[0])
        keep = seen[:, None]     # a culled Gaussian's record takes no part
        rec.backward(torch.where(keep, leaf.grad, 0.0))
        return [img[None], *(p.grad for p in leaves)]
    tile, out = case["tile"], []
    net = _net_doubles(case, seed) if kind == "net_fill" else None
    with torch.no_grad():
        for cam, gaze in zip(cams, gazes.astype(np.float64)):
            tx, ty = -(-cam.width // tile), -(-cam.height // tile)
            rec, rect, seen = _project(params, cam, tile)
            gid, first, counts = _lists(rec, rect, seen, tx, ty)
            img, depth = _composite(rec, gid, first, counts, cam, tile)
            if case.get("mode") == "full":
                out.append(img)
                continue
            layers = case.get("layers", 3)
            radii = [cam.fx * math.tan(math.radians(t)) for t in THETAS[layers]]
            lv = _tile_levels(cam, tile, gaze, radii, LEVELS[layers])
            if kind == "rounds":
                early = np.float64(np.float32(gaze) + np.float32(0.06 * case["width"]))
                shrunk = [max(0.0, r - EXPECTED_PX[0]) for r in radii]
                lv = torch.maximum(lv, _tile_levels(cam, tile, early, shrunk, LEVELS[layers]))
            k = int(case.get("count_frac", 0.0) * tx * ty)
            if k >= 1:
                c = counts.view(ty, tx)
                heavy = (c > 0) & (c >= torch.sort(counts, descending=True)[0][k - 1])
                lv = torch.where(heavy & ((lv == 2) | (lv == 3)), lv - 1, lv)
            frame, live = _foveate(img, lv, tile, case.get("fill", 0))
            if net is not None:
                full = _predict(frame[None], depth[None], *net, case["arch"])[0]
                frame = torch.where(live[:, :, None], frame, full)
            out.append(frame)
    img = torch.stack(out)
    return [img, None] if kind == "rounds" else img
