"""Performance cases of the render path.

What users of this library have it do, through its public entry points: single frames from 10,000 to 6,000,000
Gaussians (``Renderer.forward``, its packed-record and quad variants, ``FramePipeline`` from host memory), one
differentiable frame (``render_differentiable`` and ``backward()``), one fused L2 training step
(``Renderer.train_step_l2``), a training step over many views (``BatchRenderer``, eager and as a CUDA graph), and
the (tile, depth) pair sort alone.

Scenes are drawn on the GPU from the seed with the distributions of ``synthetic.uniform_scene`` (the small workload)
and ``synthetic.cluster_scene`` (the others): clusters with anisotropic spreads, log-normal scales, 40 % of the
opacities near zero, degree-3 SH. ``exact`` renders the same inputs in plain torch in 64 bits, gradients by autograd.
"""
import math

import numpy as np
import torch

from paper_2602_03207_gb300 import batch, capi, render
from paper_2602_03207_gb300 import synthetic as S

KEYS = ("means", "log_scales", "quats", "opacity_logits", "sh")


def listed():
    return [
        # A preview-sized frame (synthetic.small_forward): launches and host work count.
        {"name": "frame 10k 256x256", "kind": "frame", "scene": "uniform", "n": 10_000, "width": 256, "height": 256,
         "tile": 16, "digit_bits": 8, "bg": 0.0},
        # The benchmark's frame: a viewer at 1080p.
        {"name": "frame 1M 1080p", "kind": "frame", "scene": "cluster", "n": 1_000_000, "width": 1920, "height": 1080,
         "tile": 16, "digit_bits": 9, "bg": 0.0},
        # A large capture at 4K (synthetic.uhd_scene).
        {"name": "frame 6M 2160p", "kind": "frame", "scene": "cluster", "n": 6_000_000, "width": 3840, "height": 2160,
         "tile": 16, "digit_bits": 8, "bg": 0.0},
        # The packed-record variant on an odd-sized frame with an odd number of splats over a grey background.
        {"name": "packed 100003 1237x701", "kind": "packed", "scene": "cluster", "n": 100_003, "width": 1237,
         "height": 701, "tile": 16, "digit_bits": 8, "bg": 0.5},
        # The paper's own design (global depth sort, quads) on the benchmark's frame.
        {"name": "quads 1M 1080p", "kind": "quads", "scene": "cluster", "n": 1_000_000, "width": 1920, "height": 1080,
         "tile": 16, "digit_bits": 8, "bg": 0.0},
        # Frames of a scene that lives in host memory (the benchmark's end-to-end path).
        {"name": "host 1M 1080p", "kind": "host", "scene": "cluster", "n": 1_000_000, "width": 1920, "height": 1080,
         "tile": 16, "digit_bits": 8, "bg": 0.0},
        # A small differentiable frame, forward and backward through autograd.
        {"name": "autograd 10k 256x256", "kind": "autograd", "scene": "uniform", "n": 10_000, "width": 256,
         "height": 256, "tile": 16, "digit_bits": 8, "bg": 0.0},
        # The training workload (synthetic.grad_scene) with a user's own loss, through autograd.
        {"name": "autograd 500k 720p", "kind": "autograd", "scene": "cluster", "n": 500_000, "width": 1280,
         "height": 720, "tile": 16, "digit_bits": 8, "bg": 0.0},
        # The same workload through the fused L2 training step.
        {"name": "train_l2 500k 720p", "kind": "train_l2", "scene": "cluster", "n": 500_000, "width": 1280,
         "height": 720, "tile": 16, "digit_bits": 8, "bg": 0.0},
        # A small batch of uneven views, one eager training step of the separate calls.
        {"name": "batch 6x300k eager", "kind": "batch", "scene": "cluster", "n": 300_000, "views": 6, "tile": 16,
         "digit_bits": 9, "fused": False, "graph": False, "bg": 0.0},
        # The batched workload (synthetic.batch_scene, batch_views): 64 uneven views, the fused step as a CUDA graph.
        {"name": "batch 64x2M graph", "kind": "batch", "scene": "cluster", "n": 2_000_000, "views": 64, "tile": 16,
         "digit_bits": 11, "fused": True, "graph": True, "bg": 0.0},
        # The pair sort alone (synthetic.sort_keys): 4,194,304 keys over the 8,160 tiles of a 1080p frame.
        {"name": "sort 4M", "kind": "sort", "n": 4_194_304, "tiles": 8160, "digit_bits": 8, "sort": "segmented"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any kind, sizes spread over their logarithm."""
    kind = rng.choice(["frame", "frame", "packed", "quads", "host", "autograd", "autograd", "train_l2", "train_l2",
                       "batch", "batch", "sort"])
    digit_bits = rng.choice([8, 9, 11])
    if kind == "sort":
        return {"kind": kind, "n": _log(rng, 10_000, 8_000_000), "tiles": _log(rng, 256, 32_400),
                "digit_bits": digit_bits, "sort": rng.choice(["segmented", "segmented", "lsd"])}
    tile = rng.choice([16, 16, 16, 8, 32])
    bg = rng.choice([0.0, 0.0, 0.5, 1.0])
    if kind == "batch":
        views = _log(rng, 2, 32)
        return {"kind": kind, "scene": "cluster", "n": _log(rng, 10_000, min(2_000_000, 24_000_000 // views)),
                "views": views, "tile": tile, "digit_bits": digit_bits, "fused": rng.random() < 0.5,
                "graph": rng.random() < 0.5, "bg": bg}
    most = {"frame": 6_000_000, "host": 1_000_000}.get(kind, 2_000_000)
    width = _log(rng, 256, 3840)
    return {"kind": kind, "scene": "cluster", "n": _log(rng, 10_000, most), "width": width,
            "height": max(144, min(2160, int(width * rng.uniform(0.5, 1.0)))), "tile": tile,
            "digit_bits": digit_bits, "bg": bg}


# ------------------------------------------------------------------ inputs

def _box(case):
    """Scene side: larger captures are larger places (20 units up to 2M Gaussians, 60 at 6M)."""
    return 60.0 if case["n"] > 3_000_000 else 20.0


def _scene(case, seed):
    n = case["n"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    kw = {"generator": g, "device": "cuda", "dtype": torch.float64}
    q = torch.randn(n, 4, **kw)
    quats = q / q.norm(dim=1, keepdim=True)
    if case["scene"] == "uniform":  # synthetic.uniform_scene
        means = torch.rand(n, 3, **kw) * 2 - 1
        log_scales = torch.randn(n, 3, **kw) * 0.5 - 4.0
        logits = torch.randn(n, **kw) * 1.5
    else:  # synthetic.cluster_scene
        box, clusters = _box(case), 64
        scale = box / 20.0
        centres = (torch.rand(clusters, 3, **kw) - 0.5) * box
        rot = torch.linalg.qr(torch.randn(clusters, 3, 3, **kw).cpu())[0].cuda()
        std = (torch.rand(clusters, 3, **kw) * 1.7 + 0.3) * scale
        which = torch.randint(0, clusters, (n,), generator=g, device="cuda")
        local = torch.randn(n, 3, **kw) * std[which]
        means = centres[which] + (rot[which] * local[:, None, :]).sum(-1)
        log_scales = torch.randn(n, 3, **kw) * 0.8 - 5.0 + math.log(scale)
        low = torch.rand(n, **kw) < 0.4
        sig = torch.exp(torch.rand(n, **kw) * math.log(0.05 / 1e-4) + math.log(1e-4))
        # N(0, 1.5) conditioned on sigma >= 0.05, by its inverse distribution function
        least = 0.5 * (1.0 + math.erf((math.log(0.05) - math.log(0.95)) / 1.5 / math.sqrt(2.0)))
        u = (least + (1.0 - least) * torch.rand(n, **kw)).clamp(max=1.0 - 1e-12)
        logits = torch.where(low, torch.log(sig) - torch.log1p(-sig), 1.5 * math.sqrt(2.0) * torch.erfinv(2 * u - 1))
    sh = torch.randn(n, 16, 3, **kw) * 0.1
    sh[:, 0] *= 5.0
    out = {"means": means, "log_scales": log_scales, "quats": quats, "opacity_logits": logits, "sh": sh}
    return {k: v.to(torch.float32).contiguous() for k, v in out.items()}


def _cams(case, seed):
    rng = np.random.default_rng(seed)
    bg = (case["bg"],) * 3
    if case["scene"] == "uniform":
        w, h = case["width"], case["height"]
        view = np.concatenate([np.eye(3), [[rng.uniform(-0.1, 0.1)], [rng.uniform(-0.1, 0.1)], [3.0]]], axis=1)
        return [{"viewmat": view.astype(np.float32), "fx": float(w), "fy": float(w), "cx": w / 2.0, "cy": h / 2.0,
                 "width": w, "height": h, "znear": float(np.float32(0.2)), "bg": bg}]
    box = _box(case)
    cams = []
    for v in range(case.get("views", 1)):
        w, h = case.get("width"), case.get("height")
        if w is None:  # uneven views: the sizes of synthetic.batch_views, the same for every seed
            size = np.random.default_rng(200 + v)
            w, h = int(size.integers(320, 1921)), int(size.integers(240, 1081))
        az = rng.uniform(0.0, 2.0 * math.pi)
        pos = (1.25 * box * math.cos(az), 1.25 * box * math.sin(az), 0.25 * box)
        cams.append(S.look_at_camera(pos, (0.0, 0.0, 0.0), w, h, bg=bg))
    return cams


def _sort_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["n"]
    tile = torch.randint(0, case["tiles"], (n,), generator=g, device="cuda", dtype=torch.int64)
    depth = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 59.0 + 1.0
    bits = depth.to(torch.float32).view(torch.int32).to(torch.int64)
    return (tile << 31) | bits, torch.arange(n, device="cuda", dtype=torch.int32)


def _target(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    return torch.rand(shape, generator=g, device="cuda")


def _renderer(case):
    # 8-pixel tiles need room for more pairs per splat than the default
    cap = 12 * case["n"] if case["tile"] == 8 else None
    return render.Renderer(case["n"], case["width"], case["height"], tile=case["tile"],
                           digit_bits=case["digit_bits"], key_capacity=cap, packed=case["kind"] == "packed")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sort":
        keys, vals = _sort_inputs(case, seed)
        cfg = capi.config(digit_bits=case["digit_bits"], flags=render.SORT_FLAGS[case["sort"]])
        cam = capi.camera(S.small_forward()[1])
        work_bytes = capi.ws_workspace_bytes(0, case["n"], cam, cfg)
        return {"kind": kind, "keys": keys, "vals": vals, "n": case["n"], "cfg": cfg,
                "end_bit": 31 + max(1, math.ceil(math.log2(case["tiles"]))),
                "num": torch.tensor([case["n"], 0, 0, 0], dtype=torch.int32, device="cuda"),
                "k": [torch.empty_like(keys) for _ in range(2)], "v": [torch.empty_like(vals) for _ in range(2)],
                "work": torch.zeros(work_bytes, dtype=torch.uint8, device="cuda")}
    scene, cams = _scene(case, seed), _cams(case, seed)
    state = {"kind": kind, "scene": scene, "cam": cams[0]}
    if kind == "batch":
        cap = 8 * case["n"] * len(cams) if case["tile"] == 8 else None
        b = batch.BatchRenderer(case["n"], cams, tile=case["tile"], digit_bits=case["digit_bits"], key_capacity=cap,
                                fused=case["fused"])
        state["batch"] = b
        state["target"] = _target(b.total_pix * 3, seed)
        state["graph"] = b.capture(scene, state["target"]) if case["graph"] else None
    elif kind == "host":
        state["scene"] = {k: v.cpu().pin_memory() for k, v in scene.items()}
        cap = 12 * case["n"] if case["tile"] == 8 else None
        state["pipe"] = render.FramePipeline(case["n"], case["width"], case["height"], slots=2, tile=case["tile"],
                                             digit_bits=case["digit_bits"], key_capacity=cap)
        state["frames"] = [torch.empty(case["height"], case["width"], 3).pin_memory() for _ in range(2)]
    else:
        state["r"] = _renderer(case)
        if kind in ("autograd", "train_l2"):
            state["target"] = _target((case["height"], case["width"], 3), seed)
        if kind == "autograd":
            state["scene"] = {k: v.requires_grad_() for k, v in scene.items()}
    return state


def run(state):
    kind, scene = state["kind"], state.get("scene")
    if kind in ("frame", "packed"):
        return {"image": state["r"].forward(scene, state["cam"])}
    if kind == "quads":
        return {"image": state["r"].forward_quads(scene, state["cam"])}
    if kind == "host":
        frames = state["frames"]
        frames.append(frames.pop(0))  # the pipeline's slots take turns, and so do the images
        state["pipe"].submit(scene, state["cam"], frames[0])
        return {"image": frames[0]}
    if kind == "autograd":
        for p in scene.values():
            p.grad = None
        image = render.render_differentiable(scene, state["r"], state["cam"])
        (0.5 * (image - state["target"]).square().sum()).backward()
        return {"image": image, "grads": {k: p.grad for k, p in scene.items()}}
    if kind == "train_l2":
        grads = state["r"].train_step_l2(scene, state["cam"], state["target"])
        return {"image": state["r"].image, "grads": grads}
    if kind == "batch":
        b = state["batch"]
        if state["graph"] is not None:
            state["graph"].replay()
        else:
            b.step(scene, state["target"])
        return {"image": b.image, "grads": b.grads}
    # the sort takes its input buffers as scratch: each pass starts from a fresh list
    k, v = state["k"], state["v"]
    k[0].copy_(state["keys"])
    v[0].copy_(state["vals"])
    alt = capi.ws_sort(state["num"], state["n"], 0, state["end_bit"], k[0], v[0], k[1], v[1], state["cfg"],
                       state["work"])
    return {"keys": k[int(alt)], "vals": v[int(alt)]}


# ------------------------------------------------------------------ work

def work(case):
    """Bytes: of the clustered scene 76 % of the Gaussians pass the opacity test and 63 % are visible; a visible one
    is read whole (236 B), one culled later without its SH record, one culled by opacity costs its logit. Outputs
    once: the image, and for a training step the target read and every gradient written. Operations: 11 per pixel
    centre inside a splat's extent box up to the 1/255 test and 8 for each of the pi/4 that composite; in a backward
    11 more and 43 for each that composites."""
    n = case["n"]
    if case["kind"] == "sort":
        return {"bytes": 24.0 * n, "flops": 0.0}
    opaque, visible = (0.76, 0.63) if case["scene"] == "cluster" else (1.0, 1.0)
    backward = case["kind"] in ("autograd", "train_l2", "batch")
    read = n * (4 + opaque * 40 + visible * 192)
    views, width = case.get("views", 1), case.get("width", 1120)  # 1120x660: the mean of the uneven views
    pixels = views * width * case.get("height", 660)
    # evaluations: 4 E[q_c] sqrt(Sigma'_xx Sigma'_yy) pixel centres in a visible splat's box, E[q_c] about 6
    if case["scene"] == "cluster":  # pixels per unit at the scene's centre times a typical scale
        s = width / (2.0 * math.tan(math.radians(30.0))) / (1.25 * _box(case)) * math.exp(-5.0) * _box(case) / 20.0
        var = s * s * math.exp(2.0 * 0.8 * 0.8)
    else:
        s = width / 3.0 * math.exp(-4.0)
        var = s * s * math.exp(2.0 * 0.5 * 0.5)
    evals = views * visible * n * 4.0 * 6.0 * (0.3 + 0.6 * var)
    nbytes = read + pixels * 12 * (2 if backward else 1)
    if backward:
        nbytes += n * 236
    return {"bytes": float(nbytes), "flops": float(evals * (17.3 + (44.8 if backward else 0.0)))}


# ------------------------------------------------------------------ 64-bit values

def _basis(d):
    """Real SH of degree 3 with the Condon-Shortley phase, index l * l + l + m."""
    x, y, z = d.unbind(1)
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    c1, c2 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / (4 * pi))
    c20, c22 = math.sqrt(5 / (16 * pi)), math.sqrt(15 / (16 * pi))
    c30, c31 = math.sqrt(7 / (16 * pi)), math.sqrt(21 / (32 * pi))
    c32, c33 = math.sqrt(105 / (4 * pi)), math.sqrt(35 / (32 * pi))
    return torch.stack([
        torch.full_like(x, math.sqrt(1 / (4 * pi))), -c1 * y, c1 * z, -c1 * x,
        c2 * x * y, -c2 * y * z, c20 * (2 * zz - xx - yy), -c2 * x * z, c22 * (xx - yy),
        -c33 * y * (3 * xx - yy), c32 * x * y * z, -c31 * y * (4 * zz - xx - yy),
        c30 * z * (2 * zz - 3 * xx - 3 * yy), -c31 * x * (4 * zz - xx - yy), 0.5 * c32 * z * (xx - yy),
        -c33 * x * (xx - 3 * yy)], dim=1)


def _image64(scene, p, cam, dilation=0.3, guard=1.3):
    """The frame in 64 bits, (H, W, 3): every splat evaluated at every pixel of its extent, composited per pixel in
    (float32 depth, index) order. `scene`: the float32 inputs, which decide order and culling; `p`: the same in 64
    bits, which gradients flow into."""
    W, H = cam["width"], cam["height"]
    fx, fy, cx, cy = cam["fx"], cam["fy"], cam["cx"], cam["cy"]
    view = torch.as_tensor(np.asarray(cam["viewmat"], dtype=np.float32), device="cuda")
    R, t = view[:, :3].double(), view[:, 3].double()
    bg = torch.tensor(cam["bg"], device="cuda", dtype=torch.float64)
    with torch.no_grad():
        x, y, z = scene["means"].unbind(1)
        depth = ((view[2, 0] * x + view[2, 1] * y) + view[2, 2] * z) + view[2, 3]
        live = (scene["opacity_logits"].double() >= -math.log(254.0)) & (depth > cam["znear"])
        live &= scene["quats"].abs().amax(1) > 0
        ids = live.nonzero().squeeze(1)
        ids = ids[torch.argsort(depth[ids], stable=True)]
    take = lambda k: p[k].index_select(0, ids)  # noqa: E731
    m = take("means")
    tc = m @ R.T + t
    rz = 1.0 / tc[:, 2]
    ux, uy = tc[:, 0] * rz, tc[:, 1] * rz
    mx, my = fx * ux + cx, fy * uy + cy
    lx, ly = guard * 0.5 * W / fx, guard * 0.5 * H / fy
    zero = torch.zeros_like(rz)
    J = torch.stack([torch.stack([fx * rz, zero, -fx * ux.clamp(-lx, lx) * rz], 1),
                     torch.stack([zero, fy * rz, -fy * uy.clamp(-ly, ly) * rz], 1)], 1)
    q = take("quats")
    qw, qx, qy, qz = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    rot = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                       2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                       2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)], 1).view(-1, 3, 3)
    V = (J @ R) @ (rot * take("log_scales").exp()[:, None, :])
    sxx = V[:, 0].square().sum(1) + dilation
    syy = V[:, 1].square().sum(1) + dilation
    sxy = (V[:, 0] * V[:, 1]).sum(1)
    det = sxx * syy - sxy * sxy
    a, b, c = syy / det, -sxy / det, sxx / det
    sigma = torch.sigmoid(take("opacity_logits"))
    eye = -(R.T @ t)
    d = m - eye
    Y = _basis(d / d.norm(dim=1, keepdim=True))
    rgb = ((take("sh") * Y[:, :, None]).sum(1) + 0.5).clamp(min=0.0)
    with torch.no_grad():
        qc = (2.0 * (math.log(255.0) + torch.log(sigma))).clamp(min=0.0) * 1.0001 + 1e-6
        ex, ey = (qc * sxx).sqrt(), (qc * syy).sqrt()
        x0 = (mx - ex - 0.5).ceil().clamp(0, W).long()
        x1 = (mx + ex - 0.5).floor().clamp(-1, W - 1).long()
        y0 = (my - ey - 0.5).ceil().clamp(0, H).long()
        y1 = (my + ey - 0.5).floor().clamp(-1, H - 1).long()
        w, h = (x1 - x0 + 1).clamp(min=0), (y1 - y0 + 1).clamp(min=0)
        count = w * h
        ends = count.cumsum(0)
        who, where, first, total = [], [], 0, int(ends[-1]) if len(ends) else 0
        done = 0
        while done < total:  # about 64M (splat, pixel) candidates at a time
            last = min(len(ends), int(torch.searchsorted(ends, done + 64_000_000)) + 1)
            part = torch.arange(first, last, device="cuda").repeat_interleave(count[first:last])
            j = torch.arange(part.numel(), device="cuda") + done - (ends[part] - count[part])
            jy = j // w[part]
            py, px = y0[part] + jy, x0[part] + j - jy * w[part]
            dx, dy = px + 0.5 - mx[part], py + 0.5 - my[part]
            power = a[part] * dx * dx + 2 * b[part] * dx * dy + c[part] * dy * dy
            keep = sigma[part] * torch.exp(-0.5 * power) >= 1.0 / 255.0
            who.append(part[keep].int())
            where.append((py * W + px)[keep].int())
            first, done = last, int(ends[last - 1])
        if not who:
            return bg.expand(H, W, 3)
        pix, order = torch.sort(torch.cat(where), stable=True)
        who = torch.cat(who)[order].long()
        del where, order
        pix = pix.long()
        start = torch.searchsorted(pix, pix)
        px, py = (pix % W) + 0.5, (pix // W) + 0.5
    g = lambda v: v.index_select(0, who)  # noqa: E731
    dx, dy = px - g(mx), py - g(my)
    alpha = (g(sigma) * torch.exp(-0.5 * (g(a) * dx * dx + 2 * g(b) * dx * dy + g(c) * dy * dy))).clamp(max=0.99)
    logs = torch.log1p(-alpha)
    before = logs.cumsum(0) - logs
    weight = alpha * torch.exp(before - before.index_select(0, start))
    image = torch.zeros(H * W, 3, device="cuda", dtype=torch.float64).index_add(0, pix, g(rgb) * weight[:, None])
    left = torch.zeros(H * W, device="cuda", dtype=torch.float64).index_add(0, pix, logs).exp()
    return (image + left[:, None] * bg).view(H, W, 3)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sort":  # whole numbers
        return None
    if case["n"] * case.get("views", 1) > 16_000_000:  # too long in 64 bits
        return None
    scene, cams = _scene(case, seed), _cams(case, seed)
    backward = kind in ("autograd", "train_l2", "batch")
    p = {k: v.double().requires_grad_(backward) for k, v in scene.items()}
    if not backward:
        with torch.no_grad():  # (the packed records' 8-bit colours and 16-bit axes are part of their error)
            return {"image": _image64(scene, p, cams[0])}
    sizes = [c["width"] * c["height"] * 3 for c in cams]
    target = _target(sum(sizes), seed) if kind == "batch" else \
        _target((case["height"], case["width"], 3), seed).view(-1)
    images = []
    for c, goal in zip(cams, target.double().split(sizes)):
        image = _image64(scene, p, c)
        if image.requires_grad:
            (0.5 * (image.view(-1) - goal).square().sum()).backward()
        images.append(image.detach())
    grads = {k: p[k].grad if p[k].grad is not None else torch.zeros_like(p[k]) for k in KEYS}
    return {"image": torch.cat([i.view(-1) for i in images]) if kind == "batch" else images[0], "grads": grads}
