"""ws_cull_sort_tiles: the compaction fused into the first partition pass of
the segmented tile sort gives the offsets, key count, sorted pairs, tile
ranges and status of ws_cull followed by ws_sort_tiles, bit for bit; past
the key capacity it flags the frame and leaves only valid pairs."""
import numpy as np
import pytest

from paper_2602_03207_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def _frames(scene_np, cam, tile=16, digit_bits=9, key_capacity=None, flags=0):
    import torch
    from paper_2602_03207_gb300 import capi, render
    dev = render.scene_to_device(scene_np)
    n = scene_np["means"].shape[0]
    c = capi.camera(cam)
    out = []
    for fused in (False, True):
        r = render.Renderer(n, cam["width"], cam["height"], tile=tile, digit_bits=digit_bits,
                            key_capacity=key_capacity, flags=flags)
        r.preprocess(dev, c)
        if fused:
            r.cull_sort(c)
            assert getattr(r, "_fused_cull", True), "the fused call should apply"
        else:
            r.cull(c)
            r.sort()
        torch.cuda.synchronize()
        k = min(int(r.num_keys[0].item()), r.key_capacity)
        out.append({"offsets": r.offsets[:n + 1].cpu().numpy(), "num_keys": r.num_keys[:1].cpu().numpy(),
                    "keys": r.sorted_keys[:k].cpu().numpy(), "vals": r.sorted_vals[:k].cpu().numpy(),
                    "ranges": r.ranges[:r.tx * r.ty].cpu().numpy(),
                    "status": capi.ws_read_status(r.workspace, clear=False), "r": r})
    return out


def _same(a, b):
    for k in ("offsets", "num_keys", "keys", "vals", "ranges", "status"):
        np.testing.assert_array_equal(np.asarray(b[k]), np.asarray(a[k]), err_msg=k)


@pytest.mark.parametrize("case", ["hd0", "hd3", "train", "small4", "small9", "ragged"])
def test_fused_cull_sort_equals_separate_calls(case):
    """First digits of 7 (1080p), 6 (720p), 4 (256 tiles at 4-bit digits: two
    passes), 8 (256 tiles at 9-bit digits: the whole partition in the
    compaction) and 6 bits (35 tiles of a ragged 100x75 image)."""
    if case.startswith("hd"):
        scene, cam, kw = S.hd_scene(), S.hd_camera(int(case[2])), {}
    elif case == "train":
        scene, cam, _ = S.grad_scene()
        kw = {}
    elif case == "ragged":
        scene, cam = S.small_forward()
        cam = dict(cam, width=100, height=75)
        kw = {"key_capacity": 40 * len(scene["means"])}
    else:
        scene, cam = S.small_forward()
        kw = {"digit_bits": int(case[5:]), "key_capacity": 40 * len(scene["means"])}
    a, b = _frames(scene, cam, **kw)
    assert a["num_keys"][0] > 0
    _same(a, b)


def test_fused_cull_sort_rows_wider_than_the_digit_range():
    """Large splats: at 1280x720 (80-tile rows, 6-bit first digit) 719 of
    2,000 rectangles have rows wider than the 64 digits, so a row adds a full
    turn of the digits plus a run that may wrap; at 256x256 with 4-bit digits
    496 have 16-tile rows, exactly one turn. Also with the culling switched
    off (rectangles clamped into the grid)."""
    from paper_2602_03207_gb300 import capi
    scene = S.uniform_scene(2000, seed=5, log_scale_mean=-1.0, log_scale_std=0.4)
    cam = S.look_at_camera((2.4, -0.8, 0.7), (0.0, 0.0, 0.0), 1280, 720)
    for flags in (0, capi.WS_CFG_NO_AABB_CULL | capi.WS_CFG_NO_OPACITY_CULL):
        a, b = _frames(scene, cam, key_capacity=8_000_000, flags=flags)
        assert not (a["status"] & capi.WS_FLAG_CAPACITY)
        _same(a, b)
    _, cam = S.small_forward()
    scene = S.uniform_scene(3000, seed=5, log_scale_mean=-1.0, log_scale_std=0.4)
    a, b = _frames(scene, cam, digit_bits=4, key_capacity=600_000)
    assert not (a["status"] & capi.WS_FLAG_CAPACITY)
    _same(a, b)


@pytest.mark.parametrize("case", ["culled", "one_tile", "two_tiles"])
def test_fused_cull_sort_degenerate_frames(case):
    """A frame whose every splat is culled (no pairs), a 12x10 image (one
    tile) and a 30x10 image (two tiles): the fused call gives what the two
    calls give."""
    scene, cam = S.small_forward()
    scene = {k: v[:2000].copy() for k, v in scene.items()}
    if case == "culled":
        scene["opacity_logits"][:] = -7.0
    else:
        cam = dict(cam, width=12 if case == "one_tile" else 30, height=10)
    a, b = _frames(scene, cam, key_capacity=64 * 2000)
    _same(a, b)
    if case == "culled":
        assert int(a["num_keys"][0]) == 0


def test_fused_cull_sort_uhd():
    """6,000,000 Gaussians at 3840x2160: 15 tile bits, first digit 8."""
    a, b = _frames(S.uhd_scene(), S.uhd_camera(3))
    _same(a, b)


def test_fused_cull_sort_past_capacity_keeps_valid_pairs():
    """More pairs than the key capacity: the frame is flagged, the count is
    the capacity, and every stored pair names a Gaussian of the frame and a
    tile of the grid (the compaction falls back to slot order), so the
    rasterisation that follows reads only valid records."""
    import torch
    from paper_2602_03207_gb300 import capi
    scene, cam = S.small_forward()
    n = len(scene["means"])
    a, b = _frames(scene, cam, key_capacity=1024)
    for fr in (a, b):
        assert fr["status"] & capi.WS_FLAG_CAPACITY
        assert int(fr["num_keys"][0]) == 1024
        assert (fr["vals"].view(np.uint32) < n).all()
        tiles = fr["keys"].view(np.uint64) >> np.uint64(31)
        assert (tiles < fr["r"].tx * fr["r"].ty).all()
    r = b["r"]
    r.rasterize(capi.camera(cam))
    torch.cuda.synchronize()
    assert np.isfinite(r.image.cpu().numpy()).all()


@pytest.mark.parametrize("n", [1, 16 * 1024, 16 * 1024 + 1, 2048 * 1024, 2048 * 1024 + 1])
@pytest.mark.parametrize("room", [1.0, 0.5])
def test_offsets_at_the_edges_of_each_scan(n, room):
    """Each way an emission finds its first slot (the counts, the chunk sums or
    their scan) on both sides of its limit: offsets, count, flag and pairs
    against a cumulative sum, also where half of the pairs fit."""
    import torch
    from paper_2602_03207_gb300 import capi
    rng = np.random.default_rng(n)
    wide = rng.integers(0, 4, n)  # tiles of a one-row rectangle; 0 culls
    rect = np.zeros((n, 4), np.uint16)
    rect[:, 0] = rng.integers(0, 12, n)
    rect[:, 1] = rect[:, 3] = rng.integers(0, 16, n)
    rect[:, 2] = rect[:, 0] + np.maximum(wide, 1) - 1
    depth = rng.uniform(1.0, 9.0, n).astype(np.float32)
    total = int(wide.sum())
    cap = max(1, int(total * room))
    cam = capi.camera(dict(S.small_forward()[1], width=256, height=256))
    cfg = capi.config()
    dev = lambda a: torch.from_numpy(a).cuda()
    offsets = torch.zeros(n + 4, dtype=torch.int32, device="cuda")
    keys = torch.zeros(cap + 2, dtype=torch.int64, device="cuda")
    vals = torch.zeros(cap + 4, dtype=torch.int32, device="cuda")
    num = torch.zeros(4, dtype=torch.int32, device="cuda")
    work = torch.zeros(capi.ws_workspace_bytes(n, cap, cam, cfg), dtype=torch.uint8, device="cuda")
    capi.ws_cull(n, dev(wide.astype(np.int32)), dev(rect.view(np.int16)), dev(depth), cam, cfg, offsets, keys, vals,
                 cap, num, work)
    first = np.concatenate([[0], np.cumsum(wide)])
    np.testing.assert_array_equal(offsets[:n + 1].cpu().numpy(), first)
    kept = min(cap, total)
    assert int(num[0]) == kept
    assert capi.ws_read_status(work) == int(total > cap)
    gid = np.repeat(np.arange(n), wide)[:kept]
    tile = rect[gid, 1].astype(np.uint64) * 16 + rect[gid, 0] + (np.arange(kept) - first[gid]).astype(np.uint64)
    np.testing.assert_array_equal(vals[:kept].cpu().numpy(), gid)
    np.testing.assert_array_equal(keys[:kept].cpu().numpy().view(np.uint64),
                                  (tile << np.uint64(31)) | depth[gid].view(np.uint32).astype(np.uint64))
    assert not keys[kept:].any() and not vals[kept:].any()


@pytest.mark.parametrize("kind", ["few", "many", "fits", "one_more", "large"])
def test_emission_of_rectangles_of_every_size(kind):
    """The slot map's ways: a thread's few pairs, a thread with more than 32, a
    chunk of exactly 4,096 pairs and of one more, and a rectangle of more."""
    import torch
    from paper_2602_03207_gb300 import capi
    rng = np.random.default_rng(len(kind))
    n, tx = 2500, 256
    w, h = rng.integers(1, 4, n), rng.integers(1, 3, n)
    live = rng.random(n) < 0.6
    if kind == "many":
        w[::37], h[::37] = rng.integers(5, 60, n)[::37], rng.integers(1, 5, n)[::37]
    elif kind in ("fits", "one_more"):
        live[:1024], w[:1024], h[:1024] = True, 4, 1
        if kind == "one_more":
            w[500] = 5
    elif kind == "large":
        live[700], w[700], h[700] = True, 90, 100
    x, y = rng.integers(0, tx - w + 1), rng.integers(0, 256 - h + 1)
    rect = np.stack([x, y, x + w - 1, y + h - 1], 1).astype(np.uint16)
    touched = np.where(live, w * h, 0)
    depth = rng.uniform(1.0, 9.0, n).astype(np.float32)
    total = int(touched.sum())
    cam, cfg = capi.camera(dict(S.small_forward()[1], width=16 * tx, height=4096)), capi.config()
    dev = lambda a: torch.from_numpy(a).cuda()
    offsets = torch.zeros(n + 4, dtype=torch.int32, device="cuda")
    keys = torch.zeros(total + 2, dtype=torch.int64, device="cuda")
    vals = torch.zeros(total + 4, dtype=torch.int32, device="cuda")
    num = torch.zeros(4, dtype=torch.int32, device="cuda")
    work = torch.zeros(capi.ws_workspace_bytes(n, total, cam, cfg), dtype=torch.uint8, device="cuda")
    capi.ws_cull(n, dev(touched.astype(np.int32)), dev(rect.view(np.int16)), dev(depth), cam, cfg, offsets, keys,
                 vals, total, num, work)
    gid = np.repeat(np.arange(n), touched)
    j = np.arange(total) - np.repeat(np.cumsum(touched) - touched, touched)
    tile = (y[gid] + j // w[gid]) * tx + x[gid] + j % w[gid]
    assert int(num[0]) == total and capi.ws_read_status(work) == 0
    np.testing.assert_array_equal(vals[:total].cpu().numpy(), gid)
    np.testing.assert_array_equal(keys[:total].cpu().numpy().view(np.uint64),
                                  (tile.astype(np.uint64) << np.uint64(31)) | depth[gid].view(np.uint32))


@pytest.mark.parametrize("sort", ["segmented", "lsd", "lookback"])
@pytest.mark.parametrize("size", [(16, 16), (100, 75)], ids=["one_tile", "ragged"])
def test_whole_frame_calls_equal_staged_calls(sort, size):
    """A frame, a packed frame and a training step as one call against the
    stages called one by one: the same bits, and the same ranges and pairs
    kept for later calls."""
    import torch
    from paper_2602_03207_gb300 import capi, render
    scene, cam = S.small_forward()
    cam = dict(cam, width=size[0], height=size[1])
    dev = render.scene_to_device(scene)
    n = len(scene["means"])
    target = torch.rand(size[1], size[0], 3, device="cuda")
    for packed in (False, True):
        a, b = (render.Renderer(n, *size, key_capacity=64 * n, packed=packed, sort=sort) for _ in range(2))
        c = capi.camera(cam)
        a.preprocess(dev, c)
        a.cull(c)
        a.sort()
        a.rasterize(c)
        b.forward(dev, cam)
        assert a.sorted_in_alt == b.sorted_in_alt and a.raster_cfg.flags == b.raster_cfg.flags
        for name in ("image", "t_final", "n_contrib", "ranges"):
            assert torch.equal(getattr(a, name), getattr(b, name)), name
        if not packed:
            ga = a.train_pass_l2(dev, cam, target)
            gb = b.train_step_l2(dev, cam, target)
            assert all(torch.equal(ga[k], gb[k]) for k in ga) and torch.equal(a.image, b.image)
