"""The blends' visit streams at the sizes where they can go wrong: list lengths
around the staging batches (96 in the backward, 128 in the forward), the spans
of the backward (8 splats that reach every sub-block fill its rows), tile
counts around the one from which the backward orders its tiles, and infinite
or NaN values, which must reach only the splats that they belong to."""
import numpy as np
import pytest

import oracle
from helpers import compare_image, fetch, gpu_frame
from paper_2602_03207_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

GRAD_RTOL = 1e-3


def _scene(n, seed, log_scale):
    """n splats in front of a small camera, log-scales around log_scale."""
    s = S.uniform_scene(n, seed=seed, extent=0.6, log_scale_mean=log_scale, log_scale_std=0.3)
    s["opacity_logits"] = np.clip(s["opacity_logits"], -3.0, 3.0)
    return s


def _cam(width, height, f=64.0, bg=(0.2, 0.4, 0.1)):
    view = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, 3]], dtype=np.float32)
    return {"viewmat": view, "fx": f, "fy": f, "cx": width / 2.0, "cy": height / 2.0, "width": width,
            "height": height, "znear": float(np.float32(0.2)), "bg": bg}


def _check(scene, cam, tile, capacity):
    import torch
    from paper_2602_03207_gb300 import render
    g = gpu_frame(scene, cam, tile=tile, key_capacity=capacity)
    ref = oracle.render(scene, cam, tile=tile)
    stats = compare_image(fetch(g), ref)
    assert stats["n_bad"] == 0, stats
    target = np.random.default_rng(5).random((cam["height"], cam["width"], 3)).astype(np.float32)
    dev = render.scene_to_device(scene)
    r = render.Renderer(len(scene["means"]), cam["width"], cam["height"], tile=tile, key_capacity=capacity)
    grads = {k: v.clone() for k, v in r.train_step_l2(dev, cam, torch.as_tensor(target).cuda()).items()}
    r.check_status()
    img = r.forward(dev, cam)
    sep = r.backward(dev, cam, img - torch.as_tensor(target).cuda())
    want = oracle.loss_grad(scene, cam, target, tile=tile)["grads"]
    for k, v in grads.items():
        assert torch.equal(v, sep[k]), k
        a, b = v.cpu().numpy().astype(np.float64).ravel(), want[k].ravel()
        assert np.linalg.norm(a - b) <= GRAD_RTOL * max(np.linalg.norm(b), 1e-12), k


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("n", [1, 8, 9, 32, 33, 64, 65, 96, 97, 128, 129, 193, 300])
def test_list_lengths_around_the_batches(tile, n):
    """Splats of several pixels over one and a half tiles a side: every list
    close to n long, most splats reaching every sub-block."""
    cam = _cam(tile + tile // 2 + 1, tile + 3)
    _check(_scene(n, 10 + n, -1.2), cam, tile, 64 * n + 64)


@pytest.mark.parametrize("tile,width,height", [(8, 256, 255), (8, 259, 253), (16, 509, 515)])
def test_tile_counts_around_the_ordering(tile, width, height):
    """1,024 tiles and a few more or fewer (33 x 32 and 32 x 33 included)."""
    cam = _cam(width, height, f=float(width))
    _check(_scene(800, 3, -3.5), cam, tile, 100_000)


@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("n", [576, 577, 1152, 1153, 2500])
def test_long_lists_walked_in_segments(tile, n):
    """Lists of about n (576 to a segment) with a key capacity from which the
    backward splits them: against the oracle, and against the unsplit walk to
    the rounding of a product and a sum per segment."""
    import torch
    from paper_2602_03207_gb300 import render
    cam = _cam(tile + 5, tile)
    scene = _scene(n, n, -2.2)
    scene["opacity_logits"] -= 3.0  # faint, so that the last of them still show
    _check(scene, cam, tile, 1 << 20)
    dev = render.scene_to_device(scene)
    target = torch.rand(cam["height"], cam["width"], 3, generator=torch.Generator().manual_seed(4)).cuda()
    got = []
    for capacity in (1 << 20, 64 * n):
        r = render.Renderer(n, cam["width"], cam["height"], tile=tile, key_capacity=capacity)
        got.append({k: v.clone() for k, v in r.train_step_l2(dev, cam, target).items()})
    for k in got[0]:
        assert torch.linalg.norm(got[0][k] - got[1][k]) <= 1e-5 * torch.linalg.norm(got[1][k]), k


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite_gradient_stays_with_its_pixel(value):
    """dL/dimage infinite or NaN at one pixel: the splats composited there get
    non-finite gradients, every other splat the bits it gets with a zero
    there. A splat is composited there iff a gradient of one at this pixel
    alone reaches its colour."""
    import torch
    from paper_2602_03207_gb300 import render
    cam = _cam(40, 37)
    scene = render.scene_to_device(_scene(400, 21, -3.0))
    r = render.Renderer(400, 40, 37, key_capacity=20_000)
    r.forward(scene, cam)
    d = torch.randn(37, 40, 3, generator=torch.Generator().manual_seed(1)).cuda()
    d[18, 17] = 0.0
    plain = r.backward(scene, cam, d)
    one = torch.zeros_like(d)
    one[18, 17] = 1.0
    there = r.backward(scene, cam, one)["sh"].abs().sum((1, 2)) > 0
    d[18, 17] = value
    bad = r.backward(scene, cam, d)
    assert there.any() and not there.all()
    for k, v in bad.items():
        assert torch.equal(v[~there], plain[k][~there]), k
    assert not torch.isfinite(bad["sh"][there]).all(dim=(1, 2)).any()


def test_non_finite_colour_stays_with_its_splat():
    """An infinite SH coefficient makes one splat's colour infinite: with a
    finite dL/dimage, the splats that share no pixel with it keep the bits
    they have without it."""
    import torch
    from paper_2602_03207_gb300 import render
    cam = _cam(40, 37)
    scene = render.scene_to_device(_scene(400, 22, -3.0))
    r = render.Renderer(400, 40, 37, key_capacity=20_000)
    r.forward(scene, cam)
    d = torch.randn(37, 40, 3, generator=torch.Generator().manual_seed(2)).cuda()
    plain = r.backward(scene, cam, d)
    g = int((r.tiles_touched[:400] > 0).nonzero()[7])
    # the pixels that splat g composites: where the image changes with its colour
    base = r.forward(scene, cam).clone()
    sh = scene["sh"].clone()
    scene["sh"][g, 0] += 1.0
    touched = (r.forward(scene, cam) != base).any(-1)
    scene["sh"].copy_(sh)
    own = torch.zeros_like(d)
    own[touched] = 1.0
    r.forward(scene, cam)
    shared = r.backward(scene, cam, own)["sh"].abs().sum((1, 2)) > 0
    scene["sh"][g, 0] = float("inf")
    r.forward(scene, cam)
    bad = r.backward(scene, cam, d)
    assert shared[g] and not shared.all()
    for k, v in bad.items():
        assert torch.equal(v[~shared], plain[k][~shared]), k


def _sharing(r, scene, cam, g, bump):
    """Which splats composite a pixel that splat g composites (one where the
    image moves with g's colour): those whose colour a gradient of one at these
    pixels alone reaches. Also those pixels."""
    import torch
    base = r.forward(scene, cam).clone()
    sh = scene["sh"].clone()
    scene["sh"][g, 0] += bump
    pixels = (r.forward(scene, cam) != base).any(-1)
    scene["sh"].copy_(sh)
    r.forward(scene, cam)
    one = torch.zeros_like(base)
    one[pixels] = 1.0
    return r.backward(scene, cam, one)["sh"].abs().sum((1, 2)) > 0, pixels


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("value,scale", [(np.inf, 1.0), (1e30, 1e10)], ids=["infinite", "overflowing"])
@pytest.mark.parametrize("tile,capacity", [(16, 1 << 20), (16, 60_000), (8, 1 << 20), (32, 1 << 20)])
def test_non_finite_colour_stays_with_its_splat_across_segments(tile, capacity, value, scale, masked):
    """The farthest visible splat of a list of more than 1,152 gets an infinite colour,
    or a finite one whose product with dL/dimage overflows, where the list is
    cut into segments and where it is not: the splats in front that share no
    pixel with it keep the bits they have without it."""
    import torch
    from paper_2602_03207_gb300 import render
    side = {8: 8, 16: 16, 32: 24}[tile]
    n = {8: 8000, 16: 5000, 32: 3000}[tile]
    cam = _cam(side, side)
    s = _scene(n, 31, -3.8)
    s["opacity_logits"] = np.random.default_rng(2).uniform(-5.2, -4.4, n).astype(np.float32)
    scene = render.scene_to_device(s)
    r = render.Renderer(n, side, side, tile=tile, key_capacity=capacity)
    r.forward(scene, cam)
    first, last = (int(x) for x in r.ranges[0])
    assert last - first > 1152
    for g in r.sorted_vals[first:last].flip(0).tolist():  # the farthest that covers a pixel centre
        shared, pixels = _sharing(r, scene, cam, g, 1000.0)
        if pixels.any():
            break
    live = r.tiles_touched[:n] > 0
    assert shared[g] and (live & ~shared).sum() > 100
    d = scale * torch.randn(side, side, 3, generator=torch.Generator().manual_seed(3)).cuda()
    if masked:
        d[pixels] = 0.0
    plain = r.backward(scene, cam, d)
    assert all(torch.isfinite(v).all() for v in plain.values())
    scene["sh"][g, 0] = value
    r.forward(scene, cam)
    bad = r.backward(scene, cam, d)
    for k, v in bad.items():
        assert torch.equal(v[~shared], plain[k][~shared]), k


def test_infinite_background_stays_behind_what_is_composited():
    """An infinite background with a finite dL/dimage: colour gradients do not
    depend on it, and splats that composite no pixel keep zero gradients."""
    import torch
    from paper_2602_03207_gb300 import render
    s = _scene(500, 23, -3.0)
    s["opacity_logits"][400:] = -5.52  # an extent of a tenth of a pixel: most cover no pixel centre
    scene = render.scene_to_device(s)
    grads = []
    for bg in ((0.2, 0.4, 0.1), (float("inf"),) * 3):
        cam = _cam(40, 37, bg=bg)
        r = render.Renderer(500, 40, 37, key_capacity=20_000)
        r.forward(scene, cam)
        d = torch.randn(37, 40, 3, generator=torch.Generator().manual_seed(2)).cuda()
        grads.append(r.backward(scene, cam, d))
    plain, bad = grads
    none = (plain["sh"].abs().sum((1, 2)) == 0) & (r.tiles_touched[:500] > 0)
    assert none.sum() > 20
    assert torch.equal(bad["sh"], plain["sh"])
    for k, v in bad.items():
        assert not v[none].any(), k


def _spread(n, dense, width, height, tile):
    """n splats of about two pixels spread over the image but its last tile,
    `dense` more in one tile."""
    rng = np.random.default_rng(n)
    s = _scene(n + dense, 5, -4.2)
    s["opacity_logits"] = rng.uniform(-5.2, -4.0, n + dense).astype(np.float32)
    px, py, z = rng.uniform(0, width, n), rng.uniform(0, height, n), rng.uniform(2.5, 3.5, n + dense)
    last = (px > width - tile - 8) & (py > height - tile - 8)
    py[last] -= tile + 8
    px = np.concatenate([px, rng.uniform(5 * tile + 4, 6 * tile - 4, dense)])
    py = np.concatenate([py, rng.uniform(3 * tile + 4, 4 * tile - 4, dense)])
    s["means"] = np.stack([(px - width / 2) * z / 64, (py - height / 2) * z / 64, z - 3], 1).astype(np.float32)
    return s


def test_segments_longer_than_the_shortest_and_ranges_of_empty_tiles():
    """600 lists of about 670, one of thousands more and none in the last tile:
    segments of more than 576 positions, against the uncut walk; and the same
    bits when the caller's ranges hold (0, 0) for the empty tile, as when they
    hold its place in the list."""
    import torch
    from paper_2602_03207_gb300 import render
    width, height, n, dense, tile = 800, 768, 400_000, 5000, 32
    scene = render.scene_to_device(_spread(n, dense, width, height, tile))
    cam = _cam(width, height)
    d = torch.randn(height, width, 3, generator=torch.Generator().manual_seed(6)).cuda()
    got = []
    for capacity in (1 << 20, (1 << 20) - 4):
        r = render.Renderer(n + dense, width, height, tile=tile, key_capacity=capacity)
        r.forward(scene, cam)
        r.check_status()
        length = r.ranges[:, 1] - r.ranges[:, 0]
        assert int(length[-1]) == 0 and int((length > 576).sum()) > 512 and int(length.max()) > 4000
        got.append(r.backward(scene, cam, d))
        if capacity == 1 << 20:
            r.ranges[length == 0] = 0
            again = r.backward(scene, cam, d)
            assert all(torch.equal(again[k], got[0][k]) for k in again)
    for k in got[0]:
        assert torch.linalg.norm(got[0][k] - got[1][k]) <= 1e-5 * torch.linalg.norm(got[1][k]), k


@pytest.mark.parametrize("tile", [8, 16, 32])
def test_batched_long_lists_walked_in_segments(tile):
    """Uneven views whose lists are cut: the separate calls, the fused step and
    its persistent grid give the same bits, and the sum of the views' uncut
    gradients to rounding."""
    import torch
    from paper_2602_03207_gb300 import batch, render
    n = 6000
    cams = [_cam(40, 24), _cam(24, 41, f=48.0), _cam(33, 17, f=80.0)]
    s = _scene(n, 41, -3.8)
    s["opacity_logits"] = np.random.default_rng(2).uniform(-5.2, -4.4, n).astype(np.float32)
    scene = render.scene_to_device(s)
    target = [torch.rand(c["height"], c["width"], 3, generator=torch.Generator().manual_seed(i)).cuda()
              for i, c in enumerate(cams)]
    grads = []
    for kw in ({}, {"fused": True}, {"fused": True, "persistent": True}):
        b = batch.BatchRenderer(n, cams, tile=tile, key_capacity=3 << 20, **kw)
        grads.append({k: v.clone() for k, v in b.step(scene, b.pack(target)).items()})
        b.check_status()
        assert int((b.ranges[:, 1] - b.ranges[:, 0]).max()) > 1200
    for g in grads[1:]:
        assert all(torch.equal(g[k], grads[0][k]) for k in g)
    want = None
    for c, goal in zip(cams, target):
        r = render.Renderer(n, c["width"], c["height"], tile=tile, key_capacity=1_000_000)
        one = r.train_step_l2(scene, c, goal)
        r.check_status()
        want = {k: v.clone() if want is None else want[k] + v for k, v in one.items()}
    for k in want:
        assert torch.linalg.norm(grads[0][k] - want[k]) <= 1e-5 * torch.linalg.norm(want[k]), k
