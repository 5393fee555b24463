"""Host logic of the Python binding (no GPU): tile grids, the sort's bit
range and the configuration flags."""
import pytest

from paper_2602_03207_gb300 import capi, render


def test_tile_grid_and_key_bits():
    assert render.tile_grid(1920, 1080, 16) == (120, 68)
    assert render.tile_grid(3840, 2160, 16) == (240, 135)
    assert render.tile_grid(1, 1, 16) == (1, 1)
    # keys are (tile << 31) | depth bits: 13 tile bits at 1080p, 15 at 2160p
    assert render.key_end_bit(1920, 1080, 16) == 31 + 13
    assert render.key_end_bit(3840, 2160, 16) == 31 + 15
    assert render.key_end_bit(16, 16, 16) == 31  # one tile: the depth bits alone
    assert render.key_end_bit(32, 16, 16) == 32
    # every tile id fits below the end bit
    for w, h, t in ((1920, 1080, 8), (1280, 720, 32), (257, 255, 16)):
        tx, ty = render.tile_grid(w, h, t)
        assert tx * ty - 1 < 1 << (render.key_end_bit(w, h, t) - 31)


def test_config_flags():
    assert render.config_flags(0, "segmented") == capi.WS_CFG_SORT_SEGMENTED
    assert render.config_flags(0, "lsd") == 0
    assert render.config_flags(0, "lookback") == capi.WS_CFG_SORT_LOOKBACK
    assert render.config_flags(capi.WS_CFG_FIXED_RADIUS, "lsd") == capi.WS_CFG_FIXED_RADIUS
    with pytest.raises(ValueError):
        render.config_flags(0, "bitonic")


def _camera(width, height):
    from paper_2602_03207_gb300 import synthetic as S
    return dict(S.small_forward()[1], width=width, height=height)


@pytest.mark.parametrize("width,height", [(65, 48), (64, 49), (640, 480), (16, 1000)])
def test_cameras_that_do_not_fit_are_refused(width, height):
    """The calls size the image and the tile grid by the camera: one larger
    than the renderer is refused before anything is launched."""
    import torch
    r = render.Renderer(10, 64, 48, device="cpu")
    cam, image = _camera(width, height), torch.zeros(height, width, 3)
    calls = [lambda: r.train_step_l2({}, cam, image), lambda: r.train_pass_l2({}, cam, image),
             lambda: r.backward({}, cam, image), lambda: r.forward_quads({}, cam), lambda: r.forward({}, cam),
             lambda: r.rasterize(capi.camera(cam)), lambda: r.cull_sort(capi.camera(cam))]
    for call in calls:
        with pytest.raises(ValueError, match="camera resolution"):
            call()


def test_camera_of_another_frame_is_refused():
    """A backward by another grid than the pairs were binned for."""
    import torch
    r = render.Renderer(10, 64, 48, device="cpu")
    r._frame = (64, 48)
    cam, image = _camera(48, 48), torch.zeros(48, 48, 3)
    for call in (lambda: r.backward({}, cam, image), lambda: r.train_pass_l2({}, cam, image)):
        with pytest.raises(ValueError, match="camera resolution"):
            call()


@pytest.mark.parametrize("shape,dtype", [((48, 64), "float32"), ((47, 64, 3), "float32"), ((48, 64, 3), "float16"),
                                         ((48, 64, 3), "float64")])
def test_images_of_another_size_or_type_are_refused(shape, dtype):
    import torch
    r = render.Renderer(10, 64, 48, device="cpu")
    cam, image = _camera(64, 48), torch.zeros(shape, dtype=getattr(torch, dtype))
    for call in (lambda: r.train_step_l2({}, cam, image), lambda: r.train_pass_l2({}, cam, image),
                 lambda: r.backward({}, cam, image)):
        with pytest.raises(ValueError, match="must be float32"):
            call()
