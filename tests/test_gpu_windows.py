"""Primary-hit features of windows of every shape, and inputs whose indices pass 32 bits."""
import ctypes as C
import dataclasses

import pytest
import torch

pytestmark = pytest.mark.gpu


def _scene():
    from paper_2407_19977_gb300 import api, scenes
    return api.Scene(scenes.cornell_box(seed=1, width=640, height=480, max_depth=2))


@pytest.mark.parametrize("crop", [(0, 0, 640, 480), (3, 5, 1, 470), (3, 5, 600, 1), (10, 20, 9, 211), (10, 20, 95, 5),
                                  (7, 9, 121, 37), (0, 0, 8, 4), (639, 479, 1, 1)])
def test_features_of_a_window_are_those_of_the_frame(crop):
    g = _scene()
    x0, y0, w, h = crop
    full = g.features(2, seed=3)
    assert torch.equal(g.features(2, seed=3, crop=crop), full[y0:y0 + h, x0:x0 + w])


@pytest.mark.parametrize("width,height", [(1, (1 << 29) + 5), ((1 << 30) + 33, 1), (3, 477218600)])
def test_features_of_a_window_of_many_thin_rows(width, height):
    """Windows whose padded tiles, or whose output's floats, outnumber 32 bits."""
    from paper_2407_19977_gb300 import native as N
    from paper_2407_19977_gb300.api import make_camera, _ptr, _stream_handle
    if torch.cuda.mem_get_info()[0] < (width * height * 48) + (8 << 30):
        pytest.skip("needs the output's memory")
    g = _scene()
    cam = dataclasses.replace(g.desc.camera, width=width, height=height)
    out = torch.empty(height * width * 12, dtype=torch.float32, device="cuda")
    out[-12 * 4096:] = -1.0
    out[:12 * 4096] = -1.0
    N.call("pt_render_features", g.h, C.byref(make_camera(cam)), 0, 0, width, height, 0, 1, C.c_uint64(3), _ptr(out),
           _stream_handle())
    k = 512
    crop_w, crop_h = (k, 1) if height == 1 else (width, k)
    first = g.features(1, seed=3, camera=cam, crop=(0, 0, crop_w, crop_h)).reshape(-1)
    last = g.features(1, seed=3, camera=cam, crop=(width - crop_w, height - crop_h, crop_w, crop_h)).reshape(-1)
    assert torch.equal(out[:first.numel()], first)
    assert torch.equal(out[-last.numel():], last)


@pytest.mark.parametrize("where", [200000, -1, (1 << 32) + 7])
def test_texels_past_32_bits_are_checked(where):
    """An environment of more than 2^32 floats with one negative texel is refused wherever it lies."""
    from paper_2407_19977_gb300 import native as N
    from paper_2407_19977_gb300.api import _ptr, _stream_handle
    w, h = 65536, 21846
    if torch.cuda.mem_get_info()[0] < 3 * w * h * 12:
        pytest.skip("needs the environment's memory twice")
    v = torch.tensor([[0, 0, 0], [1, 0, 0], [0, 1, 0]], dtype=torch.float32, device="cuda")
    idx = torch.tensor([0, 1, 2], dtype=torch.int32, device="cuda")
    mid = torch.zeros(1, dtype=torch.int32, device="cuda")
    mats = (N.pt_openpbr * 1)()
    from paper_2407_19977_gb300 import scenes
    mats[0].v[:] = [float(x) for x in scenes.diffuse((.5, .5, .5))]
    env = torch.zeros(w * h * 3, dtype=torch.float32, device="cuda")
    env[where] = -1.0
    out = C.c_void_p()
    with pytest.raises(Exception):
        N.call("pt_scene_create", _ptr(v), 3, _ptr(idx), 1, _ptr(mid), mats, 1, None, 0, _ptr(env), w, h, 1,
               _stream_handle(), C.byref(out))
    assert b"env texel" in N.load().pt_last_error()
