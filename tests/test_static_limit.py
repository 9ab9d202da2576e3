"""Which frames sixdgs_render_fwd_static takes, at the edges of its limit.

Runs where no GPU is visible: a frame within the limit then stops at the device
lookup (ERR_CUDA), one beyond it is refused (ERR_WORKSPACE), and neither
launches anything."""

import ctypes

import pytest
import torch

import synth

sx = pytest.importorskip("paper_2410_04974_gb300")
from paper_2410_04974_gb300 import _lib  # noqa: E402
from paper_2410_04974_gb300.render import camera_array, make_settings  # noqa: E402


@pytest.mark.skipif(torch.cuda.is_available(), reason="a frame within the limit would be rendered")
@pytest.mark.parametrize("n,views,w,h,tile,taken", [
    (225_925, 1, 800, 800, (16, 16), True),
    (225_926, 1, 800, 800, (16, 16), False),
    (56_504, 4, 256, 256, (16, 16), True),
    (56_505, 4, 256, 256, (16, 16), False),
    (1_000, 1, 16_000, 16_384, (8, 8), True),       # 4.1 million tiles
    (8, 1, 16_384, 16_384, (8, 8), False),          # 4.2 million
])
def test_frames_at_the_edges_of_the_limit(n, views, w, h, tile, taken):
    lib = _lib.load()
    settings = make_settings(tile=tile)
    scene = _lib.Scene()
    scene.n, scene.sh_degree = n, 3
    for k in sx.PARAM_NAMES:
        setattr(scene, k, 256)                      # never read
    cams = camera_array([synth.look_at_camera((4.0, 0.0, 0.0), w, h)] * views)
    code = lib.sixdgs_render_fwd_static(n, 3, ctypes.byref(scene), cams, views, ctypes.byref(settings),
                                        ctypes.c_void_p(256), ctypes.c_void_p(256), ctypes.c_void_p(0))
    assert code == (_lib.ERR_CUDA if taken else _lib.ERR_WORKSPACE)
