"""Frames of many tiles in the fixed workspace of sixdgs_render_fwd_static, which
holds their tile state a band of tiles at a time."""

import ctypes
import os
import struct

import pytest
import torch

import synth

sx = pytest.importorskip("paper_2410_04974_gb300")
from paper_2410_04974_gb300 import _lib, build  # noqa: E402
from paper_2410_04974_gb300.render import camera_array, make_settings  # noqa: E402


def test_the_library_holds_no_more_than_the_stated_array():
    """The device array has a place of the same size among the host library's
    zero-initialised data (.bss)."""
    if not os.path.exists(build.LIB):
        build.build()
    with open(build.LIB, "rb") as f:
        elf = f.read()
    shoff, = struct.unpack_from("<Q", elf, 0x28)
    entsize, count, names = struct.unpack_from("<HHH", elf, 0x3A)
    heads = [struct.unpack_from("<IIQQQQ", elf, shoff + i * entsize) for i in range(count)]
    name0 = heads[names][4]
    bss = sum(h[5] for h in heads if elf[name0 + h[0]:elf.index(b"\0", name0 + h[0])] == b".bss")
    assert _lib.STATIC_WS_BYTES <= bss < _lib.STATIC_WS_BYTES + (1 << 20)


@pytest.mark.gpu
@pytest.mark.parametrize("n,log_scale,sizes,bands,status", [
    (150_000, -4.5, [(8192, 8192)], 5, 0),            # 1.05 million tiles
    (700, -5.0, [(4100, 3000), (2051, 4099), (64, 40), (8000, 6001)], 2, 0),      # bands that cross views
    (12_001, -4.5, [(2000, 1777)] * 10, 2, 0),        # views divided among the projection's CTAs
    (40, -5.5, [(16_000, 13_000)], 6, 0),             # 3.25 million tiles, almost all empty
    (40, 0.0, [(16_000, 13_000)], 6, 1 << _lib.ERR_CAPACITY),
])
@pytest.mark.parametrize("extra", [{}, {"count_pairs": True, "persistent": True, "store_aux": True}], ids=["plain", "extra"])
def test_banded_frames_equal_the_staged_calls(n, log_scale, sizes, bands, status, extra):
    tile = (8, 8)
    scene = synth.scene_cube(n, 3)
    scene.l_raw[:3] += log_scale                      # a few tiles a Gaussian: the call plans 4 a pair and 4,096
    scene.l_raw[6:] = 0.0
    scene.opacity_logit += 3.0
    cams = [synth.look_at_camera((4.0, 0.3 * k, 0.2), *s) for k, s in enumerate(sizes)]
    settings = make_settings(tile=tile, **extra)
    params = sx.params_to_device(scene)
    r = sx.Renderer(scene.n, scene.sh_degree, cams, tile=tile, inference=True)
    ref = r.forward(params, check=False)
    torch.cuda.synchronize()
    assert int(r.status.item()) == status and r.counts()[1] >= n // 4
    assert 56 * int(r.plan.total_tiles) > (bands - 1) * (_lib.STATIC_WS_BYTES - 144 * int(r.plan.n_pairs))
    images = torch.empty_like(ref)
    word = torch.zeros(1, dtype=torch.int32, device="cuda")
    sc = _lib.Scene()
    sc.n, sc.sh_degree = scene.n, scene.sh_degree
    for k in sx.PARAM_NAMES:
        setattr(sc, k, params[k].data_ptr())
    for again in range(2):
        images.fill_(-1.0)
        code = _lib.load().sixdgs_render_fwd_static(
            scene.n, scene.sh_degree, ctypes.byref(sc), camera_array(cams), len(cams), ctypes.byref(settings),
            ctypes.c_void_p(images.data_ptr()), ctypes.c_void_p(word.data_ptr()),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        assert code == _lib.OK
        assert int(word.item()) == status
        word.zero_()
        if status == 0:      # (a cut list holds whichever entries came first)
            assert torch.equal(images, ref)
