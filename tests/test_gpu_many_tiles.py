"""Frames of very many tiles or duplicates: the list scan with more blocks than the chip holds
at once."""

import numpy as np
import pytest
import torch

import synth
from tests.test_gpu_binning import _expected

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")
from paper_2410_04974_gb300 import _lib  # noqa: E402

SCAN_TILE = 256   # tiles of a block of the list scan


def test_lists_of_a_scan_of_more_blocks_than_are_resident():
    w, h = 4608, 6144
    props = torch.cuda.get_device_properties(0)
    blocks = (w // 8) * (h // 8) / SCAN_TILE
    assert blocks > props.multi_processor_count * (2048 // SCAN_TILE)
    scene = synth.scene_cube(900, 5)
    r = sx.Renderer(scene.n, scene.sh_degree, [synth.look_at_camera((4.0, 0.3, 0.2), w, h)], tile=(8, 8),
                    dup_capacity=8 << 20)
    r.condition_project(sx.params_to_device(scene))
    for again in range(3):
        r.bin_sort()
        torch.cuda.synchronize()
        assert int(r.status.item()) == 0
        pairs, tiles, ranges = _expected(r)
        assert r.counts()[1] == pairs.size > 100_000 and len(np.unique(tiles)) > 100_000
        np.testing.assert_array_equal(r.ranges().cpu().numpy(), ranges)
        np.testing.assert_array_equal(r.sorted_pairs().cpu().numpy(), pairs)


def test_more_duplicates_in_one_scan_block_than_32_bits_count():
    """17 million Gaussians on each of 256 tiles: the total is beyond the
    capacity, and has to be reported as such."""
    n = 17_000_000
    one = synth.scene_cube(1, 5, sh_degree=0)
    one.mu_p[:] = 0.0
    one.l_raw[:3] += np.log(40.0)             # covers the image
    one.opacity_logit[:] = 3.0
    params = {k: t.expand(*t.shape[:-1], n).contiguous() for k, t in sx.params_to_device(one).items()}
    r = sx.Renderer(n, 0, [synth.look_at_camera((4.0, 0.0, 0.0), 128, 128)], tile=(8, 8), lambda_opa=0.0,
                    dup_capacity=80_000_000, inference=True)
    r.condition_project(params)
    assert int(r.ntiles().min().item()) == SCAN_TILE
    r.bin_sort()
    torch.cuda.synchronize()
    assert int(r.status.item()) == 1 << _lib.ERR_CAPACITY
    assert r.counts()[1] & 0xffffffff == 0xffffffff            # n * 256, saturated
    ranges = r.ranges().cpu().numpy()
    assert ranges.min() >= 0 and ranges.max() == 80_000_000
