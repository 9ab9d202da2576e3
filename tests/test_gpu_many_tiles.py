"""Frames of very many tiles: the list scan with more blocks than the chip holds
at once."""

import numpy as np
import pytest
import torch

import synth
from tests.test_gpu_binning import _expected

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")

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
