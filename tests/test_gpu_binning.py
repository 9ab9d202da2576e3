"""The per-tile lists against a NumPy sort of the same frame's rectangles and
depths, at the sizes where the binning takes another path: lists of one entry,
at the limits of the sorting teams (64 to 4,096 entries), above them (runs
merged by one CTA, then by a cluster of them), rectangles of one tile and of hundreds, and
equal depths (a few, and whole lists of them)."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")
from paper_2410_04974_gb300 import _lib  # noqa: E402


def _expected(r):
    """(sorted pairs, their tiles, ranges) from the workspace's rectangles."""
    n = r.n
    nt = r.ntiles().cpu().numpy()
    vis = np.flatnonzero(nt)
    rect = r.rects().cpu().numpy().view(np.uint16)[vis].astype(np.int64)
    depth = r._section(_lib.WS_DEPTHKEY, torch.int32, int(r.plan.n_pairs)).cpu().numpy().view(np.uint32)[vis]
    view = vis // n
    tx = np.array([-(-w // r.settings.tile_w) for (_, w) in r.sizes])[view]
    off = np.array(r.tile_offsets())[view]
    w = rect[:, 1] - rect[:, 0]
    assert np.array_equal(w * (rect[:, 3] - rect[:, 2]), nt[vis])
    rep = np.repeat(np.arange(vis.size), nt[vis])
    local = np.arange(rep.size) - np.repeat(np.cumsum(nt[vis]) - nt[vis], nt[vis])
    tile = off[rep] + (rect[rep, 2] + local // w[rep]) * tx[rep] + rect[rep, 0] + local % w[rep]
    order = np.lexsort((vis[rep], depth[rep], tile))
    tiles = tile[order]
    total = int(r.plan.total_tiles)
    start = np.searchsorted(tiles, np.arange(total), "left")
    end = np.searchsorted(tiles, np.arange(total), "right")
    ranges = np.where((end > start)[:, None], np.stack([start, end], 1), 0)
    return vis[rep][order], tiles, ranges


@pytest.mark.parametrize("kind,n,views,size,spread", [
    ("cube", 1, 1, (64, 64), 1.0),
    ("cube", 127, 2, (33, 17), 1.0),
    ("cube", 3001, 9, (97, 65), 1.0),         # 9 views: the 48-camera set-up launch, three short segments each
    ("cube", 1500, 7, (97, 65), 1.0),         # views divided among CTAs: 3, 3 and 1
    ("cube", 3000, 1, (1920, 1080), 1.0),     # rectangles of dozens of tiles
    ("shell", 30_000, 1, (128, 128), 1.0),    # lists of several hundred
    ("shell", 9_000, 2, (48, 32), 1.0),       # lists of one to four thousand
    ("shell", 60_000, 1, (24, 24), 1.0),      # lists of 1,632, 6,500, 6,525 and 19,122
    ("shell", 300_000, 1, (24, 24), 1.0),     # of 7,944 to 95,749: merged by a CTA, by a cluster
    ("cube", 20_000, 1, (64, 64), 0.0),       # every depth equal: lists sorted by id alone
    ("cube", 20_000, 1, (64, 64), 1e-6),      # a handful of depths
])
def test_lists_equal_a_numpy_sort(kind, n, views, size, spread):
    scene = synth.scene_cube(n, 5) if kind == "cube" else synth.scene_shell(n, 5, dp_sigma=0.1)
    if spread < 1.0:
        # no position-direction coupling: the depth is that of mu_p, on a plane facing the camera
        scene.l_raw[[9, 10, 11, 12, 13, 14, 16, 17, 18]] = 0.0
        scene.mu_p[0] *= spread
    cams = [synth.look_at_camera((4.0 * np.cos(k), 4.0 * np.sin(k), 0.0), *size) for k in range(views)]
    r = sx.Renderer(scene.n, scene.sh_degree, cams)
    params = sx.params_to_device(scene)
    r.forward(params)
    for again in range(2):                      # the binning may be run again on the same projection
        pairs, tiles, ranges = _expected(r)
        counts = r.counts()
        assert counts[0] == int((r.ntiles() > 0).sum()) and counts[1] == pairs.size
        np.testing.assert_array_equal(r.ranges().cpu().numpy(), ranges)
        np.testing.assert_array_equal(r.sorted_pairs().cpu().numpy(), pairs)
        key = r._section(_lib.WS_SORTEDKEY, torch.int32, int(counts[1]))
        np.testing.assert_array_equal(key.cpu().numpy(), tiles)
        if kind == "shell" and size == (24, 24):
            length = ranges[:, 1] - ranges[:, 0]
            assert length.max() > 16384 and ((length > 4096) & (length <= 16384)).any()
        r.bin_sort()
        torch.cuda.synchronize()
    assert int(r.status.item()) == 0
