"""The projection's forms and the counting of large rectangles: the lists of a
frame against a NumPy sort of its rectangles, its records against those of the
views one by one, and the division of the work that leads to each form."""

import numpy as np
import pytest
import torch

import synth
from tests.test_bin_rules import rules  # noqa: F401
from tests.test_gpu_binning import _expected

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")

BIG_RECT, BIG_LIST, FILL, WIDE = 16, 128, 608, 8   # bin.cuh, project.cu
STAGE = 128                                        # Gaussians of a CTA


def _lists(r):
    pairs, tiles, ranges = _expected(r)
    assert r.counts()[1] == pairs.size and int(r.status.item()) == 0
    np.testing.assert_array_equal(r.ranges().cpu().numpy(), ranges)
    np.testing.assert_array_equal(r.sorted_pairs().cpu().numpy(), pairs)


def _cams(views, size):
    return [synth.look_at_camera((4.0 * np.cos(k), 4.0 * np.sin(k), 0.3), *size) for k in range(views)]


@pytest.mark.parametrize("n,views,threads", [(39_001, 3, 128), (38_916, 9, 256)])
def test_more_large_rectangles_than_a_cta_lists(rules, n, views, threads):  # noqa: F811
    """Where the count is not left to a kernel of its own."""
    scene = synth.scene_cube(n, 5, sh_degree=1)
    scene.l_raw[:3] += np.log(2.0)
    scene.l_raw[:3, ::4] -= np.log(20.0)          # small ones among them
    r = sx.Renderer(n, 1, _cams(views, (400, 272)), tile=(8, 8), lambda_opa=0.0, dup_capacity=32 << 20, inference=True)
    (parts, per_cta, segments, *_), = rules([(n, views, int(r.plan.total_tiles), 152)])
    assert parts == 1 and segments >= FILL // 2 and (per_cta >= WIDE) == (threads == 256)
    r.condition_project(sx.params_to_device(scene))
    r.bin_sort()
    nt = r.ntiles().cpu().numpy().reshape(views, n)
    big = [int((nt[:, g:g + STAGE] > BIG_RECT).sum()) for g in range(0, n, STAGE)]
    assert max(big) > BIG_LIST and bool(((nt > 0) & (nt <= BIG_RECT)).any())
    _lists(r)


@pytest.mark.parametrize("n,views,split", [(6_700, 5, 3), (3_001, 20, 2)])
def test_large_rectangles_left_to_their_own_kernel_by_views_divided_among_ctas(rules, n, views, split):  # noqa: F811
    scene = synth.scene_cube(n, 5, sh_degree=0)
    r = sx.Renderer(n, 0, _cams(views, (640, 424)), tile=(8, 16), dup_capacity=32 << 20, inference=True)
    tiles = int(r.plan.total_tiles)
    (parts, per_cta, segments, *_), = rules([(n, views, tiles, 152)])
    assert parts > 1 and per_cta == split and segments < FILL // 2 and tiles > 1024 * views
    r.condition_project(sx.params_to_device(scene))
    r.bin_sort()
    nt = r.ntiles().cpu().numpy()
    assert bool((nt > BIG_RECT).any()) and bool(((nt > 0) & (nt <= BIG_RECT)).any())
    _lists(r)


@pytest.mark.parametrize("n", [40_004, 40_001])           # bulk copies of the planes, plain loads
@pytest.mark.parametrize("learn", [False, True])
def test_staged_projection_with_256_threads_cached_and_not(rules, n, learn):  # noqa: F811
    """A CTA with 8 views or more: two threads a Gaussian share its state."""
    views, degree = 17, 2
    scene = synth.scene_cube(n, 5, sh_degree=degree)
    scene.l_raw[:3] -= np.log(4.0)
    if learn:
        scene = synth.with_learnable_lambda(scene, 10)
    cams = _cams(views, (72, 40))
    params = sx.params_to_device(scene)
    (parts, per_cta, *_), = rules([(n, views, 15 * views, 152)])
    assert parts == 1 and per_cta >= WIDE
    frames = []
    for p in (params, dict(params, cond_cache=sx.condition_cache(params))):
        r = sx.Renderer(n, degree, cams, inference=True)
        img = r.forward(p)
        _lists(r)
        frames.append((r.ntiles().clone(), r.records().clone(), img))
    seen = frames[0][0] > 0
    assert torch.equal(frames[0][0], frames[1][0]) and torch.equal(frames[0][1][seen], frames[1][1][seen])
    assert torch.equal(frames[0][2], frames[1][2])
    # the views one by one: the single-view form of the projection, whose compiler may contract a product and a sum
    # otherwise, so a rectangle edge or a visibility can differ, and a record by its rounding
    nt, rec, _ = frames[0]
    nt, rec = nt.view(views, n), rec.view(views, n, 12)
    for v in (0, 7, 16):
        one = sx.Renderer(n, degree, [cams[v]], inference=True)
        one.condition_project(params)
        nt1, rec1 = one.ntiles(), one.records()
        assert int(((nt[v] > 0) != (nt1 > 0)).sum()) <= 4 and int((nt[v] != nt1).sum()) <= 16
        both = (nt[v] > 0) & (nt1 > 0)
        a, b = rec[v][both].double(), rec1[both].double()
        scale = b.abs().mean(0, keepdim=True) + b.abs()
        assert float(((a - b).abs() / scale).max()) <= 1e-3 and int(both.sum()) > 1000
