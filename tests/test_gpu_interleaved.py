"""Frames beside one another: two renderers in turn on one stream, each on a
stream of its own, and an eager frame between the replays of a captured one,
with other kernels in between, against the same frames alone.  Outside capture
a frame's kernels are set up while their predecessor, whosever it is, ends."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")


def _frame(n, views, size, seed):
    scene = synth.scene_shell(n, seed, dp_sigma=0.1)
    scene.l_raw[:3] += np.log(3.0)
    cams = synth.hemisphere_cameras(views, [size] * views)
    r = sx.Renderer(scene.n, scene.sh_degree, cams)
    params = sx.params_to_device(scene)
    img = r.forward(params)
    target = torch.rand(img.shape, generator=torch.Generator().manual_seed(seed)).cuda()
    f = {"r": r, "params": params, "target": target, "img": torch.empty_like(img), "grads": r.new_grads(params)}
    _step(f)
    torch.cuda.synchronize()
    f["want"] = (f["img"].clone(), {k: g.clone() for k, g in f["grads"].items()}, float(r.loss.item()))
    return f


def _step(f, stream=None):
    f["r"].step(f["params"], f["img"], f["target"], None, f["grads"], stream)


def _check(f):
    img, grads, loss = f["want"]
    assert torch.equal(f["img"], img) and int(f["r"].status.item()) == 0
    assert abs(float(f["r"].loss.item()) - loss) <= 1e-9 * abs(loss)
    for k, g in grads.items():     # sums of atomic additions, in another order
        assert float((f["grads"][k] - g).norm()) <= 1e-5 * float(g.norm()), k
    f["img"].fill_(-1.0)
    for g in f["grads"].values():
        g.fill_(-1.0)


def test_two_renderers_in_turn_on_one_stream_with_kernels_between():
    a, b = _frame(20_000, 2, (200, 136), 1), _frame(3_001, 5, (97, 65), 2)
    for _ in range(4):
        for f in (a, b):
            for g in f["grads"].values():
                g.fill_(7.0)        # read by nothing, overwritten by the frame that follows
            _step(f)
        scaled = a["img"] * 2.0     # reads the frame before the one before
        torch.cuda.synchronize()
        assert torch.equal(scaled, a["want"][0] * 2.0)
        _check(a)
        _check(b)


def test_two_renderers_on_two_streams():
    a, b = _frame(20_000, 2, (200, 136), 1), _frame(60_000, 4, (160, 120), 2)
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(6):
        for _ in range(3):
            _step(a, sa)
            _step(b, sb)
        torch.cuda.synchronize()
        _check(a)
        _check(b)


def test_eager_frames_between_the_replays_of_a_captured_one():
    a, b = _frame(20_000, 2, (200, 136), 1), _frame(3_001, 5, (97, 65), 2)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        _step(a)
    for _ in range(4):
        graph.replay()
        _step(b)
        graph.replay()
        torch.cuda.synchronize()
        _check(a)
        _check(b)
