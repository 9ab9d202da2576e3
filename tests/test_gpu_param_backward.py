"""The per-Gaussian backward over many cameras in one frame (view masks of
several words, CTAs whose Gaussians have very different numbers of views, a
ragged last CTA, planes that cannot be copied in bulk) against the same views
one frame each, accumulated."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")


@pytest.mark.parametrize("n,views,degree,learn", [
    (1, 2, 3, False), (129, 33, 0, True), (257, 64, 2, False), (1000, 40, 3, True), (4099, 5, 1, False), (300, 256, 3, False)])
def test_many_views_equal_the_views_one_by_one(n, views, degree, learn):
    scene = synth.scene_cube(n, 9, sh_degree=degree)
    if learn:
        scene = synth.with_learnable_lambda(scene, 10)
    rng = np.random.default_rng(4)
    scene.opacity_logit = rng.normal(0.0, 3.0, n).astype(np.float32)   # seen by all views, by some, by none
    sizes = [((33, 17), (16, 40))[k % 2] for k in range(views)]
    cams = synth.hemisphere_cameras(views, sizes)
    params = sx.params_to_device(scene)
    dimg = [torch.as_tensor(g).cuda() for g in synth.random_grad_images(cams, 5)]
    r = sx.Renderer(n, degree, cams)
    grads = r.backward(params, r.forward(params), r.pack(dimg))
    total = r.new_grads(params)
    for t in total.values():
        t.zero_()
    for cam, g in zip(cams, dimg):
        one = sx.Renderer(n, degree, [cam])
        one.backward(params, one.forward(params), one.pack([g]), grads=total, accumulate=True)
    torch.cuda.synchronize()
    assert int(r.status.item()) == 0
    assert set(grads) == set(total) and ("lambda_raw" in grads) == learn
    for k in grads:
        # a Gaussian's gradient is a sum of at most `views` terms, in the same order on both sides but for the
        # pixel sums' atomics: float32 rounding of sums of that length (and of the terms' own cancellation)
        scale = float(total[k].norm()) + 1e-30
        assert float((grads[k] - total[k]).norm()) <= 1e-5 * scale, k
