"""The blend's kernels for frames of few Gaussians over many tiles (lists of at
most 32 entries staged by every warp for itself, twin blocks walked together)
against its kernels for any other frame: the same visible Gaussians with and
without enough invisible ones beside them to change the kernels.  Images bit for
bit, gradients up to the order of their sums."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")

SPARSE_PAIRS = 8      # raster.cu: fewer pairs than this a tile


def _scenes(n, n_more, log_scale):
    few, more = synth.scene_cube(n, 5, sh_degree=1), synth.scene_cube(n_more, 6, sh_degree=1)
    few.l_raw[:3] += log_scale
    more.opacity_logit[:] = -40.0
    for name, plane in few.planes().items():
        more.planes()[name][..., :n] = plane
    return few, more


@pytest.mark.parametrize("n,log_scale", [(420, 0.6), (12, 2.0), (250, 3.0)], ids=["mixed", "few", "huge"])
@pytest.mark.parametrize("tile,size,batch", [((16, 16), (211, 133), 512), ((8, 8), (130, 67), 512), ((8, 8), (130, 67), 64),
                                             ((32, 16), (330, 200), 512), ((16, 16), (211, 133), 32),
                                             ((8, 16), (97, 131), 96), ((32, 8), (200, 90), 1024)])
@pytest.mark.parametrize("store_aux", [False, True])
def test_sparse_and_dense_kernels_agree(n, log_scale, tile, size, batch, store_aux):
    tiles = -(-size[0] // tile[0]) * -(-size[1] // tile[1])
    n = min(n, SPARSE_PAIRS * tiles - 1)
    cams = [synth.look_at_camera((4.0, 0.3, 0.2), *size)]
    out = []
    for scene in _scenes(n, SPARSE_PAIRS * tiles + 130, log_scale):
        assert (scene.n // SPARSE_PAIRS < tiles) == (scene.n == n)
        r = sx.Renderer(scene.n, 1, cams, tile=tile, batch=batch, store_aux=store_aux, dup_capacity=1 << 20, lambda_opa=0.1)
        params = sx.params_to_device(scene)
        img = r.forward(params)
        gen = torch.Generator().manual_seed(3)
        target, dimg = torch.rand(img.shape, generator=gen).cuda(), torch.randn(img.shape, generator=gen).cuda()
        own = r.backward(params, img, dimg)                     # blend_bwd after raster_fwd
        fused, grads = torch.empty_like(img), r.new_grads(params)
        r.step(params, fused, target, None, grads)              # the fused kernel
        torch.cuda.synchronize()
        assert int(r.status.item()) == 0 and torch.equal(fused, img)
        length = (r.ranges()[:, 1] - r.ranges()[:, 0]).cpu().numpy()
        out.append((img, float(r.loss.item()), {k: g[..., :n] for k, g in own.items()},
                    {k: g[..., :n] for k, g in grads.items()}, length))
    (img, loss, own, fused, length), (img_d, loss_d, own_d, fused_d, length_d) = out
    assert np.array_equal(length, length_d) and (length.max() > 32 if log_scale != 2.0 else 0 < length.max() <= 12)
    assert torch.equal(img, img_d) and abs(loss - loss_d) <= 1e-12 * loss_d + 1e-15
    for got, want in ((own, own_d), (fused, fused_d)):
        for k in got:
            # a parameter's gradient: float32 sums over the pixels of its tiles, in another order
            assert float((got[k] - want[k]).norm()) <= 1e-5 * float(want[k].norm()) + 1e-12, k
