"""The blend's culling of list entries by 4x4 blocks must drop no entry that a
pixel composites: the image against a plain float64 evaluation of every record
at every pixel, for round, thin, tiny and huge Gaussians, every tile shape and
ragged images."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

sx = pytest.importorskip("paper_2410_04974_gb300")

EPS = 2.0 ** -24


def _scene(kind, n, seed):
    scene = synth.scene_cube(n, seed)
    rng = np.random.default_rng(seed + 1)
    # alpha_cond stays below exp(4.5) / 255, so that the alpha >= 1/255 ellipse lies within the 3-sigma
    # square and a pixel's entries do not depend on the tile shape
    scene.opacity_logit = np.minimum(rng.normal(-1.5, 1.0, n), -0.65).astype(np.float32)
    if kind == "thin":            # one long axis, two of a pixel or less, tilted by the off-diagonals
        scene.l_raw[:3] = np.log(np.float32(0.004))
        scene.l_raw[0] = np.log(rng.uniform(0.1, 1.5, n)).astype(np.float32)
        scene.l_raw[[6, 7]] = 2.0 * np.arctanh(rng.uniform(-0.7, 0.7, (2, n))).astype(np.float32)
    elif kind == "tiny":
        scene.l_raw[:3] -= 4.0
    elif kind == "huge":
        scene.l_raw[:3] += 3.0
    return scene


@pytest.mark.parametrize("kind", ["round", "thin", "tiny", "huge"])
@pytest.mark.parametrize("tile,size,batch", [((16, 16), (77, 61), 512), ((8, 8), (77, 61), 32), ((32, 16), (130, 35), 64),
                                             ((16, 8), (50, 90), 1024), ((8, 16), (33, 64), 128), ((32, 8), (64, 33), 96)])
def test_blocks_drop_no_composited_entry(kind, tile, size, batch):
    scene = _scene(kind, 400, 11)
    cam = synth.look_at_camera((4.0, 0.3, 0.2), *size)
    r = sx.Renderer(scene.n, scene.sh_degree, [cam], tile=tile, batch=batch)
    img = r.split(r.forward(sx.params_to_device(scene)))[0].double()
    vis = r.ntiles() > 0
    rec = r.records()[vis].double()
    rec = rec[torch.argsort(rec[:, 11], stable=True)]
    y, x = torch.meshgrid(torch.arange(size[1], device="cuda"), torch.arange(size[0], device="cuda"), indexing="ij")
    dx = rec[:, 0, None, None] - (x + 0.5)
    dy = rec[:, 1, None, None] - (y + 0.5)
    qa, qb, qc, lo = (rec[:, i, None, None] for i in (2, 3, 4, 5))
    q = qa * dx * dx + qb * dx * dy + qc * dy * dy + lo
    # a pixel's q in float32: each of its five operations rounds a value of at most S + |lo|, the offsets are
    # rounded once
    err = 8 * EPS * (qa.abs() * dx * dx + qc.abs() * dy * dy + lo.abs())
    border = (q - np.log2(1.0 / 255.0)).abs() <= err
    alpha = torch.where(q >= np.log2(1.0 / 255.0), torch.exp2(q), torch.zeros_like(q))
    after = torch.cumprod(1.0 - alpha, 0)
    border |= (after - 1e-4).abs() <= 1e-4 * (1e-3 + err.sum(0))
    alpha = torch.where(after < 1e-4, torch.zeros_like(alpha), alpha)
    T = torch.cumprod(1.0 - alpha, 0)
    before = torch.cat([torch.ones_like(T[:1]), T[:-1]])
    ref = torch.einsum("nhw,nc->chw", alpha * before, rec[:, 6:9]) + T[-1]
    # alpha is off by ln 2 err (and ex2's two ulp), every product and sum of the chain by half an ulp
    tol = ((0.7 * err + 8 * EPS) * alpha / (1 - alpha)).sum(0) * 2 + 4 * EPS * (1 + (alpha > 0).sum(0))
    bad = ((img - ref).abs() > tol) & ~border.any(0)
    assert float(border.any(0).double().mean()) < 0.2
    assert not bool(bad.any()), (int(bad.sum()), float(((img - ref).abs() - tol).max()))
