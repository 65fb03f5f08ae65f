"""Views whose tiles' lists are all about as long (random Gaussians over the whole view), at tile counts
around the number of CTAs that run at a time, where the work list goes as whole tiles with a last part of
halves, or all whole: every tile once, the image bit for bit that of one pixel a thread (no halves), and the
gradients within the rounding of the sums' order."""
import numpy as np
import pytest
import torch

from synth import frustum_scene, random_target

from gpu_helpers import cuda, new_map, rotated_cam

pytestmark = pytest.mark.gpu


def sizes():
    """(width, height, views): tiles of 16 px just below, at and above one wave of 6 CTAs an SM (152 SMs),
    with a short and a long last part of a wave, and just past three waves."""
    return [(16 * 38, 16 * 24 - 16, 1), (16 * 38, 16 * 24, 1), (16 * 38 + 1, 16 * 24, 1), (333, 251, 3),
            (640, 480, 1), (800, 600, 1), (640, 480, 2), (16 * 38, 16 * 24, 3), (16 * 38, 16 * 24 + 1, 3)]


@pytest.mark.parametrize("width,height,views", sizes())
def test_even_lists(width, height, views):
    n = 40_000
    p, cam = frustum_scene(n=n, width=width, height=height, fx=width * 0.9, fy=width * 0.9, cx=width / 2,
                           cy=height / 2, seed=1, logscale_mean=-4.5)
    cams, tg = [cam] * views, cuda(random_target(width, height, seed=2, n_views=views))
    outs = []
    for ppt in (2, 1):
        gm = new_map(n, views=views, W=width, H=height, tile_size=16, pixels_per_thread=ppt)
        gm.set_params(cuda(p))
        shots = [gm.render(cams, want_T=True, want_argmax=True)]
        bins, _ = gm.debug_pairs()
        gm.loss(tg)
        gm.backward()
        grads = [gm.grads()]
        for _ in range(2):                     # a direct iteration and a replay, from the same map
            rgb = torch.full((views, 3, height, width), float("nan"), device="cuda")
            gm.set_params(cuda(p))
            for _ in range(2):
                rgb.fill_(float("nan"))
                gm.iterate(cams, tg, rgb_out=rgb)
            shots.append((rgb,))
            grads.append(gm.grads())
        outs.append((shots, grads))
        gm.close()
    tiles = views * ((width + 15) // 16) * ((height + 15) // 16)
    assert 4 * np.bincount(bins, minlength=tiles).max() * tiles <= 7 * len(bins)
    assert torch.equal(outs[0][0][0][0], outs[1][0][0][0])
    for a, b in zip(outs[0][0][0], outs[1][0][0]):
        assert torch.equal(a, b)
    for a, b in zip(outs[0][0][1:], outs[1][0][1:]):
        assert torch.isfinite(a[0]).all() and torch.isfinite(b[0]).all()
    for a, b in zip(outs[0][1][:1], outs[1][1][:1]):
        # float32 sums of up to a few thousand pixel terms a Gaussian in another order
        assert float((a - b).norm()) <= 1e-5 * float(b.norm())


def test_replays_of_other_cameras():
    """A replay of other cameras writes the list of its own ranges (in another kernel, by 256 threads)."""
    n, width, height = 40_000, 640, 480
    p, cam = frustum_scene(n=n, width=width, height=height, fx=width * 0.9, fy=width * 0.9, cx=width / 2,
                           cy=height / 2, seed=1, logscale_mean=-4.5)
    cams = [cam, rotated_cam(cam, [0.01, -0.01, 0.02], [0.02, 0.0, 0.0]), rotated_cam(cam, [0, 0.01, 0], [0, 0, 0.1])]
    tg = cuda(random_target(width, height, seed=2))
    gm = new_map(n, W=width, H=height, tile_size=16, pixels_per_thread=2, lr=(0.0,) * 5)
    ref = new_map(n, W=width, H=height, tile_size=16, pixels_per_thread=1)
    for m in (gm, ref):
        m.set_params(cuda(p))
    rgb = torch.empty(1, 3, height, width, device="cuda")
    for k in (0, 0, 1, 2, 2, 0, 1):
        rgb.fill_(float("nan"))
        gm.iterate(cams[k], tg, rgb_out=rgb)
        assert torch.equal(rgb, ref.render(cams[k])), k
    assert torch.equal(gm.params(), cuda(p))
