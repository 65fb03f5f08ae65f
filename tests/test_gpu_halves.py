"""Compositing with long tiles taken as two halves (16 x 2 layout): a view that mixes whole and halved
tiles against the FP64 oracle and bit for bit against 8-px tiles, and non-finite values, which stay
with the pixels and Gaussians they belong to although a thread's pixels are worked on together."""
import numpy as np
import pytest
import torch

from synth import frustum_scene, random_target

from gpu_helpers import GRAD_FLOOR_DEEP, cuda, new_map, rotated_cam
from test_gpu_fused import _longest_list, check_iteration, iterate_once, oracle_ref

pytestmark = pytest.mark.gpu

W, H = 490, 277       # 31 x 18 = 558 tiles: more than half of the 6 CTAs an SM, so not all are halved


def mixed_scene():
    """1,500 Gaussians over the view and 900 faint ones around one pixel, whose tiles' lists span two
    staging batches; the last tile row and column are cut by the image's edge."""
    a, cam = frustum_scene(n=1500, width=W, height=H, fx=300, fy=300, cx=W / 2, cy=H / 2, seed=5)
    b, _ = frustum_scene(n=900, width=40, height=30, fx=300, fy=300, cx=20 - 30, cy=15 + 20, seed=6,
                         logscale_mean=-3.0, opacity_mean=-3.0)
    return np.concatenate([a, b], axis=1), cam, random_target(W, H, seed=2)


def test_whole_and_halved_tiles_against_the_oracle():
    p, cam, tg = mixed_scene()
    out = iterate_once(p, [cam], tg, tile_size=16, pixels_per_thread=2)
    assert _longest_list(out) > 512
    g, near, excl = oracle_ref(p, [cam], tg)
    check_iteration(out, g, near, excl, p, max_near=1e-2, floor_frac=GRAD_FLOOR_DEEP)
    ref = iterate_once(p, [cam], tg, tile_size=8, pixels_per_thread=1)
    np.testing.assert_array_equal(out["rgb"], ref["rgb"])
    # the separate calls take the same items
    gm = new_map(p.shape[1], W=W, H=H, tile_size=16, pixels_per_thread=2)
    gm.set_params(cuda(p))
    rgb, T, top = gm.render(cam, want_T=True, want_argmax=True)
    gm.loss(cuda(tg))
    gm.backward()
    out["grads"], out["grad2d"] = gm.grads().cpu().numpy(), gm.debug_grad2d()
    check_iteration(out, g, near, excl, p, max_near=1e-2, floor_frac=GRAD_FLOOR_DEEP)
    g8 = new_map(p.shape[1], W=W, H=H, tile_size=8, pixels_per_thread=1)
    g8.set_params(cuda(p))
    for a, b in zip((rgb, T, top), g8.render(cam, want_T=True, want_argmax=True)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("size", [(160, 120), (W, H)])
@pytest.mark.parametrize("cfg", [dict(tile_size=16, pixels_per_thread=1), dict(tile_size=16, pixels_per_thread=2),
                                 dict(tile_size=16, pixels_per_thread=4), dict(tile_size=8, pixels_per_thread=1),
                                 dict(tile_size=8, pixels_per_thread=2), dict(deterministic=1)])
def test_nonfinite_upstream_gradient_stays_with_its_pixel(size, cfg):
    w, h = size
    p, cam = frustum_scene(n=2000, width=w, height=h, fx=150, fy=150, cx=w / 2, cy=h / 2, seed=8)
    gm = new_map(p.shape[1], W=w, H=h, **cfg)
    gm.set_params(cuda(p))
    gm.render(cam)
    up = torch.zeros(1, 3, h, w, device="cuda")
    up[0, :, h // 2, w // 3] = 1.0
    gm.backward(up)
    touched = gm.grads()[11:14] != 0            # the Gaussians that blend in that pixel
    assert 0 < touched[0].sum() < p.shape[1] // 4
    for bad in (float("nan"), float("inf")):
        up[0, :, h // 2, w // 3] = bad
        gm.backward(up)
        assert torch.equal(~torch.isfinite(gm.grads()[11:14]), touched)
        assert not (~torch.isfinite(gm.grads())).any(dim=0)[~touched[0]].any()


@pytest.mark.parametrize("cfg", [dict(tile_size=16, pixels_per_thread=2), dict(tile_size=16, pixels_per_thread=4),
                                 dict(tile_size=8, pixels_per_thread=2)])
def test_nonfinite_colour_stays_with_its_pixels(cfg):
    """A Gaussian with an infinite colour: the loss and gradients of what it does not touch are those
    without it."""
    p, cam = frustum_scene(n=600, seed=9)
    p[10, 0] = -2.0
    small, n = p.copy(), p.shape[1]
    small[11:14, 0] = 0.5
    up = torch.ones(1, 3, 120, 160, device="cuda")
    grads, images = [], []
    for q in (small, p):
        if q is p:
            q[11, 0] = np.inf
        gm = new_map(n, **cfg)
        gm.set_params(cuda(q))
        images.append(gm.render(cam))
        gm.backward(up)
        grads.append(gm.grads())
    hit = ~torch.isfinite(images[1][0, 0])
    assert 0 < hit.sum() < 4000
    assert torch.equal(images[0][0, 0][~hit], images[1][0, 0][~hit])
    finite = torch.isfinite(grads[1]).all(dim=0)
    assert not finite[0] and finite.sum() > n // 4
    torch.testing.assert_close(grads[1][:, finite], grads[0][:, finite], rtol=1e-3, atol=1e-3)


@pytest.mark.parametrize("cfg", [dict(tile_size=16, pixels_per_thread=2), dict(tile_size=16, pixels_per_thread=1),
                                 dict(deterministic=1)])
def test_replays_that_change_their_cameras(cfg):
    """A replayed iteration takes the work list the one before left, or, for other cameras, one of its own:
    each image is that of a render of the same view."""
    p, cam, tg = mixed_scene()
    cams = [cam, rotated_cam(cam, [0.05, -0.04, 0.0], [0.1, 0.0, 0.1]), rotated_cam(cam, [-0.06, 0.05, 0.02], [0.0, 0.1, 0.0])]
    still = dict(lr=(0.0,) * 5, **cfg)
    gm, ref = new_map(p.shape[1], W=W, H=H, **still), new_map(p.shape[1], W=W, H=H, **still)
    for m in (gm, ref):
        m.set_params(cuda(p))
    want = [ref.render(c) for c in cams]
    rgb = torch.empty(1, 3, H, W, device="cuda")
    for v in [0, 0, 0, 1, 2, 2, 1, 0, 1, 1]:
        rgb.fill_(-1.0)
        gm.iterate(cams[v], cuda(tg), rgb_out=rgb)
        assert torch.equal(rgb, want[v]), v
