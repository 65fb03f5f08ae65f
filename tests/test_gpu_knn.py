"""The 3 nearest points behind the plain initialisation, at the edges of its chunks and query groups,
against float64: log-scale = ln of the RMS distance (2e-6, the float32 distance's rounding), and the
appending of more points than its CTA takes in one round."""
import numpy as np
import pytest
import torch

from synth import frustum_scene

from gpu_helpers import cuda, new_map

pytestmark = pytest.mark.gpu


def log_scale(pts, ref, own):
    d2 = ((pts[:, None, :].astype(np.float64) - ref[None].astype(np.float64)) ** 2).sum(-1)
    d2 = np.where(np.isfinite(d2), d2, np.inf)
    if own:
        np.fill_diagonal(d2, np.inf)
    d2 = np.sort(d2, axis=1)[:, :3]
    cnt = np.isfinite(d2).sum(1)
    s = np.where(np.isfinite(d2), d2, 0.0).sum(1)
    rms = np.where(cnt > 0, np.sqrt(s / np.maximum(cnt, 1)), 0.01)
    return np.clip(np.log(np.maximum(rms, 1e-30)), -7.0, -1.0)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 33, 257, 1500])
def test_init_map_scales(n):
    pts = np.random.default_rng(n).uniform(-0.05, 0.05, (n, 3)).astype(np.float32)
    if n > 4:
        pts[3] = pts[1]                      # a distance of zero
    gm = new_map(n)
    gm.init_map(cuda(pts), cuda(np.zeros((n, 3))))
    got = gm.params().cpu().numpy()
    np.testing.assert_allclose(got[3], log_scale(pts, pts, True), atol=2e-6, rtol=0)
    np.testing.assert_array_equal(got[0:3], pts.T)


@pytest.mark.parametrize("n_ref,n", [(0, 3), (1, 1), (2, 5), (31, 4), (257, 33), (1025, 100), (70_000, 7), (300, 2500)])
def test_insert_scales_and_order(n_ref, n):
    rng = np.random.default_rng(n_ref + n)
    p, cam = frustum_scene(n=max(n_ref, 1), seed=4)
    p = p[:, :n_ref]
    p[10] = -20.0                            # faint: every point is inserted, by the opacity gate
    if n_ref > 30:
        p[0, 5] = np.nan                     # a mean that is no point's neighbour
    pts = np.stack([rng.uniform(-1, 1, n), rng.uniform(-1, 1, n), rng.uniform(1, 5, n)], 1).astype(np.float32)
    pts[::7, 2] *= -1.0                      # behind the camera: kept by the gate
    gm = new_map(n_ref + n)
    gm.set_params(cuda(p))
    count, mask = gm.insert(cam, torch.zeros(3, 120, 160, device="cuda"), cuda(pts), return_mask=True)
    assert count == n and bool(mask.all()) and gm.n == n_ref + n
    got = gm.params().cpu().numpy()[:, n_ref:]
    np.testing.assert_array_equal(got[0:3], pts.T)
    np.testing.assert_allclose(got[3], log_scale(pts, p[0:3].T, False), atol=2e-6, rtol=0)


@pytest.mark.parametrize("n", [4096, 4097, 9001])
def test_append_in_order(n):
    """Around the number of points from which the appending takes them in several CTAs: part of them
    behind opaque Gaussians, the others appended in order."""
    rng = np.random.default_rng(n)
    p, cam = frustum_scene(n=60, seed=4)
    p[10] = 6.0
    pts = np.stack([rng.uniform(-1, 1, n), rng.uniform(-1, 1, n), rng.uniform(1, 5, n)], 1).astype(np.float32)
    gm = new_map(60 + n)
    gm.set_params(cuda(p))
    count, mask = gm.insert(cam, torch.zeros(3, 120, 160, device="cuda"), cuda(pts), return_mask=True)
    mask = mask.cpu().numpy()
    assert 0 < count == mask.sum() < n and gm.n == 60 + count
    np.testing.assert_array_equal(gm.params().cpu().numpy()[0:3, 60:], pts[mask].T)


def test_a_second_split_uses_the_buffers_of_the_first():
    """Splits swap the parameters between two sets of buffers: three in a row from one map equal the
    same splits of fresh maps."""
    rng = np.random.default_rng(3)
    p, cam = frustum_scene(n=500, seed=2)
    gm = new_map(4000, clarity_sigma=3.0)
    gm.set_params(cuda(p))
    for k in range(3):
        fresh = new_map(4000, clarity_sigma=3.0)
        fresh.set_params(gm.params())
        nz = cuda(rng.normal(size=(gm.n, 2, 3)))
        for m in (gm, fresh):
            m.count_dominant(cam)
        assert gm.densify(nz) == fresh.densify(nz) > 0
        assert torch.equal(gm.params(), fresh.params())


@pytest.mark.parametrize("size", [(160, 120), (490, 277)])
@pytest.mark.parametrize("cfg", [dict(), dict(tile_size=16, pixels_per_thread=1), dict(tile_size=16, pixels_per_thread=4),
                                 dict(tile_size=8, pixels_per_thread=1), dict(deterministic=1), dict(pair_capacity=64)])
def test_gate_is_that_of_the_whole_render(size, cfg):
    """The opacity gate composites only the tiles that hold a point: its decisions are those of the
    transmittance of a whole render, away from pixel borders and the threshold."""
    w, h = size
    p, cam = frustum_scene(n=3000, width=w, height=h, fx=150, fy=150, cx=w / 2, cy=h / 2, seed=3, opacity_mean=2.0)
    n = 700
    rng = np.random.default_rng(5)
    z = rng.uniform(0.5, 4, n)
    px, py = rng.integers(-5, w + 5, n), rng.integers(-5, h + 5, n)
    pts = np.stack([(px + 0.1 - w / 2) * z / 150, (py - 0.1 - h / 2) * z / 150, z], 1).astype(np.float32)
    gm = new_map(3000 + n, W=w, H=h, **cfg)
    gm.set_params(cuda(p))
    T = gm.render(cam, want_T=True)[1][0].cpu().numpy()
    inside = (px >= 0) & (px < w) & (py >= 0) & (py < h)
    opac = np.where(inside, 1.0 - T[np.clip(py, 0, h - 1), np.clip(px, 0, w - 1)], 0.0)
    thresh = 0.9
    gm2 = new_map(3000 + n, W=w, H=h, insert_opacity=thresh, **cfg)
    gm2.set_params(cuda(p))
    count, mask = gm2.insert(cam, torch.zeros(3, h, w, device="cuda"), cuda(pts), return_mask=True)
    sure = np.abs(opac - thresh) > 1e-6
    want = ~(inside & (opac > thresh))
    assert 20 < (~want).sum() and want.sum() > 20
    np.testing.assert_array_equal(mask.cpu().numpy()[sure], want[sure])
    assert count == int(mask.sum())
