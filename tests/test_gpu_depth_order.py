"""The (view, tile, depth, id) order of the pairs at the sizes where the sort changes its way: the
one-CTA depth sort's last size and the first beyond it, more blocks than a scatter or the emission
adds up itself,
several views, depths over a 32-bit range of keys, all depths equal, and nothing visible."""
import numpy as np
import pytest

from synth import frustum_scene

from gpu_helpers import cuda, new_map, rotated_cam

pytestmark = pytest.mark.gpu


def check_order(gm, cams, n):
    bins, vals = gm.debug_pairs()
    proj = [gm.debug_projection(v) for v in range(len(cams))]
    tiles = np.concatenate([p[7] for p in proj]).astype(np.int64)
    depth = np.concatenate([p[5] for p in proj])
    assert len(bins) == tiles.sum()
    np.testing.assert_array_equal(np.bincount(vals, minlength=len(tiles)), tiles)   # each item, once a tile
    key = bins.astype(np.int64) * len(tiles) + vals
    assert len(np.unique(key)) == len(key)
    d, v = depth[vals], vals.astype(np.int64)
    same = bins[1:] == bins[:-1]
    assert np.all(bins[1:] >= bins[:-1])
    assert np.all((d[1:] > d[:-1])[same] | ((d[1:] == d[:-1]) & (v[1:] > v[:-1]))[same])
    return len(bins)


@pytest.mark.parametrize("n,views", [(1, 1), (255, 1), (1025, 1), (8192, 1), (8193, 1), (4096, 2), (4097, 2),
                                     (30_001, 1), (300_000, 1), (60_000, 3)])
@pytest.mark.parametrize("depths", ["near", "wide", "equal"])
def test_pair_order(n, views, depths):
    p, cam = frustum_scene(n=n, width=320, height=240, fx=300, fy=300, cx=160, cy=120, seed=n, logscale_mean=-5.0)
    rng = np.random.default_rng(n + 1)
    z = {"near": p[2], "wide": 10.0 ** rng.uniform(-0.6, 30, n), "equal": np.full(n, 2.0)}[depths]
    p[0:2] *= (z / p[2])[None]
    p[2] = z
    p = p.astype(np.float32)
    cams = [cam] + [rotated_cam(cam, [0.02 * k, -0.03 * k, 0.0], [0.0, 0.0, 0.0]) for k in range(1, views)]
    gm = new_map(n, views=views, W=320, H=240)
    gm.set_params(cuda(p))
    gm.render(cams)
    assert check_order(gm, cams, n) > 0 or depths == "wide"


@pytest.mark.parametrize("n", [100, 9000])
def test_nothing_visible(n):
    p, cam = frustum_scene(n=n)
    p[2] = -1.0
    gm = new_map(n)
    gm.set_params(cuda(p))
    assert float(gm.render(cam).abs().max()) == 0.0
    assert check_order(gm, [cam], n) == 0


@pytest.mark.parametrize("n", [16384 * 256, 16384 * 256 + 1, 17000 * 256 + 17])
def test_many_blocks(n):
    """Around the number of item blocks from which the emission reads a scan of their tile sums."""
    p, cam = frustum_scene(n=n, width=160, height=120, fx=150, fy=150, cx=80, cy=60, seed=3, logscale_mean=-6.0)
    gm = new_map(n, pair_capacity=8 * n)
    gm.set_params(cuda(p.astype(np.float32)))
    gm.render(cam)
    assert check_order(gm, [cam], n) > n // 2
