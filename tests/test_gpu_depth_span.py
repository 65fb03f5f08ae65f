"""Depths whose keys span more than 27 bits, so that each of the general depth sort's three digits is wider
than nine (and the small one's passes five): visible in numbers, and their pairs in order."""
import numpy as np
import pytest

from synth import frustum_scene

from gpu_helpers import cuda, new_map
from test_gpu_depth_order import check_order

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1025, 8192, 8193, 30_001, 300_000])
def test_wide_key_ranges(n):
    p, cam = frustum_scene(n=n, width=320, height=240, fx=300, fy=300, cx=160, cy=120, seed=n, logscale_mean=-5.0)
    z = 10.0 ** np.random.default_rng(n + 1).uniform(-0.6, 30, n)
    p[0:2] *= (z / p[2])[None]
    p[2] = z
    gm = new_map(n, W=320, H=240)
    gm.set_params(cuda(p.astype(np.float32)))
    gm.render(cam)
    assert check_order(gm, [cam], n) > n // 2
    proj = gm.debug_projection(0)
    key = proj[5][proj[7] > 0].astype(np.float32).view(np.uint32).astype(np.int64)
    assert len(key) > n // 2 and int(key.max() - key.min()).bit_length() > 27
