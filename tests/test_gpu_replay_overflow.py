"""A replay that overflows its pair buffer composites nothing: black image, the loss of a black image, and a
map (parameters, moments, densification statistics) that is not touched; after the report it iterates on."""
import numpy as np
import pytest
import torch

from paper_2504_02437_gb300 import _native as N
from synth import frustum_scene, random_target

from gpu_helpers import cuda, new_map, rotated_cam

pytestmark = pytest.mark.gpu


def state(gm, path):
    """The checkpoint without its host-side count of iteration calls (bytes 24 to 27)."""
    gm.save(str(path))
    raw = path.read_bytes()
    return raw[:24] + raw[28:]


@pytest.mark.parametrize("cfg", [dict(), dict(tile_size=8), dict(deterministic=1)])
def test_overflowing_replay(cfg, tmp_path):
    p, cam = frustum_scene(n=3000, seed=12)
    far = rotated_cam(cam, [0.0, 0.0, 0.0], [0.0, 0.0, -6.0])      # sees a handful of them
    tg = cuda(random_target(160, 120, seed=13))
    gm = new_map(3000, pair_capacity=64, **cfg)
    gm.set_params(cuda(p))
    loss, rgb = torch.empty(3, device="cuda"), torch.empty(1, 3, 120, 160, device="cuda")
    for _ in range(2):
        gm.iterate(far, tg, loss, rgb)
    before = state(gm, tmp_path / "a")
    gm.iterate(cam, tg, loss, rgb)
    assert state(gm, tmp_path / "b") == before
    assert int(torch.count_nonzero(rgb)) == 0
    want = float(tg.double().abs().mean())
    # 3HW sums of magnitudes in float32, per thread, warp, CTA: their number's logarithm times 2^-24
    assert abs(float(loss[1]) - want) <= 32 * 2.0 ** -24 * want
    with pytest.raises(N.GSError) as e:
        gm.iterate(cam, tg, loss, rgb)
    assert e.value.code == N.GS_ERR_CAPACITY
    assert state(gm, tmp_path / "c") == before
    gm.iterate(cam, tg, loss, rgb)
    assert state(gm, tmp_path / "d") != before and int(torch.count_nonzero(rgb)) > 0
