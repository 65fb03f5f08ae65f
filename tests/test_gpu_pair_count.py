"""More than 2^32 (tile, Gaussian) pairs, from Gaussians that fill a large screen: refused with
GS_ERR_CAPACITY by a render, a first iteration and (after the fact) a replay, without growing the pair
buffers and without touching the map."""
import numpy as np
import pytest
import torch

from paper_2504_02437_gb300 import _native as N
from synth import Camera

from gpu_helpers import cuda, new_map

pytestmark = pytest.mark.gpu

# (Gaussians, image side): 8-px tiles times Gaussians just past 2^32, by the depth sort of small maps
# (at most 8,192 items) and by the general one
SIZES = [(4200, 8192), (16500, 4096)]


def scene(n, side):
    r = np.random.RandomState(n)
    p = np.zeros((14, n))
    p[0:3] = r.uniform(-0.1, 0.1, (3, n))
    p[3:6] = 0.0                          # sigma 1 at z = 1: one image side in pixels
    p[6] = 1.0
    p[11:14] = 0.5
    near = Camera(side, side, float(side), float(side), side / 2, side / 2, np.eye(3), np.array([0.0, 0.0, 1.0]))
    far = Camera(side, side, float(side), float(side), side / 2, side / 2, np.eye(3), np.array([0.0, 0.0, 4000.0]))
    assert n * (side // 8) ** 2 > 2 ** 32
    return cuda(p), near, far


def code_of(call):
    with pytest.raises(N.GSError) as e:
        call()
    return e.value.code


@pytest.mark.parametrize("n,side", SIZES)
@pytest.mark.parametrize("det", [0, 1])
def test_too_many_pairs_are_refused(n, side, det):
    p, near, far = scene(n, side)
    gm = new_map(n, W=side, H=side, tile_size=8, deterministic=det)
    gm.set_params(p)
    tg = torch.zeros(1, 3, side, side, device="cuda")
    loss = torch.empty(3, device="cuda")
    free = torch.cuda.mem_get_info()[0]
    with pytest.raises(N.GSError) as e:
        gm.render(near)
    assert e.value.code == N.GS_ERR_CAPACITY
    assert code_of(lambda: gm.loss(tg)) == N.GS_ERR_STATE
    assert code_of(lambda: gm.iterate(near, tg, loss)) == N.GS_ERR_CAPACITY
    assert torch.equal(gm.params(), p)
    for _ in range(2):
        gm.iterate(far, tg, loss)
    torch.cuda.synchronize()
    q = gm.params()
    gm.iterate(near, tg, loss)            # a replay: reported by the next call
    torch.cuda.synchronize()
    assert torch.equal(gm.params(), q)
    assert code_of(lambda: gm.iterate(far, tg, loss)) == N.GS_ERR_CAPACITY
    gm.iterate(far, tg, loss)
    torch.cuda.synchronize()
    assert not torch.equal(gm.params(), q)
    assert free - torch.cuda.mem_get_info()[0] < 8 * 2 ** 30   # images and own buffers, no 64 GB of pairs
    gm.close()
