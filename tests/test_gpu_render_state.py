"""Loss and adjoint want a whole render before them: an iteration (which keeps no transmittance, and in a
replay uses a work list of its own), an insertion, a split or a new map ends the last one's state."""
import pytest
import torch

from paper_2504_02437_gb300 import _native as N
from paper_2504_02437_gb300.api import rasterize
from synth import Camera, frustum_scene, random_target

from gpu_helpers import cuda, new_map, rotated_cam

pytestmark = pytest.mark.gpu


def refused(call):
    with pytest.raises(N.GSError) as e:
        call()
    return e.value.code == N.GS_ERR_STATE


def setup(**cfg):
    p, cam = frustum_scene(n=500, seed=3)
    gm = new_map(600, views=3, **cfg)
    gm.set_params(cuda(p))
    cams = [cam, rotated_cam(cam, [0.02, -0.03, 0.0], [0.03, 0.0, 0.05]), rotated_cam(cam, [0, 0.02, 0], [0, 0, 0])]
    return gm, p, cam, cams


@pytest.mark.parametrize("cfg", [dict(), dict(lambda_photo=0.2), dict(deterministic=1), dict(tile_size=0)])
def test_backward_after_an_iteration_is_refused(cfg):
    gm, p, cam, cams = setup(**cfg)
    small = Camera(24, 20, cam.fx, cam.fy, 12.0, 10.0, cam.R, cam.t)
    tg, up = cuda(random_target(24, 20)), torch.ones(1, 3, 20, 24, device="cuda")
    for _ in range(3):                       # the first direct, then replays, a larger render before each
        gm.render(cams)
        gm.iterate(small, tg)
        assert refused(lambda: gm.backward(up)) and refused(lambda: gm.loss(tg)) and refused(gm.backward)
        assert refused(gm.step)
    gm.render(small)
    gm.loss(tg)
    gm.backward()
    gm.step()


def test_autograd_after_an_iteration_is_refused():
    gm, p, cam, cams = setup()
    P = cuda(p).requires_grad_(True)
    img = rasterize(P, gm, cams)
    gm.iterate(cam, cuda(random_target(160, 120)))
    assert refused(lambda: img.sum().backward())


def test_what_else_ends_a_render():
    gm, p, cam, cams = setup(clarity_sigma=1e9)
    tg = cuda(random_target(160, 120))
    gm.render(cam)
    gm.insert(cam, tg[0], torch.full((2, 3), 50.0, device="cuda"))
    assert refused(lambda: gm.loss(tg))
    gm.render(cam)
    gm.densify()
    assert refused(lambda: gm.loss(tg))
    gm.render(cam)
    gm.set_params(cuda(p))
    assert refused(lambda: gm.backward(tg))
    gm.count_dominant(cam)                   # its image is scratch; its state takes an upstream gradient
    assert refused(lambda: gm.loss(tg))
    gm.backward(tg)
    a = gm.grads()
    gm.render(cam)
    gm.backward(tg)
    assert torch.allclose(a, gm.grads(), rtol=1e-3, atol=1e-6 * float(a.abs().max()))


def test_an_empty_map_still_has_a_render():
    gm, p, cam, cams = setup()
    gm.set_params(cuda(p[:, :0]))
    gm.iterate(cam, cuda(random_target(160, 120)))
    gm.render(cam)
    gm.loss(cuda(random_target(160, 120)))
    gm.backward()
    gm.step()
