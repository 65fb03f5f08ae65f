"""A render that outgrows its pair buffer while it already runs, and the one-launch replacement of the
map: both bit for bit what a fresh map of ample size gives."""
import pytest
import torch

from synth import frustum_scene, random_target

from gpu_helpers import cuda, new_map

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [dict(), dict(tile_size=8, pixels_per_thread=1), dict(deterministic=1)])
@pytest.mark.parametrize("n", [2000, 20_000])
def test_render_that_outgrows_the_pair_buffer(n, cfg):
    p, cam = frustum_scene(n=n, seed=n)
    small, ample = new_map(n, pair_capacity=64, **cfg), new_map(n, **cfg)
    outs = []
    for gm in (small, ample):
        gm.set_params(cuda(p))
        outs.append(gm.render(cam, want_T=True, want_argmax=True))
        gm.loss(cuda(random_target(160, 120)))
        gm.backward()
        outs.append(gm.render(cam, want_T=True, want_argmax=True))
    for other in outs[1:]:
        for a, b in zip(outs[0], other):
            assert torch.equal(a, b)


@pytest.mark.parametrize("n,cap", [(1, 1), (3, 9), (4, 4), (5, 1027), (2001, 2001)])
def test_set_params_is_a_fresh_map(n, cap):
    p, cam = frustum_scene(n=n, seed=7)
    tg = cuda(random_target(160, 120))
    used, fresh = new_map(cap, deterministic=1, clarity_sigma=1e9), new_map(cap, deterministic=1, clarity_sigma=1e9)
    q, _ = frustum_scene(n=min(cap, n + 3), seed=8)
    used.set_params(cuda(q))
    for _ in range(3):
        used.iterate(cam, tg)
    used.count_dominant(cam)
    used.set_params(cuda(p))
    fresh.set_params(cuda(p))
    assert torch.equal(used.params(), cuda(p))
    for _ in range(3):
        assert torch.equal(used.iterate(cam, tg), fresh.iterate(cam, tg))
    assert torch.equal(used.params(), fresh.params())
