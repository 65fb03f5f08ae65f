"""Pair buffers that cannot grow: the failure is made on the host, the call reports GS_ERR_OOM, nothing is
composited from buffers that are not there, and the next call grows them and gives, bit for bit, what a
fresh map of ample size gives."""
import pytest
import torch

from paper_2504_02437_gb300 import _native as N
from synth import frustum_scene, random_target

from gpu_helpers import cuda, new_map

pytestmark = pytest.mark.gpu

BUFFERS = [(0, k) for k in (1, 2, 3, 4)] + [(1, k) for k in (1, 4, 5, 6)]   # (deterministic, which one fails)


def code_of(gm, call):
    with pytest.raises(N.GSError) as e:
        call()
    return e.value.code


@pytest.mark.parametrize("det,nth", BUFFERS)
def test_render_after_a_failed_growth(det, nth):
    p, cam = frustum_scene(n=3000, seed=5)
    tg = cuda(random_target(160, 120))
    small, ample = new_map(3000, pair_capacity=64, deterministic=det), new_map(3000, deterministic=det)
    for gm in (small, ample):
        gm.set_params(cuda(p))
    assert small.lib.gs_debug_fail_pair_alloc(small.ctx, nth) == N.GS_OK
    assert code_of(small, lambda: small.render(cam)) == N.GS_ERR_OOM
    assert code_of(small, lambda: small.loss(tg)) == N.GS_ERR_STATE
    assert small.lib.gs_debug_fail_pair_alloc(small.ctx, nth) == N.GS_OK   # again, from no buffers at all
    assert code_of(small, lambda: small.render(cam)) == N.GS_ERR_OOM
    for a, b in zip(small.render(cam, want_T=True, want_argmax=True), ample.render(cam, want_T=True, want_argmax=True)):
        assert torch.equal(a, b)
    for gm in (small, ample):
        gm.loss(tg)
        gm.backward()
    if det:
        assert torch.equal(small.grads(), ample.grads())


@pytest.mark.parametrize("nth", [1, 6])
def test_iteration_after_a_failed_growth(nth):
    p, cam = frustum_scene(n=3000, seed=6)
    tg = cuda(random_target(160, 120))
    small, ample = new_map(3000, pair_capacity=64, deterministic=1), new_map(3000, deterministic=1)
    for gm in (small, ample):
        gm.set_params(cuda(p))
    assert small.lib.gs_debug_fail_pair_alloc(small.ctx, nth) == N.GS_OK
    assert code_of(small, lambda: small.iterate(cam, tg)) == N.GS_ERR_OOM
    for _ in range(3):
        assert torch.equal(small.iterate(cam, tg), ample.iterate(cam, tg))
    assert torch.equal(small.params(), ample.params())
