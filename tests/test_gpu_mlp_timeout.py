"""A bounded wait of the learned initialiser that gives up (made to, at once, at each wait of a launch in
turn; its copies and products are waited for before the CTA leaves): what the launch would have written
is not used, the calls after it report GS_ERR_TIMEOUT, and an insertion it happens in leaves the map."""
import numpy as np
import pytest
import torch

from paper_2504_02437_gb300 import _native as N
from paper_2504_02437_gb300.api import MLP
from synth import frustum_scene

from gpu_helpers import cuda, new_map

pytestmark = pytest.mark.gpu


def code_of(call):
    with pytest.raises(N.GSError) as e:
        call()
    return e.value.code


def rows(n, seed):
    r = np.random.default_rng(seed)
    return cuda(r.uniform(0, 1, (n, 80))), cuda(r.normal(size=(n, 16)))


@pytest.mark.parametrize("n", [40, 20_000])      # passes of 32 and of 64 rows, one and several a CTA
@pytest.mark.parametrize("nth", [1, 2, 3, 4, 5, 6, 7])
def test_training(nth, n):
    m = MLP(seed=2)
    x, y = rows(n, 1)
    m.backward(x, y)
    before, grads = m.params(), m.grads()
    assert m.lib.gs_debug_mlp_give_up(m.handle, nth) == N.GS_OK
    loss = m.backward(x, y)
    try:
        m.step(1e-2)                              # enqueued, or refused when the flag is already there
    except N.GSError as e:
        assert e.code == N.GS_ERR_TIMEOUT
    torch.cuda.synchronize()
    assert torch.isnan(loss).all()
    assert torch.equal(m.params(), before) and torch.equal(m.grads(), grads)
    assert m.lib.gs_debug_mlp_give_up(m.handle, 0) == N.GS_OK
    for call in (lambda: m.step(1e-2), lambda: m.backward(x, y), lambda: m.forward(x)):
        assert code_of(call) == N.GS_ERR_TIMEOUT
    assert torch.equal(m.params(), before)
    other = MLP(seed=2)                           # the GPU and other handles are as before
    assert torch.equal(other.backward(x, y).isfinite(), torch.ones(1, dtype=torch.bool, device="cuda"))
    assert torch.equal(other.grads(), grads)


@pytest.mark.parametrize("nth", [1, 2, 3, 4])
def test_insertion(nth):
    p, cam = frustum_scene(n=300, seed=4)
    m = MLP(seed=3)
    gm = new_map(400)
    gm.set_params(cuda(p))
    gm.set_initializer(m)
    image, pts = torch.rand(3, 120, 160, device="cuda"), torch.full((5, 3), 40.0, device="cuda")
    assert m.lib.gs_debug_mlp_give_up(m.handle, nth) == N.GS_OK
    assert code_of(lambda: gm.insert(cam, image, pts)) == N.GS_ERR_TIMEOUT
    assert gm.n == 300 and torch.equal(gm.params(), cuda(p))
    assert m.lib.gs_debug_mlp_give_up(m.handle, 0) == N.GS_OK
    assert code_of(lambda: gm.insert(cam, image, pts)) == N.GS_ERR_TIMEOUT   # refused before any work
    gm.set_initializer(MLP(seed=3))
    assert gm.insert(cam, image, pts) == 5
    assert gm.n == 305 and torch.equal(gm.params()[:, :300], cuda(p))
