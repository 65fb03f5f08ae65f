"""The learned initialiser at batch sizes on the edges of its passes (32 or 64 rows a CTA, one or
several passes) and with unaligned input, against the FP64 oracle within the bounds of
test_gpu_mlp.py, and its gradient bit for bit repeatable."""
import numpy as np
import pytest
import torch

import oracle as O

from gpu_helpers import cuda
from test_gpu_mlp import _feats, _mlp

pytestmark = pytest.mark.gpu


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("rows", [lambda s: 1, lambda s: 31, lambda s: 33, lambda s: 96, lambda s: 32 * s,
                                  lambda s: 32 * s + 1, lambda s: 64 * s, lambda s: 64 * s + 65])
def test_rows_at_the_edges_of_passes(rows):
    n = rows(_sms())
    m = _mlp(3)
    flat = m.params().cpu().numpy().astype(np.float64)
    f = _feats(n, 4)
    tg = np.random.default_rng(5).normal(size=(n, 16)).astype(np.float32)
    tg[:, 11:] = 0
    ref = O.mlp_forward(flat, f.astype(np.float64))
    y = m.forward(cuda(f)).cpu().numpy()
    scale = np.abs(ref[:, :11]).max()
    assert np.abs(y[:, :11] - ref[:, :11]).max() <= 1e-2 * scale
    np.testing.assert_array_equal(y[:, 11:], 0.0)
    loss = float(m.backward(cuda(f), cuda(tg)).cpu()[0])
    g = m.grads()
    L, gref = O.mlp_loss_and_grad(flat, f.astype(np.float64), tg.astype(np.float64))
    assert abs(loss - L) <= 1e-3 * L
    o = 0
    for shape in O.MLP_SHAPES:
        k = int(np.prod(shape))
        a, b = g[o:o + k].cpu().numpy(), gref[o:o + k]
        floor = 1e-2 * max(np.abs(b).max(), 1e-30)
        assert (np.abs(a - b) / np.maximum(np.abs(b), floor)).max() <= 1e-2, shape
        o += k
    # features that start off a 16-byte boundary, and a second run
    shifted = torch.empty(n * 80 + 1, device="cuda")[1:].view(n, 80)
    shifted.copy_(cuda(f))
    assert shifted.data_ptr() % 16 != 0
    m.backward(shifted, cuda(tg))
    assert torch.equal(m.grads(), g)
