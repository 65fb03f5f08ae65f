"""The projection's adjoint for elongated Gaussians, by itself: the compositing's screen gradients as the
library holds them, taken back to the parameters in float64 by the oracle's projection, against the
library's gradients.

A projection whose axes have variances in the ratio kappa is inverted and its inverse taken back. Float32
parameters cannot do better than a few roundings times sqrt(kappa): a rounding of the rotation or of a
projected axis turns the long axis towards the short one by 2^-24 of its own length, sqrt(kappa) 2^-24 of
the short one's. The bound allows eight of them over each group's norm; arithmetic in the covariance's
entries, whose determinant and products cancel, loses kappa instead (1e-3 to 6e-2 on such scenes).
"""
import numpy as np
import pytest
import torch

import oracle as O
from synth import Camera

from gpu_helpers import GROUPS, cam_f32, cuda, new_map, rotated_cam

pytestmark = pytest.mark.gpu

CAM = cam_f32(Camera(160, 120, 150.0, 150.0, 80.0, 60.0, np.eye(3), np.array([0.0, 0.0, 1.0])))
VIEWS = [CAM, rotated_cam(CAM, [0.02, -0.03, 0.01], [0.03, 0.0, 1.05]),
         rotated_cam(CAM, [-0.01, 0.02, 0.3], [-0.02, 0.01, 0.95])]


def needles(seed, n=200):
    """Thin Gaussians 0.2 to 0.6 long, about one unit from the camera."""
    r = np.random.RandomState(seed)
    p = np.zeros((14, n))
    p[0:3] = r.uniform(-0.25, 0.25, (3, n))
    s = np.stack([r.uniform(0.2, 0.6, n), r.uniform(0.004, 0.02, n), r.uniform(0.004, 0.02, n)])
    p[3:6] = np.log(np.take_along_axis(s, np.argsort(r.rand(3, n), axis=0), axis=0))
    p[6:10] = r.normal(size=(4, n))
    p[10] = r.normal(size=n) - 1.0
    p[11:14] = r.uniform(0, 1, (3, n))
    return p.astype(np.float32)


@pytest.mark.parametrize("views", [1, 3])
@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("seed", [0, 1])
def test_adjoint_of_elongated_projections(seed, det, views):
    p, cams = needles(seed), VIEWS[:views]
    n = p.shape[1]
    gm = new_map(n, views=views, deterministic=det)
    gm.set_params(cuda(p))
    gm.render(cams)
    gm.backward(cuda(np.random.RandomState(seed + 10).normal(size=(views, 3, 120, 160))))
    got = gm.grads().cpu().numpy().astype(np.float64)
    screen = gm.debug_grad2d().astype(np.float64)
    gm.close()

    P = torch.as_tensor(p, dtype=torch.float64).requires_grad_(True)
    kappa = 1.0
    for cam, g in zip(cams, screen):
        pr = O.project(P, cam)
        seen = np.abs(g).sum(0) > 0
        ev = np.linalg.eigvalsh(pr["cov2d"].detach().numpy()[seen])
        kappa = max(kappa, float((ev[:, 1] / ev[:, 0]).max()))
        torch.autograd.backward([pr[k] for k in ("u", "v", "a", "b", "c")], [torch.as_tensor(g[k]) for k in range(5)])
    want = P.grad.numpy()
    assert kappa > 1000, kappa
    tol = 8 * 2.0 ** -24 * np.sqrt(kappa)
    for name in ("mean", "logscale", "quat"):
        sl = GROUPS[name]
        err = np.linalg.norm(got[sl] - want[sl]) / np.linalg.norm(want[sl])
        assert err <= tol, (name, err, tol)
