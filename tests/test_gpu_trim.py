"""Map management keeps scratch and a second set of buffers from call to call; gs_trim gives them back, and
the calls after it do what they did before."""
import pytest
import torch

from synth import frustum_scene, random_target

from gpu_helpers import cuda, new_map

pytestmark = pytest.mark.gpu

CAP = 400_000          # a second set of parameters and moments: 67 MB


def grow(gm, p, cam, trim):
    gm.set_params(p)
    out = []
    for k in range(3):
        gm.iterate(cam, cuda(random_target(160, 120)))
        gm.count_dominant(cam)
        split = gm.densify()
        if trim:
            gm.trim()
        count = gm.insert(cam, torch.full((3, 120, 160), 0.5, device="cuda"), torch.full((4, 3), 30.0 + k, device="cuda"))
        if trim:
            gm.trim()
            gm.trim()
        out.append((split, count, gm.params()))
    return out


def test_trim_gives_back_and_changes_nothing():
    p, cam = frustum_scene(n=2000, seed=9)
    p = cuda(p)
    maps = [new_map(CAP, deterministic=1, clarity_sigma=8.0, pair_capacity=1 << 20) for _ in range(2)]
    kept, trimmed = (grow(gm, p, cam, t) for gm, t in zip(maps, (False, True)))
    for (s0, c0, a), (s1, c1, b) in zip(kept, trimmed):
        assert s0 > 0 and (s0, c0) == (s1, c1) and torch.equal(a, b)
    free = torch.cuda.mem_get_info()[0]
    maps[0].trim()
    assert torch.cuda.mem_get_info()[0] - free > 0.9 * 3 * 14 * 4 * CAP
    free = torch.cuda.mem_get_info()[0]
    maps[1].trim()
    assert torch.cuda.mem_get_info()[0] == free
    assert torch.equal(maps[0].params(), kept[-1][2])
