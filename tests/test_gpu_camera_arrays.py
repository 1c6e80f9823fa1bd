"""Camera arrays of every length and kind of host memory: cameras in pinned memory are read when the stream reaches
the call, as any copy from them is."""
import ctypes as C

import numpy as np
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _tree(pot):
    return pot.Tree.from_scene(S.scene_random(11, 5, 1, p_occ=0.3, lo=(-1.5,) * 3, size=3.0, sigma_mu=1.0))


@pytest.mark.parametrize("n_cams,size", [(1, 33), (8, 16), (9, 16), (200, 9), (257, 9), (1030, 8)])
def test_many_cameras(n_cams, size):
    """One call for all cameras against one call each; the array is overwritten as soon as the call returns."""
    import torch
    import paper_2103_14024_gb300 as pot
    tree = _tree(pot)
    views = S.make_cameras(S.hemisphere_c2ws(3, n_cams), size, size, 1.4 * size)
    cams = pot.make_cameras(views)
    torch.cuda._sleep(2_000_000)
    rgb = pot.render(tree, cams, gamma=1e-4)
    weight = pot.visibility(tree, cams)
    C.memset(cams, 0, C.sizeof(cams))
    want = torch.zeros_like(weight)
    for i in range(n_cams):
        assert torch.equal(rgb[i:i + 1], pot.render(tree, views[i:i + 1], gamma=1e-4))
        pot.visibility(tree, views[i:i + 1], max_weight=want)
    assert torch.equal(weight, want)
    pot.check()


@pytest.mark.parametrize("n_cams", [1, 8, 9, 40])
def test_pinned_cameras_follow_the_stream(n_cams):
    import torch
    import paper_2103_14024_gb300 as pot
    tree, size = _tree(pot), 24
    first, second = (S.make_cameras(S.hemisphere_c2ws(seed, n_cams), size, size, 1.4 * size) for seed in (1, 2))
    want = pot.render(tree, second), pot.visibility(tree, second)
    assert not torch.equal(want[0], pot.render(tree, first))
    held = torch.empty(n_cams * C.sizeof(pot.Camera), dtype=torch.uint8, pin_memory=True)
    cams = (pot.Camera * n_cams).from_address(held.data_ptr())
    later = torch.from_numpy(np.ascontiguousarray(second).view(np.uint8).copy()).cuda()
    for call, ref in ((pot.render, want[0]), (pot.visibility, want[1])):
        C.memmove(cams, np.ascontiguousarray(first).ctypes.data, held.numel())
        torch.cuda.synchronize()
        torch.cuda._sleep(20_000_000)
        held.copy_(later, non_blocking=True)  # behind the sleep, ahead of the call
        got = call(tree, cams)
        torch.cuda.synchronize()
        assert torch.equal(got, ref)
    pot.check()
