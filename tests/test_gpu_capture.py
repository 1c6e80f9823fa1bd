"""pot_render in a stream capture: the graph reads the caller's camera array at each replay, whether the call has
few cameras or many, few tiles or many, and clears its own tile counter."""
import ctypes as C

import numpy as np
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cams,size", [(1, 40), (8, 33), (9, 33), (12, 256)])
def test_captured_render_reads_cameras_at_replay(n_cams, size):
    import torch
    import paper_2103_14024_gb300 as pot
    tree = pot.Tree.from_scene(S.scene_random(11, 5, 1, p_occ=0.3, lo=(-1.5,) * 3, size=3.0, sigma_mu=1.0))
    views = [S.make_cameras(S.hemisphere_c2ws(seed, n_cams), size, size, 1.4 * size) for seed in (1, 2)]
    held = torch.empty(n_cams * C.sizeof(pot.Camera), dtype=torch.uint8, pin_memory=True)
    cams = (pot.Camera * n_cams).from_address(held.data_ptr())

    def show(k):
        C.memmove(cams, np.ascontiguousarray(views[k]).ctypes.data, held.numel())

    want = [pot.render(tree, v, gamma=1e-4) for v in views]
    assert not torch.equal(want[0], want[1])
    rgb = torch.empty_like(want[0])
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    show(0)
    with torch.cuda.graph(graph):
        pot.render(tree, cams, rgb=rgb, gamma=1e-4)
    for k in (0, 1, 0):
        show(k)
        rgb.fill_(-1.0)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(rgb, want[k])
    pot.check()
