"""Filtering and a training step in a stream capture: scratch comes from the graph's own allocations, sums start at
zero and cameras are read at each replay."""
import ctypes as C

import numpy as np
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _tree(pot):
    return pot.Tree.from_scene(S.scene_random(11, 5, 1, p_occ=0.3, lo=(-1.5,) * 3, size=3.0, sigma_mu=1.0))


@pytest.mark.parametrize("n_cams,size", [(1, 40), (9, 33), (12, 256)])
def test_captured_visibility(n_cams, size):
    import torch
    import paper_2103_14024_gb300 as pot
    tree = _tree(pot)
    views = [S.make_cameras(S.hemisphere_c2ws(seed, n_cams), size, size, 1.4 * size) for seed in (1, 2)]
    held = torch.empty(n_cams * C.sizeof(pot.Camera), dtype=torch.uint8, pin_memory=True)
    cams = (pot.Camera * n_cams).from_address(held.data_ptr())
    want = [pot.visibility(tree, v) for v in views]
    weight = torch.zeros_like(want[0])
    C.memmove(cams, np.ascontiguousarray(views[0]).ctypes.data, held.numel())
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        pot.visibility(tree, cams, max_weight=weight)
    for k in (0, 1, 0):
        C.memmove(cams, np.ascontiguousarray(views[k]).ctypes.data, held.numel())
        weight.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(weight, want[k])
    pot.check()


@pytest.mark.parametrize("n", [3000, 90001])
def test_captured_training_calls(n):
    import torch
    import paper_2103_14024_gb300 as pot
    tree = _tree(pot)
    o, d = (torch.from_numpy(a).cuda() for a in S.random_rays(5, n, radius=4.0, spread=1.0))
    target = torch.rand((n, 3), device="cuda")
    rays = dict(gamma=1e-3, near=0.5, far=8.0)
    rec = pot.SegmentRecords.for_rays(n, 32)
    L, K = tree.info()["n_leaves"], tree.info()["sh_dim"]
    buf = [dict(rgb=torch.empty_like(o), loss=torch.empty(1, device="cuda"), gs=torch.zeros(L, device="cuda"),
                gh=torch.zeros((L, K, 3), device="cuda")) for _ in range(2)]
    grad = torch.empty_like(o)

    def run():
        a, b = buf
        pot.render_rays_record(tree, o, d, rec, rgb=a["rgb"], **rays)
        loss, _ = pot.loss_mse(a["rgb"], target, grad=grad)
        a["loss"].copy_(loss)
        pot.render_backward_recorded(tree, o, d, grad, a["rgb"], rec, grad_sigma=a["gs"], grad_sh=a["gh"], **rays)
        pot.render_mse_backward(tree, o, d, target, rgb=b["rgb"], loss=b["loss"], grad_sigma=b["gs"], grad_sh=b["gh"],
                                **rays)

    run()
    torch.cuda.synchronize()
    want = [{k: v.clone() for k, v in x.items()} for x in buf]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    for _ in range(3):
        for x in buf:
            for v in x.values():
                v.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for x, w in zip(buf, want):
            assert torch.equal(x["rgb"], w["rgb"])
            assert abs(float(x["loss"]) - float(w["loss"])) <= 2.0 ** -22 * float(w["loss"])
            for k in ("gs", "gh"):  # float reductions in another order
                assert float((x[k] - w[k]).abs().max()) <= 1e-4 * float(w[k].abs().max())
    pot.check()
