"""Boxes of every size whose voxels are normal floats, from any distance that floats resolve, against the float64
oracle: lengths, densities and cell lookups do not depend on the scale."""
import numpy as np
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [5, 9, 12])
@pytest.mark.parametrize("size", [3e-34, 1e-31, 1e-29, 1e-25, 1e-23, 1e-10, 1e10, 1e30])
def test_walk_box_scale(oracle_mod, depth, size):
    import torch
    import paper_2103_14024_gb300 as pot
    R = 1 << depth
    lo = -0.5 * size
    rng = np.random.default_rng(depth)
    near = rng.integers(R // 2 - 6, R // 2 + 6, (1500, 3))
    v = np.unique(np.concatenate([near, rng.integers(0, R, (500, 3))]), axis=0)
    codes = np.sort(S.morton_encode(v[:, 0], v[:, 1], v[:, 2], depth))
    sigma = (np.exp(rng.normal(0, 1, len(codes))) * R / 8 / size).astype(np.float32)
    sc = S.Scene(depth, (lo,) * 3, size, 1, codes, sigma, rng.normal(0, 1, (len(codes), 4, 3)).astype(np.float32))
    tree, ot = pot.Tree.from_scene(sc), oracle_mod.build_sparse(sc)
    u = rng.normal(size=(1200, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    at = size / R * rng.uniform(-5, 5, (1200, 3))
    back = np.where(np.arange(1200) % 3 == 0, 0.0, np.where(np.arange(1200) % 3 == 1, 1.5, 40.0))
    o = (at - (back * size)[:, None] * u).astype(np.float32)
    d = (u * np.exp(rng.uniform(-9, 9, 1200))[:, None]).astype(np.float32)
    ref = oracle_mod.render_rays(ot, o, d, bg=(0.1, 0.2, 0.3), far=3.0e38)["rgb"]
    assert np.abs(ref - np.float32((0.1, 0.2, 0.3))).max() > 0.1
    for cells in ("none", "brick", "dense"):
        if cells == "brick" and depth > 11 or cells == "dense" and depth > 10:
            continue
        tree.set_cell_index(cells)
        rgb = pot.render_rays(tree, torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), bg=(0.1, 0.2, 0.3))
        pot.check()
        assert np.abs(rgb.cpu().numpy() - ref).max() <= 1e-4
    # from far away the box is not seen
    if size < 1.0:
        rgb = pot.render_rays(tree, torch.full((3, 3), 3e8, device="cuda"), torch.eye(3, device="cuda") - 0.5)
        assert not rgb.any()
    tree.free()
