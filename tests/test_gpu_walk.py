"""The walk through the octree where it can go wrong: directions in all octants with zero, tiny and huge
components, rays along faces and through edges and corners, origins on planes, inside and far away, boxes of
extreme sizes, every cell lookup (dense index, bricks, child-array descent), against the float64 oracle."""
import itertools

import numpy as np
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu
TOL = 1e-4  # the parity bound of fp32 renders


@pytest.fixture(scope="module")
def pot():
    import torch
    assert torch.cuda.is_available()
    import paper_2103_14024_gb300 as P
    P.lib()
    return P


def _scene(depth, lo, size):
    """A random tree; deep grids hold a random block around the centre and scattered voxels."""
    if depth <= 6:
        return S.scene_random(400 + depth, depth, 1, p_occ=0.35, lo=(lo,) * 3, size=size, sigma_mu=1.5 - np.log(size))
    rng = np.random.default_rng(depth)
    R = 1 << depth
    near = rng.integers(R // 2 - 6, R // 2 + 6, (1500, 3))
    far = rng.integers(0, R, (500, 3))
    v = np.unique(np.concatenate([near, far]), axis=0)
    codes = np.sort(S.morton_encode(v[:, 0], v[:, 1], v[:, 2], depth))
    sigma = np.exp(rng.normal(np.log(R / 8 / size), 1.0, len(codes))).astype(np.float32)
    sh = rng.normal(0, 1, (len(codes), 4, 3)).astype(np.float32)
    return S.Scene(depth, (lo,) * 3, size, 1, codes, sigma, sh)


def _rays(depth, lo, size):
    """Rays in units of the box [lo, lo + size): aimed at faces, edges, corners and voxel interiors around the centre."""
    rng = np.random.default_rng(7 * depth)
    R = 1 << depth
    h = size / R
    mid = lo + size / 2
    o, d = [], []
    # all octants, with components scaled to nothing one by one, from planes and from generic points
    for signs in itertools.product((-1, 1), repeat=3):
        for tiny in (1.0, 1e-3, 1e-8, 1e-17, 1e-30, 0.0):
            for axes in ((), (0,), (1,), (2,), (0, 1), (1, 2), (0, 2)):
                u = np.array(signs) * rng.uniform(0.3, 1.0, 3)
                u[list(axes)] *= tiny
                if not np.any(np.abs(u) > 0.1):
                    continue
                at = mid + h * rng.integers(-3, 4, 3)                 # a corner of the grid
                if rng.random() < 0.5:
                    at = at + h * rng.uniform(0, 1, 3)
                o.append(at - 1.5 * size * u)
                d.append(u)
    # origins inside the box, and far outside it
    for back in (0.0, 0.2, 1e3):
        for _ in range(120):
            u = rng.normal(size=3)
            u /= np.linalg.norm(u)
            o.append(mid + h * rng.integers(-4, 5, 3) * rng.uniform(0.9, 1.0) - back * size * u)
            d.append(u)
    o, d = np.array(o, np.float32), np.array(d)
    d = (d * np.exp(rng.uniform(-9, 9, len(d)))[:, None]).astype(np.float32)  # not unit length
    return o, d


def _close(gpu, ref):
    assert np.abs(gpu - ref).max() <= TOL


@pytest.mark.parametrize("depth", [1, 2, 3, 5, 6, 9, 11, 12])
def test_walk_special_rays(pot, oracle_mod, depth):
    import torch
    lo, size = -1.0, 2.0
    sc = _scene(depth, lo, size)
    tree, ot = pot.Tree.from_scene(sc), oracle_mod.build_sparse(sc)
    o, d = _rays(depth, lo, size)
    do, dd = torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda()
    ref = oracle_mod.render_rays(ot, o, d, bg=(0.1, 0.2, 0.3))
    first = None
    for cells in ("none", "brick", "dense"):
        if cells == "brick" and not 3 <= depth <= 11 or cells == "dense" and depth > 10:
            continue
        tree.set_cell_index(cells)
        rgb, tf = pot.render_rays(tree, do, dd, bg=(0.1, 0.2, 0.3), want_t_final=True)
        pot.check()
        _close(rgb.cpu().numpy(), ref["rgb"])
        _close(tf.cpu().numpy(), ref["t_final"])
        if first is not None:
            assert torch.equal(rgb, first[0]) and torch.equal(tf, first[1])
        first = rgb, tf
    # clipped ranges: near and far cut the same segments
    reach = 1.5 * size
    rgb = pot.render_rays(tree, do, dd, near=reach, far=reach + 0.3 * size)
    _close(rgb.cpu().numpy(), oracle_mod.render_rays(ot, o, d, near=reach, far=reach + 0.3 * size)["rgb"])


@pytest.mark.parametrize("size", [1e-6, 3e-3, 7.0, 1e5])
def test_walk_box_sizes(pot, oracle_mod, size):
    import torch
    lo = -0.5 * size
    sc = _scene(5, lo, size)
    tree, ot = pot.Tree.from_scene(sc), oracle_mod.build_sparse(sc)
    o, d = _rays(5, lo, size)
    rgb = pot.render_rays(tree, torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda())
    pot.check()
    _close(rgb.cpu().numpy(), oracle_mod.render_rays(ot, o, d)["rgb"])
