"""Where a walk starts: direction components too small to move a ray, origins just above a voxel's lower plane seen
from the side that the ray leaves through, and entries along slow axes, against the float64 oracle."""
import itertools

import numpy as np
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu
TOL = 1e-4  # the parity bound of fp32 renders


def _compare(pot, oracle_mod, sc, o, d, kinds):
    import torch
    tree, ot = pot.Tree.from_scene(sc), oracle_mod.build_sparse(sc)
    ref = oracle_mod.render_rays(ot, o, d, bg=(0.1, 0.2, 0.3))
    for cells in kinds:
        tree.set_cell_index(cells)
        rgb, tf = pot.render_rays(tree, torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), bg=(0.1, 0.2, 0.3),
                                  want_t_final=True)
        pot.check()
        assert np.abs(rgb.cpu().numpy() - ref["rgb"]).max() <= TOL
        assert np.abs(tf.cpu().numpy() - ref["t_final"]).max() <= TOL
    tree.free()


@pytest.mark.parametrize("small", [1e-37, 1.2e-38, 1e-39, 1e-42, 1e-45])
def test_components_below_the_normal_floats(oracle_mod, small):
    """An axis with a subnormal component does not move, whatever the component's sign, and is not mirrored."""
    import paper_2103_14024_gb300 as pot
    lo, size = -1.0, 2.0
    sc = S.scene_random(431, 5, 1, p_occ=0.35, lo=(lo,) * 3, size=size, sigma_mu=1.5)
    rng = np.random.default_rng(5)
    o, d = [], []
    for signs in itertools.product((-1, 1), repeat=3):
        for axes in ((0,), (1,), (2,), (0, 1), (1, 2), (0, 2)):
            for scale in (1.0, 1e-3, 1e3):
                u = np.array(signs) * rng.uniform(0.3, 1.0, 3)
                at = lo + size * rng.uniform(0.05, 0.45, 3)  # below the centre: its mirror is another voxel
                start = at - 3.0 * u
                start[list(axes)] = at[list(axes)]
                u *= scale
                u[list(axes)] = np.array(signs)[list(axes)] * small
                o.append(start)
                d.append(u)
    o, d = np.array(o).astype(np.float32), np.array(d).astype(np.float32)
    assert (d != 0).all() and (d < 0).any()
    _compare(pot, oracle_mod, sc, o, d, ("none", "brick", "dense"))


@pytest.mark.parametrize("depth", [5, 9, 12])
@pytest.mark.parametrize("lo", [0.0, -0.25])
def test_origins_just_above_low_planes(oracle_mod, depth, lo):
    """Viewers inside the box, 1e-7 to 1e-3 voxels above a plane, looking down along one axis or more: the sliver of
    the first voxel counts.  Densities make a voxel opaque, so that at depth 12 a skipped 1e-4 voxels would show."""
    import paper_2103_14024_gb300 as pot
    R = 1 << depth
    h = 1.0 / R
    rng = np.random.default_rng(depth)
    v = rng.integers(1, max(2, R // 8), (400, 3))
    v = np.unique(v, axis=0)
    codes = np.sort(S.morton_encode(v[:, 0], v[:, 1], v[:, 2], depth))
    sc = S.Scene(depth, (lo,) * 3, 1.0, 1, codes, np.full(len(codes), 30.0 * R, np.float32),
                 rng.normal(0, 1, (len(codes), 4, 3)).astype(np.float32))
    o, d = [], []
    for i in range(4000):
        c = v[i % len(v)]
        f = np.where(rng.random(3) < 0.6, 10.0 ** rng.uniform(-7, -3, 3), rng.uniform(0.1, 0.9, 3))
        o.append(lo + h * (c + f))
        u = rng.normal(size=3)
        down = rng.random(3) < 0.7
        d.append(np.where(down, -np.abs(u), u))
    o, d = np.array(o).astype(np.float32), np.array(d).astype(np.float32)
    _compare(pot, oracle_mod, sc, o, d, ["none"] + ["brick"] * (3 <= depth <= 11) + ["dense"] * (depth <= 10))


@pytest.mark.parametrize("depth", [6, 9, 12])
@pytest.mark.parametrize("slow", [1e-2, 1e-4, 1e-6])
def test_entries_through_a_slow_axis(oracle_mod, depth, slow):
    """Rays nearly parallel to two faces of the box that enter through one of them: the box's plane times on that axis
    are large and nearly cancel.  A layer of opaque voxels under each face shows which voxel was entered."""
    import paper_2103_14024_gb300 as pot
    R = 1 << depth
    h = 1.0 / R
    rng = np.random.default_rng(int(-np.log10(slow)) + 100 * depth)
    n = min(R, 64)
    base = R // 2 - n // 2
    i, j = np.meshgrid(np.arange(n) + base, np.arange(n) + base, indexing="ij")
    v = np.unique(np.concatenate([np.roll(np.stack([np.full(i.size, layer), i.ravel(), j.ravel()], 1), a, axis=1)
                                  for a in range(3) for layer in (0, R - 1)]), axis=0)
    codes = np.sort(S.morton_encode(v[:, 0], v[:, 1], v[:, 2], depth))
    sc = S.Scene(depth, (0.0,) * 3, 1.0, 1, codes, np.full(len(codes), 30.0 * R, np.float32),
                 rng.normal(0, 1, (len(codes), 4, 3)).astype(np.float32))
    o, d = [], []
    for k in range(1500):
        a, up = k % 3, k // 3 % 2
        u = rng.normal(size=3)
        u[(a + 1) % 3] = rng.choice([-1.0, 1.0])
        u[a] = slow * rng.uniform(0.5, 2.0) * (1.0 if up else -1.0)
        at = h * (base + n * rng.uniform(0.2, 0.8, 3))
        at[a] = 0.0 if up else 1.0
        o.append(at - u * rng.uniform(0.01, 1.0))
        d.append(u)
    o, d = np.array(o).astype(np.float32), np.array(d).astype(np.float32)
    _compare(pot, oracle_mod, sc, o, d, ["none"] + ["brick"] * (3 <= depth <= 11) + ["dense"] * (depth <= 10))


@pytest.mark.parametrize("small", [1.5e-38, 1e-37, 1e-36, 1e-32])
def test_slow_axis_outside_its_slab(oracle_mod, small):
    """An origin outside the box on an axis along which the ray hardly moves: the box's plane times leave the float
    range, and the ray misses the box."""
    import paper_2103_14024_gb300 as pot
    lo, size = -1.0, 2.0
    sc = S.scene_random(431, 5, 1, p_occ=0.35, lo=(lo,) * 3, size=size, sigma_mu=1.5)
    rng = np.random.default_rng(6)
    o, d = [], []
    for k in range(600):
        a = k % 3
        u = rng.normal(size=3)
        at = lo + size * rng.uniform(0.1, 0.9, 3)
        start = at - 3.0 * u
        start[a] = at[a] if k % 2 else rng.choice([-1, 1]) * 10.0 ** rng.uniform(0.1, 4.0)
        u[a] = small * rng.choice([-1, 1])
        o.append(start)
        d.append(u)
    o, d = np.array(o).astype(np.float32), np.array(d).astype(np.float32)
    _compare(pot, oracle_mod, sc, o, d, ("none", "brick", "dense"))


@pytest.mark.parametrize("small", [0.0, 1e-45, 1e-39, 1e-36])
def test_side_of_a_plane(oracle_mod, small):
    """An origin on a voxel's plane, or the box's, belongs to the side that even the smallest component heads for."""
    import paper_2103_14024_gb300 as pot
    lo, size = -1.0, 2.0
    sc = S.scene_random(432, 5, 1, p_occ=0.35, lo=(lo,) * 3, size=size, sigma_mu=1.5)
    rng = np.random.default_rng(7)
    o, d = [], []
    for k in range(990):
        a = k % 3
        u = rng.normal(size=3)
        start = lo + size * rng.uniform(0.1, 0.9, 3) - 3.0 * u
        start[a] = lo + size / 32 * (k // 6 % 33)
        u[a] = small * (1.0 if k // 3 % 2 else -1.0)
        o.append(start)
        d.append(u)
    o, d = np.array(o).astype(np.float32), np.array(d).astype(np.float32)
    _compare(pot, oracle_mod, sc, o, d, ("none", "brick", "dense"))
