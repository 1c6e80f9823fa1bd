"""A leaf whose SH coefficients hold a NaN: pixels that composite it say so, all others are as without it."""
import numpy as np
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
def test_nan_coefficient_shows(dtype):
    import torch
    import paper_2103_14024_gb300 as pot
    sc = S.scene_random(61, 4, 1, p_occ=0.3, sigma_mu=0.0)
    sh = sc.sh.copy()
    sh[len(sh) // 2, 2, 1] = np.nan  # one channel
    o, d = (torch.from_numpy(a).cuda() for a in S.random_rays(61, 4000, radius=3.0, spread=0.9))
    good, tree = (pot.Tree.from_scene(s, dtype=dtype) for s in (sc, sc.replace(sh=sh)))
    rgb, want = pot.render_rays(tree, o, d), pot.render_rays(good, o, d)
    assert torch.equal(rgb[:, 0], want[:, 0]) and torch.equal(rgb[:, 2], want[:, 2])
    shown = torch.isnan(rgb[:, 1])
    assert shown.any() and not shown.all() and torch.equal(rgb[~shown, 1], want[~shown, 1])
    pot.check()
