"""The loss of pot_render_mse_backward against its own colours in float64: split tiles (1,000 rays), whole tiles
(20,011, 77,824) and tiles drawn from a counter (100,003 and 2^18 rays).  A ray's error is 3 squares summed in float
and a warp's 32 are summed by 5 shuffles, at most 11 roundings of 2^-24 with the last one of the result; the rest of
the sum adds nothing to that, whatever the number of rays."""
import numpy as np
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu
BOUND = 11 * 2.0 ** -24


@pytest.mark.parametrize("n", [1, 1000, 20011, 77824, 100003, 1 << 18])
@pytest.mark.parametrize("leaves", [False, True])
def test_fused_loss_does_not_drift(n, leaves):
    import torch
    import paper_2103_14024_gb300 as pot
    sc = S.scene_random(71, 5, 2, p_occ=0.35, sigma_mu=1.5, sigma_s=1.0, sh_std=0.8)
    if not leaves:  # every warp adds the same value, whose rounding errors then add up too
        sc = sc.replace(morton=sc.morton[:0], sigma=sc.sigma[:0], sh=sc.sh[:0])
    tree = pot.Tree.from_scene(sc)
    o, d = S.random_rays(71, n, radius=3.0, spread=0.9)
    target = np.random.default_rng(n).uniform(size=(n, 3)) if leaves else np.full((n, 3), 0.37)
    o, d, target = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (o, d, target))
    rgb = torch.empty_like(o)
    loss = torch.full((1,), -1.0, device="cuda")
    for _ in range(2):  # the sum starts anew at each call
        pot.render_mse_backward(tree, o, d, target, rgb=rgb, loss=loss, bg=(0.1, 0.2, 0.9))
        want = float(((rgb.double() - target.double()) ** 2).mean())
        assert abs(float(loss) - want) <= BOUND * want
    pot.check()
