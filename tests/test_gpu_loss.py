"""The losses of pot_render_mse_backward and pot_loss_mse against the colours they are of in float64: split tiles
(1,000 rays), whole tiles (20,011), tiles drawn from a counter (77,824 rays and more), and one to several values per
thread.  A ray's error is 3 squares summed in float (a thread's up to 3) and a warp's 32 are summed by 5 shuffles, at
most 11 roundings of 2^-24 with the last one of the result; the rest of the sum adds nothing to that, whatever the
number of rays."""
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


@pytest.mark.parametrize("n", [1, 1000, 20011, 200003, 1 << 20])
def test_loss_mse_does_not_drift(n):
    import torch
    import paper_2103_14024_gb300 as pot
    gen = torch.Generator(device="cuda").manual_seed(n)
    loss = torch.full((1,), -1.0, device="cuda")
    for rgb, target in ((torch.rand((n, 3), device="cuda", generator=gen), torch.rand((n, 3), device="cuda", generator=gen)),
                        (torch.full((n, 3), 0.1, device="cuda"), torch.full((n, 3), 0.37, device="cuda"))):
        want = float(((rgb.double() - target.double()) ** 2).mean())
        for _ in range(2):
            loss, grad = pot.loss_mse(rgb, target)
            assert abs(float(loss) - want) <= BOUND * want
            assert torch.allclose(grad, 2.0 / (3 * n) * (rgb - target), rtol=1e-6, atol=0.0)
    loss, _ = pot.loss_mse(rgb[:0], target[:0], grad=torch.empty((0, 3), device="cuda"))
    assert float(loss) == 0.0
