"""Items of one batch whose outputs share memory: the groups write in their order (ascending SH degree here), also
when the first group's launch is long and the second one's short."""
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("as_t_final", [False, True])
@pytest.mark.parametrize("order", [(0, 1), (1, 0)])
def test_later_group_stands(order, as_t_final):
    import torch
    import paper_2103_14024_gb300 as pot
    sizes = (800, 8)
    trees = [pot.Tree.from_scene(S.scene_random(30 + deg, 6, deg, p_occ=0.3, lo=(-1.5,) * 3, size=3.0, sigma_mu=0.0))
             for deg in range(2)]
    cams = [S.make_cameras(S.hemisphere_c2ws(9 + k, 1), w, w, 1.4 * w) for k, w in enumerate(sizes)]
    large = pot.render(trees[0], cams[0])[0].reshape(-1)
    small, small_t = (x[0].reshape(-1) for x in pot.render(trees[1], cams[1], want_t_final=True))
    last = large.numel() - (small_t if as_t_final else small).numel()  # the pixels that the long group writes last
    want = large.clone()
    want[last:] = small_t if as_t_final else small
    buf, side = torch.empty_like(large), torch.empty_like(small)
    first = (trees[0], cams[0][0], buf, (0.0, 0.0, 0.0), 0.0, None)
    second = (trees[1], cams[1][0], side if as_t_final else buf[last:], (0.0, 0.0, 0.0), 0.0,
              buf[last:] if as_t_final else None)
    for _ in range(5):
        buf.fill_(-1.0)
        pot.render_batch([(first, second)[k] for k in order])
        assert torch.equal(buf, want)
    pot.check()
