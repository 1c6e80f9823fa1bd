"""Groups of one batch overlap on the GPU: what follows the call on its stream must still see every group's pixels,
also when a long group's last blocks outlive the short groups launched after it."""
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(640, 8), (640, 8, 8), (8, 640, 16), (24, 8, 640)])
def test_next_work_sees_all_groups(sizes):
    import torch
    import paper_2103_14024_gb300 as pot
    trees = [pot.Tree.from_scene(S.scene_random(30 + deg, 6, deg, p_occ=0.3, lo=(-1.5,) * 3, size=3.0, sigma_mu=0.0))
             for deg in range(len(sizes))]  # a group per SH degree, launched in this order
    cams = [S.make_cameras(S.hemisphere_c2ws(9 + k, 1), w, w, 1.4 * w) for k, w in enumerate(sizes)]
    want = [pot.render(t, c)[0] for t, c in zip(trees, cams)]
    outs = [torch.empty_like(w) for w in want]
    items = [(t, c[0], o, (0.0, 0.0, 0.0), 0.0, None) for t, c, o in zip(trees, cams, outs)]
    for _ in range(4):
        for o in outs:
            o.fill_(-1.0)
        pot.render_batch(items)
        seen = [o.clone() for o in outs]
        for o in outs:
            o.zero_()  # a late store of the batch would show in the next check
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(seen, want))
        assert all(not o.any() for o in outs)
    pot.check()
