"""pot_render_batch in a stream capture: the graph keeps the descriptors that its copy reads at each replay, for as
long as it lives, whatever the host's heap holds by then."""
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [(40,), (96, 24, 64), (16,) * 40])
def test_captured_batch_replays(widths):
    import torch
    import paper_2103_14024_gb300 as pot
    trees = [pot.Tree.from_scene(S.scene_random(30 + deg, 5, deg, p_occ=0.3, lo=(-1.5,) * 3, size=3.0, sigma_mu=1.0))
             for deg in range(3)]  # up to a group per SH degree
    cams = [S.make_cameras(S.hemisphere_c2ws(9 + k, 1), w, w, 1.4 * w) for k, w in enumerate(widths)]
    want = [pot.render(trees[k % 3], c)[0] for k, c in enumerate(cams)]
    outs = [torch.empty_like(w) for w in want]
    items = [(trees[k % 3], c[0], o, (0.0, 0.0, 0.0), 0.0, None) for k, (c, o) in enumerate(zip(cams, outs))]
    pot.render_batch(items)
    torch.cuda.synchronize()
    graphs = []
    for _ in range(2):
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1]):
            pot.render_batch(items)
    for step in range(6):
        # blocks of the descriptors' size, taken and filled in case they had been given back to the heap
        churn = [b"\xff" * (64 + 16 * k) for k in range(2000)]
        for o in outs:
            o.fill_(-1.0)
        graphs[step % len(graphs)].replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(outs, want))
        del churn
        if step == 3:
            del graphs[0]
    pot.check()
