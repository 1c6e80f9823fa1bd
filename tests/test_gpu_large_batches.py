"""Explicit-ray and filtering calls with more tiles than one wave of warps takes: warps draw tiles from a counter and
reuse their rows, stack and record blocks.  Compared with the same rays in calls that are one wave each, at sizes
around the lines between the two (16 warps per SM, 12 in the backward, 32 rays each) and well above them, ragged."""
import pytest

from paper_2103_14024_gb300 import synth as S

pytestmark = pytest.mark.gpu
RAYS = dict(bg=(0.2, 0.4, 0.6), gamma=1e-3, near=0.2, far=8.0)
PIECE = 30011


def _wave(torch, warps):
    return warps * torch.cuda.get_device_properties(0).multi_processor_count * 32


def _close(torch, a, b):
    """The bar of gradients, whose summation order varies: 1e-4 of the largest value."""
    assert float((a - b).abs().max()) <= 1e-4 * float(b.abs().max())


@pytest.mark.parametrize("cells", ["none", "brick", "dense"])
@pytest.mark.parametrize("warps,over", [(12, 0), (12, 1), (16, 0), (16, 1), (16, 31), (16, 22179)])
def test_rays_above_one_wave(cells, warps, over):
    import torch
    import paper_2103_14024_gb300 as pot
    n = _wave(torch, warps) + over
    tree = pot.Tree.from_scene(S.scene_random(91, 5, 3, p_occ=0.35, sigma_mu=1.5, sigma_s=1.0, sh_std=0.8))
    tree.set_cell_index(cells)
    o, d = (torch.from_numpy(a).cuda() for a in S.random_rays(91, n, radius=3.0, spread=0.9))
    gen = torch.Generator(device="cuda").manual_seed(n)
    grad, target = (torch.rand((n, 3), device="cuda", generator=gen) for _ in range(2))
    cuts = [(a, min(a + PIECE, n)) for a in range(0, n, PIECE)]
    want, want_t, want_g, want_m = [], [], None, None
    for a, b in cuts:
        rgb, t = pot.render_rays(tree, o[a:b], d[a:b], want_t_final=True, **RAYS)
        want.append(rgb)
        want_t.append(t)
        want_g = pot.render_backward(tree, o[a:b], d[a:b], grad[a:b], rgb_fwd=rgb,
                                     **({} if want_g is None else dict(grad_sigma=want_g[0], grad_sh=want_g[1])), **RAYS)
        mse = (rgb - target[a:b]) * (2.0 / (3 * n))
        want_m = pot.render_backward(tree, o[a:b], d[a:b], mse, rgb_fwd=rgb,
                                     **({} if want_m is None else dict(grad_sigma=want_m[0], grad_sh=want_m[1])), **RAYS)
    want, want_t = torch.cat(want), torch.cat(want_t)
    rgb, t = pot.render_rays(tree, o, d, want_t_final=True, **RAYS)
    assert torch.equal(rgb, want) and torch.equal(t, want_t)
    for fwd in (want, None):
        got = pot.render_backward(tree, o, d, grad, rgb_fwd=fwd, **RAYS)
        _close(torch, got[0], want_g[0])
        _close(torch, got[1], want_g[1])
    rgb = torch.empty_like(o)
    _, gs, gh = pot.render_mse_backward(tree, o, d, target, rgb=rgb, **RAYS)
    assert torch.equal(rgb, want)
    _close(torch, gs, want_m[0])
    _close(torch, gh, want_m[1])
    # records that fit, and a buffer that overflows into the walking backward
    for records in (pot.SegmentRecords.for_rays(n, 32), pot.SegmentRecords(40 * pot.SEGMENT_BLOCK)):
        rgb, t = pot.render_rays_record(tree, o, d, records, want_t_final=True, **RAYS)
        assert torch.equal(rgb, want) and torch.equal(t, want_t)
        assert records.overflowed() == (records.capacity == 40 * pot.SEGMENT_BLOCK)
        got = pot.render_backward_recorded(tree, o, d, grad, rgb, records, **RAYS)
        _close(torch, got[0], want_g[0])
        _close(torch, got[1], want_g[1])
    pot.check()
    tree.free()


@pytest.mark.parametrize("cells", ["none", "brick", "dense"])
def test_filter_above_one_wave(cells):
    import torch
    import paper_2103_14024_gb300 as pot
    tree = pot.Tree.from_scene(S.scene_random(92, 6, 1, p_occ=0.3, lo=(-1.5,) * 3, size=3.0, sigma_mu=1.0))
    tree.set_cell_index(cells)
    views = S.make_cameras(S.hemisphere_c2ws(5, 3), 401, 400, 560.0)
    got = pot.visibility(tree, views)
    want = torch.zeros_like(got)
    for i in range(3):
        small = views[i:i + 1].copy()
        for row in range(0, 400, 100):  # 100 rows at a time: one wave each, the same pixels by a shifted centre
            part = small.copy()
            part["height"], part["cy"] = 100, small["cy"] - row
            pot.visibility(tree, part, max_weight=want)
    assert torch.equal(got, want)
    pot.check()
    tree.free()
