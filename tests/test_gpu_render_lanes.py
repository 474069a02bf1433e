"""The render kernels give a lane 2, 4 or 8 pixels by the number of sub-blocks of the launch: the
choice changes how work is laid out, never what a pixel computes."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

# width of a 1024-pixel-high, nearly empty companion frame that brings a batch into each class
# (sub-blocks are 8x8 pixels): nothing, forward 2 / backward 4, forward 4 / backward 4 pixels per
# lane, forward 4 / backward 8, forward 8 / backward 8
COMPANIONS = (0, 512, 1008, 1200, 2304)


def _run(tile, grad_limit, companion):
    import torch
    from paper_2308_04079_gb300 import Frame, FrameBatch, GaussianTensors, make_config
    g, cam = S.tiny_scene(31, n=900, width=203, height=117, deg=2, log_scale_mean=-2.8, opacity_logit_std=3.0)
    e, ecam = S.tiny_scene(32, n=3, width=max(companion, 8), height=1024, deg=2)
    cfg = make_config(tile=tile, grad_limit=grad_limit)
    sets = [(g, cam)] + ([(e, ecam)] if companion else [])
    gts = [GaussianTensors.from_numpy(x).prepared() for x, _ in sets]
    frames = [Frame(t.n, c, cfg, capacity=1 << 17) for t, (_, c) in zip(gts, sets)]
    b = FrameBatch(frames, gts)
    b.ensure_binned()
    outs = b.outputs()
    b.render_forward((0.1, 0.2, 0.3), outs)
    dl = [torch.from_numpy(S.upstream_grad(33 + i, c.height, c.width)).cuda() for i, (_, c) in enumerate(sets)]
    grads = [f.new_grads(t) for f, t in zip(frames, gts)]
    b.render_backward((0.1, 0.2, 0.3), dl, outs, grads)
    pairs = frames[0].status()[1].blended_pairs
    return [o.cpu().numpy() for o in outs[0]], {k: v.cpu().numpy().astype(np.float64) for k, v in grads[0].items()}, pairs


@pytest.mark.parametrize("tile", [(16, 16), (16, 8), (8, 8)])
@pytest.mark.parametrize("grad_limit", [0, 3])
def test_pixels_per_lane_change_nothing(tile, grad_limit):
    want, wgrads, wpairs = _run(tile, grad_limit, 0)
    assert wpairs > 0
    for companion in COMPANIONS[1:]:
        got, grads, pairs = _run(tile, grad_limit, companion)
        for a, b in zip(got, want):
            assert np.array_equal(a, b), companion
        assert pairs == wpairs
        for k, w in wgrads.items():
            # the same terms summed in another order: fp32 sums of up to ~1e3 terms
            assert np.linalg.norm(grads[k] - w) <= 1e-5 * np.linalg.norm(w), (companion, k)


@pytest.mark.parametrize("companion", COMPANIONS)
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_a_pixel_without_a_finite_gradient_spoils_only_what_it_blends(bad, companion):
    import torch
    from paper_2308_04079_gb300 import Frame, FrameBatch, GaussianTensors, make_config
    g, cam = S.tiny_scene(34, n=40, width=64, height=64, deg=0, log_scale_mean=-4.0, log_scale_std=0.2)
    e, ecam = S.tiny_scene(35, n=3, width=max(companion, 8), height=1024, deg=0)
    sets = [(g, cam)] + ([(e, ecam)] if companion else [])
    gts = [GaussianTensors.from_numpy(x).prepared() for x, _ in sets]
    frames = [Frame(t.n, c, make_config(), capacity=1 << 16) for t, (_, c) in zip(gts, sets)]
    b = FrameBatch(frames, gts)
    b.ensure_binned()
    outs = b.outputs()
    b.render_forward((0.0, 0.0, 0.0), outs)
    base = [torch.from_numpy(S.upstream_grad(36, c.height, c.width)).cuda() for _, c in sets]
    res = []
    for value in (0.0, bad):
        dl = [d.clone() for d in base]
        dl[0][:, 30, 33] = value
        grads = [f.new_grads(t) for f, t in zip(frames, gts)]
        b.render_backward((0.0, 0.0, 0.0), dl, outs, grads)
        res.append(grads[0]["opacities"].cpu().numpy())
    hit = ~np.isfinite(res[1])
    assert hit.sum() < 40 // 2
    clean = ~hit
    assert np.allclose(res[1][clean], res[0][clean], rtol=1e-4, atol=1e-5 * np.abs(res[0]).max())
