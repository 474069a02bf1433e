"""Values so large that a product overflows stay with the pixels that blend the splat.  In the
backward pass the lanes of a group run through a splat together, also those whose pixel does not
blend it: whatever the magnitude of a colour, a dL/dimage or a conic, these add nothing to the splat
and keep their own recurrence."""
from types import SimpleNamespace

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

C0 = 0.28209479177387814      # the constant SH basis function
# width of a 1024-pixel-high companion frame that brings the batch to 2, 4 or 8 pixels per lane in
# the backward pass: its 8x8 sub-blocks and the 64 of the tested frame lie below 3,000, between
# 3,000 and 16,000, above 16,000
COMPANIONS = (0, 512, 2304)
# two splats within one 8x8 sub-block, the second in front: each covers the 3x3 pixels around its own
AT = ((18, 18), (22, 22))


def _camera(width, height, cx, cy):
    return SimpleNamespace(width=width, height=height, fx=64.0, fy=64.0, cx=cx, cy=cy, R=np.eye(3), t=np.zeros(3),
                           near=0.2)


def _gaussians(colours):
    z = np.array([2.0, 1.0])[: len(colours)]
    uv = np.array(AT, np.float64)[: len(colours)] + 0.5
    means = np.stack([(uv[:, 0] - 32) / 64 * z, (uv[:, 1] - 32) / 64 * z, z], 1)
    n = len(colours)
    return SimpleNamespace(means=means, scales=np.repeat(0.002 * z[:, None], 3, 1), quats=np.tile([1.0, 0, 0, 0], (n, 1)),
                           opacities=np.full(n, 0.9), sh=np.array(colours)[:, None, None] / C0 * np.ones((1, 1, 3)),
                           sh_degree=0)


def _batch(g, companion, grad_limit=0, **cfg):
    from paper_2308_04079_gb300 import Frame, FrameBatch, GaussianTensors, make_config
    sets = [(g, _camera(64, 64, 32.0, 32.0))]
    if companion:
        e, ecam = S.tiny_scene(35, n=3, width=companion, height=1024, deg=0)
        sets.append((e, ecam))
        groups = 64 + companion // 8 * 128
        assert (groups < 16000) == (companion == 512) and groups >= 3000
    gts = [GaussianTensors.from_numpy(x).prepared() for x, _ in sets]
    frames = [Frame(t.n, c, make_config(grad_limit=grad_limit, **cfg), capacity=1 << 16)
              for t, (_, c) in zip(gts, sets)]
    b = FrameBatch(frames, gts)
    b.ensure_binned()
    outs = b.outputs()
    b.render_forward((0.0, 0.0, 0.0), outs)
    return b, outs


def _run(colours, dl_back, dl_front, companion, grad_limit):
    """Gradients with dL/dimage = dl_back on the pixels of the first splat, dl_front elsewhere."""
    import torch
    b, outs = _batch(_gaussians(colours), companion, grad_limit)
    covered = outs[0][2].cpu().numpy() > 0
    back, front = np.zeros((64, 64), bool), np.zeros((64, 64), bool)
    for m, (x, y) in zip((back, front), AT):
        m[y - 1:y + 2, x - 1:x + 2] = True
    assert np.array_equal(covered, back | front) and not (back & front).any()
    dl = [torch.zeros_like(o[0]) for o in outs]
    dl[0].copy_(torch.from_numpy(np.where(back, np.float32(dl_back), np.float32(dl_front))))
    grads = [f.new_grads(t) for f, t in zip(b.frames, b.gaussians)]
    b.render_backward((0.0, 0.0, 0.0), dl, outs, grads)
    return {k: v.cpu().numpy() for k, v in grads[0].items()}


def _same(got, want, row):
    # the same products and sums up to the path chosen for the splat: a few roundings of nine terms
    for k in want:
        assert np.all(np.isfinite(want[k][row])) and np.all(np.isfinite(got[k][row])), k
        assert np.allclose(got[k][row], want[k][row], rtol=1e-5, atol=1e-5 * np.abs(want[k][row]).max()), k
    assert np.any(want["opacities"][row] != 0)


@pytest.mark.parametrize("companion", COMPANIONS)
@pytest.mark.parametrize("grad_limit", [0, 3])
@pytest.mark.parametrize("colour,dl", [(1e25, 1e25), (1e35, 1e10), (1e29, 1e29), (1e17, 1e22)])
def test_a_wild_colour_leaves_the_pixels_that_do_not_blend_it(colour, dl, grad_limit, companion):
    got = _run((colour, 0.5), 0.0, dl, companion, grad_limit)
    want = _run((1.0, 0.5), 0.0, dl, companion, grad_limit)
    _same(got, want, 1)
    assert all(np.all(v[0] == 0) for v in got.values())    # its own pixels have no gradient


@pytest.mark.parametrize("companion", COMPANIONS)
@pytest.mark.parametrize("grad_limit", [0, 3])
@pytest.mark.parametrize("colour,dl", [(1e25, 1e25), (1e17, 1e22), (1e22, 1e17)])
def test_a_wild_splat_gets_nothing_from_the_pixels_that_do_not_blend_it(colour, dl, grad_limit, companion):
    got = _run((colour, 0.5), 1.0, dl, companion, grad_limit)
    want = _run((colour, 0.5), 1.0, 1.0, companion, grad_limit)
    _same(got, want, 0)


@pytest.mark.parametrize("companion", COMPANIONS)
def test_an_infinite_conic_leaves_its_sums_finite(companion):
    """Without dilation, a splat 2e-21 pixels wide: its conic's factor is infinite, so the form is
    infinite or not a number at every pixel.  The former are skipped and add nothing; the latter blend
    with the clamped alpha, which has a colour gradient only."""
    import torch
    g = _gaussians((1.0,))
    g.means = np.array([[0.0, 0.0, 1.0]])
    g.scales = np.array([[3e-23, 1e-2, 1e-2]])
    b, outs = _batch(g, companion, dilation=0.0, tile_rule="rect")
    fr = b.frames[0]
    fr.set_camera(_camera(64, 64, 17.5, 17.5))
    b.ensure_binned()
    b.render_forward((0.0, 0.0, 0.0), outs)
    assert np.isinf(fr.view("conic_opacity", torch.float32, 4).cpu().numpy()[0])
    last = outs[0][2].cpu().numpy()[16:24, 16:24]
    assert np.any(last > 0) and np.any(last == 0)          # some pixels of its sub-block blend it
    grads = [f.new_grads(t) for f, t in zip(b.frames, b.gaussians)]
    b.render_backward((0.0, 0.0, 0.0), [torch.ones_like(o[0]) for o in outs], outs, grads)
    sums = fr.view("grad2d", torch.float32, 12).cpu().numpy()[:9]
    assert np.all(sums[:6] == 0) and np.all(np.isfinite(sums[6:])) and np.all(sums[6:] != 0)
