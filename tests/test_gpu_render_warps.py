"""The groups of a render warp work together in ways that depend on the frame: they take the careful
path of the blend as one, their gradient sums are added as one where they walk the same splats, and
their pixels are loaded and stored in an order that follows the image's width and the buffers'
alignment.  None of it changes what a pixel or a Gaussian gets."""
import numpy as np
import pytest

import oracle
import synthetic as S
from test_gpu_backward import _check

pytestmark = pytest.mark.gpu

# 4, 8 pixels per lane in the backward pass: between 3,000 and 16,000 sub-blocks of 8x8, and above
SIZES = [(640, 480), (1920, 1080)]
TILES = [(16, 16), (16, 8), (8, 8)]


def _ocfg(tile):
    return oracle.cfg_array(tile_w=tile[0], tile_h=tile[1])


# ---- the order in which a lane's pixels are loaded and stored ----

def _pass(g, cam, companion, shift, grad_limit):
    """Outputs and gradients with every buffer `shift` words past an aligned address, in guard words."""
    import torch
    from paper_2308_04079_gb300 import Frame, FrameBatch, GaussianTensors, make_config
    e, ecam = S.tiny_scene(32, n=3, width=max(companion, 8), height=1024, deg=2)
    cfg = make_config(grad_limit=grad_limit)
    sets = [(g, cam)] + ([(e, ecam)] if companion else [])
    gts = [GaussianTensors.from_numpy(x).prepared() for x, _ in sets]
    frames = [Frame(t.n, c, cfg, capacity=1 << 17) for t, (_, c) in zip(gts, sets)]
    b = FrameBatch(frames, gts)
    b.ensure_binned()
    guards = []

    def shifted(n, dtype, data=None):
        raw = torch.full((n + 16,), 77, dtype=dtype, device="cuda")
        guards.append((raw, shift, n))
        v = raw[shift:shift + n]
        assert v.data_ptr() % 16 == 4 * shift
        if data is not None:
            v.copy_(torch.from_numpy(np.ascontiguousarray(data).reshape(-1)))
        return v

    outs, dl = [], []
    for i, (_, c) in enumerate(sets):
        P = c.width * c.height
        outs.append((shifted(3 * P, torch.float32), shifted(P, torch.float32), shifted(P, torch.int32)))
        dl.append(shifted(3 * P, torch.float32, S.upstream_grad(33 + i, c.height, c.width)))
    b.render_forward((0.1, 0.2, 0.3), outs)
    grads = [f.new_grads(t) for f, t in zip(frames, gts)]
    b.render_backward((0.1, 0.2, 0.3), dl, outs, grads)
    pairs = frames[0].status()[1].blended_pairs
    for raw, s, n in guards:
        assert torch.all(raw[:s] == 77) and torch.all(raw[s + n:] == 77)
    return [o.cpu().numpy() for o in outs[0]], {k: v.cpu().numpy().astype(np.float64) for k, v in grads[0].items()}, pairs


# companions (1024 rows high) that bring the launch to 4 and 8 pixels per lane in both passes
@pytest.mark.parametrize("grad_limit", [0, 3])
@pytest.mark.parametrize("width", [1, 7, 8, 9, 202, 203, 204, 208])
def test_widths_and_alignments_change_nothing(width, grad_limit):
    g, cam = S.tiny_scene(41, n=400, width=width, height=45, deg=1, log_scale_mean=-2.8, opacity_logit_std=3.0)
    want, wgrads, wpairs = _pass(g, cam, 0, 0, grad_limit)
    for companion, shift in [(0, 1), (0, 2), (880, 0), (880, 1), (880, 2), (2304, 0), (2304, 1), (2304, 2), (2304, 3)]:
        groups = companion // 8 * 128 + (width + 15) // 16 * 2 * 3 * 2
        if companion:
            assert 12000 <= groups < 16000 if companion == 880 else groups >= 26000
        got, grads, pairs = _pass(g, cam, companion, shift, grad_limit)
        for a, w in zip(got, want):
            assert np.array_equal(a, w), (companion, shift)
        assert pairs == wpairs
        for k, w in wgrads.items():
            # the same terms summed in another order: fp32 sums of up to ~1e4 terms of both signs
            assert np.linalg.norm(grads[k] - w) <= 1e-5 * max(np.linalg.norm(w), 1e-30), (companion, shift, k)


# ---- groups that walk the same splats add as one ----

@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("W,H", SIZES)
def test_splats_that_cover_every_sub_block(W, H, tile):
    """Forty splats larger than the frame: every group of every warp walks the same positions, over a
    full window of 32 and a partial one."""
    from paper_2308_04079_gb300 import make_config
    g, cam = S.tiny_scene(42, n=40, width=W, height=H, deg=1, log_scale_mean=0.7, log_scale_std=0.2)
    g.opacities = (np.asarray(g.opacities) * 0.2).astype(np.float32)
    _check(g, cam, (0.1, 0.3, 0.2), S.upstream_grad(43, H, W), cfg=make_config(tile=tile), ocfg=_ocfg(tile),
           label=f"frame-filling {W}x{H} {tile[0]}x{tile[1]}")


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("W,H", SIZES)
def test_tiles_with_a_splat_each(W, H, tile):
    """One splat in the middle of every tile, within the tile: the groups of a warp that holds several
    tiles walk the same positions of their lists, which name different splats."""
    from paper_2308_04079_gb300 import make_config
    tw, th = tile
    TX, TY = W // tw, H // th
    x, y = (v.reshape(-1) for v in np.meshgrid((np.arange(TX) + 0.5) * tw, (np.arange(TY) + 0.5) * th))
    n = x.size
    rng = np.random.default_rng(44)
    z = rng.uniform(1.0, 3.0, n)
    f = float(W)
    quats = rng.normal(size=(n, 4))
    g = S.Gaussians(means=np.stack([(x - W / 2) / f * z, (y - H / 2) / f * z, z], 1).astype(np.float32),
                    scales=(rng.uniform(0.1, 0.7, (n, 3)) * z[:, None] / f).astype(np.float32),
                    quats=(quats / np.linalg.norm(quats, axis=1, keepdims=True)).astype(np.float32),
                    opacities=rng.uniform(0.1, 0.95, n).astype(np.float32),
                    sh=rng.normal(0.5, 0.2, (n, 1, 3)).astype(np.float32), sh_degree=0)
    cam = S.Camera(W, H, f, f, W / 2, H / 2, np.eye(3, dtype=np.float32), np.zeros(3, np.float32))
    _check(g, cam, (0.0, 0.0, 0.0), S.upstream_grad(45, H, W), cfg=make_config(tile=tile), ocfg=_ocfg(tile),
           label=f"a splat per tile {W}x{H} {tw}x{th}")
