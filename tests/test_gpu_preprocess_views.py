"""A batch's views of one scene share a thread per Gaussian where the blocks fill whole waves (on 152
SMs 608 blocks each, 0.9 of one or two waves) and are worked through one by one where they do not:
either way every view's screen-space Gaussians are those of the frame alone, bit for bit, whatever
else is in the batch."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


def _scene(seed, n, deg, isotropic):
    from paper_2308_04079_gb300 import GaussianTensors
    g, _ = S.tiny_scene(seed, n=n, deg=deg, box=1.5)
    t = GaussianTensors.from_numpy(g).prepared()
    if isotropic:
        t = GaussianTensors(t.means, t.scales[:, 0].contiguous(), None, t.opacities, t.sh, deg)
    return t


def _state(fr):
    import torch
    n = fr.n
    st = fr.status()[1]
    return [st.num_visible, st.num_nonfinite] + [
        fr.view(k, torch.int32, c * n).clone() for k, c in
        (("xy", 4), ("depth", 1), ("conic_opacity", 4), ("rgb", 4), ("radius", 1), ("tau", 1))]


# 547 and 548, 608 and 609 blocks with the other scene's two
@pytest.mark.parametrize("isotropic", [False, True])
@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 700, 139_520, 139_521, 155_136, 155_137])
def test_views_equal_the_frames_alone(n, deg, isotropic):
    import torch
    from paper_2308_04079_gb300 import Frame, FrameBatch, make_config
    a, b = _scene(81, n, deg, isotropic), _scene(82, 300, deg, isotropic)
    a.means[n // 2] = float("nan")                       # culled and counted, in every view
    cams = [S.orbit_camera(3.0, 0.4 * v, 0.1 * v, 320 + 16 * v, 200) for v in range(4)]
    sets = [(a, cams[0]), (b, cams[1]), (a, cams[2]), (b, cams[0]), (a, cams[3])]
    cfg = make_config(isotropic=isotropic)
    frames = [Frame(g.n, c, cfg, capacity=1 << 16) for g, c in sets]
    FrameBatch(frames, [g for g, _ in sets]).preprocess()
    for fr, (g, c) in zip(frames, sets):
        alone = Frame(g.n, c, cfg, capacity=1 << 16)
        alone.preprocess(g)
        for x, y in zip(_state(fr), _state(alone)):
            assert torch.equal(x, y) if torch.is_tensor(x) else x == y
    assert frames[0].status()[1].num_nonfinite == 1
