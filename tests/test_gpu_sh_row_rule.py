"""Which SH rows the per-Gaussian backward stages in shared memory: those of a single view that are
neither short, nor a multiple of four floats, nor longer than 48, unless the gradients are
accumulated.  On both sides of each line the gradients are those of the vector path on padded rows,
and a batch's are the sums over its views."""
import numpy as np
import pytest

import synthetic as S
from test_gpu_sh_rows import test_staged_rows_equal_vector_rows as _check_rows

pytestmark = pytest.mark.gpu


# rows of 9, 12, 15, 18, 36, 39, 45 and 48 floats
@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("deg,stride,shift", [(0, 3, 0), (1, 4, 3), (1, 5, 0), (0, 6, 1), (2, 12, 1), (2, 13, 0),
                                              (0, 15, 2), (2, 15, 0), (3, 16, 1)])
@pytest.mark.parametrize("n", [257, 700])
def test_rows_on_both_sides_of_the_rule(n, deg, stride, shift, accumulate):
    _check_rows(n, deg, stride, shift, False, accumulate)


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("deg,stride", [(0, 1), (1, 5), (2, 9), (2, 15)])
def test_a_batch_sums_its_views(deg, stride, accumulate):
    import torch
    from paper_2308_04079_gb300 import Frame, FrameBatch, GaussianTensors
    g, _ = S.tiny_scene(71, n=700, width=96, height=80, deg=deg)
    cams = [S.orbit_camera(3.0, 0.3 * v, 0.1, 96, 80) for v in range(3)]
    t = GaussianTensors.from_numpy(g).prepared()
    sh = torch.zeros(g.n, stride, 3, device="cuda")
    sh[:, : t.sh.shape[1]] = t.sh
    t = GaussianTensors(t.means, t.scales, t.quats, t.opacities, sh, deg)
    bg = (0.1, 0.2, 0.3)
    dl = [torch.from_numpy(S.upstream_grad(72 + v, 80, 96)).cuda() for v in range(3)]
    frames = [Frame(t.n, c, capacity=1 << 16) for c in cams]
    b = FrameBatch(frames, [t] * 3)
    b.ensure_binned()
    outs = b.outputs()
    b.render_forward(bg, outs)
    got, want = frames[0].new_grads(t), frames[0].new_grads(t)
    for v in (*got.values(), *want.values()):
        v.fill_(0.5)
    b.render_backward(bg, dl, outs, [got] * 3, accumulate)
    for v, f in enumerate(frames):
        f.render_backward(t, bg, dl[v], outs[v][1], outs[v][2], want, accumulate or v > 0)
    for k in got:
        x, w = got[k].double(), want[k].double()
        # three views' terms in another order, each view's own sums by atomics
        assert float(torch.linalg.norm(x - w)) <= 1e-5 * float(torch.linalg.norm(w)), k
    assert torch.equal(got["sh"][:, (deg + 1) ** 2:], want["sh"][:, (deg + 1) ** 2:])
