"""SH rows that are not whole 16-byte vectors (degrees 0 and 2, or a shifted buffer) go through
shared memory in the per-Gaussian backward: the gradients are those of the vector path on the
same rows padded to whole vectors, bit for bit (same accumulators, same arithmetic)."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("isotropic", [False, True])
@pytest.mark.parametrize("deg,stride,shift", [(0, 1, 0), (0, 1, 1), (2, 9, 0), (2, 9, 3), (1, 4, 1), (3, 16, 2), (2, 17, 0)])
@pytest.mark.parametrize("n", [1, 255, 257, 700])
def test_staged_rows_equal_vector_rows(n, deg, stride, shift, isotropic, accumulate):
    import torch
    from paper_2308_04079_gb300 import Frame, GaussianTensors, make_config
    g, cam = S.tiny_scene(60 + n, n=n, width=96, height=80, deg=deg)
    gt = GaussianTensors.from_numpy(g).prepared()
    if isotropic:
        gt = GaussianTensors(gt.means, gt.scales[:, 0].contiguous(), None, gt.opacities, gt.sh, deg)
    D = (deg + 1) ** 2

    def rows(width, offset):   # the same coefficients in rows of `width`, the buffer shifted by `offset` floats
        buf = torch.full((offset + n * width * 3,), 0.25, device="cuda")
        sh = buf[offset:].view(n, width, 3)
        sh[:, :D] = gt.sh
        return GaussianTensors(gt.means, gt.scales, gt.quats, gt.opacities, sh, deg)

    a, b = rows(stride, shift), rows(4 * ((stride + 3) // 4), 0)
    fr = Frame(n, cam, make_config(isotropic=isotropic))
    fr.ensure_binned(a)
    img, T, last = fr.outputs()
    fr.render_forward((0.0, 0.0, 0.0), img, T, last)
    d = torch.from_numpy(S.upstream_grad(61, cam.height, cam.width)).cuda()
    fr.render_backward_tiles((0.0, 0.0, 0.0), d, T, last)
    out = []
    for x in (a, b):
        grads = fr.new_grads(x)
        if x is a and shift:
            grads["sh"] = torch.empty(shift + x.sh.numel(), device="cuda")[shift:].view(x.sh.shape)
        for v in grads.values():
            if v is not None:
                v.fill_(0.5)
        fr.render_backward_gaussians(x, grads, accumulate)
        out.append(grads)
    for k in out[0]:
        if out[0][k] is None:
            continue
        p, q = (o[k].cpu().numpy() for o in out)
        if k == "sh":
            assert np.array_equal(p[:, :D], q[:, :D])
            assert np.all(p[:, D:] == (0.5 if accumulate else 0.0))
        else:
            assert np.array_equal(p, q), k
