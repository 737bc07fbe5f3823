"""Gradients whose lower moments cancel exactly, so that only the second moments are left: a splat seen by four
pixels at its corners whose image gradients alternate in sign turns, and neither moves nor grows.

Against FP64 autograd of the oracle, 2e-3 norm-wise (the bar of test_gpu_render.py).
"""
import numpy as np
import pytest
import torch

from oracle import render as OR
from paper_2408_03538_gb300 import api, scenes as S

pytestmark = pytest.mark.gpu


def quadrupole_frame(k):
    """One splat, wider than high, centred on pixel (4, 1); +1 and -1 alternate at the four pixels diagonal to it."""
    sc = S.isotropic_scene(1, 3)
    sc.means[:] = (0.0, 0.0, 2.0)
    sc.scales[:] = (0.5, 0.3, 0.4)
    sc.quats[:] = (1.0, 0.0, 0.0, 0.0)
    sc.opacity[:] = 0.5
    cam = S.Camera(rot=np.eye(3, dtype=np.float32), trans=np.zeros(3, np.float32), fx=8.0, fy=8.0, cx=4.0, cy=1.0,
                   width=16, height=8, position=np.zeros(3, np.float32))
    dimg = np.zeros((k, 3, 8, 16), np.float32)
    for x, y, v in ((3, 0, 1.0), (5, 0, -1.0), (3, 2, -1.0), (5, 2, 1.0)):
        dimg[:, :, y, x] = v
    return sc, cam, np.ones((k, 1, 3), np.float32), dimg


@pytest.mark.parametrize("k", [1, 2, 9])
def test_render_backward_keeps_second_moments(k):
    sc, cam, colors, dimg = quadrupole_frame(k)
    g = api.GaussianTensors.from_scene(sc)
    col, bg = torch.from_numpy(colors).cuda(), torch.zeros(3, device="cuda")
    _, state = api.render(g, col, cam, bg, max_pairs=64)
    dq = api.render_backward(g, col, cam, bg, state, torch.from_numpy(dimg).cuda())[2].cpu().double()
    ps = [torch.tensor(np.asarray(a, np.float64), requires_grad=True)
          for a in (sc.means, sc.scales, sc.quats, sc.opacity, colors)]
    ref = torch.autograd.grad((OR.render(*ps, cam, bg=(0.0, 0.0, 0.0)) * torch.tensor(dimg, dtype=torch.float64)).sum(),
                              ps[2])[0]
    assert float(ref.norm()) > 0.1 * k
    assert float((dq - ref).norm()) <= 2e-3 * float(ref.norm())
