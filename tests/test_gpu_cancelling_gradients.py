"""Gradients whose lower moments cancel exactly, so that only the second moments are left: a splat seen by four
pixels at its corners whose image gradients alternate in sign turns, and neither moves nor grows; so does an
occluder met by four parallel rays whose gradients alternate.

Against FP64 autograd of the oracle, 2e-3 norm-wise (the bar of test_gpu_render.py).
"""
import numpy as np
import pytest
import torch

import oracle
from oracle import render as OR, transfer_torch as TT
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


def quadrupole_rays():
    """An occluder, wider than deep, and four receivers below its corners that look up along z: the gradients of their
    first coefficients alternate in sign."""
    sc = S.isotropic_scene(5, 4)
    sc.means[0] = 0.0
    sc.means[1:] = [(x, y, -2.0) for x in (-0.25, 0.25) for y in (-0.125, 0.125)]
    sc.scales[0] = (0.5, 0.25, 0.5)
    sc.scales[1:] = 0.03125
    sc.quats[:] = (1.0, 0.0, 0.0, 0.0)
    sc.opacity[:] = (0.5, 0.25, 0.25, 0.25, 0.25)
    sc.normals[0] = (0.0, 0.0, -1.0)
    sc.normals[1:] = (0.0, 0.0, 1.0)
    dP = np.zeros((5, 4), np.float32)
    dP[1:, 0] = (1.0, -1.0, -1.0, 1.0)
    return sc, np.array([[0.0, 0.0, 1.0]], np.float32), dP


def test_transfer_backward_keeps_second_moments():
    sc, dirs, dP = quadrupole_rays()
    g = api.GaussianTensors.from_scene(sc)
    out = api.precompute_transfer_backward(g, api.build_bvh(g), torch.from_numpy(dirs).cuda(), 1,
                                           torch.from_numpy(dP).cuda(), t_min=0.0)
    ps = [torch.tensor(np.asarray(getattr(sc, f), np.float64), requires_grad=True)
          for f in ("means", "scales", "quats", "opacity", "normals")]
    P = TT.transfer_P(*ps, dirs, oracle.sh(1, dirs))
    ref = torch.autograd.grad((P * torch.as_tensor(dP.astype(np.float64))).sum(), ps)[2]
    assert float(ref.norm()) > 0.1
    assert float((out["d_quats"].cpu().double() - ref).norm()) <= 2e-3 * float(ref.norm())
