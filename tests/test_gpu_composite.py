"""The rasteriser's forward and backward at the sizes where its warps, groups and lists have edges:
colour groups that are full, one over and one short, images that end inside a tile and inside a warp's
pixels, lists longer than one group of splats, needle-thin splats, and splats behind opaque ones.

Against FP64 autograd of the oracle's renderer: PSNR >= 50 dB and 2e-3 norm-wise per gradient, the
bars of test_gpu_render.py.
"""
import numpy as np
import pytest
import torch

from oracle import render as OR
from paper_2408_03538_gb300 import api, scenes as S

pytestmark = pytest.mark.gpu


def _check(sc, cam, k, bg):
    rng = np.random.default_rng(k)
    colors = rng.uniform(0, 1, (k, sc.n, 3)).astype(np.float32)
    dimg = rng.standard_normal((k, 3, cam.height, cam.width)).astype(np.float32)
    g = api.GaussianTensors.from_scene(sc)
    col, bgd = torch.from_numpy(colors).cuda(), torch.tensor(bg, dtype=torch.float32, device="cuda")
    st = api.Status()
    img, state = api.render(g, col, cam, bgd, status=st, max_pairs=400_000)
    got = api.render_backward(g, col, cam, bgd, state, torch.from_numpy(dimg).cuda())
    torch.cuda.synchronize()
    assert st.read() == 0
    ps = [torch.tensor(np.asarray(a, np.float64), requires_grad=True)
          for a in (sc.means, sc.scales, sc.quats, sc.opacity, colors)]
    ref = OR.render(*ps, cam, bg=bg)
    assert OR.psnr(img.cpu().numpy(), ref.detach().numpy(), peak=1.0) >= 50.0
    grads = torch.autograd.grad((ref * torch.tensor(dimg, dtype=torch.float64)).sum(), ps)
    for a, r, name in zip(got, grads, ("means", "scales", "quats", "opacity", "colors")):
        assert float((a.cpu().double() - r).norm()) <= 2e-3 * float(r.norm()), name


@pytest.mark.parametrize("k", [1, 2, 4, 5, 8, 9, 17])
def test_composite_color_groups(k):
    sc = S.surface_scene(700, 60 + k)
    sc.means *= 0.4
    _check(sc, S.look_at_camera((0, -4.0, 2.0), (0, 0, 0.2), 40, 61, 45), k, (0.2, 0.1, 0.3))


@pytest.mark.parametrize("w,h", [(1, 1), (16, 16), (17, 4), (9, 33), (40, 31)])
def test_composite_image_edges(w, h):
    sc = S.surface_scene(400, 70)
    sc.means *= 0.4
    _check(sc, S.look_at_camera((0, -3.0, 1.5), (0, 0, 0.2), 40, w, h), 3, (0.0, 0.0, 0.0))


@pytest.mark.parametrize("thin,opacity", [(1.0, 0.05), (100.0, 0.5), (1.0, 1.5)])
def test_composite_thin_faint_and_opaque_splats(thin, opacity):
    sc = S.surface_scene(900, 71)
    sc.means *= 0.25
    sc.scales[:, 0] /= np.float32(thin)
    sc.opacity = np.minimum(sc.opacity * np.float32(opacity), np.float32(0.995))
    _check(sc, S.look_at_camera((0, -3.0, 1.5), (0, 0, 0.2), 45, 48, 40), 2, (0.5, 0.5, 0.5))
