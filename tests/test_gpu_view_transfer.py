"""The view transfer and its gradient at the edges of its direction chunks (32 at a time, four read ahead) and of its
SH rows (1 to 13 words of four), up to the largest direction set, against the FP64 oracle on the same visibility.

Tolerances as in test_gpu_training.py: 2e-4 norm-wise per receiver + 1e-6; gradients 2e-4 of the largest.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_03538_gb300 import api, scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2, 3, 4, 6])
@pytest.mark.parametrize("n_dirs", [1, 31, 33, 128, 129, 161, 1024])
def test_view_transfer_direction_chunks(order, n_dirs):
    rng = np.random.default_rng(1000 * order + n_dirs)
    sc = S.surface_scene(75, 30 + order)
    sc.roughness = rng.uniform(0.15, 1.0, sc.n).astype(np.float32)
    sc.metallic = rng.uniform(0.0, 1.0, sc.n).astype(np.float32)
    dirs = S.direction_set(n_dirs, 11)
    V = (rng.uniform(0, 1, (sc.n, n_dirs)) * (rng.uniform(0, 1, (sc.n, n_dirs)) < 0.8)).astype(np.float32)
    cam = (0.7, -4.0, 6.2)
    g, d = api.GaussianTensors.from_scene(sc), torch.from_numpy(dirs).cuda()
    Vd, C = torch.from_numpy(V).cuda(), (order + 1) ** 2
    dt = rng.normal(size=(sc.n, C)).astype(np.float32)
    t = api.training_transfer(g, Vd, d, order, cam).cpu().numpy()
    dr, dm = api.training_transfer_backward(g, Vd, d, order, cam, torch.from_numpy(dt).cuda())
    args = (sc, dirs, order, np.arange(sc.n), V.astype(np.float64), np.asarray(cam, np.float32))
    ref = oracle.training_transfer(*args)
    assert np.all(np.linalg.norm(t - ref, axis=1) <= 2e-4 * np.linalg.norm(ref, axis=1) + 1e-6)
    gr, gm = oracle.training_transfer_grad(*args, dt)
    for got, want in ((dr, gr), (dm, gm)):
        assert np.all(np.abs(got.cpu().numpy() - want) <= 2e-4 * np.abs(want).max() + 2e-4 * np.abs(want))
