"""The transfer backward's own paths: without shadows (a warp per receiver), and packet lists that are continued.

Against FP64: closed form of the unshadowed gradient, 1e-5 norm-wise; FP64 autograd of the oracle's transfer,
2e-3 norm-wise (the bar of test_gpu_transfer.py).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_03538_gb300 import api, scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,n,dirs", [(1, 1, 1), (3, 5, 33), (2, 130, 7), (5, 66, 64), (6, 3, 1024)])
def test_unshadowed_backward(order, n, dirs):
    """d n_i = sum over the directions above the horizon of w (dP_i . Y(w_s)) w_s; every other gradient 0. Sums of up
    to 1,024 FP32 terms, each a dot product of up to 49: a few hundred roundings of 6e-8 at most, below 1e-5."""
    sc, d = S.isotropic_scene(n, 900 + n), S.direction_set(dirs, 12)
    g = api.GaussianTensors.from_scene(sc)
    dP = np.random.default_rng(n).standard_normal((n, (order + 1) ** 2)).astype(np.float32)
    out = api.precompute_transfer_backward(g, api.build_bvh(g), torch.from_numpy(d).cuda(), order,
                                           torch.from_numpy(dP).cuda(), shadow=False)
    d64 = d.astype(np.float64)
    up = sc.normals.astype(np.float64) @ d64.T > 0
    G = np.where(up, 4 * np.pi / dirs * (dP.astype(np.float64) @ oracle.sh(order, d).T), 0.0)
    ref = G @ d64
    scale = max(np.linalg.norm(np.abs(G) @ np.abs(d64)), 1e-30)
    assert np.linalg.norm(out["d_normals"].cpu().double().numpy() - ref) <= 1e-5 * scale
    for f in ("means", "scales", "quats", "opacity"):
        assert not out["d_" + f].any()
