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


FIELDS = ("means", "scales", "quats", "opacity", "normals")


def _crowd(n, seed, spread, opacity):
    sc = S.surface_scene(n, seed)
    sc.means *= np.float32(spread)
    sc.opacity *= np.float32(opacity)
    return sc


def _cutoff_bound(sc, dirs, G, t_min):
    """Largest change of every opacity gradient by the cut-off. A ray that ends below t_min takes the transmittance
    of its hits so far, less than t_min, for its own, and its later hits get nothing: either way each hit's
    |g| V / (1 - alpha) exp(-D^2 / 2) is off by at most |g| t_min / (1 - alpha)."""
    f64 = lambda a: torch.tensor(np.asarray(a, np.float64))
    mu, op = f64(sc.means), f64(sc.opacity)
    R = torch.tensor(oracle.quat_rot(sc.quats.astype(np.float64)))
    A = R.transpose(1, 2) / f64(sc.scales)[:, :, None]
    bound = torch.zeros(sc.n, dtype=torch.float64)
    for s, w in enumerate(dirs.astype(np.float64)):
        a = A @ torch.tensor(w)
        u = torch.einsum("jkl,ijl->ijk", A, mu[:, None] - mu[None])
        t = -(u * a).sum(-1) / (a * a).sum(-1)
        d2 = ((u + t[..., None] * a) ** 2).sum(-1)
        hit = (t > 0) & (d2 <= 9.0)
        hit.fill_diagonal_(False)
        al = op * torch.exp(-0.5 * d2)
        bound += (G[:, s, None].abs() * torch.where(hit, t_min / (1 - al), 0.0)).sum(0)
    return bound


@pytest.mark.parametrize("n,spread,opacity,dirs,t_min,continued", [
    (2600, 0.02, 0.02, 5, 0.0, True),      # lists of more than 2,048 leaves
    (2600, 0.02, 0.02, 5, 1e-5, True),     # ... and with rays that end at a cut-off
    (700, 0.2, 0.95, 9, 1e-3, False)])     # opaque splats, several windows, most rays end early
def test_lists_and_cutoff(n, spread, opacity, dirs, t_min, continued):
    """2e-3 norm-wise per field of FP64 autograd (which has no cut-off), and with a cut-off the opacity gradient
    within its bound besides. The counter of continued walks says that the lists overflow where they are meant to."""
    from oracle import transfer_torch as TT

    sc, d, order = _crowd(n, 43, spread, opacity), S.direction_set(dirs, 9), 1
    g = api.GaussianTensors.from_scene(sc)
    w = np.random.default_rng(n).standard_normal((n, 4)).astype(np.float32)
    stats = torch.zeros(10, dtype=torch.int64, device="cuda")
    out = api.precompute_transfer_backward(g, api.build_bvh(g), torch.from_numpy(d).cuda(), order,
                                           torch.from_numpy(w).cuda(), t_min=t_min, stats=stats)
    assert (int(stats[1]) > 0) == continued
    ps = [torch.tensor(np.asarray(getattr(sc, f), np.float64), requires_grad=True) for f in FIELDS]
    Y = oracle.sh(order, d)
    ref = dict(zip(FIELDS, torch.autograd.grad((TT.transfer_P(*ps, d, Y) * torch.tensor(w.astype(np.float64))).sum(), ps)))
    c = np.maximum(sc.normals.astype(np.float64) @ d.T.astype(np.float64), 0.0)
    G = torch.tensor(4 * np.pi / dirs * (w.astype(np.float64) @ Y.T) * c)
    bound = _cutoff_bound(sc, d, G, t_min)
    for f in FIELDS if t_min == 0.0 else ("opacity",):
        err = (out["d_" + f].cpu().double() - ref[f]).norm()
        assert float(err) <= 2e-3 * float(ref[f].norm()) + float(bound.norm() if f == "opacity" else 0.0), f


def test_second_batch_of_receivers():
    """More than 2^26 rays go in batches of receivers. Half of the directions at a time fits one batch, and the
    weights 4 pi / S make the whole the mean of its halves; the sums are atomic, 1e-5 norm-wise."""
    n, dirs = 66_000, 1024
    sc, d = S.isotropic_scene(n, 44), torch.from_numpy(S.direction_set(dirs, 13)).cuda()
    sc.scales *= np.float32(0.5)
    g = api.GaussianTensors.from_scene(sc)
    bvh = api.build_bvh(g)
    dP = torch.randn((n, 4), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    keep = torch.zeros(n, dtype=torch.bool, device="cuda")
    keep[bvh.view("order", torch.int32, (n,)).long()[torch.arange(60_000, n, 3, device="cuda")]] = True  # both batches
    dP = (dP * keep[:, None]).contiguous()
    whole = api.precompute_transfer_backward(g, bvh, d, 1, dP)
    parts = [api.precompute_transfer_backward(g, bvh, d[at].contiguous(), 1, dP) for at in (slice(0, 512), slice(512, 1024))]
    for f in ("means", "scales", "opacity", "normals"):  # (round splats: the rotation gradient is 0 but for rounding)
        ref = 0.5 * (parts[0]["d_" + f].double() + parts[1]["d_" + f].double())
        assert float((whole["d_" + f].double() - ref).norm()) <= 1e-5 * float(ref.norm()), f


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_normal_gradient_of_many_directions(seed):
    """512 directions of few hits each: a term g V w_s has some six roundings of 2^-25 on average, 2^-23 at most in
    all but rare terms, and sums over the directions keep that: 2^-23 norm-wise. A sum in 32 bits adds twice as much."""
    from oracle import transfer_torch as TT

    rng, n, dirs = np.random.default_rng(seed), 500, 512
    sc = S.isotropic_scene(n, 20 + seed)
    sc.means *= np.float32(3.0)
    sc.scales = (0.6 * sc.scales * np.exp(rng.normal(0, 0.3, sc.scales.shape))).astype(np.float32)
    d, w = S.direction_set(dirs, 3), rng.standard_normal((n, 9)).astype(np.float32)
    g = api.GaussianTensors.from_scene(sc)
    got = api.precompute_transfer_backward(g, api.build_bvh(g), torch.from_numpy(d).cuda(), 2,
                                           torch.from_numpy(w).cuda(), t_min=0.0)["d_normals"].cpu().double()
    f64 = [torch.tensor(np.asarray(getattr(sc, f), np.float64)) for f in FIELDS]
    V = TT.transfer_V(*f64, d).numpy()
    ref = torch.tensor((4 * np.pi / dirs * (w.astype(np.float64) @ oracle.sh(2, d).T) * V) @ d.astype(np.float64))
    assert float((got - ref).norm()) <= 2.0 ** -23 * float(ref.norm())
