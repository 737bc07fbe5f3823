"""The packet walk's staging, quick test and index search at the sizes where they can go wrong: windows
and packets that are just full or one over, several scenes inside a window, needle-thin splats (the
quick test's margin), many hits on a ray (more rounds than one buffer holds).

Tolerances as in test_gpu_transfer.py: 1e-4 norm-wise per receiver plus the oracle's allowance; the
index matrix bit-exact on unflagged rays.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2408_03538_gb300 import api, scenes as S

pytestmark = pytest.mark.gpu


def _check(sc, offs, dirs, order, sizes):
    g = api.GaussianTensors.from_scene(sc)
    st = api.Status()
    bvh = api.build_bvh(g, torch.from_numpy(offs).cuda(), status=st)
    d = torch.from_numpy(dirs).cuda()
    out = api.precompute_transfer(g, bvh, d, order, bounce=True, status=st)
    P0 = api.precompute_transfer(g, bvh, d, order, status=st)["P"]
    torch.cuda.synchronize()
    assert st.read() == 0
    floor = 1e-3 * oracle.unoccluded_norm(order)
    for b, n in enumerate(sizes):
        at = np.arange(offs[b], offs[b + 1])
        ref = oracle.transfer(sc.subset(at), dirs, order, np.arange(n), bounce=True)
        lim = 1e-4 * np.maximum(np.linalg.norm(ref["P"], axis=1), floor) + ref["allow_P"]
        for P in (out["P"], P0):
            assert np.all(np.linalg.norm(P.cpu().numpy()[at] - ref["P"], axis=1) <= lim)
        T = out["T"].cpu().numpy()[at]
        lim = 1e-4 * np.maximum(np.linalg.norm(ref["T"].reshape(n, -1), axis=1), floor)
        lim = lim + np.linalg.norm(ref["allow_T"], axis=1)
        assert np.all(np.linalg.norm((T - ref["T"]).reshape(n, -1), axis=1) <= lim)
        clean = (ref["flags"] & (oracle.RF_AMBIG_HIT | oracle.RF_AMBIG_ARGMAX)) == 0
        idx = out["idx"].cpu().numpy()[at]
        np.testing.assert_array_equal(np.where(idx >= 0, idx - offs[b], idx)[clean], ref["idx"][clean])


@pytest.mark.parametrize("sizes", [[31], [64], [65], [129], [40, 1, 30, 90], [500]])
def test_packet_windows_against_oracle(sizes):
    parts = [S.surface_scene(n, 300 + n) for n in sizes]
    for p in parts:
        p.means *= 0.25  # crowded: hits in the tens per ray
    sc, offs = S.concat_scenes(parts)
    _check(sc, offs, S.direction_set(37, 5), 2, sizes)


@pytest.mark.parametrize("thin", [1.0, 30.0, 300.0])
def test_packet_thin_splats_against_oracle(thin):
    sc = S.surface_scene(900, 41)
    sc.means *= 0.3
    sc.scales[:, 2] = sc.scales[:, :2].min(axis=1) / np.float32(thin)
    sc.scales[::3, 0] /= np.float32(thin)
    _check(sc, np.array([0, sc.n], np.int64), S.direction_set(48, 6), 3, [sc.n])


def test_packet_many_hits_per_ray():
    """Faint splats: rays pass tens of them before the index matrix is settled."""
    sc = S.surface_scene(1500, 42)
    sc.means *= 0.2
    sc.opacity *= np.float32(0.1)
    _check(sc, np.array([0, sc.n], np.int64), S.direction_set(24, 7), 1, [sc.n])


GRADS = ("means", "scales", "quats", "opacity", "normals")


def _grads_against_autograd(parts, dirs, order, t_min):
    """The packet backward of several scenes in one call against FP64 autograd of each scene's
    brute-force P (tolerance of test_gpu_transfer.py: 2e-3 norm-wise per field)."""
    from oracle import transfer_torch as TT

    sc, offs = S.concat_scenes(parts)
    g = api.GaussianTensors.from_scene(sc)
    st = api.Status()
    bvh = api.build_bvh(g, torch.from_numpy(offs).cuda(), status=st)
    w = np.random.default_rng(sc.n).standard_normal((sc.n, (order + 1) ** 2)).astype(np.float32)
    w[::7] = 0.0  # receivers without a gradient
    out = api.precompute_transfer_backward(g, bvh, torch.from_numpy(dirs).cuda(), order, torch.from_numpy(w).cuda(),
                                           t_min=t_min, status=st)
    torch.cuda.synchronize()
    assert st.read() == 0
    for b, p in enumerate(parts):
        at = slice(int(offs[b]), int(offs[b + 1]))
        ps = [torch.tensor(np.asarray(getattr(p, f), np.float64), requires_grad=True) for f in GRADS]
        P = TT.transfer_P(*ps, dirs, oracle.sh(order, dirs))
        ref = torch.autograd.grad((P * torch.as_tensor(w[at].astype(np.float64))).sum(), ps, allow_unused=True)
        top = max(float(r.norm()) for r in ref if r is not None)
        for f, r in zip(GRADS, ref):
            a = out["d_" + f].cpu().double()[at]
            r = torch.zeros_like(a) if r is None else r
            assert float((a - r).norm()) <= 2e-3 * max(float(r.norm()), 1e-3 * top), (b, f)


@pytest.mark.parametrize("sizes", [[33], [64, 65], [1, 130, 2, 257]])
def test_packet_backward_windows(sizes):
    parts = [S.surface_scene(n, 500 + n) for n in sizes]
    for p in parts:
        p.means *= 0.3
    _grads_against_autograd(parts, S.direction_set(29, 8), 2, 0.0)


def test_packet_backward_list_overflow():
    """More hit leaves per packet than the kernel keeps at a time (2,048): faint splats all over
    one another, so that the list is continued by further walks."""
    sc = S.surface_scene(2600, 43)
    sc.means *= 0.02
    sc.opacity *= np.float32(0.02)
    _grads_against_autograd([sc], S.direction_set(5, 9), 1, 0.0)


@pytest.mark.parametrize("sizes", [[255], [256], [600], [200, 100, 213]])
def test_packet_backward_wide_windows(sizes):
    """Backward windows that are full, one short and in part; normals at random, so that a packet's rays come from
    all over its window."""
    parts = [S.isotropic_scene(n, 700 + n) for n in sizes]
    for p in parts:
        p.scales *= np.float32(1.5)
        p.scales[:, 0] *= np.float32(0.7)
        p.scales[:, 1] *= np.float32(1.2)
    _grads_against_autograd(parts, S.direction_set(31, 10), 2, 0.0)
