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


@pytest.mark.parametrize("n,width", [(1, 64), (700, 64), (4096, 250), (4097, 250), (60_000, 640), (700_000, 1920)])
def test_pair_order(n, width):
    """The sorted (tile, depth) pairs: ascending keys, equal keys by index, every key its splat's tile
    and depth, each splat in exactly the tiles of its rectangle, ranges and prefix sums to match (one-block,
    self-summing and scanned passes of the sort)."""
    sc = S.isotropic_scene(n, 80)
    sc.scales *= np.float32(0.3)
    sc.means[1::2] = sc.means[: sc.n // 2 * 2 : 2][: sc.means[1::2].shape[0]]  # equal depths
    cam = S.look_at_camera((0, -3.5, 1.0), (0, 0, 0), 45, width, width // 2)
    g = api.GaussianTensors.from_scene(sc)
    st = api.Status()
    _, s = api.render(g, torch.zeros((1, n, 3), device="cuda"), cam, torch.zeros(3, device="cuda"), status=st,
                      max_pairs=64 * n + 4096)
    assert st.read() == 0
    m, gx, gy = s.n_pairs(), (width + 15) // 16, (width // 2 + 15) // 16
    key = s.view("pair_keys", torch.int64, (s.max_pairs,))[:m]
    ids = s.view("pair_ids", torch.int32, (s.max_pairs,))[:m].long()
    assert m > 0 and bool((key[1:] >= key[:-1]).all())
    assert bool((ids[1:] > ids[:-1])[key[1:] == key[:-1]].all())
    depth = s.view("depth", torch.float32, (n,))
    assert torch.equal(key & 0xffffffff, depth[ids].view(torch.int32).long())
    xy, r = s.view("mean2d", torch.float32, (n, 2)), s.view("radius", torch.int32, (n,)).float()
    tile = key >> 32
    lo = torch.floor((xy[ids] - r[ids, None]) / 16)
    hi = torch.floor((xy[ids] + r[ids, None]) / 16)
    t2 = torch.stack([tile % gx, tile // gx], 1)
    assert bool(((t2 >= lo) & (t2 <= hi)).all())
    on = r > 0
    lim = torch.tensor([gx, gy], device="cuda", dtype=torch.float32)
    side = torch.minimum(torch.floor((xy + r[:, None]) / 16) + 1, lim).clamp(min=0) - torch.minimum(
        torch.floor((xy - r[:, None]) / 16).clamp(min=0), lim)
    area = torch.where(on, side[:, 0] * side[:, 1], torch.zeros_like(r)).long()
    assert torch.equal(torch.bincount(ids, minlength=n), area)
    assert torch.equal(s.view("tiles_touched", torch.int32, (n,)).long(), torch.cumsum(area, 0))
    ranges = s.view("ranges", torch.int32, (gx * gy, 2)).long()
    assert torch.equal(ranges[:, 1] - ranges[:, 0], torch.bincount(tile, minlength=gx * gy))


@pytest.mark.parametrize("n", [4096, 4097, 524_288, 524_289, 1_300_001])
def test_bvh_sort_sizes(n):
    """The 64-bit keys of the BVH at the ends of the sort's ranges: sorted, and stable by construction
    (the low bits are the index)."""
    g = api.GaussianTensors.from_scene(S.isotropic_scene(n, 81))
    bvh = api.build_bvh(g)
    key = bvh.view("keys", torch.int64, (n,))
    order = bvh.view("order", torch.int32, (n,)).long()
    assert bool((key[1:] > key[:-1]).all()) and torch.equal(key & ((1 << 27) - 1), order)
    assert torch.equal(torch.sort(order).values, torch.arange(n, device="cuda"))


@pytest.mark.parametrize("w,h", [(1, 1), (17, 4), (61, 45), (640, 360)])
@pytest.mark.parametrize("k", [2, 5, 16, 23, 32])
def test_color_groups_and_rows_agree(w, h, k):
    """Every group of colour sets blends with the same weights: k sets at once equal k renders of one set, bit
    for bit; so do the normals that the geometry maps blend from rows."""
    sc = S.isotropic_scene(1501, 90)
    cam = S.look_at_camera((0, -3.5, 1.0), (0, 0, 0), 45, w, h)
    g = api.GaussianTensors.from_scene(sc)
    colors = torch.rand((k, sc.n, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(k))
    colors[1] = g.normals
    bg = torch.zeros(3, device="cuda")
    st = api.Status()
    img, s = api.render(g, colors, cam, bg, max_pairs=400_000, status=st)
    assert st.read() == 0
    for l in range(k):
        one, s1 = api.render(g, colors[l : l + 1].contiguous(), cam, bg, max_pairs=400_000)
        assert torch.equal(one[0], img[l]), l
        for field, dt in (("final_T", torch.float32), ("n_contrib", torch.int32)):
            assert torch.equal(s.view(field, dt, (h, w)), s1.view(field, dt, (h, w)))
    tight, _ = api.render(g, colors, cam, bg, max_pairs=s.n_pairs(), status=st)  # the colours read in place
    assert st.read() == 0 and torch.equal(tight, img)
    _, normal, _ = api.render_geometry(g, cam, max_pairs=400_000)
    assert torch.equal(normal, img[1])


@pytest.mark.parametrize("seed", [0, 1, 2])
@pytest.mark.parametrize("k", [1, 3])
def test_needle_gradients(seed, k):
    """Scales that differ by e^1.4 at random, in any direction: along a needle's long axis the offsets of its pixels
    are large and what they add to the gradients small."""
    sc, rng = S.isotropic_scene(900, 10 + seed), np.random.default_rng(seed)
    sc.scales = (1.6 * sc.scales * np.exp(rng.normal(0, 1.4, sc.scales.shape))).astype(np.float32)
    q = rng.normal(size=(sc.n, 4))
    sc.quats = (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)
    sc.opacity = np.clip(sc.opacity * (1 + seed), 0, 0.99).astype(np.float32)
    _check(sc, S.look_at_camera((0, -4.0, 1.5), (0, 0, 0), 50, 160, 90), k, (0.2, 0.2, 0.2))
