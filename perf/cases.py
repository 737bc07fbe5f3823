"""The calls whose speed counts: the precomputed transfer of a Gaussian scene (visibility, bounces,
glossy matrices), its differentiable form, relit frames forward and backward, many lights in pixel
space, the training stage's per-view step and batched scenes, from a thousand splats to a million.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes what a
caller holds before the call, ``run`` is one pass through the public API, ``work`` the bytes and
operations a pass cannot do without, and ``exact`` the same results in 64 bits from plain torch.
"""
import math
import random

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2408_03538_gb300 import api, scenes as S

DEV = "cuda"


def listed():
    return [
        # one small object, visibility only: the edit-and-preview call, where launches and latency count
        dict(name="transfer-tiny", kind="transfer", scene="volume", n=1024, order=2, dirs=64, bounce=False,
             glossy=False),
        # a scanned surface scene with one bounce, the ordinary precompute
        dict(name="transfer-surface-100k", kind="transfer", scene="surface", n=100_000, order=3, dirs=256,
             bounce=True, glossy=False),
        # the largest single-GPU scene: ten instances, shadow + bounce + glossy matrices
        dict(name="transfer-tiled-1m", kind="transfer", scene="tiled", n=1_000_000, order=3, dirs=256, bounce=True,
             glossy=True),
        # the visibility cache that training makes once per scene (a dense volume, odd size)
        dict(name="visibility-60k", kind="visibility", scene="volume", n=60_001, order=3, dirs=128),
        # geometry optimisation through the shadowed transfer: forward and backward
        dict(name="difftransfer-volume", kind="difftransfer", scene="volume", n=100_003, order=3, dirs=128,
             through="shadow"),
        # the same through one self-transfer bounce on a surface
        dict(name="difftransfer-bounce", kind="difftransfer", scene="surface", n=40_000, order=3, dirs=256,
             through="bounce"),
        # a thumbnail of a small object, forward and backward: launches and latency
        dict(name="frame-tiny", kind="frame", scene="volume", n=1024, order=2, lights=1, width=256, height=256,
             rgb=False),
        # differentiable relighting of a dense volume at full HD: one forward and backward frame
        dict(name="frame-300k", kind="frame", scene="volume", n=300_000, order=3, lights=1, width=1920, height=1080,
             rgb=False),
        # interactive relighting: a few lights of a surface scene, colours and images, forward only
        dict(name="lights-surface-100k", kind="lights", scene="surface", n=100_000, order=3, lights=8, width=1920,
             height=1080, precision="fp32"),
        # a light turntable: 64 lights of the million-splat scene in pixel space, glossy splats among them
        dict(name="relit-64-tiled-1m", kind="relit", scene="tiled", n=1_000_000, order=3, lights=64, width=1920,
             height=1080, precision="bf16x3"),
        # one training iteration's transfer and normal supervision: view transfer forward and backward,
        # depth and normal maps, pseudo-normal, normal loss
        dict(name="training-300k", kind="training", scene="surface", n=300_000, order=3, dirs=256, width=1920,
             height=1080),
        # several scenes of uneven size in one call per stage: relit frames, losses and gradients
        dict(name="batched-8", kind="batched", scene="volume", n=400_000, scenes=8, order=3, lights=4, width=1280,
             height=720),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["transfer", "transfer", "visibility", "difftransfer", "frame", "frame", "lights", "relit",
                       "training", "batched"])
    size = rng.choice([(1920, 1080), (1280, 720), (801, 603), (640, 360), (333, 257)])
    if kind in ("transfer", "visibility"):
        c = dict(kind=kind, scene=rng.choice(["volume", "surface"]), n=_log(rng, 1000, 200_000),
                 order=rng.choice([1, 2, 3, 3, 4]), dirs=rng.choice([33, 64, 100, 128, 255, 256]))
        if kind == "transfer":
            c["bounce"] = rng.random() < 0.6
            c["glossy"] = c["order"] <= 3 and rng.random() < 0.4
        return c
    if kind == "difftransfer":
        return dict(kind=kind, scene=rng.choice(["volume", "surface"]), n=_log(rng, 1000, 60_000),
                    order=rng.choice([1, 2, 3]), dirs=rng.choice([33, 64, 128, 256]),
                    through=rng.choice(["shadow", "bounce", "glossy"]))
    if kind == "frame":
        return dict(kind=kind, scene=rng.choice(["volume", "surface"]), n=_log(rng, 1000, 300_000),
                    order=rng.choice([1, 2, 3, 4]), lights=rng.choice([1, 1, 2, 3, 5, 8]), width=size[0],
                    height=size[1], rgb=rng.random() < 0.5)
    if kind == "lights":
        return dict(kind=kind, scene=rng.choice(["volume", "surface"]), n=_log(rng, 1000, 300_000),
                    order=rng.choice([1, 2, 3, 5]), lights=rng.choice([1, 3, 8, 17]), width=size[0], height=size[1],
                    precision=rng.choice(["fp32", "bf16x3"]))
    if kind == "relit":
        return dict(kind=kind, scene="surface", n=_log(rng, 1000, 500_000), order=rng.choice([2, 3, 4]),
                    lights=rng.choice([5, 16, 33, 64]), width=size[0], height=size[1],
                    precision=rng.choice(["fp32", "bf16x3"]))
    if kind == "training":
        return dict(kind=kind, scene=rng.choice(["volume", "surface"]), n=_log(rng, 1000, 500_000),
                    order=rng.choice([2, 3]), dirs=rng.choice([64, 100, 256]), width=size[0], height=size[1])
    b = rng.choice([2, 5, 8, 16])
    return dict(kind=kind, scene="volume", n=_log(rng, 2000 * b, 30_000 * b), scenes=b, order=rng.choice([2, 3]),
                lights=rng.choice([1, 3, 4, 8]), width=640, height=360)


# ---- inputs ---------------------------------------------------------------------------------------
CAMERAS = {"volume": ((0.0, -3.5, 1.5), (0.0, 0.0, 0.0), 50.0), "surface": ((0.0, -7.0, 3.0), (0.0, 0.0, 0.8), 45.0),
           "tiled": ((0.0, -40.0, 14.0), (0.0, 0.0, 0.0), 45.0)}
PRECISION = {"fp32": 0, "bf16x3": 1}


def _volume(n, seed):
    """A cloud of splats; optimisation leaves none of them round."""
    sc = S.isotropic_scene(n, seed)
    sc.scales = (sc.scales * np.exp(np.random.default_rng(seed + 7).normal(0.0, 0.3, (n, 3)))).astype(np.float32)
    return sc


def _scene(case, seed):
    if case["scene"] == "volume":
        sc = _volume(case["n"], seed)
    elif case["scene"] == "surface":
        sc = S.surface_scene(case["n"], seed)
    else:
        sc = S.tiled_scene(seed, base_n=case["n"] // 10)
    rng = np.random.default_rng(seed + 1)
    sc.glossy_mask = (rng.permutation(sc.n) < (3 * sc.n) // 10).astype(np.uint8)
    sc.roughness = rng.uniform(0.15, 1.0, sc.n).astype(np.float32)
    sc.metallic = rng.uniform(0.0, 1.0, sc.n).astype(np.float32)
    return sc


def _camera(case, seed):
    eye, target, fov = CAMERAS[case["scene"]]
    turn = 0.2 * math.sin(seed)  # the view moves a little with the seed
    eye = (eye[0] * math.cos(turn) - eye[1] * math.sin(turn), eye[0] * math.sin(turn) + eye[1] * math.cos(turn), eye[2])
    return S.look_at_camera(eye, target, fov, case["width"], case["height"])


def _sh(d, order):
    """Real spherical harmonics [.., (order+1)^2] of unit directions, Condon-Shortley phase, l*l+l+m."""
    x, y, z = d[..., 0], d[..., 1], d[..., 2]
    Y = [None] * (order + 1) ** 2
    re, im, qmm = torch.ones_like(x), torch.zeros_like(x), 1.0
    for m in range(order + 1):
        if m:
            re, im = re * x - im * y, re * y + im * x
            qmm *= -(2 * m - 1)
        q2, q1 = None, torch.full_like(x, qmm)
        for l in range(m, order + 1):
            if l == m + 1:
                q2, q1 = q1, (2 * m + 1) * z * q1
            elif l > m + 1:
                q2, q1 = q1, ((2 * l - 1) * z * q1 - (l + m - 1) * q2) / (l - m)
            K = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            if m == 0:
                Y[l * l + l] = K * q1
            else:
                Y[l * l + l + m] = math.sqrt(2) * K * q1 * re
                Y[l * l + l - m] = math.sqrt(2) * K * q1 * im
    return torch.stack(Y, -1)


def _transfer_rows(normals, order, gen, rgb):
    """Transfer rows as a precompute leaves them: the clamped-cosine lobe about the normal, dimmed by
    the occlusion, with the occluders' higher bands on top."""
    n = normals.shape[0]
    A = [math.pi, 2 * math.pi / 3, math.pi / 4, 0.0, -math.pi / 24, 0.0, math.pi / 64]
    band = torch.tensor([A[l] for l in range(order + 1) for _ in range(2 * l + 1)], device=DEV)
    T = _sh(normals, order) * band * (0.2 + 0.8 * torch.rand((n, 1), device=DEV, generator=gen))
    T = T + 0.05 * torch.randn(T.shape, device=DEV, generator=gen)
    if not rgb:
        return T.contiguous()
    T = T[:, None, :] * torch.ones((1, 3, 1), device=DEV)
    return (T + 0.05 * torch.rand((n, 3, 1), device=DEV, generator=gen) * T.abs().mean()).contiguous()


def _state(g, colors, cam):
    """A render state with room for this view's pairs and a quarter more, sized by one render."""
    room = max(64 * g.n, 1 << 16)
    while True:
        st = api.Status()
        _, s = api.render(g, colors, cam, torch.zeros(3, device=DEV), max_pairs=room, status=st)
        if st.read() == 0:
            return int(s.n_pairs() * 1.25) + 4096
        room *= 2


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    s = dict(case=case)
    kind, order = case["kind"], case["order"]
    if kind == "batched":
        w = np.exp(np.random.default_rng(case["n"]).uniform(0.0, math.log(8.0), case["scenes"]))
        sizes = np.floor(case["n"] * w / w.sum()).astype(int)
        sizes[-1] = case["n"] - sizes[:-1].sum()
        merged, offs = S.concat_scenes([_volume(int(n), seed * 1000 + b) for b, n in enumerate(sizes)])
        g = api.GaussianTensors.from_scene(merged)
        s.update(g=g, offs_host=offs, offs=torch.from_numpy(offs).to(DEV), k=case["lights"])
        s["T"] = _transfer_rows(g.normals, order, gen, rgb=False)
        s["L"] = torch.from_numpy(np.stack([S.env_lights(case["lights"], order, seed + 10 + b)
                                            for b in range(case["scenes"])])).to(DEV)
        s["cams"] = [_camera(case, seed + b) for b in range(case["scenes"])]
        s["bg"] = torch.zeros(3, device=DEV)
        s["target"] = 0.4 * torch.rand((case["scenes"], case["lights"], 3, case["height"], case["width"]), device=DEV,
                                       generator=gen)
        room = 64 * g.n
        colors = api.relight_batched(s["T"], g.albedo, s["offs"], s["L"], order)
        while True:
            st, probe = api.Status(), api.RenderState(g.n, case["width"], case["height"], room, DEV, case["scenes"])
            api.render_batched(g, s["offs"], colors, case["lights"], s["cams"], s["bg"], probe, status=st)
            if st.read() == 0:
                break
            room *= 2
        s["state"] = api.RenderState(g.n, case["width"], case["height"], int(probe.n_pairs() * 1.25) + 4096, DEV,
                                     case["scenes"])
        return s
    sc = _scene(case, seed)
    g = api.GaussianTensors.from_scene(sc)
    s["g"] = g
    if "dirs" in case:
        s["dirs"] = torch.from_numpy(S.direction_set(case["dirs"], seed + 2)).to(DEV)
    if "lights" in case:
        s["L"] = torch.from_numpy(S.env_lights(case["lights"], order, seed + 3)).to(DEV)
    if "width" in case:
        s["cam"] = _camera(case, seed)
        s["bg"] = torch.full((3,), 0.1, device=DEV)
    if kind == "difftransfer":
        C = (order + 1) ** 2
        shape = (g.n, 3, C) if case["through"] == "bounce" else (g.n, C)
        s["up"] = torch.randn(shape, device=DEV, generator=gen)
        if case["through"] == "glossy":
            ng = int(g.glossy_mask.sum())
            s["up_M"] = torch.randn((ng, C, C), device=DEV, generator=gen)
    elif kind == "frame":
        s["T"] = _transfer_rows(g.normals, order, gen, case["rgb"])
        colors = api.relight(s["T"], g.albedo, s["L"], order)
        s["max_pairs"] = _state(g, colors, s["cam"])
        s["up"] = torch.randn((case["lights"], 3, case["height"], case["width"]), device=DEV, generator=gen) / 1e3
    elif kind in ("lights", "relit"):
        s["T"] = _transfer_rows(g.normals, order, gen, rgb=True)
        C = (order + 1) ** 2
        s["ids"] = torch.nonzero(g.glossy_mask).flatten().to(torch.int32)
        fall = torch.tensor([1.0 / (l + 1) ** 2 for l in range(order + 1) for _ in range(2 * l + 1)], device=DEV)
        rows = s["T"][s["ids"].long(), 0]
        s["M"] = (rows[:, :, None] * (3.5 * (torch.arange(C, device=DEV) == 0))[None, None, :]
                  + 0.2 * torch.randn((rows.shape[0], C, C), device=DEV, generator=gen) * fall[:, None]
                  * fall[None, :]).contiguous()
        s["cam_pos"] = torch.from_numpy(np.asarray(s["cam"].position, np.float32)).to(DEV)
        pairs = _state(g, api.relight(s["T"], g.albedo, s["L"][:1].contiguous(), order), s["cam"])
        s["state"] = api.RenderState(g.n, case["width"], case["height"], pairs)
    elif kind == "training":
        n, d = g.n, case["dirs"]
        # visibility as the cache holds it: 0 below the horizon, blocked rays (exactly 0 or below 2^-30),
        # open ones between 0 and 1
        u = torch.rand((n, d), device=DEV, generator=gen)
        v = torch.rand((n, d), device=DEV, generator=gen) ** 2
        v = torch.where(u < 0.3, v * 2.0 ** -30, v)
        v = torch.where(u < 0.05, torch.zeros_like(v), v)
        s["V"] = torch.where(g.normals @ s["dirs"].T > 0, v, torch.zeros_like(v)).contiguous()
        s["up"] = torch.randn((n, (order + 1) ** 2), device=DEV, generator=gen)
        s["cam_pos"] = tuple(float(x) for x in s["cam"].position)
        pairs = _state(g, torch.zeros((1, n, 3), device=DEV), s["cam"])
        s["state"] = api.RenderState(n, case["width"], case["height"], pairs)
    return s


# ---- one pass -------------------------------------------------------------------------------------
def run(s):
    case, g = s["case"], s["g"]
    kind, order = case["kind"], case["order"]
    if kind == "transfer":
        bvh = api.build_bvh(g)
        out = api.precompute_transfer(g, bvh, s["dirs"], order, bounce=case["bounce"], glossy=case["glossy"])
        return {k: out[k] for k in ("P", "T", "idx", "M") if k in out}
    if kind == "visibility":
        out = api.precompute_visibility(g, api.build_bvh(g), s["dirs"], order)
        return {"V": out["V"], "P": out["P"]}
    if kind == "difftransfer":
        names = ["means", "scales", "quats", "opacity", "normals"]
        if case["through"] == "bounce":
            names.append("albedo")
        elif case["through"] == "glossy":
            names += ["roughness", "metallic"]
        x = {f: getattr(g, f).detach().requires_grad_(f in names) for f in
             ("means", "scales", "quats", "opacity", "normals", "albedo", "roughness", "metallic")}
        geo = [x[f] for f in ("means", "scales", "quats", "opacity", "normals")]
        if case["through"] == "shadow":
            out = {"P": api.shadowed_transfer(*geo, x["albedo"], s["dirs"], order)}
            up = [s["up"]]
        elif case["through"] == "bounce":
            out = {"T": api.bounce_transfer(*geo, x["albedo"], s["dirs"], order)}
            up = [s["up"]]
        else:
            P, M = api.glossy_transfer(*geo, x["roughness"], x["metallic"], g.glossy_mask, x["albedo"], s["dirs"], order)
            out = {"P": P, "M": M}
            up = [s["up"], s["up_M"]]
        grads = torch.autograd.grad(list(out.values()), [x[f] for f in names], up)
        return {**{k: v.detach() for k, v in out.items()}, **{"d_" + f: v for f, v in zip(names, grads)}}
    if kind == "frame":
        names = ("means", "scales", "quats", "opacity", "albedo")
        x = [getattr(g, f).detach().requires_grad_() for f in names]
        Lsh, T = s["L"].detach().requires_grad_(), s["T"].detach().requires_grad_()
        img = api.relit_render(*x, Lsh, T, g.normals, s["cam"], order, bg=s["bg"], max_pairs=s["max_pairs"])
        grads = torch.autograd.grad(img, x + [Lsh, T], s["up"])
        return {"image": img.detach(), **{"d_" + f: v for f, v in zip(names + ("L", "T"), grads)}}
    if kind == "lights":
        colors = api.relight(s["T"], g.albedo, s["L"], order, precision=PRECISION[case["precision"]],
                             glossy_ids=s["ids"], M=s["M"], means=g.means, cam_pos=s["cam_pos"])
        img, _ = api.render(g, colors, s["cam"], s["bg"], state=s["state"])
        return {"colors": colors, "image": img}
    if kind == "relit":
        img, _ = api.render_relit(g, s["T"], s["L"], s["cam"], order, bg=s["bg"], precision=PRECISION[case["precision"]],
                                  glossy_ids=s["ids"], M=s["M"], state=s["state"])
        return {"image": img}
    if kind == "training":
        t = api.training_transfer(g, s["V"], s["dirs"], order, s["cam_pos"])
        dr, dm = api.training_transfer_backward(g, s["V"], s["dirs"], order, s["cam_pos"], s["up"])
        depth, normal, _ = api.render_geometry(g, s["cam"], state=s["state"])
        pseudo = api.pseudo_normal(depth, s["cam"])
        loss, dN = api.normal_loss(normal, pseudo)
        return {"t": t, "d_roughness": dr, "d_metallic": dm, "depth": depth, "normal": normal, "pseudo": pseudo,
                "loss": loss, "dN": dN}
    k = s["k"]
    colors = api.relight_batched(s["T"], g.albedo, s["offs"], s["L"], order)
    images = api.render_batched(g, s["offs"], colors, k, s["cams"], s["bg"], s["state"])
    losses, dimg = api.l2_loss_batched(images, s["target"])
    dm, ds, dq, do, dcol = api.render_backward_batched(g, s["offs"], colors, k, s["cams"], s["bg"], s["state"], dimg)
    da, _, dL = api.relight_backward_batched(s["T"], g.albedo, s["offs"], s["L"], order, dcol)
    return {"images": images, "losses": losses, "d_means": dm, "d_scales": ds, "d_quats": dq, "d_opacity": do,
            "d_albedo": da, "dL": dL}


# ---- what a pass cannot do without ------------------------------------------------------------------
def work(case):
    n, C = case["n"], (case["order"] + 1) ** 2
    kind = case["kind"]
    geo = 17 * 4 * n  # means, scales, quats, opacity, normals, albedo
    px = case.get("width", 0) * case.get("height", 0)
    k = case.get("lights", 1)
    if kind in ("transfer", "visibility", "difftransfer"):
        d = case["dirs"]
        rays = n * d / 2  # the directions above the splat's horizon
        base = n / 10 if case["scene"] == "tiled" else n
        hits = min(60.0, 0.009 * base) if case["scene"] == "volume" else min(80.0, 8e-4 * base)
        by, fl = geo + 4 * n * C, rays * (40 * hits + 2 * C)
        through = case.get("through")
        if kind == "visibility":
            by += 4 * n * d
        if case.get("bounce") or through == "bounce":
            by += 12 * n * C + 4 * n * d
            fl += rays * 6 * C
        if case.get("glossy") or through == "glossy":
            by += 0.3 * n * 4 * C * C
            fl += 0.3 * n * ((d / 2) * (d / 2) * (100 + 2 * C) + d * C * C)
        if kind == "difftransfer":
            by += geo + 4 * n * C * (3 if through == "bounce" else 1)
            fl += rays * hits * 100
        return {"bytes": by, "flops": fl}
    if kind == "training":
        d = case["dirs"]
        by = 2 * (4 * n * d + 32 * n + 4 * n * C) + 8 * n + geo + px * 4 * (4 + 4 + 3 + 3)
        return {"bytes": by, "flops": n * d / 6 * (2 * 100 + 4 * C) + px * 20 * 40}
    if kind == "batched":
        px *= case["scenes"]
    tch = 3 if kind in ("lights", "relit") or case.get("rgb") else 1
    by = geo + 4 * n * C * tch + 12 * k * px
    fl = 6.0 * n * C * k + px * 40 * (20 + 6 * k)
    if kind in ("lights", "relit"):
        by += 0.3 * n * 4 * C * C + (12 * k * n if kind == "lights" else 0)
    if kind in ("frame", "batched"):
        by += geo + 12 * k * px + (4 * n * C * tch if kind == "frame" else 12 * k * px)
        fl += 2 * fl
    return {"bytes": by, "flops": fl}


# ---- the same in 64 bits ------------------------------------------------------------------------------
TILE = 16


def _rot(q):
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def _project(means, scales, quats, cam):
    W = torch.as_tensor(np.asarray(cam.rot, np.float64), device=DEV)
    p = means @ W.T + torch.as_tensor(np.asarray(cam.trans, np.float64), device=DEV)
    x, y, z = p.unbind(1)
    ok = z > cam.near
    z1 = torch.where(ok, z, torch.ones_like(z))
    lx, ly = 0.65 * cam.width / cam.fx, 0.65 * cam.height / cam.fy
    tx, ty = (x / z1).clamp(-lx, lx) * z1, (y / z1).clamp(-ly, ly) * z1
    o = torch.zeros_like(z)
    J = torch.stack([cam.fx / z1, o, -cam.fx * tx / z1 ** 2, o, cam.fy / z1, -cam.fy * ty / z1 ** 2], 1).view(-1, 2, 3)
    B = J @ W @ _rot(quats) * scales[:, None, :]
    cov = B @ B.transpose(1, 2)
    a, b, c = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = a * c - b * b
    conic = torch.stack([c / det, -b / det, a / det], 1)
    mid = 0.5 * (a + c)
    r = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1)))).detach()
    m2 = torch.stack([cam.fx * x / z1 + cam.cx, cam.fy * y / z1 + cam.cy], 1)
    return m2, conic, z.detach(), r, ok


def _tile_lists(m2, r, z, ok, gx, gy):
    lo = torch.floor((m2.detach() - r[:, None]) / TILE)
    hi = torch.floor((m2.detach() + r[:, None]) / TILE) + 1
    lim = torch.tensor([gx, gy], device=DEV, dtype=lo.dtype)
    lo, hi = torch.minimum(lo.clamp(min=0), lim).long(), torch.minimum(hi.clamp(min=0), lim).long()
    ids = torch.nonzero(ok).flatten()
    ids = ids[torch.sort(z[ids], stable=True).indices]
    w = (hi - lo)[ids].clamp(min=0)
    cnt = w[:, 0] * w[:, 1]
    who = torch.repeat_interleave(torch.arange(ids.numel(), device=DEV), cnt)
    at = torch.arange(who.numel(), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[who]
    tx, ty = lo[ids[who], 0] + at % w[who, 0], lo[ids[who], 1] + at // w[who, 0]
    tile, perm = torch.sort(ty * gx + tx, stable=True)
    lens = torch.bincount(tile, minlength=gx * gy)
    return ids[who[perm]], torch.cumsum(lens, 0) - lens, lens


def _block(T, px, m2, conic, op, feat, g, live):
    """`g.shape[1]` splats of each tile, front to back: the colour they add and the transmittance left."""
    d = m2[g][:, None] - px[:, :, None]
    con = conic[g][:, None]
    power = -0.5 * (con[..., 0] * d[..., 0] ** 2 + con[..., 2] * d[..., 1] ** 2) - con[..., 1] * d[..., 0] * d[..., 1]
    a = (op[g][:, None] * torch.exp(power)).clamp(max=0.99)
    a = torch.where((power <= 0) & (a >= 1 / 255) & live[:, None], a, torch.zeros_like(a))
    P = T[..., None] * torch.cumprod(1 - a, -1)
    keep = P >= 1e-4
    before = torch.cat([T[..., None], P[..., :-1]], -1)
    left = torch.where(keep, P, torch.full_like(P, math.inf)).amin(-1)
    stop = ~keep.all(-1)
    wgt = torch.where(keep, a * before, torch.zeros_like(a))
    return torch.bmm(wgt, feat[g]), torch.where(torch.isinf(left), T, left), stop


def _raster(m2, conic, z, r, ok, op, feat, bg, cam):
    """[K,H,W] of the splats' features [n,K], composited front to back, 16 x 16 tiles."""
    W, H = cam.width, cam.height
    gx, gy = (W + TILE - 1) // TILE, (H + TILE - 1) // TILE
    lst, start, lens = _tile_lists(m2, r, z, ok, gx, gy)
    t = torch.arange(gx * gy, device=DEV)
    q = torch.arange(TILE * TILE, device=DEV)
    px = torch.stack([(t % gx)[:, None] * TILE + (q % TILE)[None], (t // gx)[:, None] * TILE + (q // TILE)[None]],
                     -1).double()
    T = torch.ones(px.shape[:2], dtype=torch.float64, device=DEV)
    done = torch.zeros(px.shape[:2], dtype=torch.bool, device=DEV)
    acc = torch.zeros(*px.shape[:2], feat.shape[1], dtype=torch.float64, device=DEV)
    step = 32
    for j0 in range(0, int(lens.max()) if lst.numel() else 0, step):
        on = torch.nonzero((lens > j0) & ~done.all(1)).flatten()
        if not on.numel():
            break
        j = j0 + torch.arange(step, device=DEV)
        live = j[None] < lens[on][:, None]
        g = lst[(start[on][:, None] + j[None]).clamp(max=lst.numel() - 1)]
        Tin = torch.where(done[on], torch.zeros_like(T[on]), T[on])
        args = (Tin, px[on], m2, conic, op, feat, g, live)
        add, left, stop = checkpoint(_block, *args, use_reentrant=False) if torch.is_grad_enabled() else _block(*args)
        was = done[on][..., None]
        acc = acc.index_add(0, on, torch.where(was, torch.zeros_like(add), add))
        T = T.index_copy(0, on, torch.where(done[on], T[on], left))
        done = done.index_copy(0, on, done[on] | stop)
    img = acc + T[..., None] * bg
    img = img.view(gy, gx, TILE, TILE, -1).permute(4, 0, 2, 1, 3).reshape(feat.shape[1], gy * TILE, gx * TILE)
    return img[:, :H, :W]


def _relit(albedo, T, L):
    """[k,n,3] = (albedo / pi) (T . L)."""
    T = T if T.dim() == 3 else T[:, None, :].expand(-1, 3, -1)
    return albedo[None] / math.pi * torch.einsum("ncm,kcm->knc", T, L)


def _image(x, L, T, cam, bg):
    col = _relit(x["albedo"], T, L)
    k, n = col.shape[:2]
    feat = col.permute(1, 0, 2).reshape(n, 3 * k)
    img = _raster(*_project(x["means"], x["scales"], x["quats"], cam), x["opacity"], feat, bg.repeat(k), cam)
    return img.view(k, 3, cam.height, cam.width)


def _kernel(n, wi, v, rough, metal):
    """k(w_i, v) = (1 - m) + pi f_s of unit normals, [.., n] x directions."""
    u = n / n.norm(dim=-1, keepdim=True)
    h = wi + v
    h = h / h.norm(dim=-1, keepdim=True)
    xi, xo = (u * wi).sum(-1), (u * v).sum(-1)
    a = rough ** 2
    den = (u * h).sum(-1) ** 2 * (a * a - 1) + 1
    D = a * a / (math.pi * den ** 2)
    F = 0.04 + 0.96 * (1 - (v * h).sum(-1).clamp(0, 1)) ** 5
    kk = a / 2
    g = 1 / ((xi * (1 - kk) + kk) * (xo * (1 - kk) + kk))
    return (1 - metal) + math.pi / 4 * D * F * g


def _visibility(g, dirs):
    """V [n,S] by testing every ray against every splat: the 3-sigma ellipsoid's nearest approach."""
    A = _rot(g["quats"]).transpose(1, 2) / g["scales"][:, :, None]
    n = A.shape[0]
    V = torch.zeros((n, dirs.shape[0]), dtype=torch.float64, device=DEV)
    for s, w in enumerate(dirs):
        a = A @ w
        dd = (a * a).sum(1)
        up = torch.nonzero(g["normals"] @ w > 0).flatten()
        for part in torch.split(up, max(1, 30_000_000 // n)):
            u = g["means"][part][:, None] - g["means"][None]
            b = torch.einsum("nij,rnj->rni", A, u)
            t = -(b * a).sum(-1) / dd
            d2 = ((b + t[..., None] * a) ** 2).sum(-1)
            al = torch.where((t > 0) & (d2 <= 9), g["opacity"] * torch.exp(-0.5 * d2), torch.zeros_like(d2))
            al[torch.arange(part.numel(), device=DEV), part] = 0
            v = torch.prod(1 - al, 1)
            V[part, s] = v
    return V


def exact(case, seed):
    s = prepare(case, seed)
    kind, order, n = case["kind"], case["order"], case["n"]
    f64 = {f: getattr(s["g"], f).double() for f in ("means", "scales", "quats", "opacity", "normals", "albedo",
                                                    "roughness", "metallic") if getattr(s["g"], f) is not None}
    if kind in ("transfer", "visibility", "difftransfer"):
        d = s["dirs"].double()
        if n * n * d.shape[0] > 1.5e10 or kind == "difftransfer":
            return None
        V = _visibility(f64, d)
        wgt = 4 * math.pi / d.shape[0] * (f64["normals"] @ d.T).clamp(min=0)
        out = {"P": (V * wgt) @ _sh(d, order)}
        if kind == "visibility":
            return {"V": V, **out}
        if case["bounce"]:
            out.update(T=None, idx=None)
        if case["glossy"]:
            out["M"] = None
        return out
    if kind == "frame":
        names = ("means", "scales", "quats", "opacity", "albedo")
        x = {f: f64[f].requires_grad_() for f in names}
        L, T = s["L"].double().requires_grad_(), s["T"].double().requires_grad_()
        img = _image(x, L, T, s["cam"], s["bg"].double())
        grads = torch.autograd.grad(img, list(x.values()) + [L, T], s["up"].double())
        return {"image": img.detach(), **{"d_" + f: v for f, v in zip(names + ("L", "T"), grads)}}
    if kind in ("lights", "relit"):
        T, ids = s["T"].double(), s["ids"].long()
        v = torch.as_tensor(np.asarray(s["cam"].position, np.float64), device=DEV) - f64["means"][ids]
        te = torch.einsum("gab,gb->ga", s["M"].double(), _sh(v / v.norm(dim=1, keepdim=True), order))
        T[ids] = te[:, None, :].expand(-1, 3, -1)
        with torch.no_grad():
            if kind == "lights":
                img = _image(f64, s["L"].double(), T, s["cam"], s["bg"].double())
                return {"colors": _relit(f64["albedo"], T, s["L"].double()), "image": img}
            feat = (f64["albedo"][:, :, None] / math.pi * T).reshape(n, -1)  # [n, 3 C], then the transmittance
            feat = torch.cat([feat, torch.zeros((n, 1), dtype=torch.float64, device=DEV)], 1)
            back = torch.zeros(feat.shape[1], dtype=torch.float64, device=DEV)
            back[-1] = 1.0
            TI = _raster(*_project(f64["means"], f64["scales"], f64["quats"], s["cam"]), f64["opacity"], feat, back,
                         s["cam"])
            H, W = TI.shape[1:]
            img = torch.empty((case["lights"], 3, H, W), dtype=torch.float64, device=DEV)
            for c in range(3):
                rows = TI[:-1].view(3, -1, H * W)[c]
                img[:, c] = (s["L"].double()[:, c] @ rows).view(-1, H, W) + float(s["bg"][c]) * TI[-1]
            return {"image": img}
    if kind == "training":
        d = s["dirs"].double()
        Y = _sh(d, order)
        cam = torch.as_tensor(np.asarray(s["cam_pos"], np.float32).astype(np.float64), device=DEV)
        ts, drs, dms = [], [], []
        for i0 in range(0, n, 20_000):
            at = slice(i0, i0 + 20_000)
            r, m = f64["roughness"][at].requires_grad_(), f64["metallic"][at].requires_grad_()
            nn = f64["normals"][at]
            v = cam - f64["means"][at]
            v = v / v.norm(dim=1, keepdim=True)
            c = nn @ d.T
            on = (c > 0) & ((nn * v).sum(1) > 0)[:, None]
            k = _kernel(nn[:, None], d[None], v[:, None], r[:, None], m[:, None])
            f = torch.where(on, k * c * s["V"][at].double(), torch.zeros_like(k))
            t = 4 * math.pi / d.shape[0] * f @ Y
            gr, gm = torch.autograd.grad(t, [r, m], s["up"][at].double())
            ts.append(t.detach())
            drs.append(gr)
            dms.append(gm)
        camera = s["cam"]
        with torch.no_grad():
            pr = _project(f64["means"], f64["scales"], f64["quats"], camera)
            feat = torch.cat([pr[2][:, None], f64["normals"]], 1)
            maps = _raster(*pr, f64["opacity"], feat, torch.zeros(4, dtype=torch.float64, device=DEV), camera)
        # the pseudo-normal amplifies the depth map's last bits by the focal length: no value of its own
        return {"t": torch.cat(ts), "d_roughness": torch.cat(drs), "d_metallic": torch.cat(dms), "depth": maps[0],
                "normal": maps[1:], "pseudo": None, "loss": None, "dN": None}
    names = ("means", "scales", "quats", "opacity", "albedo")
    imgs, losses, grads, dLs = [], [], [], []
    for b in range(case["scenes"]):
        at = slice(int(s["offs_host"][b]), int(s["offs_host"][b + 1]))
        x = {f: f64[f][at].requires_grad_() for f in names}
        L = s["L"][b].double().requires_grad_()
        img = _image(x, L, s["T"][at].double(), s["cams"][b], s["bg"].double())
        loss = ((img - s["target"][b].double()) ** 2).mean()
        gr = torch.autograd.grad(loss, list(x.values()) + [L])
        imgs.append(img.detach())
        losses.append(loss.detach())
        grads.append(gr[:5])
        dLs.append(gr[5])
    cat = [torch.cat([gr[j] for gr in grads]) for j in range(5)]
    return {"images": torch.stack(imgs), "losses": torch.stack(losses), "dL": torch.stack(dLs),
            **{"d_" + f: v for f, v in zip(names, cat)}}
