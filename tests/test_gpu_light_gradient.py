"""dL of the relight backward at the edges of its batches (128 and 32 Gaussians), chunks (2,048) and light groups (1
and 4 lights a thread, the passes of each order), one scene and many, against FP64 sums.

Bound per output: a chain of at most 2,048 products and the partial sums after it, 2,100 roundings of 2^-24 of the sum
of magnitudes.
"""
import math

import pytest
import torch

from paper_2408_03538_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2, 3, 4, 6])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 9, 17])
@pytest.mark.parametrize("tch", [1, 3])
@pytest.mark.parametrize("sizes", [[1], [129, 2049], [31, 33, 5000]])
def test_light_gradient_sums(order, k, tch, sizes):
    C, n = (order + 1) ** 2, sum(sizes)
    gen = torch.Generator("cuda").manual_seed(100 * order + k)
    f = lambda *s: torch.randn(s, device="cuda", generator=gen)
    T = f(n, C) if tch == 1 else f(n, 3, C)
    albedo, L = f(n, 3).abs(), f(len(sizes), k, 3, C)
    offs = torch.tensor([sum(sizes[:b]) for b in range(len(sizes) + 1)], dtype=torch.int64, device="cuda")
    dcol = [f(k, m, 3) for m in sizes]
    _, _, many = api.relight_backward_batched(T, albedo, offs, L, order, torch.cat([d.flatten() for d in dcol]))
    for b, m in enumerate(sizes):
        at = slice(int(offs[b]), int(offs[b]) + m)
        Tb = (T[at] if tch == 3 else T[at][:, None, :].expand(m, 3, C)).double()
        w = dcol[b].double() * albedo[at].double() / math.pi
        ref = torch.einsum("lic,icm->lcm", w, Tb)
        lim = 2100 * 2.0 ** -24 * torch.einsum("lic,icm->lcm", w.abs(), Tb.abs())
        _, _, one = api.relight_backward(T[at].contiguous(), albedo[at].contiguous(), L[b].contiguous(), order, dcol[b])
        for got in (one, many[b]):
            assert bool(((got.double() - ref).abs() <= lim).all())
