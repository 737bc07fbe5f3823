"""The two forms of the glossy colours, a block per few splats and a thread per splat, at the sizes where the choice
between them changes: the same sums in the same order, so the same bits."""
import pytest
import torch

from paper_2408_03538_gb300 import api, scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,n,k", [(6, 30_001, 1), (6, 29_999, 5), (6, 15_000, 129), (3, 62_500, 128), (3, 31_251, 256)])
def test_forms_agree(order, n, k):
    C, gen = (order + 1) ** 2, torch.Generator("cuda").manual_seed(n)
    f = lambda *s: torch.randn(s, device="cuda", generator=gen)
    T, M, means, albedo = f(n, C), f(n, C, C), f(n, 3), f(n, 3).abs()
    L = torch.from_numpy(S.env_lights(k, order, 5)).cuda()
    ids = torch.randperm(n, device="cuda", generator=gen).to(torch.int32)
    cam = torch.tensor([0.0, -7.0, 3.0], device="cuda")
    kw = dict(means=means, cam_pos=cam)
    all_ = api.relight(T, albedo, L, order, glossy_ids=ids, M=M, **kw)
    part = torch.empty_like(all_)
    for at in range(0, n, 5000):  # few enough for a block per few splats
        one = api.relight(T, albedo, L, order, glossy_ids=ids[at:at + 5000].contiguous(),
                          M=M[at:at + 5000].contiguous(), **kw)
        j = ids[at:at + 5000].long()
        part[:, j] = one[:, j]
    assert torch.equal(all_, part)
