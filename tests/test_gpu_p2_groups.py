"""Batches of p = 2 transforms and interpolations whose last group of functions is
larger or shorter than the others: every function as in a call of its own."""
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


# 64 MB hold 64 functions of 2^18, 32 of 2^19, 16 of 2^20 and 8 of 2^21 FP32 or int32
# points: one group up to half as many again, then two
@pytest.mark.parametrize("m,batch,groups", [(18, 64, 1), (18, 96, 1), (18, 97, 2), (19, 48, 1), (20, 25, 2), (20, 41, 3), (21, 12, 1),
                                            (21, 21, 3)])
def test_groups(dwt, dev, m, batch, groups):
    N, s = 1 << m, 3
    plan = dwt.dwt_plan(2, m, s, S.small_net(2, m, s, index=490))
    g = torch.Generator(device=dev).manual_seed(m)
    x = torch.randn((batch, N), device=dev, generator=g)
    xi = torch.randint(-1000, 1000, (batch, N), dtype=torch.int32, device=dev, generator=g)
    for call, inp, t in ((dwt.dwt_forward, x, dwt.DWT_F32), (dwt.dwt_inverse, xi, dwt.DWT_I32)):
        y = torch.empty_like(inp)
        n0 = dwt.dwt_launch_count()
        call(plan, inp, y, batch, N, N, t, t)
        assert dwt.dwt_launch_count() - n0 == 2 * groups
        one = torch.empty_like(inp[:1])
        for b in (0, batch // 2, batch - 1):
            call(plan, inp[b:b + 1], one, 1, N, N, t, t)
            assert torch.equal(one[0].view(torch.int32), y[b].view(torch.int32)), b
    c = torch.empty_like(x)
    var = torch.empty((batch, 2, s + 1), dtype=torch.float64, device=dev)
    dim = torch.empty((batch, 2), dtype=torch.int32, device=dev)
    dwt.dwt_interpolate(plan, x, c, None, batch, N, dwt.DWT_F32, dwt.DWT_WEIGHT_INV_SQ_WAVENUMBER, var=var, dim=dim)
    for b in (0, batch // 2, batch - 2, batch - 1):
        c1, v1, d1 = torch.empty_like(x[:1]), torch.empty_like(var[:1]), torch.empty_like(dim[:1])
        dwt.dwt_interpolate(plan, x[b:b + 1], c1, None, 1, N, dwt.DWT_F32, dwt.DWT_WEIGHT_INV_SQ_WAVENUMBER, var=v1, dim=d1)
        assert torch.equal(c1[0].view(torch.int32), c[b].view(torch.int32)) and torch.equal(v1[0], var[b]) and torch.equal(d1[0], dim[b])
