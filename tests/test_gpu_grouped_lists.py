"""Grouped transforms of more jobs than one launch's parameters hold: bit-identical
to the own calls, forward and inverse."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


# 32 jobs travel with the launch, longer lists through device memory; one-tile
# sizes (2^12) and generic passes (2^9, 3^5)
@pytest.mark.parametrize("p,m,n", [(2, 12, 32), (2, 12, 33), (2, 9, 32), (2, 9, 33), (2, 9, 97), (3, 5, 33)])
def test_long_lists_bit_identical(dwt, dev, p, m, n):
    N = p ** m
    plans = [dwt.dwt_plan(p, m, 2, S.small_net(p, m, 2, index=500 + i), dwt.DWT_PLAN_TRANSFORM_ONLY) for i in range(3)]
    tt, dt = (torch.float32, dwt.DWT_F32) if p == 2 else (torch.complex64, dwt.DWT_C64)
    g = torch.Generator(device=dev).manual_seed(7)
    for own, grouped in ((dwt.dwt_forward, dwt.dwt_forward_grouped), (dwt.dwt_inverse, dwt.dwt_inverse_grouped)):
        jobs, refs = [], []
        for i in range(n):
            b = 1 + i % 2
            x = torch.randn((b, N), dtype=tt, device=dev, generator=g)
            out, ref = torch.zeros_like(x), torch.zeros_like(x)
            own(plans[i % 3], x, ref, b, N, N, dt, dt)
            jobs.append((plans[i % 3], x, out, b, N, N))
            refs.append(ref)
        grouped(jobs, dt, dt)
        for i, (job, ref) in enumerate(zip(jobs, refs)):
            assert torch.equal(job[2], ref), i
