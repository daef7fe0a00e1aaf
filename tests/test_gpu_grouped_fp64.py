"""Grouped FP64 transforms of p = 2 nets: jobs of 2^12 points and more share their
launches, and every element is the one of the job's own call."""
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


# one pass and 1 .. 9 high digits, two high passes (2^22), generic passes beside them
# (2^5, 2^11); lists within the 32 jobs that travel with a launch, and longer ones
@pytest.mark.parametrize("ms,launches", [([12] * 32, 1), ([12] * 33, 1), ([13] * 32, 2), ([12, 13, 14, 15, 16], 2),
                                         ([12, 17, 5, 18, 19, 11, 20, 21, 12, 22], 3), ([13, 12] * 50, 2)])
def test_fp64_jobs_share_launches(dwt, dev, ms, launches):
    plans = {m: dwt.dwt_plan(2, m, 1, S.small_net(2, m, 1), dwt.DWT_PLAN_TRANSFORM_ONLY) for m in set(ms)}
    g = torch.Generator(device=dev).manual_seed(11)
    t = dwt.DWT_F64
    for own, grouped in ((dwt.dwt_forward, dwt.dwt_forward_grouped), (dwt.dwt_inverse, dwt.dwt_inverse_grouped)):
        jobs, refs = [], []
        for i, m in enumerate(ms):
            b, N = (1 + i % 3) if m < 20 else 1, 1 << m
            ld_in, ld_out = N + i % 2, N + (i + 1) % 3
            x = torch.randn((b, ld_in), dtype=torch.float64, device=dev, generator=g)
            ref = torch.full((b, ld_out), 7.0, dtype=torch.float64, device=dev)
            own(plans[m], x, ref, b, ld_in, ld_out, t, t)
            if i % 5 == 4:   # in place
                ref = torch.full_like(x, 7.0)
                ref[:, N:] = x[:, N:]
                own(plans[m], x, ref, b, ld_in, ld_in, t, t)
                jobs.append((plans[m], x, x, b, ld_in, ld_in))
            else:
                jobs.append((plans[m], x, torch.full((b, ld_out), 7.0, dtype=torch.float64, device=dev), b, ld_in, ld_out))
            refs.append(ref)
        jobs.append((plans[ms[0]], None, None, 0, 1 << ms[0], 1 << ms[0]))   # batch 0: skipped
        small = [len(dwt.dwt_plan_passes(plans[m], 8)) for m in set(ms) if m < 12]
        n0 = dwt.dwt_launch_count()
        grouped(jobs, t, t)
        assert dwt.dwt_launch_count() - n0 == launches + max(small, default=0)
        for i, (job, ref) in enumerate(zip(jobs, refs)):
            assert torch.equal(job[2].view(torch.int64), ref.view(torch.int64)), (i, ms[i])
