"""A function's spline variances do not depend on the other functions of its call
(within one form of the contraction), whatever the number of groups and launches."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


# one group of functions against several (each with its waves of tiles), and more
# functions than the tiles' sums of one launch hold (2^26 doubles: 8192 functions of
# 128 tables in 64 tiles)
@pytest.mark.parametrize("p,m,s,B,few", [(2, 17, 12, 100, 33), (3, 9, 16, 65, 20), (2, 12, 64, 8232, 40)])
def test_variances_do_not_depend_on_the_batch(dwt, dev, p, m, s, B, few):
    N = p ** m
    plan = dwt.dwt_plan(p, m, s, S.small_net(p, m, s, index=480 + m), dwt.DWT_PLAN_TRANSFORM_ONLY)
    dwt.dwt_spline_prepare(plan, 2.0, 0.9 / np.arange(1, s + 1) ** 1.2)
    base = torch.from_numpy(S.uniform(S.stream_seed(73, S.P_VALUES, m), few * N).reshape(few, N) - 0.5).to(dev)

    def call(n):
        f = base[torch.arange(n, device=dev) % few]
        v = torch.empty((2, n, s + 1), dtype=torch.float64, device=dev)
        d = torch.empty((n, 2), dtype=torch.int32, device=dev)
        dwt.dwt_spline(plan, f, f if p == 2 else None, n, N, v[0], v[1], d)
        return v, d

    v0, d0 = call(few)
    v, d = call(B)
    assert torch.isfinite(v0).all() and (v0[0, :, -1] > 0).all()
    for b in range(0, B, few):
        n = min(few, B - b)
        assert torch.equal(v[:, b:b + n], v0[:, :n]) and torch.equal(d[b:b + n], d0[:n])
