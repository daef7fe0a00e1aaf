"""dwt_spline of few functions or few dimensions: the variance contraction in FP64
instead of digits, on both sides of the line between them."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _run(dwt, dev, plan, fs, s):
    B, N = fs.shape
    f = torch.from_numpy(fs).to(dev)
    c = torch.empty((B, N), dtype=torch.float64 if plan.p == 2 else torch.complex128, device=dev)
    v = torch.empty((2, B, s + 1), dtype=torch.float64, device=dev)
    d = torch.empty((B, 2), dtype=torch.int32, device=dev)
    dwt.dwt_profile_reset()
    dwt.dwt_profile_enable(True)
    dwt.dwt_spline(plan, f, c, B, N, v[0], v[1], d)
    torch.cuda.synchronize()
    dwt.dwt_profile_enable(False)
    fam = [n for n in ("spline_dots", "spline_dots_fp64", "spline_scale") if dwt.dwt_profile_query(n)[0]]
    dwt.dwt_profile_reset()
    return v.cpu().numpy(), d.cpu().numpy(), c.cpu().numpy(), fam


# the most functions of a round of 32 tables in FP64 and the least in digits, fewer
# tables, several rounds; labels: less than a tile (2^4, 5^3), a remainder (3^7), many
@pytest.mark.parametrize("p,m,s,few,many", [(2, 13, 16, 9, 10), (2, 11, 5, 30, 31), (2, 4, 20, 15, 33), (3, 7, 16, 9, 32),
                                            (5, 3, 64, 9, 32), (2, 15, 1, 64, 0), (2, 12, 2, 1, 0), (3, 9, 40, 11, 32)])
def test_few_functions(dwt, dev, orc, p, m, s, few, many):
    N = p ** m
    C = S.small_net(p, m, s, index=470 + m)
    Y = orc.net_points(p, m, C)
    gamma = 0.9 / np.arange(1, s + 1) ** 1.2
    plan = dwt.dwt_plan(p, m, s, C, dwt.DWT_PLAN_TRANSFORM_ONLY)
    dwt.dwt_spline_prepare(plan, 2.0, gamma)
    B = max(few, many)
    cf = S.uniform(S.stream_seed(72, S.P_COEFFS, m), B * s).reshape(B, s) / np.arange(1, s + 1)
    fs = np.stack([orc.eval_product(p, m, Y, x) for x in cf])
    v, d, c, fam = _run(dwt, dev, plan, fs[:few], s)
    assert fam == ["spline_dots_fp64"]
    for b in sorted({0, few // 2, few - 1}):
        r = orc.spline(p, m, Y, fs[b], 2.0, gamma)
        tot = r["var_trc"][-1]
        # as the other variance tests of the spline, and as well as the quotients
        # f~ / K~ are conditioned (both sides compute them in FP64)
        tol = 1e-9 + 1e-16 * np.prod(1.0 + gamma) / r["Ktil"].real.min()
        assert np.all(np.abs(v[0, b] - r["var_trc"]) <= tol * tot) and np.all(np.abs(v[1, b] - r["var_sup"]) <= tol * tot)
        assert np.linalg.norm(c[b].real - r["c"].real) <= tol * np.linalg.norm(r["c"].real)
    # one at a time: the same to the last bit
    for b in (0, few - 1):
        v1, d1, c1, _ = _run(dwt, dev, plan, fs[b:b + 1], s)
        assert np.array_equal(v1[:, 0], v[:, b]) and np.array_equal(d1[0], d[b]) and np.array_equal(c1[0], c[b])
    if many:
        w, e, _, fam = _run(dwt, dev, plan, fs[:many], s)
        assert fam == ["spline_dots"]
        n = min(few, many)
        # either form within 2^-48 of a tile's sum of magnitudes, the tiles' sums within
        # 2^-44; tables that cancel are held against the total
        tot = v[0, :n, -1][:, None]
        assert np.all(np.abs(w[:, :n] - v[:, :n]) <= 2.0 ** -43 * tot)
