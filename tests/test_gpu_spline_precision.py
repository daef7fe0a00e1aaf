"""The variance contraction of dwt_spline keeps FP64's relative precision when the
numbers of a tile differ widely: its inputs (tables and coefficients) are formed
here to the last bit and summed in 80 bits."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _transform(x, m):
    """The FP64 forward transform as the library rounds it for p = 2, m = 12 .. 20:
    exact sums over the 12 low digits rounded once, then over the others."""
    one = 1 << 220
    v = np.array([[int(a * 2.0 ** 100) * (one >> 100) if a * 2.0 ** 100 == np.floor(a * 2.0 ** 100) else
                   int(a * 2.0 ** 160) * (one >> 160) for a in row] for row in x], dtype=object)
    n = 1 << m
    h = 1
    while h < n:
        u = v.reshape(len(x), n // (2 * h), 2, h)
        v = np.stack((u[:, :, 0] + u[:, :, 1], u[:, :, 0] - u[:, :, 1]), 2).reshape(len(x), n)
        h *= 2
        if h in (1 << 12, n):   # int / int is rounded correctly
            y = np.array([[a / one for a in row] for row in v])
            if h < n:
                v = np.array([[int(a * 2.0 ** 160) * (one >> 160) for a in row] for row in y], dtype=object)
    return y * 2.0 ** -m


@pytest.mark.parametrize("m", [12, 16])
def test_numbers_of_very_different_size(dwt, dev, orc, m):
    p, s, N = 2, 2, 1 << m
    C = S.small_net(p, m, s, index=460)
    Y = orc.net_points(p, m, C)
    gamma = np.array([0.5, 0.25])
    # kernel data, alpha = 2 (K' and the products of two are exact, R' is 4/14 of dyadic numbers)
    i = np.arange(m + 1)
    kp = np.where(i == 0, 1.0, 1.0 - 3.0 * 2.0 ** -i)
    rp = np.where(i == 0, 4.0 / 14.0, 4.0 / 14.0 * (1.0 - 15.0 * 2.0 ** (-3.0 * i)))
    pos = np.zeros(N, dtype=int)
    pos[1:] = m - np.floor(np.log2(np.arange(1, N))).astype(int)
    x0, x1 = pos[Y[0]], pos[Y[1]]
    a0, a1 = 0.25 * rp[x0], 0.0625 * rp[x1]
    K = (1.0 + 0.5 * kp[x0]) * (1.0 + 0.25 * kp[x1])
    rows = np.stack((K, 1.0 + a0, (1.0 + a0) * (1.0 + a1), a0 + a1, a1 * a0))
    # functions: random values, one point, a smooth one, coefficients from 1 to 2^-50
    rnd = S.uniform(S.stream_seed(71, S.P_VALUES, m), N) - 0.5
    point = np.zeros(N)
    point[5] = 1.0
    h = np.arange(N)
    coef = 2.0 ** -(h % 51).astype(float)
    n = 1
    while n < N:
        u = coef.reshape(-1, 2, n)
        coef = np.stack((u[:, 0] + u[:, 1], u[:, 0] - u[:, 1]), 1).reshape(-1)
        n *= 2
    fs = np.stack((rnd, point, orc.eval_product(p, m, Y, np.array([0.9, 0.4])), np.round(coef * 2.0 ** 60) * 2.0 ** -60))
    T = _transform(rows, m)
    ft = _transform(fs, m)
    W = 1.0 / (N * T[0])
    tab = T[1:].copy()
    tab[:2, 0] -= 1.0
    c = (ft * W).astype(np.longdouble)
    v = (c * c) @ tab.astype(np.longdouble).T * np.longdouble(N) ** 2
    ref = np.stack((v[:, 0], v[:, 1], v[:, 2], v[:, 2] + v[:, 3]), 1)

    plan = dwt.dwt_plan(p, m, s, C, dwt.DWT_PLAN_TRANSFORM_ONLY)
    dwt.dwt_spline_prepare(plan, 2.0, gamma)
    # as many copies as give whole groups of functions, and a few functions alone
    for B in (64, 4, 1):
        f = torch.from_numpy(np.tile(fs, (16, 1))[:B]).to(dev)
        g = torch.empty_like(f)
        vt = torch.empty((B, s + 1), dtype=torch.float64, device=dev)
        vs = torch.empty((B, s + 1), dtype=torch.float64, device=dev)
        dwt.dwt_spline(plan, f, g, B, N, vt, vs)
        got = np.concatenate((vt.cpu().numpy()[:, 1:], vs.cpu().numpy()[:, 1:]), 1)
        want = np.tile(ref, (16, 1))[:B]
        err = np.abs((got - want) / want).astype(float)
        # a tile's sum within 2^-48 (FP64: 2^-53 for the square, the product and each of
        # the 24 additions of 4096 labels), then at most 305 tiles, lanes and a tree of
        # 2^-53 each, the factor and one more sum: below 2^-48 + 320 2^-53
        assert err.max() < 2.0 ** -48 + 320 * 2.0 ** -53, (B, err.max(0))
