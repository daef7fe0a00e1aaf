"""The FP64 transform of p = 2 nets (integer stages): elements far below their
tile's largest where the large ones cancel, and columns of very different size."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _inverse(dwt, dev, m, x):
    N = 1 << m
    plan = dwt.dwt_plan(2, m, 1, S.small_net(2, m, 1), dwt.DWT_PLAN_TRANSFORM_ONLY)
    f = torch.from_numpy(x).to(dev)
    y = torch.empty_like(f)
    dwt.dwt_inverse(plan, f, y, x.shape[0], N, N, dwt.DWT_F64, dwt.DWT_F64)
    dwt.dwt_inverse(plan, f, f, x.shape[0], N, N, dwt.DWT_F64, dwt.DWT_F64)
    assert torch.equal(f.view(torch.int64), y.view(torch.int64))
    return y.cpu().numpy()


def _fwht(x):
    n = x.shape[-1]
    h = 1
    while h < n:
        v = x.reshape(-1, n // (2 * h), 2, h)
        x = np.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), 2).reshape(-1, n)
        h *= 2
    return x


# Four parts by the digits a and b of the last pass: 1, 2^-100, whole multiples of
# 2^-200 and of 2^-400 below 2^20.  A constant part reaches one element of the low
# digits only, so that every other sum is one of whole numbers below 2^53 of the small
# parts: exact, or rounded once.  The last pass has 12 (m = 12, the only one), 4, 8, 9
# and 5 digits (m = 16, 20, 21, 22).
@pytest.mark.parametrize("m,a,b", [(12, 0, 11), (12, 5, 7), (16, 12, 15), (20, 13, 19), (21, 20, 12), (22, 17, 21)])
def test_small_elements_where_large_ones_cancel(dwt, dev, m, a, b):
    N = 1 << m
    h = np.arange(N)
    part = ((h >> a) & 1) + 2 * ((h >> b) & 1)
    k = (S.splitmix64(S.stream_seed(81, S.P_VALUES, m), N) >> np.uint64(44)).astype(np.int64)
    x = np.where(part == 0, 1.0, np.where(part == 1, 2.0 ** -100, k * np.where(part == 2, 2.0 ** -200, 2.0 ** -400)))
    got = _inverse(dwt, dev, m, x.reshape(1, N))[0]
    # the four parts apart: exact in 64-bit integers, added up exactly
    ref = [0] * N
    for q, e in ((0, 400), (1, 300), (2, 200), (3, 0)):
        s = _fwht(np.where(part == q, k if q >= 2 else 1, 0).reshape(1, N))[0]
        for i in np.nonzero(s)[0]:
            ref[i] += int(s[i]) << e
    one = 1 << 400
    ref = np.array([r / one for r in ref])   # rounded correctly
    # one rounding per pass (of a column's sums) and one more where levels are added
    assert np.all(np.abs(got - ref) <= 2.0 ** -51 * np.abs(ref))


# The columns of the high pass (one per value of the low digits) lie up to 2^-50
# apart: one exponent for a whole tile would round them all at the largest.
@pytest.mark.parametrize("m", [16, 20, 21])
def test_each_column_keeps_its_own_exponent(dwt, dev, m):
    N, low = 1 << m, 1 << 12
    u = (S.uniform(S.stream_seed(82, S.P_VALUES, m), N) - 0.5).reshape(-1, low) * 2.0 ** -(8.0 * (np.arange(low) % 12))
    # samples whose low pass delivers u, in whole multiples of 2^-58
    X = np.round(_fwht(u) * 2.0 ** 46).astype(np.int64)
    assert np.abs(X).max() < 1 << 53
    got = _inverse(dwt, dev, m, (X * 2.0 ** -58).reshape(1, N)).reshape(-1, low)
    # exact in two 64-bit halves, added in 80 bits
    hi, lo = X >> 27, X & ((1 << 27) - 1)
    ref = (_fwht(hi.reshape(1, N)).astype(np.longdouble) * 2.0 ** 27 + _fwht(lo.reshape(1, N))).reshape(-1, low) * 2.0 ** -58
    col = np.abs(ref).max(0)
    assert col.min() < 2.0 ** -45 * col.max()
    # the low pass rounds each of a column's 2^b numbers at 2^-53, the high pass each
    # result: at most 2^-53 (2^b max / largest result + 1), the largest result at least
    # 2^(b/2) rms, so 2^-53 (2^4.5 4 + 1) < 1e-14 of the column's largest
    err = np.abs(got - ref).max(0)
    assert np.all(err <= 1e-14 * col), float((err / col).max())
