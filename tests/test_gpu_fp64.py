"""The FP64 transform of p = 2 nets from 2^12 points (integer stages, one
rounding per pass): every split of the digits into passes, values whose results
are exact, special values."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _fwht(x):
    """Walsh-Hadamard transform along the last axis, in x's type."""
    n = x.shape[-1]
    h = 1
    while h < n:
        v = x.reshape(-1, n // (2 * h), 2, h)
        x = np.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), 2).reshape(-1, n)
        h *= 2
    return x


def _call(dwt, dev, m, x, inverse, pad=0):
    B, N = x.shape
    plan = dwt.dwt_plan(2, m, 1, S.small_net(2, m, 1), dwt.DWT_PLAN_TRANSFORM_ONLY)
    f = torch.zeros((B, N + pad), dtype=torch.float64, device=dev)
    f[:, :N] = torch.from_numpy(x)
    y = torch.full((B, N + pad), 3.0, dtype=torch.float64, device=dev)
    (dwt.dwt_inverse if inverse else dwt.dwt_forward)(plan, f, y, B, N + pad, N + pad, dwt.DWT_F64, dwt.DWT_F64)
    assert (y[:, N:] == 3.0).all()
    z = f.clone()
    (dwt.dwt_inverse if inverse else dwt.dwt_forward)(plan, z, z, B, N + pad, N + pad, dwt.DWT_F64, dwt.DWT_F64)
    assert torch.equal(z[:, :N].contiguous().view(torch.int64), y[:, :N].contiguous().view(torch.int64))
    return y[:, :N].cpu().numpy()


# 12: one pass; 13 .. 21: 1 .. 9 high digits; 22, 24: two high passes.  Whole
# numbers with sums below 2^53 are exact in every order; magnitudes from 1 to
# 2^26 in one tile.
@pytest.mark.parametrize("m,inverse,pad", [(12, False, 0), (12, True, 1), (13, False, 3), (14, True, 0), (15, False, 0),
                                           (16, True, 1), (17, False, 0), (18, True, 2), (19, False, 1), (20, True, 0),
                                           (21, False, 0), (22, True, 0), (24, False, 0)])
def test_exact_values(dwt, dev, m, inverse, pad):
    B, N = 2, 1 << m
    u = S.splitmix64(S.stream_seed(41, S.P_VALUES, m), B * N)
    x = ((u >> np.uint64(38)).astype(np.int64) - (1 << 25)) >> (u & np.uint64(15)).astype(np.int64)
    x = x.reshape(B, N)
    got = _call(dwt, dev, m, x.astype(np.float64), inverse, pad)
    ref = _fwht(x).astype(np.float64) * (1.0 if inverse else 2.0 ** -m)
    assert np.array_equal(got, ref)


# One rounding of 2^-53 per pass (three passes at most) and nothing else of that
# size: within 3 2^-53 of the norm, against 80-bit sums.
@pytest.mark.parametrize("m", [12, 17, 20, 22])
def test_one_rounding_per_pass(dwt, dev, m):
    N = 1 << m
    x = (S.uniform(S.stream_seed(42, S.P_VALUES, m), N) - 0.3).reshape(1, N)
    got = _call(dwt, dev, m, x, True)
    ref = _fwht(x.astype(np.longdouble))
    err = np.linalg.norm((got - ref).astype(np.float64)) / np.linalg.norm(ref.astype(np.float64))
    assert err < 3 * 2.0 ** -53


# columns of a high pass that differ by many orders keep their own precision:
# function 0 varies in the 12 low digits only, function 1 in all with a decay
def test_columns_of_different_size(dwt, dev):
    m, N = 20, 1 << 20
    h = np.arange(N)
    x = np.stack((np.where(h < 4096, 2.0 ** -(h % 40).astype(float), 0.0), 2.0 ** -(h % 64).astype(float)))
    got = _call(dwt, dev, m, x, True)
    ref = _fwht(x.astype(np.longdouble))
    assert np.abs(got - ref).max() < 1e-15 * np.abs(ref).max()


@pytest.mark.parametrize("m", [12, 16, 20])
def test_special_values(dwt, dev, m):
    N = 1 << m
    x = (S.uniform(S.stream_seed(43, S.P_VALUES, m), 4 * N) - 0.5).reshape(4, N)
    x[0, 5] = np.inf
    x[1, 7] = np.nan
    x[2, 3], x[2, N - 1] = np.inf, np.inf
    # multiples of the smallest subnormal: exact
    x[3] = np.floor(x[3] * 2.0 ** 20) * 2.0 ** -1074
    got = _call(dwt, dev, m, x, True)
    with np.errstate(invalid="ignore"):
        ref = _fwht(x)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(got[[0, 2, 3]], ref[[0, 2, 3]], equal_nan=True)
    z = _call(dwt, dev, m, np.zeros((1, N)), False)
    assert np.array_equal(z, np.zeros((1, N)))
