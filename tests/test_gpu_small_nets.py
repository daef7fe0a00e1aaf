"""The one-launch interpolation of small p = 2 nets (2^8 .. 2^14 points) and the
reduction of class partials to variances and dimensions."""
import ctypes

import numpy as np
import pytest
import torch

import synthetic as S
from conftest import rel_l2

pytestmark = pytest.mark.gpu


def _np(t):
    return t.detach().cpu().numpy()


def _classes(dwt, plan):
    _, cp = dwt.dwt_plan_tables(plan)
    cls = np.empty((plan.N, 2), dtype=np.uint8)
    rt = ctypes.CDLL("libcudart.so")
    rt.cudaMemcpy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]
    torch.cuda.synchronize()
    assert rt.cudaMemcpy(cls.ctypes.data, cp, cls.nbytes, 2) == 0
    return cls


# every size; s from one class pair to 255 (one binning warp, 64 KB of bins);
# rows that start on any element; in place; weighted or not; with or without
# the optional outputs.  Tolerances: 2 m FP32 additions per point, each within
# 2^-24 of partial sums no larger than the norm, stay below 1e-5; class sums of
# at most 2^14 positive FP32 terms in chains of at most 2^9: 2^9 2^-24 = 3e-5
# in the worst case, a tenth of it in practice.
@pytest.mark.parametrize("m,s,pad,weight,inplace", [
    (8, 1, 0, 1, False), (8, 7, 3, 0, True), (9, 64, 1, 1, False), (10, 5, 0, 1, True), (11, 17, 2, 1, False),
    (12, 255, 0, 1, False), (13, 3, 5, 0, False), (13, 24, 0, 1, True), (14, 2, 1, 1, False), (14, 255, 4, 1, True)])
def test_small_interpolate(dwt, dev, orc, m, s, pad, weight, inplace):
    p, N, B = 2, 1 << m, 3
    ld = N + pad
    C = S.small_net(p, m, s, index=40 + m)
    plan = dwt.dwt_plan(p, m, s, C)
    Y = orc.net_points(p, m, C)
    cf = S.uniform(S.stream_seed(31, S.P_COEFFS, m), B * s).reshape(B, s) / (1.0 + np.arange(s))
    f = torch.zeros((B, ld), device=dev)
    for b in range(B):
        f[b, :N] = torch.from_numpy(orc.eval_product(p, m, Y, cf[b]).astype(np.float32))
    fin = _np(f).astype(np.float64)
    cls = _classes(dwt, plan)
    W = orc.coset_leaders_dp(p, m, C)["W64"] if weight else np.ones(N)
    c = f if inplace else torch.full((B, ld), -7.0, device=dev)
    g = torch.full((B, ld), -7.0, device=dev)
    var = torch.full((B, 2, s + 1), -1.0, dtype=torch.float64, device=dev)
    dim = torch.full((B, 2), -1, dtype=torch.int32, device=dev)
    n0 = dwt.dwt_launch_count()
    dwt.dwt_interpolate(plan, f, c, g, B, ld, dwt.DWT_F32, weight, var=var, dim=dim, threshold=0.95)
    assert dwt.dwt_launch_count() == n0 + 1
    if not inplace and pad:
        assert (c[:, N:] == -7.0).all() and (g[:, N:] == -7.0).all()
    only = torch.empty((B, ld), device=dev)
    if not inplace:
        dwt.dwt_interpolate(plan, f, only, None, B, ld, dwt.DWT_F32, weight)
        assert torch.equal(only[:, :N], c[:, :N])
    for b in range(B):
        cref, gref, vt, vs, dt, ds = orc.interpolate(p, m, fin[b, :N], W, cls, s, 0.95)
        assert rel_l2(_np(c)[b, :N], cref.real) < 1e-5
        assert rel_l2(_np(g)[b, :N], gref.real) < 1e-5
        v = _np(var)[b]
        assert np.allclose(v[0], vt, rtol=3e-5, atol=1e-14 * vt[-1])
        assert np.allclose(v[1], vs, rtol=3e-5, atol=1e-14 * vt[-1])
        for got, ref, x in ((int(dim[b, 0]), dt, vt), (int(dim[b, 1]), ds, vs)):
            lo, hi = sorted((got, ref))
            assert all(abs(x[d] / vt[-1] - 0.95) < 1e-6 for d in range(lo, hi))


# one CTA or a cluster per function (s = 255: 2^15 and 2^16 points lie on the two
# sides of the line), fewer partials than lanes, odd counts; classes that add
# nothing leave the dimension at threshold 1 where the last contribution is
@pytest.mark.parametrize("p,m,s", [(2, 13, 3), (2, 15, 255), (2, 16, 255), (3, 13, 8), (2, 22, 31)])
def test_effdim_reduction(dwt, dev, orc, p, m, s):
    N, B = p ** m, 2
    plan = dwt.dwt_plan(p, m, s, S.small_net(p, m, s, index=60 + m))
    cls = _classes(dwt, plan)
    x = S.uniform(S.stream_seed(32, S.P_VALUES, m), B * N).reshape(B, N).astype(np.float32)
    x[1][cls[:, 0] > 2] = 0.0
    g = torch.from_numpy(x).to(dev)
    if p > 2:
        g = torch.complex(g, torch.zeros_like(g))
    var = torch.empty((B, 2, s + 1), dtype=torch.float64, device=dev)
    dim = torch.empty((B, 2), dtype=torch.int32, device=dev)
    dwt.dwt_effdim_packed(plan, g, B, N, dwt.DWT_F32 if p == 2 else dwt.DWT_C64, var=var, dim=dim, threshold=1.0)
    for b in range(B):
        q = x[b].astype(np.float64) ** 2
        q[0] = 0.0
        for k in range(2):
            ref = np.cumsum(np.bincount(cls[:, k], weights=q, minlength=s + 1)[:s + 1])
            assert np.allclose(_np(var)[b, k], ref, rtol=1e-5)
        v = _np(var)[b]
        assert int(dim[b, 0]) == int(np.argmax(v[0] >= v[0, -1]))
        assert int(dim[b, 1]) == (int(np.argmax(v[1] >= v[0, -1])) if (v[1] >= v[0, -1]).any() else 0)
    assert int(dim[1, 0]) <= 2
