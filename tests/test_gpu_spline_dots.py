"""The variance contraction of dwt_spline (exact digit products on the tensor
cores): sizes on both sides of its blocks, rows of very different size, special
values."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _spline(dwt, dev, plan, fs, s, with_c=True, pad=0):
    B, N = fs.shape
    f = torch.zeros((B, N + pad), dtype=torch.float64, device=dev)
    f[:, :N] = torch.from_numpy(fs)
    c = torch.zeros((B, N + pad), dtype=torch.float64 if plan.p == 2 else torch.complex128, device=dev) if with_c else None
    vt = torch.empty((B, s + 1), dtype=torch.float64, device=dev)
    vs = torch.empty((B, s + 1), dtype=torch.float64, device=dev)
    dim = torch.empty((B, 2), dtype=torch.int32, device=dev)
    dwt.dwt_spline(plan, f, c, B, N + pad, vt, vs, dim)
    return vt.cpu().numpy(), vs.cpu().numpy(), dim.cpu().numpy(), None if c is None else c[:, :N].cpu().numpy()


# fewer labels than a block (2^4), a block and a remainder (3^5 = 243, 5^4), one
# to three groups of 32 functions, one to three rounds of 32 tables
@pytest.mark.parametrize("p,m,s,B", [(2, 4, 3, 2), (2, 11, 20, 33), (3, 5, 17, 2), (5, 4, 3, 40), (2, 13, 40, 1), (2, 9, 16, 65)])
def test_sizes(dwt, dev, orc, p, m, s, B):
    N = p ** m
    C = S.small_net(p, m, s, index=400 + m)
    Y = orc.net_points(p, m, C)
    gamma = 0.9 / np.arange(1, s + 1) ** 1.2
    cf = S.uniform(S.stream_seed(64, S.P_COEFFS, m), B * s).reshape(B, s) / np.arange(1, s + 1)
    fs = np.stack([orc.eval_product(p, m, Y, cf[b]) for b in range(B)])
    plan = dwt.dwt_plan(p, m, s, C, dwt.DWT_PLAN_TRANSFORM_ONLY)
    dwt.dwt_spline_prepare(plan, 2.0, gamma)
    vt, vs, dim, c = _spline(dwt, dev, plan, fs, s, pad=1)
    vt2, vs2, dim2, _ = _spline(dwt, dev, plan, fs, s, with_c=False)
    assert np.array_equal(vt, vt2) and np.array_equal(vs, vs2) and np.array_equal(dim, dim2)
    for b in sorted({0, 1 % B, B // 2, B - 1}):
        r = orc.spline(p, m, Y, fs[b], 2.0, gamma)
        tot = r["var_trc"][-1]
        # as the other variance tests of the spline
        assert np.all(np.abs(vt[b] - r["var_trc"]) <= 1e-9 * tot)
        assert np.all(np.abs(vs[b] - r["var_sup"]) <= 1e-9 * tot)
        assert np.linalg.norm(c[b].real - r["c"].real) <= 1e-9 * np.linalg.norm(r["c"].real)


def test_rows_of_different_size_and_special_values(dwt, dev, orc):
    p, m, s, B = 2, 12, 6, 36
    N = p ** m
    C = S.small_net(p, m, s, index=420)
    f0 = orc.eval_product(p, m, orc.net_points(p, m, C), 1.0 / np.arange(1, s + 1))
    fs = np.tile(f0, (B, 1))
    # powers of two scale every variance exactly, whatever the other rows hold
    e = np.arange(B) * 20 - 360
    fs = np.ldexp(fs, e[:, None])
    fs[7, 5] = np.inf
    fs[9, 11] = np.nan
    fs[11] = 0.0
    plan = dwt.dwt_plan(p, m, s, C, dwt.DWT_PLAN_TRANSFORM_ONLY)
    dwt.dwt_spline_prepare(plan, 2.0, 0.9 / np.arange(1, s + 1))
    vt, vs, dim, _ = _spline(dwt, dev, plan, fs, s)
    ref = 18                       # scaled by 2^0
    assert np.isfinite(vt[ref]).all() and vt[ref, -1] > 0
    for b in range(B):
        if b in (7, 9):
            assert not np.isfinite(vt[b, 1:]).any() and not np.isfinite(vs[b, 1:]).any()
        elif b == 11:
            assert (vt[b] == 0).all() and (vs[b] == 0).all() and (dim[b] == 0).all()
        else:
            assert np.array_equal(vt[b], np.ldexp(vt[ref], 2 * e[b])) and np.array_equal(vs[b], np.ldexp(vs[ref], 2 * e[b]))
            assert np.array_equal(dim[b], dim[ref])


# the coefficients' buffer holds the intermediate values unless it shares memory
# with the samples: in place (p = 2), or samples inside the complex coefficients
@pytest.mark.parametrize("p,m,off", [(2, 13, 0), (2, 13, 40), (3, 6, 0), (3, 6, 729)])
def test_samples_inside_the_coefficients(dwt, dev, orc, p, m, off):
    N, s, B = p ** m, 3, 3
    C = S.small_net(p, m, s, index=430 + m)
    f0 = orc.eval_product(p, m, orc.net_points(p, m, C), 1.0 / np.arange(1, s + 1))
    fs = f0[None, :] * np.array([[1.0], [-2.5], [0.3]])
    plan = dwt.dwt_plan(p, m, s, C, dwt.DWT_PLAN_TRANSFORM_ONLY)
    dwt.dwt_spline_prepare(plan, 2.0, 0.9 / np.arange(1, s + 1))
    vt, vs, dim, c = _spline(dwt, dev, plan, fs, s)
    buf = torch.zeros(2 * B * N + 64, dtype=torch.float64, device=dev)
    f = buf[off:off + B * N].view(B, N)
    f.copy_(torch.from_numpy(fs))
    cb = buf[:B * N].view(B, N) if p == 2 else torch.view_as_complex(buf[:2 * B * N].view(B, N, 2))
    v = torch.empty((2, B, s + 1), dtype=torch.float64, device=dev)
    d = torch.empty((B, 2), dtype=torch.int32, device=dev)
    dwt.dwt_spline(plan, f, cb, B, N, v[0], v[1], d)
    assert np.array_equal(cb.cpu().numpy(), c)
    assert np.array_equal(v[0].cpu().numpy(), vt) and np.array_equal(v[1].cpu().numpy(), vs)
    assert np.array_equal(d.cpu().numpy(), dim)


def test_squares_near_the_largest_number(dwt, dev, orc):
    # rows whose squares come near the largest double, or pass it, take FP64 sums:
    # finite ones within 2^12 roundings of the scaled row, the others infinite
    p, m, s = 2, 12, 6
    C = S.small_net(p, m, s, index=440)
    f0 = orc.eval_product(p, m, orc.net_points(p, m, C), 1.0 / np.arange(1, s + 1))
    e = np.array([0, 470, 490, 500, 530, 600])
    fs = np.ldexp(f0[None, :], e[:, None])
    plan = dwt.dwt_plan(p, m, s, C, dwt.DWT_PLAN_TRANSFORM_ONLY)
    dwt.dwt_spline_prepare(plan, 2.0, 0.9 / np.arange(1, s + 1))
    vt, vs, _, _ = _spline(dwt, dev, plan, fs, s)
    with np.errstate(over="ignore"):
        for b in range(len(e)):
            for v in (vt, vs):
                want = np.ldexp(v[0], 2 * e[b])
                if e[b] >= 530:
                    assert not np.isfinite(v[b, 1:]).any()
                else:
                    assert np.allclose(v[b], want, rtol=0, atol=2.0 ** -41 * want[-1])


def test_tiles_of_several_waves(dwt, dev, orc):
    # 10 groups of functions times 1024 blocks of labels: two waves of tiles of 18
    # blocks and a shorter last one, against one function's tiles of one wave and
    # the oracle
    p, m, s, B = 2, 16, 2, 320
    C = S.small_net(p, m, s, index=450)
    Y = orc.net_points(p, m, C)
    gamma = 0.9 / np.arange(1, s + 1)
    f0 = orc.eval_product(p, m, Y, 1.0 / np.arange(1, s + 1))
    fs = f0[None, :] * (1.0 + np.arange(B)[:, None] / 64.0)
    plan = dwt.dwt_plan(p, m, s, C, dwt.DWT_PLAN_TRANSFORM_ONLY)
    dwt.dwt_spline_prepare(plan, 2.0, gamma)
    vt, vs, dim, _ = _spline(dwt, dev, plan, fs, s)
    r = orc.spline(p, m, Y, fs[319], 2.0, gamma)
    assert np.all(np.abs(vt[319] - r["var_trc"]) <= 1e-9 * r["var_trc"][-1])
    for b in (0, 31, 32, 200, 319):
        v1, w1, d1, _ = _spline(dwt, dev, plan, fs[b:b + 1], s)
        # sums of 2^10 tiles at most, rounded at 2^-53 each
        assert np.all(np.abs(vt[b] - v1[0]) <= 2.0 ** -43 * v1[0, -1]) and np.all(np.abs(vs[b] - w1[0]) <= 2.0 ** -43 * v1[0, -1])
        assert np.array_equal(dim[b], d1[0])
