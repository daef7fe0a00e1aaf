"""Workloads of the library's public calls, with their inputs, minimum work and 64-bit values.

A case names a call and its sizes:

  kind      interpolate  dwt_interpolate: forward, weight, variance classes, inverse (Sec. 3, Sec. 4)
            forward      dwt_forward (Algorithm 1)
            inverse      dwt_inverse (Algorithm 2)
            grouped      dwt_forward_grouped: several nets of different sizes in one call
            spline       dwt_spline: the FP64 kernel spline and its ANOVA variances
            request      a whole request on a net of its own: dwt_plan, dwt_eval_product,
                         dwt_interpolate, dwt_plan_destroy_async (what the serving engine runs)
  p, m, s   the digital net: p^m points in s dimensions
  batch     functions per call
  pad       elements between functions beyond p^m (ld = p^m + pad)
  dtype     element type of the samples (and of the coefficients of an inverse)

Nets are random nonsingular upper-triangular generating matrices, functions are product
functions prod_j (1 + c_j (x_j - 1/2)) sampled at the net points, the coefficients of an
inverse decay with their label, integers are uniform in -1000..1000.
"""
import math

import numpy as np
import torch

import paper_0808_0487_gb300 as dwt

DEV = "cuda"
POINTS = 1 << 29          # samples of the largest call: 32 functions of 2^24 points


def listed():
    return [
        # the paper's net of Sec. 5.2 (2^12 points): one function per call, bound by latency and launches
        dict(name="interpolate_p2_m12_s4_b1", kind="interpolate", p=2, m=12, s=4, batch=1, pad=0, dtype="f32"),
        # an ordinary net of the serving mix, an odd number of functions
        dict(name="interpolate_p2_m17_s24_b7", kind="interpolate", p=2, m=17, s=24, batch=7, pad=0, dtype="f32"),
        # the mid-sized workload, every function's passes within L2
        dict(name="interpolate_p2_m20_s16_b32", kind="interpolate", p=2, m=20, s=16, batch=32, pad=0, dtype="f32"),
        # the benchmark's step: 2 GiB in, 2 GiB out
        dict(name="interpolate_p2_m24_s32_b32", kind="interpolate", p=2, m=24, s=32, batch=32, pad=0, dtype="f32"),
        # an odd prime: real samples, complex coefficients, rows padded to a multiple of four
        dict(name="interpolate_p3_m13_s8_b4", kind="interpolate", p=3, m=13, s=8, batch=4, pad=1, dtype="f32"),
        # the transform alone, FP32, many functions
        dict(name="forward_p2_m20_f32_b32", kind="forward", p=2, m=20, s=16, batch=32, pad=0, dtype="f32"),
        # the exact integer transform, the other direction
        dict(name="inverse_p2_m20_i32_b32", kind="inverse", p=2, m=20, s=16, batch=32, pad=0, dtype="i32"),
        # one ternary transform of real samples: less than one wave of blocks per pass
        dict(name="forward_p3_m13_f32_b1", kind="forward", p=3, m=13, s=8, batch=1, pad=1, dtype="f32"),
        # complex coefficients of a quinary net back to samples (the largest p = 5 net of the serving mix)
        dict(name="inverse_p5_m9_c64_b32", kind="inverse", p=5, m=9, s=8, batch=32, pad=0, dtype="c64"),
        # a batch of small nets of different sizes in one call
        dict(name="grouped_p2_m8_15_b4", kind="grouped", p=2, m=8, m1=15, s=1, batch=4, pad=0, dtype="f32"),
        # the kernel spline of the mid-sized workload, FP64 throughout
        dict(name="spline_p2_m20_s16_b32", kind="spline", p=2, m=20, s=16, batch=32, pad=0, dtype="f64"),
        # one request of the serving mix: plan build included, one function
        dict(name="request_p2_m15_s33_b1", kind="request", p=2, m=15, s=33, batch=1, pad=0, dtype="f32"),
    ]


def draw(rng):
    kind = rng.choice(["interpolate"] * 8 + ["forward"] * 4 + ["inverse"] * 4 + ["grouped", "spline", "request", "request"])
    p = rng.choice([2] * 5 + [3] * 3 + [5] * 2 + [7, 13, 31])
    top = 24 if p == 2 and kind in ("interpolate", "forward", "inverse") else 20
    m = max(1, round(rng.uniform(8.0, top) / math.log2(p)))
    while p ** m > 1 << top:
        m -= 1
    s = round(2.0 ** rng.uniform(1.0, 6.0))
    dtype = "f32"
    if kind in ("forward", "inverse"):
        real = ["f32", "f32", "f32", "f64", "i32"] if p == 2 else ["f32", "f32", "f64"]
        dtype = rng.choice(real if p == 2 or kind == "forward" else ["c64", "c64", "c128"])
        if p > 2 and kind == "forward":
            dtype = rng.choice([dtype, "c64"])
    cap = POINTS if p == 2 and dtype in ("f32", "i32") else 1 << 25
    pad = rng.choice([0, 0, 0, 4, rng.randrange(1, 9)])
    if p == 2 and pad % 4:
        cap = 1 << 26     # rows that do not start on 16 bytes
    if dtype == "i32":
        m = min(m, 20)    # 2^m * 1000 < 2^31
    if kind == "spline":
        s, dtype, cap = min(s, 24), "f64", 1 << 24
    if kind in ("grouped", "request"):
        pad = 0
    if kind == "grouped":
        m = max(1, m // 2)
    batch = 1 if kind == "request" else max(1, round(2.0 ** rng.uniform(0.0, min(6.5, math.log2(max(1, cap // p ** m))))))
    case = dict(kind=kind, p=p, m=m, s=s, batch=batch, pad=pad, dtype=dtype)
    if kind == "grouped":
        case["m1"] = m + rng.randrange(1, 6 if p == 2 else 3)
    return case


# ---- inputs ---------------------------------------------------------------

def matrices(rng, p, m, s):
    """Nonsingular upper-triangular generating matrices, uint8 [s][m][m]."""
    C = np.triu(rng.randint(0, p, size=(s, m, m)), 1)
    d = np.arange(m)
    C[:, d, d] = rng.randint(1, p, size=(s, m)) if p > 2 else 1
    return C.astype(np.uint8)


def numerators(p, m, Cj):
    """Y_n = sum_i y_{n,i} p^(m-i) of one coordinate (int64 [p^m]), y = C_j n over F_p (Def. 1.1)."""
    Y = torch.zeros(p ** m, dtype=torch.int64, device=DEV)
    a = torch.arange(p, dtype=torch.int16, device=DEV)[:, None]
    for i in range(m):
        v = torch.zeros(1, dtype=torch.int16, device=DEV)
        for c in range(m):
            x = int(Cj[i, c])
            v = ((v[None, :] + a * x) % p if p > 2 else v[None, :] ^ (a * x)).reshape(-1)
        Y += v.long() * p ** (m - 1 - i)
    return Y


def functions(p, m, C, coef, dtype):
    """prod_j (1 + coef[b][j] (x_j - 1/2)) at the net points, [batch][p^m]."""
    f = torch.ones((coef.shape[0], p ** m), dtype=dtype, device=DEV)
    for j in range(C.shape[0]):
        x = (numerators(p, m, C[j]).double() / p ** m - 0.5).to(dtype)
        for b in range(0, f.shape[0], 8):
            f[b:b + 8] *= 1 + coef[b:b + 8, j:j + 1].to(dtype) * x
    return f


TORCH = {"f32": torch.float32, "f64": torch.float64, "i32": torch.int32, "c64": torch.complex64, "c128": torch.complex128}
CODE = {"f32": dwt.DWT_F32, "f64": dwt.DWT_F64, "i32": dwt.DWT_I32, "c64": dwt.DWT_C64, "c128": dwt.DWT_C128}


def out_type(p, dtype):
    return dtype if p == 2 else {"f32": "c64", "f64": "c128"}.get(dtype, dtype)


def samples(case, seed):
    """C, the functions' coefficients and the samples [batch][p^m] (of a grouped call: lists of them)."""
    p, m, s, B, kind, dtype = (case[k] for k in ("p", "m", "s", "batch", "kind", "dtype"))
    rng = np.random.RandomState(seed & 0x7FFFFFFF)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if kind == "grouped":
        nets = [matrices(rng, p, mm, s) for mm in range(m, case["m1"] + 1)]
        coef = torch.rand((B, s), generator=gen, dtype=torch.float64, device=DEV)
        return nets, coef, [functions(p, C.shape[1], C, coef, TORCH[dtype]) for C in nets]
    C = matrices(rng, p, m, s)
    coef = torch.rand((B, s), generator=gen, dtype=torch.float64, device=DEV)
    if m == 24:     # the benchmark's functions: coefficients about 1 / j^2
        coef = (0.5 + coef) / torch.arange(1, s + 1, dtype=torch.float64, device=DEV) ** 2
    if kind == "request":
        return C, coef, None
    if dtype == "i32":
        return C, coef, torch.randint(-1000, 1001, (B, p ** m), generator=gen, dtype=torch.int32, device=DEV)
    if kind == "inverse":
        f = torch.randn((B, p ** m), generator=gen, dtype=TORCH[dtype], device=DEV)
        f /= 1 + torch.arange(p ** m, device=DEV).to(f.real.dtype)
        return C, coef, f
    f = functions(p, m, C, coef, TORCH[{"c64": "f32", "c128": "f64"}.get(dtype, dtype)])
    if dtype in ("c64", "c128"):
        f = torch.complex(f, f.flip(0))
    return C, coef, f


def padded(x, ld):
    y = torch.zeros((x.shape[0], ld), dtype=x.dtype, device=DEV)
    y[:, :x.shape[1]] = x
    return y


def kernel_weights(s):
    return [0.9 / (j + 1) ** 1.2 for j in range(s)]


def prepare(case, seed):
    p, m, s, B, kind, dtype = (case[k] for k in ("p", "m", "s", "batch", "kind", "dtype"))
    N = p ** m
    ld = N + case["pad"]
    C, coef, f = samples(case, seed)
    st = dict(case=case, N=N, ld=ld, C=C, coef=coef)
    if kind == "grouped":
        st["plans"] = [dwt.dwt_plan(p, c.shape[1], s, c, dwt.DWT_PLAN_TRANSFORM_ONLY) for c in C]
        st["f"] = f
        st["c"] = [torch.zeros(x.shape, dtype=TORCH[out_type(p, dtype)], device=DEV) for x in f]
        st["jobs"] = [(pl, x, c, B, pl.N, pl.N) for pl, x, c in zip(st["plans"], f, st["c"])]
        return st
    if kind == "request":
        st["f"] = torch.zeros((B, ld), dtype=torch.float32, device=DEV)
    else:
        st["plan"] = dwt.dwt_plan(p, m, s, C, 0 if kind == "interpolate" else dwt.DWT_PLAN_TRANSFORM_ONLY)
        st["f"] = f if ld == N else padded(f, ld)
    st["c"] = torch.zeros((B, ld), dtype=TORCH[out_type(p, dtype)], device=DEV)
    if kind in ("interpolate", "request"):
        st["var"] = torch.zeros((B, 2, s + 1), dtype=torch.float64, device=DEV)
        st["dim"] = torch.zeros((B, 2), dtype=torch.int32, device=DEV)
    if kind == "spline":
        dwt.dwt_spline_prepare(st["plan"], 2.0, kernel_weights(s))
        st["vt"] = torch.zeros((B, s + 1), dtype=torch.float64, device=DEV)
        st["vs"] = torch.zeros((B, s + 1), dtype=torch.float64, device=DEV)
        st["dim"] = torch.zeros((B, 2), dtype=torch.int32, device=DEV)
    return st


def run(st):
    case = st["case"]
    p, m, s, B, kind, dtype = (case[k] for k in ("p", "m", "s", "batch", "kind", "dtype"))
    N, ld, f, c = st["N"], st["ld"], st["f"], st["c"]
    t_in, t_out = CODE[dtype], CODE[out_type(p, dtype)]
    if kind == "interpolate":
        dwt.dwt_interpolate(st["plan"], f, c, None, B, ld, t_in, dwt.DWT_WEIGHT_INV_SQ_WAVENUMBER, var=st["var"], dim=st["dim"])
        return c[:, :N], st["var"], st["dim"]
    if kind == "request":
        plan = dwt.dwt_plan(p, m, s, st["C"])
        dwt.dwt_eval_product(plan, st["coef"], f, B, ld, t_in)
        dwt.dwt_interpolate(plan, f, c, None, B, ld, t_in, dwt.DWT_WEIGHT_INV_SQ_WAVENUMBER, var=st["var"], dim=st["dim"])
        dwt.dwt_plan_destroy_async(plan)
        return c[:, :N], st["var"], st["dim"]
    if kind == "forward":
        dwt.dwt_forward(st["plan"], f, c, B, ld, ld, t_in, t_out)
        return c[:, :N]
    if kind == "inverse":
        dwt.dwt_inverse(st["plan"], f, c, B, ld, ld, t_in, t_out)
        return c[:, :N]
    if kind == "grouped":
        dwt.dwt_forward_grouped(st["jobs"], t_in, t_out)
        return c
    dwt.dwt_spline(st["plan"], f, c, B, ld, st["vt"], st["vs"], st["dim"])
    return c[:, :N], st["vt"], st["vs"], st["dim"]


def work(case):
    """Samples in, results and the plan's tables once each; one add (p = 2) or 8 p real operations per point and digit."""
    p, m, s, B, kind, dtype = (case[k] for k in ("p", "m", "s", "batch", "kind", "dtype"))
    size = {"f32": 4, "i32": 4, "f64": 8, "c64": 8, "c128": 16}
    e_in, e_out = size[dtype], size[out_type(p, dtype)]
    stage = 1 if p == 2 else 8 * p
    n = [p ** k for k in range(m, case.get("m1", m) + 1)]
    N = p ** m
    if kind in ("forward", "inverse", "grouped"):
        return dict(bytes=B * sum(n) * (e_in + e_out), flops=B * sum(x * k * stage for x, k in zip(n, range(m, m + len(n)))))
    if kind == "spline":
        # the weight and the 2s variance tables; a multiply-add per function, point and table
        return dict(bytes=B * N * (e_in + e_out) + (1 + 2 * s) * N * 8, flops=2 * B * N * m * stage + 4 * s * B * N)
    # the weight (4 bytes) and class (2 bytes) tables; a request computes them
    return dict(bytes=B * N * (e_in + e_out) + 6 * N, flops=2 * B * N * m * stage + (2 * s * N * m * p if kind == "request" else 0))


# ---- the same in 64 bits --------------------------------------------------

def transform(x, p, sgn):
    """sum over each digit with omega^(sgn n h), FP64 / complex128, [batch][p^m]."""
    B, N = x.shape
    S = 1
    if p > 2:
        k = torch.arange(p, dtype=torch.float64, device=DEV)
        F = torch.polar(torch.ones_like(k[:, None] * k), sgn * 2 * math.pi / p * ((k[:, None] * k) % p))
        x = x.to(torch.complex128)
    while S < N:
        v = x.reshape(B, N // (p * S), p, S)
        if p == 2:
            v = torch.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), 2)
        else:
            v = torch.stack([sum(F[h, u] * v[:, :, u] for u in range(p)) for h in range(p)], 2)
        x = v.reshape(B, N)
        S *= p
    return x


def minus(U, r, p, m):
    """U - r digit by digit over F_p."""
    if p == 2:
        return U ^ r
    V = torch.zeros_like(U)
    for i in range(m):
        pw = p ** i
        V += (U // pw % p + (p - r // pw % p)) % p * pw
    return V


def representatives(p, m, C):
    """prod_j (1 + k_j), max supp and |supp| of the representative k(H) of K(C) (Sec. 2.1) for every H:
    the least nu, then the smallest k_1, k_2, ..."""
    s, N = C.shape[0], p ** m
    pw = [p ** c for c in range(m)]
    R = [[int(sum(int(C[j, i, c]) * pw[c] for c in range(m))) for i in range(m)] for j in range(s)]
    H = torch.arange(N, dtype=torch.int32 if p == 2 else torch.int64, device=DEV)
    FAR = 250

    def spans(T, j):
        # M[i](U) = min of T over U - span of the first i rows of C_j
        M = [T]
        for i in range(m):
            idx, best = H, M[-1]
            for _ in range(p - 1):
                idx = minus(idx, R[j][i], p, m)
                best = torch.minimum(best, M[-1][idx])
            M.append(best)
        return M

    T = torch.full((N,), FAR, dtype=torch.uint8, device=DEV)
    T[0] = 0
    Ts = [T]
    for j in reversed(range(s)):
        M, T = spans(Ts[-1], j), Ts[-1].clone()
        for i in range(1, m + 1):
            # nu = i: any i-digit k_j (the ones with top digit 0 are counted with fewer digits already)
            T = torch.minimum(T, torch.where(M[i] >= FAR, M[i], M[i] + i))
        Ts.append(T)
    Ts.reverse()
    Q = torch.ones(N, dtype=torch.float64, device=DEV)
    top = torch.zeros(N, dtype=torch.uint8, device=DEV)
    num = torch.zeros(N, dtype=torch.uint8, device=DEV)
    U = H.clone()
    for j in range(s):
        M = spans(Ts[j + 1], j)
        want = Ts[j][U].to(torch.int16)
        digits = torch.full((N,), -1, dtype=torch.int16, device=DEV)
        for i in range(m + 1):
            hit = (digits < 0) & (M[i][U].to(torch.int16) + i == want)
            digits = torch.where(hit, torch.full_like(digits, i), digits)
        k = torch.zeros(N, dtype=torch.int64, device=DEV)
        for i in reversed(range(m)):
            # the digit at position i: nonzero at the top, then the smallest that keeps the target reachable
            goal = want - digits
            lead, todo = digits == i + 1, digits > i
            V = U
            for a in range(p):
                if a:
                    V = minus(V, R[j][i], p, m)
                hit = todo & (M[i][V].to(torch.int16) == goal)
                if a == 0:
                    hit &= ~lead
                k += hit * (a * pw[i])
                U = torch.where(hit, V, U)
                todo &= ~hit
        Q *= (1 + k).double()
        top = torch.where(k > 0, torch.full_like(top, j + 1), top)
        num += k > 0
    return Q, top, num


def classes(q, cls, s):
    return torch.zeros(s + 1, dtype=torch.float64, device=DEV).index_add_(0, cls.long(), q).cumsum(0)


def exact_interpolate(case, C, f):
    p, m, s, N = case["p"], case["m"], case["s"], case["p"] ** case["m"]
    Q, top, num = representatives(p, m, C)
    c, var = [], []
    for b in range(f.shape[0]):
        g = transform(f[b:b + 1].double(), p, -1) / N / (Q * Q)
        q = g.abs().square()[0]
        q[0] = 0
        var.append(torch.stack((classes(q, top, s), classes(q, num, s))))
        c.append(transform(g, p, +1))
    return torch.cat(c), torch.stack(var), None


def exact_spline(case, C, f):
    p, m, s, N = case["p"], case["m"], case["s"], case["p"] ** case["m"]
    gam = kernel_weights(s)
    rc = (p * p - p) ** 2 / ((p - 1.0) * (p ** 4 - p))      # alpha = 2
    i = torch.arange(1, m + 1, dtype=torch.float64, device=DEV)
    kp = torch.cat((torch.ones(1, dtype=torch.float64, device=DEV), 1 - p ** -i * (p * p - 1) / (p - 1.0)))
    rp = rc * torch.cat((torch.ones(1, dtype=torch.float64, device=DEV), 1 - p ** (-3.0 * i) * (p ** 4 - 1) / (p - 1.0)))
    K = torch.ones(N, dtype=torch.float64, device=DEV)
    Rd = torch.ones_like(K)
    E = [torch.ones_like(K)] + [torch.zeros_like(K) for _ in range(s)]
    R = []
    for j in range(s):
        Y = numerators(p, m, C[j])
        first = sum((Y < p ** (m - i)).long() for i in range(1, m + 1)) + 1     # position of the first nonzero digit
        first[Y == 0] = 0
        K *= 1 + gam[j] * kp[first]
        a = gam[j] ** 2 * rp[first]
        Rd = Rd * (1 + a)
        R.append(Rd)
        for q in range(j + 1, 0, -1):
            E[q] = E[q] + a * E[q - 1]
    hat = lambda x: transform(x[None], p, -1).real[0] / N  # noqa: E731
    Wk = 1 / (N * hat(K))
    Rh = [hat(x) for x in R]
    for x in Rh:
        x[0] -= 1
    Eh = [hat(x) for x in E[1:]]
    c, vt, vs = [], [], []
    for b in range(f.shape[0]):
        ct = transform(f[b:b + 1].double(), p, -1) / N * Wk
        q = ct.abs().square()[0] * float(N) ** 2
        c.append(transform(ct, p, +1))
        zero = torch.zeros((), dtype=torch.float64, device=DEV)
        vt.append(torch.stack([zero] + [(q * x).sum() for x in Rh]))
        vs.append(torch.stack([zero] + [(q * x).sum() for x in Eh]).cumsum(0))
    return torch.cat(c), torch.stack(vt), torch.stack(vs), None


def exact(case, seed):
    p, m, kind, dtype, N = case["p"], case["m"], case["kind"], case["dtype"], case["p"] ** case["m"]
    if dtype == "i32":
        return None     # whole numbers are compared as they are
    C, coef, f = samples(case, seed)
    if kind == "grouped":
        return [transform(x.to(torch.float64), p, -1) / x.shape[1] for x in f]
    if kind == "request":
        f = functions(p, m, C, coef, torch.float64).float()
    if kind in ("interpolate", "request"):
        return exact_interpolate(case, C, f)
    if kind == "spline":
        return exact_spline(case, C, f)
    f = f.to(torch.complex128 if f.is_complex() else torch.float64)
    if kind == "forward":
        return torch.cat([transform(x[None], p, -1) / N for x in f])
    return torch.cat([transform(x[None], p, +1) for x in f])
