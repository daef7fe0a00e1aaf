"""The p = 2 coset tables of 2^12 .. 2^16 labels (one cluster sweeps backwards)."""
import ctypes

import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _dense_nonsingular(m, s, index):
    """Dense generating matrices over F_2 with independent rows (unit lower times unit upper triangular)."""
    up = S.small_net(2, m, s, index=index).astype(np.int64)
    lo = np.transpose(S.small_net(2, m, s, index=index + 1), (0, 2, 1)).astype(np.int64)
    return ((lo @ up) % 2).astype(np.uint8)


# the cluster form of the p = 2 coset tables: one tile to two tiles per CTA, one
# to eight CTAs, and the first size past it; s = 1, 2 (no and one swept
# coordinate) and many; against the oracle where that is quick, and against the
# tiled form (a capped grid) everywhere
@pytest.mark.parametrize("m,s", [(12, 1), (12, 2), (12, 40), (13, 3), (14, 33), (15, 2), (16, 1), (16, 17), (17, 3)])
def test_p2_cluster_tables(dwt, dev, orc, m, s, monkeypatch):
    N, C = 2 ** m, _dense_nonsingular(m, s, 300 + m)
    rt = ctypes.CDLL("libcudart.so")
    rt.cudaMemcpy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]

    def tables():
        plan = dwt.dwt_plan(2, m, s, C)
        w, c = dwt.dwt_plan_tables(plan)
        W, cls = np.empty(N, np.float32), np.empty((N, 2), np.uint8)
        torch.cuda.synchronize()
        assert rt.cudaMemcpy(W.ctypes.data, w, W.nbytes, 2) == 0 and rt.cudaMemcpy(cls.ctypes.data, c, cls.nbytes, 2) == 0
        return W, cls

    W, cls = tables()
    monkeypatch.setenv("DWT_TILE_GRID", "64")
    W2, cls2 = tables()
    assert np.array_equal(W.view(np.uint32), W2.view(np.uint32)) and np.array_equal(cls, cls2)
    if m <= 13:
        ref = orc.coset_leaders_dp(2, m, C)
        assert np.array_equal(W.view(np.uint32), ref["W32"].view(np.uint32)) and np.array_equal(cls, ref["cls"])
