"""The breakdown test of the FP64 factorization on diagonal tiles that hold an Inf or a NaN: the scale max|S| of an Inf
is Inf, so that it is reported, and a NaN is left out of the scale, so that it does not hide a zero pivot; the same
with both tile engines."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
PIVOT = 4                                            # D3M_ERR_PIVOT


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    from paper_2002_05026_gb300 import build
    build.build()
    return torch


def _status(torch, K, p, **kw):
    from paper_2002_05026_gb300 import D3M
    s = D3M(p.colptr, p.rowidx, m=p.m, precision="fp64", max_nrhs=1, **kw)
    s.factor(torch.from_numpy(K).cuda())
    st = s.info()["status"]
    s.close()
    return st


@pytest.mark.parametrize("engine", ["digits", "fma"])
@pytest.mark.parametrize("pivot", [False, True])
@pytest.mark.parametrize("m,r,c", [(64, 40, 3), (40, 39, 39), (80, 79, 70)])
@pytest.mark.parametrize("value", [np.inf, complex(0, -np.inf)])
def test_inf_is_a_breakdown(torch_cuda, engine, pivot, m, r, c, value):
    p = synth.make_problem(2, 2, 1, m, 1.0, 0.1, 5)
    K = p.blocks_numpy().copy()
    blk = K[p.blk_off[0]:p.blk_off[0] + m * m].reshape(m, m)
    blk[c, r] = blk[r, c] = value
    assert _status(torch_cuda, K, p, pivot=pivot, fp64_engine=engine) == PIVOT


@pytest.mark.parametrize("engine", ["digits", "fma"])
@pytest.mark.parametrize("m", [64, 40])
def test_nan_does_not_hide_a_zero_pivot(torch_cuda, engine, m):
    p = synth.make_problem(2, 2, 1, m, 1.0, 0.1, 5)
    K = p.blocks_numpy().copy()
    blk = K[p.blk_off[0]:p.blk_off[0] + m * m].reshape(m, m)
    blk[0, 0] = 0.0
    blk[m - 3, m - 2] = blk[m - 2, m - 3] = np.nan
    assert _status(torch_cuda, K, p, fp64_engine=engine) == PIVOT
