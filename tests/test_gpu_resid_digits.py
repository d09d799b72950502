"""The residual's digit products at the edges of its tiles (32-column chunks, 128-row tiles, 512-column accumulation
units) and of its right-hand-side groups (8 and 16 wide): the backward error that the device reports is that of the
X it returns, taken here with extended-precision products."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    from paper_2002_05026_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("g,m,nrhs", [((3, 1, 1), 31, 25), ((2, 2, 1), 33, 17), ((2, 2, 1), 129, 9), ((2, 1, 1), 544, 8)])
def test_reported_omega_is_that_of_x(torch_cuda, g, m, nrhs):
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    p = synth.make_problem(*g, m, 1.0, 0.1, 3 + m)
    B = synth.rhs(9, p.n, nrhs) * 10.0 ** (np.arange(nrhs) % 7 - 3)      # every column has scales of its own
    s = D3M(p.colptr, p.rowidx, m=m, perm=np.asarray(O.nd_order(*g), dtype=np.int32), precision="bf16x3", max_nrhs=nrhs)
    s.factor(torch.from_numpy(p.blocks_numpy()).cuda())
    X = s.solve(torch.from_numpy(np.ascontiguousarray(B)).cuda()).cpu().numpy()
    w_dev = s.info()["omega"]
    s.close()
    A = O.dense_from_lower(O.lower_blocks(p.colptr, p.rowidx, p.blocks, p.m), p.nblk, p.m).astype(np.clongdouble)
    R = np.abs(B.astype(np.clongdouble) - A @ X.astype(np.clongdouble)).max(axis=0)
    w = (R / (np.abs(A).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(B).max(axis=0))).astype(np.float64)
    # a dropped digit product is below 2^-54 of the scales' product and a row has 2 m of them a block, so with
    # ||K||_inf of the order of m max |K| the residual is off by a few 2^-53 of the denominator, its sums by a
    # few more; ||K||_inf itself is held in FP32 sums of |K| (2%)
    assert w.max() <= 1e-12
    assert abs(w_dev - w.max()) <= 0.02 * w.max() + 16 * 2.0 ** -53, (w_dev, w)
