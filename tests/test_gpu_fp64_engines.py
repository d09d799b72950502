"""D3M_FP64 factors with the digit engine, and with the SIMT engine where a task lists more than 64 tile products.
Both against the FP64 oracle to the parity bar (1e-10), on an arrow pattern: the last block couples to every
other one, so its diagonal tile has one product per block, and one update task takes seg_group of them."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    from paper_2002_05026_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("seg_group", [1, 64, 65, 100])
@pytest.mark.parametrize("pivot", [False, True])
def test_engines_agree(torch_cuda, seg_group, pivot):
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    N, m = 80, 20
    rs = np.random.RandomState(1)
    colptr = np.append(np.arange(0, 2 * N - 1, 2), 2 * N - 1).astype(np.int64)
    rowidx, blocks = [], []
    for c in range(N):
        A = rs.randn(m, m) + 1j * rs.randn(m, m)
        blocks.append((A + A.T) / np.sqrt(8 * m) + (3.0 + 0.5j) * np.eye(m) * (1 if c < N - 1 else 4))
        rowidx.append(c)
        if c < N - 1:
            blocks.append((rs.randn(m, m) + 1j * rs.randn(m, m)) / np.sqrt(2 * m * N))
            rowidx.append(N - 1)
    vals = np.concatenate([b.T.reshape(-1) for b in blocks])          # column-major
    rowidx = np.asarray(rowidx, dtype=np.int32)
    n = N * m
    K = np.zeros((n, n), dtype=complex)
    e = 0
    for c in range(N):
        for q in range(colptr[c], colptr[c + 1]):
            r = rowidx[q]
            K[r * m:(r + 1) * m, c * m:(c + 1) * m] = blocks[q]
            K[c * m:(c + 1) * m, r * m:(r + 1) * m] = blocks[q].T
    B = rs.randn(n, 3) + 1j * rs.randn(n, 3)
    s = D3M(colptr, rowidx, m=m, precision="fp64", max_nrhs=3, seg_group=seg_group, pivot=pivot)
    s.factor(torch.from_numpy(vals).cuda())
    X = s.solve(torch.from_numpy(B).cuda()).cpu().numpy()
    Xo = np.linalg.solve(K, B)
    assert np.linalg.norm(X - Xo) <= 1e-10 * np.linalg.norm(Xo)
    if not pivot:
        F = O.block_ldlt(O.lower_blocks(colptr, rowidx, vals, m), N, m)
        last = s.pivots(N - 1, m)
        assert np.linalg.norm(last - F.D[N - 1]) <= 1e-10 * np.linalg.norm(F.D[N - 1])
    s.close()
