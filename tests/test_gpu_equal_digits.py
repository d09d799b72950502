"""Digit products of entries that repeat: with the same large digits in every entry all digit products of a level have
one sign, and the level sums reach the bounds that the kernels' exact sums rest on (2^21.5 in the residual, 2^24 in the
FP64 engine), which entries of random signs stay far below."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    from paper_2002_05026_gb300 import build
    build.build()
    return torch


def _dense_pattern(nblk):
    colptr = np.cumsum([0] + [nblk - c for c in range(nblk)]).astype(np.int64)
    rowidx = np.concatenate([np.arange(c, nblk) for c in range(nblk)]).astype(np.int32)
    return colptr, rowidx


def _lower(K, nblk, m):
    return np.concatenate([K[r * m:(r + 1) * m, c * m:(c + 1) * m].T.reshape(-1) for c in range(nblk) for r in range(c, nblk)])


@pytest.mark.parametrize("m", [512, 500])
def test_residual(torch_cuda, m):
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    v = sum(15.0 * 2.0 ** (-4 - 5 * s) for s in range(10))            # ten base-32 digits of 15 (50 bits: exact)
    nblk = 3
    n = nblk * m
    K = np.full((n, n), v * (1 + 1j)) + np.diag(np.full(n, 8.0 * n + 1j))
    x = np.stack([np.full(n, v * (1 + 1j)), np.full(n, -v * (1 + 1j)), np.full(n, v * (1 - 1j))], axis=1)
    A = K.astype(np.clongdouble)
    B = (A @ x.astype(np.clongdouble)).astype(np.complex128)
    colptr, rowidx = _dense_pattern(nblk)
    s = D3M(colptr, rowidx, m=m, precision="bf16x3", max_nrhs=3)
    s.factor(torch.from_numpy(_lower(K, nblk, m)).cuda())
    X = s.solve(torch.from_numpy(B).cuda()).cpu().numpy()
    w_dev = s.info()["omega"]
    s.close()
    R = np.abs(B.astype(np.clongdouble) - A @ X.astype(np.clongdouble)).max(axis=0)
    w = (R / (np.abs(A).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(B).max(axis=0))).astype(np.float64)
    # the bars of the reported omega: a few 2^-53 of the denominator, and FP32 sums of |K|
    assert w.max() <= 1e-12
    assert abs(w_dev - w.max()) <= 0.02 * w.max() + 16 * 2.0 ** -53, (w_dev, w)


def test_fp64_product(torch_cuda):
    # K = [[I, a J], [a J, 1000 I]], J all ones: the Schur complement 1000 I - 64 a^2 J is one digit product
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    m = 64
    v = 63.0 * 2.0 ** -6 + sum(127.0 * 2.0 ** (-6 - 8 * s) for s in range(1, 6))   # base-256 digits 63, 127, ... (46 bits)
    a = v * (1 + 1j)
    K = np.block([[np.eye(m), np.full((m, m), a)], [np.full((m, m), a), 1000.0 * np.eye(m)]])
    colptr, rowidx = _dense_pattern(2)
    s = D3M(colptr, rowidx, m=m, precision="fp64", max_nrhs=1, fp64_engine="digits")
    s.factor(torch.from_numpy(_lower(K, 2, m)).cuda())
    d = s.pivots(1, m)
    s.close()
    S = 1000.0 * np.eye(m, dtype=np.clongdouble) - m * np.clongdouble(a) * np.clongdouble(a) * np.ones((m, m))
    ref = np.zeros(m, dtype=np.clongdouble)
    for c in range(m):
        ref[c] = S[c, c]
        S[c + 1:, c + 1:] -= np.outer(S[c + 1:, c] / S[c, c], S[c + 1:, c])
    # 64 elimination steps of relative error 2^-53 each on pivots of about 1000
    assert np.abs((d - ref) / ref).max() <= 64 * 2.0 ** -53, np.abs((d - ref) / ref).max()
