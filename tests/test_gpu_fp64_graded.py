"""D3M_FP64 keeps the digits of weakly coupled unknowns: matrices whose entries differ in size by more than a
diagonal scaling explains, solved for a right-hand side on the strong unknowns only, with the error of every group of
unknowns taken against that group.

K is dense in blocks, complex symmetric, off-diagonal part of norm about 1 on a diagonal of 3; entry (i, j) is scaled by
eps^|g_i - g_j|, so that every group's response is a sum of products of that size, and an elimination in FP64 gives it
to about n 2^-53 times the growth of its sums, which a condition of 2 keeps within a small factor: 1e-13 for
n <= 384 (n 2^-53 = 4e-14).  The reference is an elimination in extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    from paper_2002_05026_gb300 import build
    build.build()
    return torch


def _extended_solve(K, b):
    A, x = K.astype(np.clongdouble), b.astype(np.clongdouble)
    n = len(A)
    for c in range(n):
        l = A[c + 1:, c] / A[c, c]
        A[c + 1:, c:] -= l[:, None] * A[c, c:][None, :]
        x[c + 1:] -= l * x[c]
    for c in range(n - 1, -1, -1):
        x[c] /= A[c, c]
        x[:c] -= A[:c, c] * x[c]
    return x


def _groups(kind, nblk, m, rs):
    if kind == "interleaved":            # both groups in every tile and every panel of a tile
        return np.arange(nblk * m) % 2
    if kind == "halves":                 # the two tiles of a block of 128: products of different scale in one task
        return (np.arange(nblk * m) % m) // (m // 2)
    return rs.randint(0, 8, nblk * m)    # eight groups


@pytest.mark.parametrize("engine", ["digits", "fma"])
@pytest.mark.parametrize("pivot", [False, True])
@pytest.mark.parametrize("kind,nblk,m", [("interleaved", 3, 64), ("interleaved", 3, 23), ("halves", 3, 128), ("decay", 3, 100)])
@pytest.mark.parametrize("eps", [2.0 ** -4, 1e-4, 1e-8, 1e-14])
def test_weakly_coupled_groups(torch_cuda, engine, pivot, kind, nblk, m, eps):
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    rs = np.random.RandomState(nblk * m)
    n = nblk * m
    g = _groups(kind, nblk, m, rs)
    G = rs.randn(n, n) + 1j * rs.randn(n, n)
    K = (G + G.T) / np.sqrt(8 * n) + (3.0 + 0.5j) * np.eye(n)
    K *= np.power(eps, np.abs(g[:, None] - g[None, :]).astype(float))
    b = (rs.randn(n) + 1j * rs.randn(n)) * (g == 0)
    colptr = np.cumsum([0] + [nblk - c for c in range(nblk)]).astype(np.int64)
    rowidx = np.concatenate([np.arange(c, nblk) for c in range(nblk)]).astype(np.int32)
    vals = np.concatenate([K[r * m:(r + 1) * m, c * m:(c + 1) * m].T.reshape(-1) for c in range(nblk) for r in range(c, nblk)])
    s = D3M(colptr, rowidx, m=m, precision="fp64", max_nrhs=1, pivot=pivot, fp64_engine=engine)
    s.factor(torch.from_numpy(vals).cuda())
    X = s.solve(torch.from_numpy(b).cuda()).cpu().numpy()
    assert s.info()["status"] == 0
    s.close()
    ref = _extended_solve(K, b)
    for q in range(g.max() + 1):
        err = np.linalg.norm((X - ref)[g == q].astype(complex)) / np.linalg.norm(ref[g == q].astype(complex))
        assert err <= 1e-13, (q, err)


@pytest.mark.parametrize("engine", ["digits", "fma"])
@pytest.mark.parametrize("pivot", [False, True])
@pytest.mark.parametrize("kind,nblk,m", [("interleaved", 3, 64), ("decay", 3, 100)])
def test_decoupled_groups(torch_cuda, engine, pivot, kind, nblk, m):
    # eps = 0: rows of different groups meet in zeros only, and what couples them stays exactly zero
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    rs = np.random.RandomState(nblk * m)
    n = nblk * m
    g = _groups(kind, nblk, m, rs)
    G = rs.randn(n, n) + 1j * rs.randn(n, n)
    K = (G + G.T) / np.sqrt(8 * n) + (3.0 + 0.5j) * np.eye(n)
    K *= g[:, None] == g[None, :]
    b = (rs.randn(n) + 1j * rs.randn(n)) * np.power(1e-6, g)
    colptr = np.cumsum([0] + [nblk - c for c in range(nblk)]).astype(np.int64)
    rowidx = np.concatenate([np.arange(c, nblk) for c in range(nblk)]).astype(np.int32)
    vals = np.concatenate([K[r * m:(r + 1) * m, c * m:(c + 1) * m].T.reshape(-1) for c in range(nblk) for r in range(c, nblk)])
    s = D3M(colptr, rowidx, m=m, precision="fp64", max_nrhs=1, pivot=pivot, fp64_engine=engine)
    s.factor(torch.from_numpy(vals).cuda())
    X = s.solve(torch.from_numpy(b).cuda()).cpu().numpy()
    if not pivot:
        L = s.factor_block(nblk - 1, 0, m, m)
        assert not L[g[(nblk - 1) * m:][:, None] != g[None, :m]].any()
    s.close()
    ref = _extended_solve(K, b)
    for q in range(g.max() + 1):
        err = np.linalg.norm((X - ref)[g == q].astype(complex)) / np.linalg.norm(ref[g == q].astype(complex))
        assert err <= 1e-13, (q, err)
