"""The FP64 tile engine of a handle: which one a handle gets, that it is reported, that either can be asked for, that
both give the oracle's solutions on uneven blocks of several tiles, and that the choice leaves room for the copy of a
host K."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu
DIGITS, FMA = 1, 2


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    from paper_2002_05026_gb300 import build
    build.build()
    return torch


def _arrow(N, m):
    """Pattern whose last block couples to every other one: its diagonal tile lists one product per block."""
    colptr = np.append(np.arange(0, 2 * N - 1, 2), 2 * N - 1).astype(np.int64)
    rowidx = np.asarray([r for c in range(N - 1) for r in (c, N - 1)] + [N - 1], dtype=np.int32)
    return dict(colptr=colptr, rowidx=rowidx, m=m)


def _uneven(sizes, seed):
    """A chain of blocks of the given sizes: pattern, lower blocks (column-major) and the dense K."""
    rs = np.random.RandomState(seed)
    N, n = len(sizes), sum(sizes)
    at = np.concatenate([[0], np.cumsum(sizes)])
    K = np.zeros((n, n), dtype=complex)
    vals, colptr, rowidx = [], [0], []
    for c in range(N):
        for r in range(c, min(c + 2, N)):
            A = (rs.randn(sizes[r], sizes[c]) + 1j * rs.randn(sizes[r], sizes[c])) / np.sqrt(8 * max(sizes))
            if r == c:
                A = A + A.T + (3.0 + 0.5j) * np.eye(sizes[c])
            K[at[r]:at[r + 1], at[c]:at[c + 1]] = A
            K[at[c]:at[c + 1], at[r]:at[r + 1]] = A.T
            vals.append(A.T.reshape(-1))
            rowidx.append(r)
        colptr.append(len(rowidx))
    return (np.asarray(colptr, dtype=np.int64), np.asarray(rowidx, dtype=np.int32), np.concatenate(vals), K)


@pytest.mark.parametrize("kw,engine", [(dict(precision="fp64"), DIGITS), (dict(precision="fp64", seg_group=64), DIGITS),
                                       (dict(precision="fp64", seg_group=65), FMA),
                                       (dict(precision="fp64", fp64_engine="fma"), FMA),
                                       (dict(precision="fp64", fp64_engine="digits"), DIGITS),
                                       (dict(precision="bf16x3"), 0)])
def test_engine_is_reported(torch_cuda, kw, engine):
    from paper_2002_05026_gb300 import D3M
    s = D3M(**_arrow(80, 4), max_nrhs=1, **kw)
    assert s.info()["fp64_engine"] == engine
    s.close()


@pytest.mark.parametrize("kw", [dict(seg_group=65, fp64_engine="digits"), dict(fp64_engine=3)])
def test_engine_refused(torch_cuda, kw):
    from paper_2002_05026_gb300 import D3M, D3MError
    with pytest.raises(D3MError) as e:
        D3M(**_arrow(80, 4), max_nrhs=1, precision="fp64", **kw)
    assert e.value.code == 1          # D3M_ERR_INVALID


@pytest.mark.parametrize("engine", ["digits", "fma"])
@pytest.mark.parametrize("pivot", [False, True])
@pytest.mark.parametrize("sizes", [(65, 1, 130), (63, 64, 17, 128)])
def test_engines_match_the_oracle(torch_cuda, engine, pivot, sizes):
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    colptr, rowidx, vals, K = _uneven(sizes, 7)
    rs = np.random.RandomState(3)
    B = rs.randn(len(K), 3) + 1j * rs.randn(len(K), 3)
    s = D3M(colptr, rowidx, blk_size=np.asarray(sizes, dtype=np.int32), precision="fp64", max_nrhs=3, pivot=pivot,
            fp64_engine=engine)
    s.factor(torch.from_numpy(vals).cuda())
    X = s.solve(torch.from_numpy(B).cuda()).cpu().numpy()
    s.close()
    Xo = np.linalg.solve(K, B)
    assert np.linalg.norm(X - Xo) <= 1e-10 * np.linalg.norm(Xo)      # the bar of the FP64 parity tests


def test_room_for_the_copy_of_a_host_k(torch_cuda):
    # a chain of eight blocks of 1024 without fill: K takes 252 MB, L's tiles 189 and the digit words 378.  With what the
    # handle needs besides the words, 4/3 of the words and 40 MB free, the words fit three quarters of the rest, but
    # would leave less than K takes.
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    p = synth.make_problem(9, 1, 1, 1024, 1.0, 0.1, 5)
    K = p.blocks_numpy()
    kw = dict(colptr=p.colptr, rowidx=p.rowidx, m=p.m, precision="fp64", max_nrhs=1)
    B = torch.from_numpy(np.ascontiguousarray(synth.rhs(9, p.n, 1))).cuda()
    sizes = {}
    for engine in ("digits", "fma"):                  # both engines' kernels are loaded before memory gets short
        s = D3M(fp64_engine=engine, **kw)
        sizes[engine] = s.info()["device_bytes"]
        s.factor(K)
        ref = s.solve(B)
        assert s.info()["status"] == 0
        s.close()
    words = sizes["digits"] - sizes["fma"]
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hog = torch.empty(free - (sizes["fma"] + words * 4 // 3 + (40 << 20)), dtype=torch.uint8, device="cuda")
    s = D3M(**kw)
    s.factor(K)                                       # the copy of a host K is allocated here
    X = s.solve(B)
    inf = s.info()
    s.close()
    del hog
    torch.cuda.empty_cache()
    assert inf["status"] == 0 and inf["fp64_engine"] == FMA
    assert torch.equal(X, ref)                        # ref is the FMA engine's
