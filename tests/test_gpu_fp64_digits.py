"""The FP64 engine's exact digit products where they can go wrong: remainders of the 64-row tiles and of the
16-column panels, and entries of very different size in one row.

A diagonal scaling K' = S K S by powers of two changes no significand of an FP64 elimination: L' = S L S^{-1} and
D' = S D S exactly.  The digit words hold a row with one scale, so the factor of K' agrees with the scaled
oracle factor only if the columns are balanced and the products aligned by their scales.

Bars: the factors of the unscaled K compared to 1e-10 in the Frobenius norm, the bar of the FP64 parity tests (the
words' 2^-55 of a row's largest entry against FP64's 2^-53 per operation leaves the elimination's own error the
larger one); for K' the same bar after undoing the scaling."""
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


@pytest.mark.parametrize("g,m", [((2, 2, 1), 15), ((2, 2, 1), 17), ((3, 2, 1), 63), ((2, 2, 1), 65), ((2, 3, 1), 128),
                                 ((2, 2, 2), 81)])
@pytest.mark.parametrize("within,between", [(0, 0), (8, 0), (8, 40)])
def test_scaled_factor(torch_cuda, g, m, within, between):
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    p = synth.make_problem(*g, m, 1.0, 0.1, 17 + m)
    perm = np.asarray(O.nd_order(*g), dtype=np.int32)
    F = O.block_ldlt(O.permute_lower(O.lower_blocks(p.colptr, p.rowidx, p.blocks, m), perm), p.nblk, m)
    # exponents within a block and between blocks, inside what the breakdown test accepts (a pivot above 1e-13 of its
    # tile's largest entry, and below 3e38)
    rs = np.random.RandomState(m)
    e = rs.randint(-within, within + 1, (p.nblk, m)) + rs.randint(-between, between + 1, (p.nblk, 1))
    K = p.blocks_numpy().copy()
    for c in range(p.nblk):
        for q in range(p.colptr[c], p.colptr[c + 1]):
            blk = K[p.blk_off[q]:p.blk_off[q + 1]].reshape(m, m)          # [column][row]
            sc = np.ldexp(1.0, e[c][:, None] + e[p.rowidx[q]][None, :])
            blk *= sc
    s = D3M(p.colptr, p.rowidx, m=m, perm=perm, precision="fp64", max_nrhs=1)
    s.factor(torch.from_numpy(K).cuda())
    assert s.info()["status"] == 0
    num = den = dn = dd = 0.0
    for (i, j), Lo in F.L.items():
        ei, ej = e[perm[i]], e[perm[j]]
        L = s.factor_block(i, j, m, m) * np.ldexp(1.0, ej[None, :] - ei[:, None])
        num += np.linalg.norm(L - Lo) ** 2
        den += np.linalg.norm(Lo) ** 2
    for j in range(p.nblk):
        d = s.pivots(j, m) * np.ldexp(1.0, -2 * e[perm[j]])
        dn += np.linalg.norm(d - F.D[j]) ** 2
        dd += np.linalg.norm(F.D[j]) ** 2
    s.close()
    assert np.sqrt(num / den) <= 1e-10 and np.sqrt(dn / dd) <= 1e-10, (np.sqrt(num / den), np.sqrt(dn / dd))


def test_nan_reaches_the_solution(torch_cuda):
    # a NaN in an off-diagonal block has no digits: the rows it reaches are NaN, as with FP64 products
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    p = synth.make_problem(2, 2, 1, 64, 1.0, 0.1, 5)
    K = p.blocks_numpy().copy()
    e = int(p.colptr[0]) + 1                                                  # an off-diagonal block
    K[p.blk_off[e] + 7] = np.nan
    s = D3M(p.colptr, p.rowidx, m=64, precision="fp64", max_nrhs=1)
    s.factor(torch.from_numpy(K).cuda())
    s.info()
    last = p.nblk - 1
    f = int(p.rowidx[e])
    assert np.isnan(s.factor_block(f, 0, 64, 64)).any()
    assert np.isnan(s.pivots(last, 64)).any() or np.isnan(s.factor_block(last, last, 64, 64)).any()
    s.close()
