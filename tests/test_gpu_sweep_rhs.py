"""The solve sweeps handle right-hand sides in groups whose size follows nrhs and the width of a level.  A column's
sums are formed in the same order in every group, so a column of a solution is bitwise the same whatever other
columns are solved with it."""
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


@pytest.mark.parametrize("g,m", [((3, 3, 1), 100), ((2, 2, 1), 130), ((1, 3, 1), 5)])
def test_columns_do_not_depend_on_their_group(torch_cuda, g, m):
    from paper_2002_05026_gb300 import D3M
    torch = torch_cuda
    p = synth.make_problem(*g, m, 1.0, 0.1, 3 + m)
    s = D3M(p.colptr, p.rowidx, m=m, perm=np.asarray(O.nd_order(*g), dtype=np.int32), precision="fp64", max_nrhs=17)
    s.factor(torch.from_numpy(p.blocks_numpy()).cuda())
    B = torch.from_numpy(np.ascontiguousarray(synth.rhs(9, p.n, 17))).cuda()
    ref = s.solve(B)
    for n in (1, 2, 3, 4, 5, 8, 9, 16):
        assert torch.equal(s.solve(B[:, :n].contiguous()), ref[:, :n]), n
    s.close()
