"""Coupling rows cut into pieces (few long rows): every piece's share of the row, its combination in
order and the reset of the row's ticket, at block counts that do not divide evenly."""
import numpy as np
import pytest
import torch

import h2gen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h2():
    import paper_1902_01829_gb300 as h2
    return h2


def to_dev(x):
    return torch.from_numpy(np.ascontiguousarray(x.T)).to("cuda:0").t()


# long rows through a small eta; k = 16 and 64 read row pairs, k = 27 the generic row mapping
SHAPES = [dict(dim=2, n=3001, m=16, p=4, eta=0.25, ell=0.1), dict(dim=3, n=2500, m=64, p=4, eta=0.9, ell=0.2),
          dict(dim=3, n=5003, m=64, p=3, eta=0.7, ell=0.2)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("nv", [1, 5, 16])
def test_split_rows_fp64(h2, shape, nv):
    A = h2gen.generate(**shape, kernel="exp", seed=31)
    assert np.max(np.diff(A.S_rowptr)) * A.k ** 2 > 1.5 * 8192  # rows that are cut
    x = h2gen.vectors(700 + nv, A.n, nv)
    M = h2.H2Matrix.from_generator(A)
    ref = oracle.matvec(A, x)
    first = M.matvec(to_dev(x)).cpu().numpy()
    assert oracle.rel_l2(first, ref) <= 1e-12
    assert np.array_equal(M.matvec(to_dev(x)).cpu().numpy(), first)  # the tickets are back at zero, the order is fixed
    M.close()
