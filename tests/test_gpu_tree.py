"""The tree phases at depths and ranks where their steps change: subtrees of one, two, four and more
leaves, fewer subtrees than a cluster, one and two tickets above the clusters, two nodes per CTA in a
ticket's first level, ranks that are not multiples of the row block or of the copy width, ragged leaves."""
import numpy as np
import pytest

import h2gen
import oracle
from fp32_tol import acc_tol, check
from oracle import quant

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def h2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1902_01829_gb300 as mod

    return mod


def to_dev(x):
    return torch.from_numpy(np.ascontiguousarray(x.T)).to("cuda:0").t()


# (dim, n, m, p): depths 1, 2, 5, 8, 9, 10 (five levels in one ticket), 11, 13 (two tickets)
SHAPES = [(2, 100, 64, 4), (2, 130, 50, 5), (1, 1000, 32, 8), (2, 4099, 17, 3), (3, 9000, 18, 3), (2, 5001, 5, 2),
          (2, 6000, 3, 1), (1, 16383, 2, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("nv", [1, 2, 4, 7, 16])
def test_tree_depths(h2, shape, nv):
    dim, n, m, p = shape
    A = h2gen.generate(dim=dim, n=n, m=m, p=p, eta=0.9, kernel="exp", ell=0.2, seed=41)
    x = h2gen.vectors(760 + nv, n, nv)
    ref = oracle.matvec(A, x)
    M = h2.H2Matrix.from_generator(A)
    for _ in range(2):  # twice: the tickets return to zero
        assert oracle.rel_l2(M.matvec(to_dev(x)).cpu().numpy(), ref) <= 1e-12
    M.close()
    for form, bases in (("int16", True), ("fp16", False)):
        M = h2.H2Matrix.from_generator(A, storage=form, bases_fp32=bases)
        ref = oracle.matvec(A, x, **quant.dequantized_arrays(A, form, bases))
        for profile in (False, True):  # the phases overlapping (up to four vectors) and in order
            M.profile(profile)
            check(oracle.rel_l2(M.matvec(to_dev(x)).cpu().numpy(), ref), acc_tol(A), (shape, nv, form, profile))
        M.close()
