"""The tree phases of large trees (2048 leaves and more, k <= 16, up to eight vectors): a warp per node. Ranks on
both sides of the lane groups, leaves of one point to 64 and ragged, the panel layout, one to eight vectors with
nodes fewer than warps in the upper levels, the vectors' parts for the MMA dense phase, phases in order and beside
one another, and the subtree levels the tuner tries."""
import numpy as np
import pytest

import h2gen
import oracle
from fp32_tol import acc_tol, check, tc_split_tol
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


# (dim, n, m, p): depths 11 (three and four vectors only), 12 and 13; k = 1, 9, 12, 16
SHAPES = [(1, 5999, 3, 7), (1, 5001, 2, 1), (1, 10001, 2, 9), (1, 150001, 37, 12), (1, 32767, 4, 16), (1, 262144, 64, 16)]
FORMS = [("int16", True), ("fp16", False), ("bf16", False)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("form, bases", FORMS)
def test_large_trees(h2, shape, form, bases):
    dim, n, m, p = shape
    A = h2gen.generate(dim=dim, n=n, m=m, p=p, eta=0.9, kernel="exp", ell=0.2, seed=44)
    assert A.q >= 11
    M = h2.H2Matrix.from_generator(A, storage=form, bases_fp32=bases)
    arrays = quant.dequantized_arrays(A, form, bases)
    for nv in (1, 2, 3, 5, 8):
        x = h2gen.vectors(960 + nv, n, nv)
        ref = oracle.matvec(A, x, **arrays)
        tc = nv == 8 and form != "int16" and m == 64  # 64-point leaves at k = 16: the tensor-core pass
        for profile in (False, True):  # the phases overlapping (up to four vectors) and in order
            M.profile(profile)
            for _ in range(2):  # the tickets return to zero
                check(oracle.rel_l2(M.matvec(to_dev(x)).cpu().numpy(), ref), acc_tol(A) + (tc_split_tol(form) if tc else 0.0),
                      (shape, nv, form, profile))
        M.profile(False)
        if nv == 3:
            y = torch.empty((nv, n), dtype=torch.float64, device="cuda:0").t()
            chosen = M.tune(to_dev(x), y)  # its last candidate's product (subtrees two levels higher) is left in y
            check(oracle.rel_l2(y.cpu().numpy(), ref), acc_tol(A), (shape, form, "tuner's last candidate"))
            assert chosen["tree_leaves"] in [1 << (A.q - L) for L in (9, 8, 7)]
    M.close()
