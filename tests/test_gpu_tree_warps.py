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


@pytest.mark.parametrize("form, bases", FORMS)
def test_batch_of_many_leaves(h2, form, bases):
    """A batch of more than 2^14 leaves takes these kernels for all its members of up to eight vectors, shallow ones and
    single leaves too, beside members of more vectors and of none."""
    sizes = [(32767, 4, 1), (20000, 2, 3), (10, 16, 2), (100, 32, 8), (2000, 2, 7), (300, 4, 16), (64, 64, 1), (5000, 40, 0)]
    As = [h2gen.generate(dim=1, n=n, m=m, p=16, eta=0.9, kernel="exp", ell=0.2, seed=45 + i) for i, (n, m, _) in enumerate(sizes)]
    assert sum(A.leaves for A in As) >= 1 << 14 and min(A.q for A in As) == 0
    B = h2.H2Batch([h2.H2Matrix.from_generator(A, storage=form, bases_fp32=bases) for A in As])
    xs = [h2gen.vectors(980 + i, A.n, max(nv, 1)) for i, (A, (_, _, nv)) in enumerate(zip(As, sizes))]
    refs = [oracle.matvec(A, x, **quant.dequantized_arrays(A, form, bases)) for A, x in zip(As, xs)]
    xd = [to_dev(x) if nv else None for x, (_, _, nv) in zip(xs, sizes)]
    narrow = [x[:, :4] if x is not None else None for x in xd]  # up to four vectors: beside the dense stream
    for tuned in (False, True):
        for vectors in (xd, narrow):
            ys = [torch.full((x.shape[1] if x is not None else 1, A.n), float("nan"), dtype=torch.float64, device="cuda:0").t()
                  for A, x in zip(As, vectors)]
            if tuned:
                B.tune(vectors, ys)
            for _ in range(2):  # the tickets return to zero
                B.matvec(vectors, ys)
                B.check()
                for A, x, y, ref in zip(As, vectors, ys, refs):
                    if x is not None:
                        check(oracle.rel_l2(y.cpu().numpy(), ref[:, :x.shape[1]]), acc_tol(A), (A.n, form, x.shape[1], tuned))
    B.close()
