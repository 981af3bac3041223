"""Coupling blocks at every level up to the root, so that the upsweep's vectors of every node reach y (uniform
points have none near the root): trees of depth 0 to 6, no dense blocks, every form; the launch parameters of a
handle, of the tuner's last candidate (whose product the tuning call leaves in y: subtrees two levels higher) and
of a batch."""
import types

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


def far_matrix(q, k, seed):
    """Random blocks: every node row couples to itself and to two others of its level."""
    rng = np.random.default_rng(seed)
    leaves, nodes = 1 << q, (2 << q) - 1
    sizes = rng.integers(1, 65, leaves)
    lo = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    cols = []
    for l in range(q + 1):
        first, count = (1 << l) - 1, 1 << l
        for i in range(count):
            cols.append(sorted({first + i, first + (i ^ 1) % count, first + int(rng.integers(count))}))
    ptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32)
    s = 1.0 / np.sqrt(k)
    return types.SimpleNamespace(
        n=int(lo[-1]), q=q, k=k, n_nodes=nodes, nS=int(ptr[-1]), nD=0, leaf_offset=lo, U=rng.uniform(-1, 1, lo[-1] * k),
        E=s * rng.uniform(-1, 1, (nodes - 1) * k * k), S_rowptr=ptr, S_colidx=np.concatenate(cols).astype(np.int32),
        S_val=s * rng.uniform(-1, 1, ptr[-1] * k * k), D_rowptr=np.zeros(leaves + 1, np.int32),
        D_colidx=np.zeros(0, np.int32), D_valoff=np.zeros(1, np.int64), D_val=np.zeros(0))


FORMS = [("fp64", False), ("int16", True), ("fp16", False)]


def reference(A, x, form, bases):
    return oracle.matvec(A, x) if form == "fp64" else oracle.matvec(A, x, **quant.dequantized_arrays(A, form, bases))


def tol(A, form, nv):
    # (k = 64, fp16, eight or more vectors: the coupling runs on the tensor cores, vectors in two parts)
    return 1e-12 if form == "fp64" else acc_tol(A) + (tc_split_tol(form) if form == "fp16" and A.k == 64 and nv >= 8 else 0.0)


@pytest.mark.parametrize("q", range(7))
@pytest.mark.parametrize("k", [5, 16, 64])
def test_every_level(h2, q, k):
    A = far_matrix(q, k, 10 * q + k)
    for form, bases in FORMS:
        M = h2.H2Matrix.from_generator(A, storage=form, bases_fp32=bases)
        for nv in (1, 4, 5, 16):
            x = h2gen.vectors(900 + nv, A.n, nv)
            ref = reference(A, x, form, bases)
            for profile in (False, True):
                M.profile(profile)
                check(oracle.rel_l2(M.matvec(to_dev(x)).cpu().numpy(), ref), tol(A, form, nv), (q, k, form, nv, profile))
            M.profile(False)
            if form != "fp64":
                xd = to_dev(x)
                y = torch.full_like(xd.t(), float("nan")).t()
                M.tune(xd, y)
                check(oracle.rel_l2(y.cpu().numpy(), ref), tol(A, form, nv), (q, k, form, nv, "tuner's last candidate"))
                check(oracle.rel_l2(M.matvec(xd).cpu().numpy(), ref), tol(A, form, nv), (q, k, form, nv, "tuned"))
        M.close()


@pytest.mark.parametrize("form,bases", FORMS[1:])
def test_batch_every_level(h2, form, bases):
    As = [far_matrix(q, 16, 70 + q) for q in range(7)]
    Ms = [h2.H2Matrix.from_generator(A, storage=form, bases_fp32=bases) for A in As]
    B = h2.H2Batch(Ms)
    for nvs in ([16, 1, 7, 16, 3, 12, 5], [1, 4, 2, 3, 1, 4, 1]):
        xs = [h2gen.vectors(930 + i, A.n, nv) for i, (A, nv) in enumerate(zip(As, nvs))]
        refs = [reference(A, x, form, bases) for A, x in zip(As, xs)]
        xd = [to_dev(x) for x in xs]
        for tuned in (False, True):
            ys = [torch.full_like(x.t(), float("nan")).t() for x in xd]
            if tuned:
                B.tune(xd, ys)
            B.matvec(xd, ys)
            B.check()
            for A, y, ref, nv in zip(As, ys, refs, nvs):
                check(oracle.rel_l2(y.cpu().numpy(), ref), tol(A, form, nv), (A.q, form, nv, tuned))
    B.close()
