"""The dense phase of passes of more than four vectors (MMA tiles): leaf sizes on both sides of every
tile, half and K-step edge in one matrix, blocks of different magnitudes, one and two halves of vectors,
FP64 and FP32 vectors, alone and in a batch with members of fewer vectors."""
import types

import numpy as np
import pytest

import h2gen
import oracle
from fp32_tol import acc_tol, check
from oracle import quant

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [1, 3, 4, 7, 8, 15, 16, 17, 31, 32, 33, 36, 47, 48, 63, 64]


@pytest.fixture(scope="module")
def h2():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1902_01829_gb300 as mod

    return mod


def dense_matrix(seed, sizes):
    """Every leaf pair a dense block (random values, block magnitudes 2^-6 .. 2^6), no coupling."""
    rng = np.random.default_rng(seed)
    sizes = rng.permutation(np.asarray(sizes))
    q, k, leaves = int(np.log2(sizes.size)), 2, sizes.size
    lo = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    drp = (np.arange(leaves + 1) * leaves).astype(np.int32)
    dci = np.tile(np.arange(leaves), leaves).astype(np.int32)
    voff = np.concatenate([[0], np.cumsum((sizes[:, None] * sizes[None, :]).ravel())]).astype(np.int64)
    D = rng.uniform(-1, 1, voff[-1]) * np.repeat(np.ldexp(1.0, rng.integers(-6, 7, leaves * leaves)), np.diff(voff))
    nodes = 2 * leaves - 1
    return types.SimpleNamespace(n=int(lo[-1]), q=q, k=k, n_nodes=nodes, nS=0, leaf_offset=lo, U=rng.uniform(-1, 1, lo[-1] * k),
                                 E=rng.uniform(-1, 1, (nodes - 1) * k * k), S_rowptr=np.zeros(nodes + 1, np.int32),
                                 S_colidx=np.zeros(0, np.int32), S_val=np.zeros(0), D_rowptr=drp, D_colidx=dci, D_valoff=voff, D_val=D)


def handle(h2, A, form):
    return h2.H2Matrix(n=A.n, depth=A.q, rank=A.k, leaf_offset=A.leaf_offset, U=A.U, E=A.E, S_rowptr=A.S_rowptr, S_colidx=A.S_colidx,
                       S_val=A.S_val, D_rowptr=A.D_rowptr, D_colidx=A.D_colidx, D_val=A.D_val, storage=form, check_cover=True)


def to_dev(x):
    return torch.from_numpy(np.ascontiguousarray(x.T)).to("cuda:0").t()


@pytest.mark.parametrize("form", ["int16", "fp16", "bf16"])
@pytest.mark.parametrize("sizes", [SIZES, [32] * 8, [64] * 4 + [36] * 4, [29, 30] * 4])
def test_leaf_sizes_and_vector_counts(h2, form, sizes):
    A = dense_matrix(len(sizes) + sum(sizes), sizes)
    M = handle(h2, A, form)
    arrays = quant.dequantized_arrays(A, form)
    for nv in (5, 8, 9, 16, 22):
        x = h2gen.vectors(780 + nv, A.n, nv) * np.ldexp(1.0, 3 * np.arange(nv) - 30)[None, :]
        check(oracle.rel_l2(M.matvec(to_dev(x)).cpu().numpy(), oracle.matvec(A, x, **arrays)), acc_tol(A), (form, nv))
        xf = x.astype(np.float32)
        y = M.matvec_f32(to_dev(xf)).cpu().numpy()
        check(oracle.rel_l2(y, oracle.matvec(A, xf.astype(np.float64), **arrays)), acc_tol(A), (form, nv, "f32"))
    M.close()


def test_batch_with_fewer_vectors(h2):
    As = [dense_matrix(i, s) for i, s in enumerate([SIZES, [32] * 8, [64] * 2, [17] * 16, [5]])]
    Ms = [handle(h2, A, "int16") for A in As]
    B = h2.H2Batch(Ms)
    nvs = [16, 1, 7, 3, 12]
    xs = [h2gen.vectors(800 + i, A.n, nv) for i, (A, nv) in enumerate(zip(As, nvs))]
    ys = B.matvec([to_dev(x) for x in xs])
    B.check()
    for A, x, y in zip(As, xs, ys):
        check(oracle.rel_l2(y.cpu().numpy(), oracle.matvec(A, x, **quant.dequantized_arrays(A, "int16"))), acc_tol(A), (A.n, x.shape[1]))
    B.close()


@pytest.mark.parametrize("sizes", [SIZES, [32] * 8, [64] * 4 + [49] * 4, [29, 30] * 4, [5]])
@pytest.mark.parametrize("span", ["narrow", "wide"])
def test_fp64_digits(h2, sizes, span):
    """FP64: blocks whose nonzero entries lie within 2^10 (the digits' path for more than four vectors; zeros,
    exact powers of two and block magnitudes 2^-200 .. 2^200 among them) and blocks that do not."""
    A = dense_matrix(50 + len(sizes), sizes)
    rng = np.random.default_rng(5)
    if span == "narrow":
        D = np.sign(A.D_val) * rng.uniform(2.0 ** -9, 1.0, A.D_val.size)
        D[rng.random(D.size) < 0.05] = 0.0
        D[rng.random(D.size) < 0.05] = 1.0
        nb = A.D_valoff.size - 1
        A.D_val = D * np.repeat(np.ldexp(1.0, np.where(rng.random(nb) < 0.1, rng.integers(-200, 201, nb), 0)), np.diff(A.D_valoff))
    M = handle(h2, A, "fp64")
    for nv in (5, 8, 9, 16, 22):
        x = h2gen.vectors(820 + nv, A.n, nv) * np.ldexp(1.0, 20 * np.arange(nv) - 160)[None, :]
        x[rng.random(x.shape) < 0.05] = 0.0
        x[: A.leaf_offset[1]] *= 2.0 ** -60  # a leaf far below the vector's largest entry
        assert oracle.rel_l2(M.matvec(to_dev(x)).cpu().numpy(), oracle.matvec(A, x)) <= 1e-12
    M.check()
    M.close()


@pytest.mark.parametrize("form", ["fp64", "int16", "fp16", "bf16"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite_entries(h2, form, bad):
    """An infinity or NaN in one vector reaches every row of that vector and no other vector."""
    A = dense_matrix(70, [32] * 4 + [49] * 4)
    A.D_val = np.sign(A.D_val) * np.maximum(np.abs(A.D_val), 2.0 ** -7 * np.max(np.abs(A.D_val)))
    M = handle(h2, A, form)
    x = h2gen.vectors(840, A.n, 9)
    clean = M.matvec(to_dev(x)).cpu().numpy()
    x[17, 3] = bad
    y = M.matvec(to_dev(x)).cpu().numpy()
    assert not np.isfinite(y[:, 3]).any()
    keep = [v for v in range(9) if v != 3]
    assert np.array_equal(y[:, keep], clean[:, keep])
    M.close()


@pytest.mark.parametrize("form", ["int16", "fp16", "bf16"])
@pytest.mark.parametrize("sizes", [SIZES, [33, 39, 40, 41, 55, 57, 63, 64]])
def test_leaf_sizes_up_to_four_vectors(h2, form, sizes):
    """The columns of leaves of more than 32 points are padded to eight rows: every remainder, streamed."""
    A = dense_matrix(sum(sizes), sizes)
    M = handle(h2, A, form)
    arrays = quant.dequantized_arrays(A, form)
    for nv in (1, 2, 4):
        x = h2gen.vectors(830 + nv, A.n, nv)
        check(oracle.rel_l2(M.matvec(to_dev(x)).cpu().numpy(), oracle.matvec(A, x, **arrays)), acc_tol(A), (form, nv))
    M.close()
