"""The dense phase row by row: |y - A x|_i against (|A| |x|)_i, where a form that is accurate only relative to a
block's or a chunk's largest entry would show: blocks of zeros and a few entries, rows far smaller than their
block's largest, vectors that span 2^40 within a leaf, a leaf far below its vector's largest entry."""
import types

import numpy as np
import pytest

import h2gen
from oracle import construct, quant

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# FP64: 64 products' share of what the digits leave out (384 2^-56 of the block's largest product) where a row is
# 2^-8 of its block: 2^-43.4; entries cut at 2^-46; a double-float sum of two blocks: 2^-46
FP64_TOL = 2.0 ** -42.5
# scaled forms: FP32 sums of 64 products (2^-18) of two blocks
FP32_TOL = 2.0 ** -17
# every remainder of the tiles, halves and K steps
EDGES = [1, 3, 4, 7, 8, 15, 16, 17, 31, 32, 33, 36, 47, 48, 63, 64]


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


def near_field(sizes, blocks):
    """A matrix of dense blocks alone: blocks {(i, j): array}."""
    sizes = np.asarray(sizes)
    k = 16 if np.all(sizes == 64) else 2  # 64-point leaves at k = 16: the panel layout of 16-bit codes
    q, leaves, nodes = int(np.log2(sizes.size)), sizes.size, 2 * sizes.size - 1
    lo = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    keys = sorted(blocks)
    drp = np.searchsorted([i for i, _ in keys], np.arange(leaves + 1)).astype(np.int32)
    D = [np.asfortranarray(blocks[key]).ravel(order="F") for key in keys]
    return types.SimpleNamespace(n=int(lo[-1]), q=q, k=k, n_nodes=nodes, nS=0, leaf_offset=lo, U=np.zeros(lo[-1] * k),
                                 E=np.zeros((nodes - 1) * k * k), S_rowptr=np.zeros(nodes + 1, np.int32),
                                 S_colidx=np.zeros(0, np.int32), S_val=np.zeros(0), D_rowptr=drp,
                                 D_colidx=np.array([j for _, j in keys], np.int32), D_val=np.concatenate(D),
                                 D_valoff=np.concatenate([[0], np.cumsum([d.size for d in D])]).astype(np.int64), keys=keys)


def handle(h2, A, form):
    return h2.H2Matrix(n=A.n, depth=A.q, rank=A.k, leaf_offset=A.leaf_offset, U=A.U, E=A.E, S_rowptr=A.S_rowptr, S_colidx=A.S_colidx,
                       S_val=A.S_val, D_rowptr=A.D_rowptr, D_colidx=A.D_colidx, D_val=A.D_val, storage=form)


def product(A, D_val, x):
    """A x and |A| |x|, FP64."""
    y, a = np.zeros_like(x), np.zeros_like(x)
    lo = A.leaf_offset
    for b, (i, j) in enumerate(A.keys):
        B = D_val[A.D_valoff[b]:A.D_valoff[b + 1]].reshape(lo[i + 1] - lo[i], -1, order="F")
        y[lo[i]:lo[i + 1]] += B @ x[lo[j]:lo[j + 1]]
        a[lo[i]:lo[i + 1]] += np.abs(B) @ np.abs(x[lo[j]:lo[j + 1]])
    return y, a


def case(kind, sizes, nv):
    rng = np.random.default_rng(len(kind) + sum(sizes))
    L = len(sizes)

    def full(i, j):
        return rng.uniform(0.5, 1.0, (sizes[i], sizes[j])) * rng.choice([-1.0, 1.0], (sizes[i], sizes[j]))

    x = rng.uniform(0.5, 1.0, (sum(sizes), nv)) * rng.choice([-1.0, 1.0], (sum(sizes), nv))
    span = np.ldexp(1.0, -rng.integers(0, 41, x.shape))
    diag = {(i, i): np.diag(np.diag(full(i, i))) for i in range(L)}
    rows = {(i, i): full(i, i) * np.ldexp(1.0, -(np.arange(sizes[i]) % 9))[:, None] for i in range(L)}
    if kind == "diagonal":
        return diag, x * span
    if kind == "rows":
        return rows, x
    if kind == "vectors":
        return {(i, i): full(i, i) for i in range(L)}, x * span
    if kind == "mixed":  # a row of both kinds of blocks
        return {**rows, **{(i, i + 1): np.eye(sizes[i], sizes[i + 1]) for i in range(L - 1)}}, x
    if kind == "small leaf":
        x[sizes[0]:] *= 2.0 ** -95
        return rows, x
    raise ValueError(kind)


@pytest.mark.parametrize("kind", ["diagonal", "rows", "vectors", "mixed", "small leaf"])
@pytest.mark.parametrize("sizes", [[64] * 4, [16] * 8, [49, 33, 17, 48], EDGES])
@pytest.mark.parametrize("nv", [4, 5, 9, 16])
def test_fp64_rows(h2, kind, sizes, nv):
    if kind == "small leaf" and nv <= 4:
        pytest.skip("the streams' float pairs lose bits from 2^-103 of the vector's largest entry times the block's on")
    blocks, x = case(kind, sizes, nv)
    A = near_field(sizes, blocks)
    M = handle(h2, A, "fp64")
    y = M.matvec(to_dev(x)).cpu().numpy()
    M.check()
    ref, bound = product(A, A.D_val, x)
    worst = np.max(np.abs(y - ref) / bound)
    assert worst <= FP64_TOL, (kind, np.log2(worst))
    M.close()


@pytest.mark.parametrize("form", ["int16", "fp16", "bf16"])
@pytest.mark.parametrize("kind", ["diagonal", "rows", "vectors", "mixed", "small leaf"])
@pytest.mark.parametrize("sizes", [[64] * 4, [16] * 8, [49, 33, 17, 48], EDGES])
@pytest.mark.parametrize("nv", [4, 5, 7, 16])
def test_scaled_rows(h2, form, kind, sizes, nv):
    if nv == 16 and form != "int16" and sizes == [64] * 4:
        pytest.skip("the tcgen05 passes hold a vector's entries relative to its largest")
    blocks, x = case(kind, sizes, nv)
    x = x.astype(np.float32)
    A = near_field(sizes, blocks)
    M = handle(h2, A, form)
    y = M.matvec_f32(to_dev(x)).cpu().numpy().astype(np.float64)
    M.check()
    ref, bound = product(A, quant.dequantized_arrays(A, form)["D_val"], x.astype(np.float64))
    worst = np.max(np.abs(y - ref) / bound)
    assert worst <= FP32_TOL, (kind, np.log2(worst))
    M.close()


@pytest.mark.parametrize("form", ["int16", "fp16"])
def test_generated_wide_blocks(h2, form):
    """Dense blocks generated on the device carry the mark of wide blocks too: every leaf pair a block, so short a
    correlation length that most rows see their own point alone, vectors that span 2^40 within a leaf; more than four
    vectors against the same codes times four (the streams: FP32 entry by entry)."""
    A = h2gen.generate(dim=2, n=700, m=32, p=4, eta=0.0, kernel="exp", ell=0.002, seed=61, coupling_values=False, dense_values=False)
    D = construct.dense_blocks(A.leaf_offset, A.D_rowptr, A.D_colidx, A.points, A.kernel, A.ell)
    A.keys = [(i, int(j)) for i in range(A.leaves) for j in A.D_colidx[A.D_rowptr[i]:A.D_rowptr[i + 1]]]
    rng = np.random.default_rng(62)
    x = (rng.uniform(0.5, 1.0, (A.n, 16)) * np.ldexp(1.0, -rng.integers(0, 41, (A.n, 16)))).astype(np.float32)
    _, bound = product(A, quant.dequantize_blocks(D, np.asarray(A.D_valoff), form), x.astype(np.float64))
    M = h2.H2Matrix.from_generator(A, storage=form, bases_fp32=True, coupling="kernel", dense="generated")
    four = M.matvec_f32(to_dev(x[:, :4])).cpu().numpy().astype(np.float64)
    for nv in (7, 16):
        y = M.matvec_f32(to_dev(x[:, :nv])).cpu().numpy().astype(np.float64)[:, :4]
        assert np.max(np.abs(y - four) / bound[:, :4]) <= 2 * FP32_TOL, (form, nv)
    M.check()
    M.close()
