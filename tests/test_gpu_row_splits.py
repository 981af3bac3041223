"""Coupling rows cut into pieces (few long rows): every piece's share of the row, its combination in
order and the reset of the row's ticket, at block counts that do not divide evenly."""
import numpy as np
import pytest
import torch

import h2gen
import oracle
from fp32_tol import acc_tol, check
from oracle import kernel_coupling, quant

KERNEL_EVAL = 2e-6  # the evaluated blocks' own error (test_gpu_kernel_coupling.py)

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


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("nv", [1, 3, 7, 16])
def test_split_rows_scaled(h2, shape, nv):
    A = h2gen.generate(**shape, kernel="exp", seed=32)
    x = h2gen.vectors(720 + nv, A.n, nv)
    M = h2.H2Matrix.from_generator(A, storage="int16", bases_fp32=True)
    ref = oracle.matvec(A, x, **quant.dequantized_arrays(A, "int16", True))
    first = M.matvec(to_dev(x)).cpu().numpy()
    check(oracle.rel_l2(first, ref), acc_tol(A), ("split rows", A.k, nv))
    assert np.array_equal(M.matvec(to_dev(x)).cpu().numpy(), first)
    M.close()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("nv", [1, 6, 16])
@pytest.mark.parametrize("kernel", ["exp", "matern32"])
def test_split_rows_evaluated(h2, shape, nv, kernel):
    A = h2gen.generate(**shape, kernel=kernel, seed=33)
    x = h2gen.vectors(740 + nv, A.n, nv)
    M = h2.H2Matrix.from_generator(A, storage="int16", bases_fp32=True, coupling="kernel")
    arrays = dict(quant.dequantized_arrays(A, "int16", True))
    arrays["S_val"] = kernel_coupling.coupling_blocks(A.chebyshev_nodes(), A.kernel, A.ell, A.S_rowptr, A.S_colidx)
    first = M.matvec(to_dev(x)).cpu().numpy()
    check(oracle.rel_l2(first, oracle.matvec(A, x, **arrays)), acc_tol(A) + KERNEL_EVAL, ("split rows, evaluated", A.k, nv, kernel))
    assert np.array_equal(M.matvec(to_dev(x)).cpu().numpy(), first)
    M.close()
