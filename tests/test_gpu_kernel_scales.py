"""Evaluated coupling blocks at the ends of the range of lengths: coordinates and correlation lengths whose squares
leave the FP32 range, together and apart (K = 0 or 1 everywhere, or ordinary values of far too large or small
lengths). The dense blocks and bases are the same ordinary ones in every case."""
import numpy as np
import pytest

import h2gen
import oracle
from fp32_tol import acc_tol, check
from oracle import kernel_coupling, quant

KERNEL_EVAL = 2e-6  # the evaluated blocks' own error (test_gpu_kernel_coupling.py)

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


@pytest.mark.parametrize("kernel", ["exp", "matern32"])
@pytest.mark.parametrize("dim,n,m,p", [(2, 1500, 32, 3), (3, 3000, 64, 4)])
@pytest.mark.parametrize("size,ell", [(1.0, 1e19), (1.0, 1e25), (1.0, 1e38), (1.0, 1e-18), (1.0, 1e-25), (1.0, 3e-38),
                                      (2.0 ** 62, 0.2 * 2.0 ** 62), (2.0 ** 124, 0.2 * 2.0 ** 124), (2.0 ** 124, 0.2),
                                      (2.0 ** 124, 3e-38), (2.0 ** -100, 0.2 * 2.0 ** -100), (2.0 ** -100, 0.2)])
def test_length_scales(h2, kernel, dim, n, m, p, size, ell):
    A = h2gen.generate(dim=dim, n=n, m=m, p=p, eta=0.9, kernel=kernel, ell=0.2, seed=51)
    cheb = A.chebyshev_nodes() * size
    M = h2.H2Matrix(n=A.n, depth=A.q, rank=A.k, leaf_offset=A.leaf_offset, U=A.U, E=A.E, S_rowptr=A.S_rowptr,
                    S_colidx=A.S_colidx, S_val=None, D_rowptr=A.D_rowptr, D_colidx=A.D_colidx, D_val=A.D_val,
                    storage="int16", bases_fp32=True, coupling_kernel=dict(kernel=kernel, ell=ell, cheb=cheb))
    arrays = dict(quant.dequantized_arrays(A, "int16", True))
    with np.errstate(over="ignore"):  # (the FP64 squares of the largest coordinates are finite)
        arrays["S_val"] = kernel_coupling.coupling_blocks(cheb, kernel, ell, A.S_rowptr, A.S_colidx)
    assert np.isfinite(arrays["S_val"]).all()
    for nv in (1, 6):
        x = h2gen.vectors(950 + nv, A.n, nv)
        y = M.matvec(torch.from_numpy(np.ascontiguousarray(x.T)).to("cuda:0").t()).cpu().numpy()
        check(oracle.rel_l2(y, oracle.matvec(A, x, **arrays)), acc_tol(A) + KERNEL_EVAL, (kernel, dim, size, ell, nv))
    M.close()
