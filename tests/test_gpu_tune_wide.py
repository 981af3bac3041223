"""Tuning for products of more than four vectors: the candidates are the ones such passes use, and the
split of the dense work over the SMs follows the members' vector counts."""
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


def empty(n, nv):
    return torch.full((nv, n), float("nan"), dtype=torch.float64, device="cuda:0").t()


# consumer warps are a choice only where a pass takes up to four vectors: 2 x 9 candidates, else 9
@pytest.mark.parametrize("nv, candidates", [(4, 18), (5, 9), (16, 9), (18, 18)])
def test_candidates_of_a_handle_and_a_batch(h2, nv, candidates):
    A = h2gen.generate(dim=2, n=2000, m=32, p=4, eta=0.9, kernel="exp", ell=0.1, seed=51)
    M = h2.H2Matrix.from_generator(A, storage="int16")
    x, y = to_dev(h2gen.vectors(900 + nv, A.n, nv)), empty(A.n, nv)

    def launches(T, product):
        T.profile(True)
        T.profile_read()
        product()
        count = T.profile_read()[1]
        T.profile(False)
        return count

    one = launches(M, lambda: M.matvec(x, y))
    assert launches(M, lambda: M.tune(x, y)) == candidates * 4 * one
    B = h2.H2Batch([M])
    one = launches(B, lambda: B.matvec([x], [y]))
    assert launches(B, lambda: B.tune([x], [y])) == (candidates * 3 + 4 * 3) * one
    B.close()
    M.close()


def test_split_of_a_batch_follows_the_vector_counts(h2):
    """A member of 16 vectors beside one eight times as large with none: by cycles alone it gets a ninth of
    the SMs, with 1 + beta nv / 16 at beta = 4 five thirteenths, and the dense phase a third of the time."""
    sizes, nvs = [8192, 65536], [16, 0]
    As = [h2gen.generate(dim=2, n=n, m=64, p=4, eta=0.9, kernel="exp", ell=0.1, seed=52 + i) for i, n in enumerate(sizes)]
    B = h2.H2Batch([h2.H2Matrix.from_generator(A, storage="int16") for A in As])
    x_np = h2gen.vectors(950, As[0].n, 16)
    xs, ys = [to_dev(x_np), None], [empty(As[0].n, 16), empty(As[1].n, 1)]

    def dense_ms():
        B.matvec(xs, ys)
        B.profile(True)
        B.profile_read()
        for _ in range(20):
            B.matvec(xs, ys)
        ms = B.profile_read()[0]["dense_expand"]
        B.profile(False)
        return ms

    before = dense_ms()
    B.tune(xs, ys)
    after = dense_ms()
    B.check()
    ref = oracle.matvec(As[0], x_np, **quant.dequantized_arrays(As[0], "int16"))
    check(oracle.rel_l2(ys[0].cpu().numpy(), ref), acc_tol(As[0]), "tuned split")
    assert after < 0.7 * before, (before, after)
    B.close()
