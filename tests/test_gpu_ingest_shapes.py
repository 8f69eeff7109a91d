"""The factor's input and its row permutation at ragged sizes: vectors of 8
entries and remainders of the conversion, one and several runs of
interchanges.  A row-permuted upper triangular matrix has exactly one
candidate for every pivot, so its L is the identity, its U is the converted
matrix itself and its permutation is known."""

import numpy as np
import pytest

from oracle import formats as OF
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2107_06200_gb300 as M
    c = M.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("u,uf", [(OF.FP32, OF.FP16), (OF.FP32, OF.BF16), (OF.FP32, OF.FP32), (OF.FP64, OF.FP32),
                                  (OF.FP64, OF.FP64), (OF.FP64, OF.FP16)])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 65, 519, 2051])
def test_permuted_triangle_is_exact(ctx, u, uf, n):
    import paper_2107_06200_gb300 as M
    rng = np.random.default_rng(n)
    U = np.triu(rng.uniform(0.5, 1.0, (n, n)), 1) / n + np.diag(rng.uniform(1.0, 2.0, n))
    where = rng.permutation(n)  # row i of U is row where[i] of A
    A = np.empty_like(U)
    A[where] = U
    f = ctx.factor(to_dev(A), u, uf, M.params_default())
    F, ipiv = f.export()
    Uf = OF.fl(OF.fl(U, u), uf)
    b = rng.standard_normal(n)
    x = f.apply(to_dev(b), OF.FP64, OF.FP64).cpu().numpy().reshape(-1)
    assert f.info == 0 and f.nonfinite == 0
    f.close()
    assert np.array_equal(F, Uf)
    perm = np.arange(n)
    for j, p in enumerate(ipiv):
        perm[[j, p]] = perm[[p, j]]
    assert np.array_equal(perm, where)
    # the permutation on the device: U x = P b; the condition number of U is
    # below (2 + 1) e (1 + 1), and the blocks' inverses square it at most
    r = Uf @ x - b[where]
    assert np.max(np.abs(r)) <= 256 * (n + 2) * 2.0 ** -53 * np.max(np.abs(x)) * 3
