"""The LU kernels at the edges of their launch shapes, against the CPU oracle:
rows per CTA at and around the panel's block sizes, one CTA and clusters,
panel widths that are not the default, ragged outer blocks, pivot ties and
zero columns.  fp32 / fp64 LUs (and bf16 / fp16 within one outer block) are
fixed operation for operation, so they are compared bit for bit."""

import numpy as np
import pytest

from oracle import formats as OF
from oracle import lu as OL
from gpu_helpers import gpu_factorization, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2107_06200_gb300 as M
    c = M.Context(0)
    yield c
    c.close()


def _matrix(n, kind):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n))
    if kind == "ties":  # many equal magnitudes: the smallest row index wins
        A = np.round(A * 2) / 2
    return A


@pytest.mark.parametrize("uf,n,nb,nbo,kind", [
    # 128 / 256 threads per CTA, one CTA, two CTAs, several
    (OF.FP32, 128, 32, 64, "random"), (OF.FP32, 129, 32, 64, "ties"), (OF.FP32, 192, 32, 64, "ties"),
    (OF.FP32, 193, 32, 64, "random"), (OF.FP32, 385, 32, 128, "ties"), (OF.FP64, 257, 16, 64, "ties"),
    # widths that leave part of a chunk or of a 16-byte vector
    (OF.FP32, 200, 13, 39, "random"), (OF.FP32, 150, 20, 100, "ties"), (OF.FP64, 140, 5, 15, "random"),
    (OF.FP32, 97, 1, 3, "random"), (OF.FP64, 90, 7, 21, "ties"),
    # bf16 / fp16 inside one outer block
    (OF.FP16, 250, 32, 256, "ties"), (OF.BF16, 191, 8, 192, "random"),
    # the 128 x 128 update tiles (n - nbo > 1408) next to the 64 x 64 ones
    (OF.FP32, 1501, 32, 64, "random")])
def test_lu_launch_shapes_are_bit_exact(ctx, uf, n, nb, nbo, kind):
    u = OF.FP64 if uf == OF.FP64 else OF.FP32
    A = _matrix(n, kind)
    fac, info, nf = gpu_factorization(ctx, A, u, uf, nb, nbo)
    Fo, ipo, info_o = OL.lu_factor(OF.fl(A, u), uf, nb, nbo)
    assert info == info_o and nf == 0
    assert np.array_equal(fac.ipiv, ipo)
    assert np.array_equal(fac.F, Fo)


def test_panel_with_two_rows_per_thread(ctx):
    """n > 8192: a CTA of the 16-CTA panel cluster holds more than 512 rows.
    The factors reproduce the matrix: |P A - L U| <= 2 (n + 2) u (|L||U|)
    elementwise (each element is a chain of at most n rounded terms and one
    rounded difference per outer block), sampled by rows, and |l_ij| <= 1."""
    import torch
    n = 8300
    g = torch.Generator(device="cuda:0")
    g.manual_seed(5)
    A = torch.randn((n, n), generator=g, dtype=torch.float32, device="cuda:0").double()
    import paper_2107_06200_gb300 as M
    f = ctx.factor(A, M.FP32, M.FP32)
    F, ipiv = f.export()
    f.close()
    assert f.info == 0 and f.nonfinite == 0
    perm = OL.ipiv_to_perm(ipiv.astype(np.int64))
    assert np.array_equal(np.sort(perm), np.arange(n))
    F = torch.from_numpy(F).cuda()
    U = torch.triu(F)
    rows = np.random.default_rng(6).choice(n, 40, replace=False)
    for i in rows:
        l = F[i].clone()
        l[i] = 1.0
        l[i + 1:] = 0.0
        assert float(l.abs().max()) <= 1.0
        e = (A[int(perm[i])] - l @ U).abs()
        assert bool((e <= 2 * (n + 2) * 2.0 ** -24 * (l.abs() @ U.abs())).all())
