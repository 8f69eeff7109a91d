"""The substitutions' inverses and scaled blocks at the edges of their block
sizes and of fp32's range, against the CPU oracle on the GPU's own factors.
Tolerance: that of the substitution parity test, 2 (n u_acc + u_store)
cond(L) cond(U) |x|_inf with componentwise condition numbers."""

import numpy as np
import pytest

from oracle import formats as OF
from oracle import lu as OL
from oracle import trsv as OT
from synth import randsvd_system
from gpu_helpers import cond_comp, gpu_factorization, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2107_06200_gb300 as M
    c = M.Context(0)
    yield c
    c.close()


def _check(ctx, A, u, uf, ariths, seed=1):
    import paper_2107_06200_gb300 as M
    n = A.shape[0]
    fac, info, nf = gpu_factorization(ctx, A, u, uf, 0, 0)
    assert info == 0 and nf == 0
    f = ctx.factor(to_dev(A), u, uf, M.params_default())
    rng = np.random.default_rng(seed)
    L, U = OL.unpack(fac.F)
    c = rng.standard_normal(n)
    y = np.linalg.solve(L, c[fac.perm])
    for arith, store in ariths:
        xg = f.apply(to_dev(c), arith, store).cpu().numpy()[:, 0]
        if arith == OF.DD:
            xo = OT.solve_factored(fac, OF.dd(c), OF.DD, OF.DD)
            xo = xo[0] + xo[1]
            uacc, ust = 2.0 ** -104, 2.0 ** -53
        else:
            cc = OF.fl(c, store).astype(np.float64) if store != OF.FP64 else c
            xo = OT.solve_factored(fac, cc, arith, store)
            uacc, ust = OF.u_of(arith), OF.u_of(store)
        tol = 2 * (n * uacc + ust) * cond_comp(L, y) * cond_comp(U, xo) * np.max(np.abs(xo))
        assert np.max(np.abs(xg - xo)) <= max(tol, 4 * ust * np.max(np.abs(xo))), (arith, store)
    f.close()


@pytest.mark.parametrize("n", [1, 7, 63, 64, 65, 130])
@pytest.mark.parametrize("uf", [OF.FP16, OF.BF16, OF.FP32, OF.FP64])
def test_block_edges(ctx, n, uf):
    """One block, ragged blocks, every factor format and arithmetic on one
    set of factors (each precision's inverses are built when first needed)."""
    A, _, _ = randsvd_system(n, 1e2 if n > 1 else 1.0, 30 + n)
    u = OF.FP64 if uf in (OF.FP32, OF.FP64) else OF.FP32
    _check(ctx, A, u, uf, [(OF.FP32, OF.FP32), (OF.DD, OF.FP64), (OF.FP64, OF.FP64), (OF.FP32, OF.FP32)])


@pytest.mark.parametrize("uf,scale", [(OF.BF16, 2.0 ** 80), (OF.BF16, 2.0 ** -80), (OF.FP32, 2.0 ** 80),
                                      (OF.FP32, 2.0 ** -80), (OF.FP32, 1.0)])
def test_block_diagonals_near_the_ends_of_fp32(ctx, uf, scale):
    """U's diagonal outside [2^-60, 2^60]: the fp32 inverse is formed in
    double-double there.  A power-of-two scale changes no rounding, so the
    solution scales exactly against the unscaled factors' bound."""
    A, _, _ = randsvd_system(150, 1e3, 41)
    _check(ctx, scale * A, OF.FP32, uf, [(OF.FP32, OF.FP32)])


@pytest.mark.parametrize("n", [1023, 1024, 1025, 1536, 1793, 2049])
@pytest.mark.parametrize("uf", [OF.FP16, OF.FP32, OF.FP64])
def test_wide_solve_edges(ctx, n, uf):
    """Around the smallest sizes of the superblock solves, whole and ragged
    last superblocks (one row, one missing), fp32 and fp64 arithmetic, and a
    16-bit storage format (which keeps the 64-row solve)."""
    A, _, _ = randsvd_system(n, 1e3, 50 + n)
    u = OF.FP64 if uf in (OF.FP32, OF.FP64) else OF.FP32
    _check(ctx, A, u, uf, [(OF.FP32, OF.FP32), (OF.FP64, OF.FP64), (OF.FP32, OF.FP16)])


@pytest.mark.parametrize("n", [3071, 3072, 3073, 3585])
def test_wide_apply_edges(ctx, n):
    """fp64 applies around the smallest size of the superblock solves, with a
    last superblock of one row and of all but one."""
    A, _, _ = randsvd_system(n, 1e3, 50 + n)
    _check(ctx, A, OF.FP32, OF.FP16, [(OF.FP64, OF.FP64)])


@pytest.mark.parametrize("n", [1023, 1024, 1025, 1535, 1793])
def test_wide_refinement_edges(ctx, n):
    """Solves around the smallest sizes of the fp32 superblock solves: the
    refinement stops when its correction is below u = 2^-24, so the backward
    error is at most 4 u."""
    A, _, _ = randsvd_system(n, 1e2, 60 + n)
    A = A.astype(np.float32).astype(np.float64)
    b = (A @ np.random.default_rng(n).standard_normal(n)).astype(np.float32).astype(np.float64)
    X, reps, st = ctx.solve(to_dev(A), to_dev(b), "fp16,fp32,fp64")
    x = X.cpu().numpy().reshape(-1)
    r = np.abs(b - A @ x).max()
    assert st == 0
    assert r <= 4 * 2.0 ** -24 * (np.abs(A).sum(1).max() * np.abs(x).max() + np.abs(b).max())
