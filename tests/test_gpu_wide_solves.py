"""The superblock substitutions through Factors.apply: MSIR_WIDE_APPLY=1
takes applies down the route of a solve, 0 keeps them on the 64-row one, so
each route can be checked by itself and against the other."""

import numpy as np
import pytest

from oracle import formats as OF
from synth import randsvd_system
from gpu_helpers import to_dev
from test_gpu_substitution_shapes import _check, ctx  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1023, 1024, 1025, 1536, 1793, 2049])
@pytest.mark.parametrize("uf", [OF.FP16, OF.BF16, OF.FP32])
def test_edges(ctx, monkeypatch, n, uf):
    """Around the smallest sizes of the superblock solves, whole and ragged
    last superblocks (one row, one missing); a 16-bit storage format (a
    64-row solve) and fp32 again on the same factors."""
    monkeypatch.setenv("MSIR_WIDE_APPLY", "1")
    A, _, _ = randsvd_system(n, 1e3, 50 + n)
    u = OF.FP64 if uf == OF.FP32 else OF.FP32
    _check(ctx, A, u, uf, [(OF.FP32, OF.FP32), (OF.FP64, OF.FP64), (OF.FP32, OF.FP16),
                           (OF.FP32, OF.FP32)])


def error_ratio(ctx, monkeypatch, A, B, u, uf, arith):
    """Geometric mean over the columns of an apply of the ratio of its mean
    error on the superblock route to that on the 64-row route, both against
    the double-double apply.  (One column's ratio is that of two sums of
    random rounding errors: of 180 columns with a mean ratio of 0.27 one is
    near 1.)"""
    import paper_2107_06200_gb300 as M
    f = ctx.factor(to_dev(A), u, uf, M.params_default())
    assert f.info == 0 and f.nonfinite == 0
    ref = f.apply(to_dev(B), OF.DD, OF.FP64).cpu().numpy()
    e = []
    for route in ("1", "0"):
        monkeypatch.setenv("MSIR_WIDE_APPLY", route)
        x = f.apply(to_dev(B), arith, arith).cpu().numpy()
        e.append(np.abs(x - ref).mean(0))
    f.close()
    return np.exp(np.log(e[0] / e[1]).mean())


def system(n, kappa, graded):
    """A, four right-hand sides of the form A x and four random ones."""
    A, B, _ = randsvd_system(n, kappa, n, nrhs=4, graded=graded, device="cuda:0")
    R = np.random.default_rng(n).standard_normal((n, 4))
    return A, B.astype(np.float32).astype(np.float64), R.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,kappa,graded", [(1025, 1e2, False), (1300, 1e8, False), (1537, 1e4, True), (2100, 1e8, True)])
@pytest.mark.parametrize("uf", [OF.FP16, OF.FP32])
def test_fp32_error_is_below_the_64_row_route(ctx, monkeypatch, n, kappa, graded, uf):
    """fp32: inverses and z are pairs, so only the final rounding of a
    component is of fp32's size, against one per 64-row block and product."""
    A, B, R = system(n, kappa, graded)
    assert error_ratio(ctx, monkeypatch, A, B, OF.FP32, uf, OF.FP32) <= 1
    assert error_ratio(ctx, monkeypatch, A, R, OF.FP32, uf, OF.FP32) <= 1


@pytest.mark.parametrize("n", [1024, 1500])
@pytest.mark.parametrize("lo,hi", [(90, -60), (-60, 90), (10, -10)])
def test_rows_that_leave_the_range_of_a_superblock(ctx, monkeypatch, n, lo, hi):
    """A = D T with T well conditioned and upper triangular, D powers of two
    that fall or rise by 2^150 within one superblock (and by 2^20, which the
    pairs hold): the products behind a superblock's inverse overflow or
    vanish, the solve does not.  A scaling by rows changes no rounding of the
    64-row solve, so T's bound holds: 2 (n u + u) cond(T, x) |x|_inf."""
    import paper_2107_06200_gb300 as M
    from gpu_helpers import cond_comp
    monkeypatch.setenv("MSIR_WIDE_APPLY", "1")
    rng = np.random.default_rng(n)
    T = np.eye(n) + np.triu(rng.uniform(-1, 1, (n, n)), 1) / np.sqrt(n)
    T = T.astype(np.float32).astype(np.float64)
    e = np.full(n, float(hi))
    e[:512] = np.round(np.linspace(lo, hi, 512))
    A = T * 2.0 ** e[:, None]
    x = rng.standard_normal(n)
    c = (A @ x).astype(np.float32).astype(np.float64)
    f = ctx.factor(to_dev(A), OF.FP32, OF.FP32, M.params_default())
    assert f.info == 0 and f.nonfinite == 0
    got = f.apply(to_dev(c), OF.FP32, OF.FP32).cpu().numpy()[:, 0]
    f.close()
    ref = np.linalg.solve(T, c * 2.0 ** -e)
    u = 2.0 ** -24
    assert np.max(np.abs(got - ref)) <= 2 * (n * u + u) * cond_comp(T, ref) * np.max(np.abs(ref))


@pytest.mark.parametrize("n,kappa,graded", [(1793, 1e2, False), (2100, 1e8, False), (2560, 1e4, True), (3100, 1e6, False)])
@pytest.mark.parametrize("uf", [OF.FP16, OF.FP32])
def test_fp64_error_is_below_the_64_row_route(ctx, monkeypatch, n, kappa, graded, uf):
    """fp64: the superblocks' inverses are the exact ones rounded to fp64, as
    the 64-row blocks' are, so the error of a solve is bounded by |X||T||x|
    on both routes and fewer roundings are left on the wide one.  (Rows
    graded by 10^+-4: right-hand sides of the same grading.)"""
    A, B, R = system(n, kappa, graded)
    assert error_ratio(ctx, monkeypatch, A, B, OF.FP32, uf, OF.FP64) <= 1
    if not graded:
        assert error_ratio(ctx, monkeypatch, A, R, OF.FP32, uf, OF.FP64) <= 1


@pytest.mark.parametrize("c", [0.15, 0.3, 0.4])
@pytest.mark.parametrize("arith", [OF.FP32, OF.FP64])
def test_ill_conditioned_superblocks(ctx, monkeypatch, c, arith):
    """U = I + c N, N uniform in [-1, 1] above the diagonal: the Skeel
    condition number of its 512-row blocks is 2^10.8, 2^18.1 and 2^25.5, on
    both sides of what the pairs and the Newton step are used for."""
    n = 1900
    rng = np.random.default_rng(1)
    A = (np.eye(n) + c * np.triu(rng.uniform(-1, 1, (n, n)), 1)).astype(np.float32).astype(np.float64)
    B = rng.standard_normal((n, 4)).astype(np.float32).astype(np.float64)
    assert error_ratio(ctx, monkeypatch, A, B, OF.FP32, OF.FP32, arith) <= 1


def test_routes_share_a_workspace(ctx, monkeypatch):
    """The wide route's construction uses the 64-row route's scaled blocks as
    scratch: each route gives the same bits before and after the other, in
    either order of first use."""
    import paper_2107_06200_gb300 as M
    n = 1793
    A, _, B = system(n, 1e3, False)
    x = {}
    for order in ("01010", "10101"):
        f = ctx.factor(to_dev(A), OF.FP32, OF.FP16, M.params_default())
        for route in order:
            monkeypatch.setenv("MSIR_WIDE_APPLY", route)
            for arith in (OF.FP64, OF.FP32):
                got = f.apply(to_dev(B), arith, arith).cpu().numpy()
                assert np.array_equal(got, x.setdefault((route, arith), got))
        f.close()
    assert not np.array_equal(x["0", OF.FP64], x["1", OF.FP64])


@pytest.mark.parametrize("n,arith", [(1300, OF.FP32), (1900, OF.FP64)])
@pytest.mark.parametrize("uf", [OF.BF16, OF.FP32])
def test_graded_columns_keep_the_wide_route(ctx, monkeypatch, n, arith, uf):
    """Columns scaled by 10^+-4 change neither the accuracy of an inverse nor
    that of a solve (x is scaled back), though Skeel's condition number of
    U's blocks is 2^30 and more.  The routes' results differ, and the wide
    one's error, component by component in units of its scale, is the smaller."""
    import paper_2107_06200_gb300 as M
    A, _, R = system(n, 1e4, False)
    d = 10.0 ** np.random.default_rng(n).uniform(-4, 4, n)
    f = ctx.factor(to_dev(A * d[None, :]), OF.FP32, uf, M.params_default())
    assert f.info == 0 and f.nonfinite == 0
    ref = f.apply(to_dev(R), OF.DD, OF.FP64).cpu().numpy()
    e = []
    for route in ("1", "0"):
        monkeypatch.setenv("MSIR_WIDE_APPLY", route)
        e.append(np.abs(f.apply(to_dev(R), arith, arith).cpu().numpy() - ref) * d[:, None])
    f.close()
    assert not np.array_equal(e[0], e[1])
    assert np.exp(np.log(e[0].mean(0) / e[1].mean(0)).mean()) <= 1
