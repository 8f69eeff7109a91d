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


def route_errors(ctx, monkeypatch, A, B, u, uf, arith):
    """Mean errors of the columns of an apply, normalised by |x|_inf, on the
    superblock and the 64-row route, against the double-double apply."""
    import paper_2107_06200_gb300 as M
    f = ctx.factor(to_dev(A), u, uf, M.params_default())
    assert f.info == 0 and f.nonfinite == 0
    ref = f.apply(to_dev(B), OF.DD, OF.FP64).cpu().numpy()
    e = []
    for route in ("1", "0"):
        monkeypatch.setenv("MSIR_WIDE_APPLY", route)
        x = f.apply(to_dev(B), arith, arith).cpu().numpy()
        e.append(np.abs(x - ref).mean(0) / np.abs(ref).max(0))
    f.close()
    return np.array(e)


def system(n, kappa, graded, nrhs=4):
    """A and right-hand sides: two of the form A x, two random ones."""
    A, B, _ = randsvd_system(n, kappa, n, nrhs=2, graded=graded, device="cuda:0")
    R = np.random.default_rng(n).standard_normal((n, 2))
    return A, np.concatenate([B, R], 1).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,kappa,graded", [(1025, 1e2, False), (1300, 1e8, False), (1537, 1e4, True), (2100, 1e8, True)])
@pytest.mark.parametrize("uf", [OF.FP16, OF.FP32])
def test_fp32_error_is_below_the_64_row_route(ctx, monkeypatch, n, kappa, graded, uf):
    """fp32: inverses and z are pairs, so only the final rounding of a
    component is of fp32's size, against one per 64-row block and product."""
    A, B = system(n, kappa, graded)
    ew, e64 = route_errors(ctx, monkeypatch, A, B, OF.FP32, uf, OF.FP32)
    assert np.all(ew <= e64), (ew / e64)
