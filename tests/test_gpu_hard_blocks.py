"""Diagonal blocks whose inverses fp32 pairs do not hold: triangles with a
Skeel condition number above 2^14."""

from fractions import Fraction

import numpy as np
import pytest

from oracle import formats as OF
from gpu_helpers import to_dev
from test_gpu_substitution_shapes import ctx  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def triangle(n, c, seed):
    """I + c N with N uniform in [-1, 1] above the diagonal, in fp32."""
    N = np.triu(np.random.default_rng(seed).uniform(-1, 1, (n, n)), 1)
    return (np.eye(n) + c * N).astype(np.float32).astype(np.float64)


def exact_inverse(T):
    """The inverse of a unit upper triangle, in fractions."""
    n = T.shape[0]
    t = [[Fraction(float(v)) for v in row] for row in T]
    X = [[Fraction(int(i == j)) for j in range(n)] for i in range(n)]
    for j in range(n):
        for i in range(j - 1, -1, -1):
            X[i][j] = -sum((t[i][k] * X[k][j] for k in range(i + 1, j + 1)), Fraction(0))
    return X


@pytest.mark.parametrize("c", [0.5, 1.2, 2.4, 2.8])
def test_fp32_apply_of_one_block(ctx, c):
    """U = fl(T^-1) for random triangles T: Skeel condition numbers 2^8 to
    2^58, and inverses that are smaller than the terms they are sums of by up
    to 2^28.  L = I and U is one block, so x = fl(fl(X) b): the rounded
    inverse and the rounded result are the only errors of fp32's size, 2 u
    |X||b| together (2.01 for the rest)."""
    import paper_2107_06200_gb300 as M
    n = 64
    U = np.triu(np.linalg.inv(triangle(n, c, 1))).astype(np.float32).astype(np.float64)
    b = np.random.default_rng(9).standard_normal(n).astype(np.float32).astype(np.float64)
    f = ctx.factor(to_dev(U), OF.FP32, OF.FP32, M.params_default())
    x = f.apply(to_dev(b), OF.FP32, OF.FP32).cpu().numpy()[:, 0]
    f.close()
    X = exact_inverse(U)
    bf = [Fraction(float(v)) for v in b]
    for i in range(n):
        exact = sum(X[i][k] * bf[k] for k in range(i, n))
        mag = sum(abs(X[i][k] * bf[k]) for k in range(i, n))
        assert abs(Fraction(float(x[i])) - exact) <= mag * Fraction(2.01 * 2.0 ** -24), i


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("spec", ["fp32,fp64,dd", "fp16,fp32,fp64"])
def test_solves_with_hard_blocks(ctx, batched, spec):
    """U with three blocks of Skeel number about 2^16 (and a ragged, weakly
    coupled rest): the refinement contracts by about u_f
    times that with fp32 factors, so its first stage converges; fp16 factors
    go on to GMRES and finer factors.  Backward error at most 2 u."""
    n = 200
    A = np.eye(n) + np.triu(np.random.default_rng(3).uniform(-1, 1, (n, n)), 1) * 2.0 ** -20
    for o, seed in ((0, 0), (64, 1), (128, 2)):
        T = triangle(64, 1.05, seed)
        assert (np.abs(np.linalg.inv(T)) @ np.abs(T).sum(1)).max() > 2.0 ** 14
        A[o:o + 64, o:o + 64] = T
    A = A.astype(np.float32).astype(np.float64)
    b = (A @ np.random.default_rng(4).standard_normal(n)).astype(np.float32).astype(np.float64)
    if batched:
        xs, reps, st = ctx.solve_batched([to_dev(A)], [to_dev(b)], spec)
        x = xs[0].cpu().numpy()
    else:
        X, reps, st = ctx.solve(to_dev(A), to_dev(b), spec)
        x = X.cpu().numpy().reshape(-1)
    assert st == 0 and reps[0]["cged"]
    if spec.startswith("fp32"):
        assert [s["alg"] for s in reps[0]["stages"]] == ["SIR"]
    u = 2.0 ** (-53 if spec.startswith("fp32") else -24)
    r = np.abs(b.astype(np.longdouble) - A.astype(np.longdouble) @ x.astype(np.longdouble)).max()
    assert r <= 2.01 * u * (np.abs(A).sum(1).max() * np.abs(x).max() + np.abs(b).max())
