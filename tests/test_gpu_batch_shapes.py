"""The batched engine's one-block substitution and block LU at the edges of
their shapes (64-row blocks, 256-row panels, 16-byte pieces): the engine runs
the same algorithm as the single-system path, so each system must go through
the same stages in as many steps (+-1) and iterations, and end with a
normwise backward error of the working precision."""

import numpy as np
import pytest

from gpu_helpers import assert_stage_parity, stages_of, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2107_06200_gb300 as M
    c = M.Context(0)
    yield c
    c.close()


def _matrix(n, kappa, rng):
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    p, _ = np.linalg.qr(rng.standard_normal((n, n)))
    return (q * kappa ** -np.linspace(0.0, 1.0, n)) @ p


@pytest.mark.parametrize("spec,kappa", [("fp16,fp32,fp64", 1e1), ("bf16,fp32,fp64", 1e1), ("fp32,fp64,dd", 1e3),
                                        ("fp16,fp32,fp64", 1e4)])
def test_engine_matches_the_single_path(ctx, spec, kappa):
    u = 2.0 ** -24 if spec.split(",")[1] == "fp32" else 2.0 ** -53
    sizes = [2, 63, 64, 65, 130, 193, 255, 256, 257, 321, 449, 509, 511, 512]
    rng = np.random.default_rng(5)
    As = [_matrix(n, min(kappa, 10.0 ** min(n, 9)), rng) for n in sizes]
    if u > 1e-10:
        As = [A.astype(np.float32).astype(np.float64) for A in As]
    bs = [A @ rng.standard_normal(A.shape[0]) for A in As]
    if u > 1e-10:
        bs = [b.astype(np.float32).astype(np.float64) for b in bs]
    xs, reps, st = ctx.solve_batched([to_dev(A) for A in As], [to_dev(b) for b in bs], spec)
    assert st == 0
    for A, b, x, rep in zip(As, bs, xs, reps):
        xh = x.cpu().numpy()
        _, one, _ = ctx.solve(to_dev(A), to_dev(b), spec)
        if kappa <= 1e3:  # far from a decision between two stages
            assert_stage_parity(stages_of(rep), stages_of(one[0]))
        # the refinement stops when its correction is below u, the residual is
        # formed in u_r: 4 u covers the last correction and x's rounding
        r = np.abs(b - A @ xh).max()
        bound = 4 * u * (np.abs(A).sum(1).max() * np.abs(xh).max() + np.abs(b).max())
        assert r <= bound, (A.shape[0], r / bound)
