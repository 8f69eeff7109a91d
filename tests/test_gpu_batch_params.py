"""The batched engine's report of the blocking it used."""

import numpy as np
import pytest

from gpu_helpers import to_dev
from test_gpu_substitution_shapes import ctx  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,nbo,used", [(0, 0, (32, 64)), (16, 32, (16, 32)), (64, 64, (32, 64))])
def test_reported_blocking(ctx, nb, nbo, used):
    """Panels are at most 32 columns wide; wider ones are split."""
    import paper_2107_06200_gb300 as M
    n = 150
    A = np.eye(n) * 4 + np.random.default_rng(0).uniform(-1, 1, (n, n)) / np.sqrt(n)
    _, reps, st = ctx.solve_batched([to_dev(A)], [to_dev(A.sum(1))], "fp16,fp32,fp64",
                                    M.params_default(nb=nb, nbo=nbo))
    assert st == 0 and (reps[0]["nb"], reps[0]["nbo"]) == used
