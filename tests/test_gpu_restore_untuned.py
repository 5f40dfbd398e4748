"""A checkpoint restored into a context whose kernel has not been chosen yet:
the timing of the candidates at its first pass leaves the history of passes
alone.  The shape is one that no other test runs, and the context that wrote
the checkpoint has its kernel pinned, so that nothing has chosen one before."""
import numpy as np
import pytest

from test_gpu_pass_shapes import BW, POW, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n", [(0, 37), (1, 37), (1, 39)])
def test_first_pass_after_a_restore_combines_the_history(precision, n):
    from paper_1811_09711_gb300 import vamp as V
    pr = problem(7, n, 5, [[BW, POW], [BW]])
    first = V.Vamp(pr, precision=precision)
    first.select_kernel(0)
    rs = []
    for it in range(3):
        rs.append(first.sample_pass(40_000, it))
        first.refine_grids()
        first.update_alpha()
    resumed = V.Vamp(pr, precision=precision)
    resumed.restore(first.checkpoint())
    rs.append(resumed.sample_pass(40_000, 3))
    I, v = np.array([r.integral for r in rs]), np.array([r.variance for r in rs])
    mean = np.sum(I / v) / np.sum(1 / v)
    # four terms, each rounded a few times
    assert rs[-1].combined == pytest.approx(mean, rel=1e-14)
    assert rs[-1].combined_sigma == pytest.approx(np.sum(1 / v) ** -0.5, rel=1e-14)
    assert rs[-1].chi2_dof == pytest.approx(np.sum((I - mean) ** 2 / v) / 3, rel=1e-9)
