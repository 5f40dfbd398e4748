"""Rebinning of rows that the general ones do not look like.

The new edge i lies where the cumulative of the measure m, linear inside each
old bin, reaches i M / n.  Over empty bins (m = 0) the cumulative is flat, and
where i M / n equals it, any place of the gap is one: so the check is of the
cumulative at the new edges, computed here in float64 from the pass's own
d-values.  Both sides round m, C and t at 2^-53 and add at most n terms:
(n + 8) 2^-53 of M each, and the edges are rounded at 2^-53 of a cumulative
whose slope per unit of x is at most n max(m): bar (n + 8) 2^-51 M + n 2^-52 max(m).
"""
import numpy as np
import pytest

from paper_1811_09711_gb300 import problems as P
from test_gpu_pass_shapes import problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1811_09711_gb300 import vamp
    vamp.load()
    return vamp


def measure(D, a=1.5):
    w = np.sqrt(D)
    r = w / w.sum()
    with np.errstate(divide="ignore", invalid="ignore"):
        m = ((r - 1.0) / np.log(r)) ** a
    return np.where(r == 0.0, 0.0, np.where(np.abs(r - 1.0) < 1e-12, 1.0, m))


def check_rows(old, new, D):
    n = D.shape[-1]
    for e0, e1, w in zip(old.reshape(-1, n + 1), new.reshape(-1, n + 1), D.reshape(-1, n)):
        assert np.all(np.isfinite(e1)) and e1[0] == 0.0 and e1[-1] == 1.0 and np.all(np.diff(e1) >= 0.0)
        m = measure(w)
        C = np.concatenate([[0.0], np.cumsum(m)])
        bar = (n + 8) * 2.0 ** -51 * C[-1] + n * 2.0 ** -52 * m.max()
        at = np.interp(e1, e0, C)
        assert np.all(np.abs(at - np.arange(n + 1) * C[-1] / n) <= bar)


@pytest.mark.parametrize("n", [20, 50, 64, 100, 256])
def test_mirror_symmetric_rows_with_empty_bins(V, n):
    """An axis that is its own mirror image, a few calls: most bins are empty."""
    d = 6
    eq = np.array([[0, 0, *range(d), *[P.EQ_INVERT] * d]], np.int32)
    for seed in range(40):
        g = V.Vamp(problem(d, n, 1, [[]], seed=seed, equivalences=eq, n_min=4), precision=V.PREC_FP64)
        old = g.get_state()["edges"]
        g.sample_pass(4 + seed % 9, seed)
        D = g.get_pass()["D"]
        g.refine_grids()
        check_rows(old, g.get_state()["edges"], D + D[..., ::-1])


@pytest.mark.parametrize("n", [20, 50, 64, 100, 256])
def test_sparse_rows_of_equal_weights(V, n):
    """f = g = 1: every call adds the same to its bins."""
    d = 8
    for seed in range(40):
        g = V.Vamp(problem(d, n, 1, [[]], seed=seed, sigma=0.0, n_min=4), precision=V.PREC_FP32_EVAL)
        old = g.get_state()["edges"]
        g.sample_pass(4 + seed % 9, seed)
        D = g.get_pass()["D"]
        assert np.all(D == np.round(D))
        g.refine_grids()
        check_rows(old, g.get_state()["edges"], D)


def huge(d, n, K, smooth=0):
    """Weights around 1e160: finite, their squares are not."""
    pr = problem(d, n, K, [[], [P.MAP_BW]], smooth=smooth)
    return pr.replace(peak_weight=pr.peak_weight * 1e160)


@pytest.mark.parametrize("smooth,a", [(0, 1.5), (1, 1.5), (0, 0.5)])
def test_infinite_d_values_keep_the_axis(V, smooth, a):
    pr = huge(3, 20, 2, smooth).replace(grid_alpha=a)
    g = V.Vamp(pr, precision=V.PREC_FP64)
    old = g.get_state()["edges"]
    r = g.sample_pass(5000, 0)
    assert np.isfinite(r.integral) and np.all(np.isinf(g.get_pass()["D"].max(axis=2)))
    g.refine_grids()
    assert np.array_equal(g.get_state()["edges"], old)
    assert g.sample_pass(5000, 0).integral == pytest.approx(r.integral, rel=1e-12)


def test_infinite_d_values_keep_the_axis_in_a_batch(V):
    prs = [huge(3, 20, 2), problem(3, 20, 2, [[], [P.MAP_BW]])]
    b = V.Batch(prs, precision=V.PREC_FP64, autotune=False)
    b.iterate([5000, 5000], 0, 1)
    uniform = np.broadcast_to(np.arange(21) / 20, (2, 3, 21))
    assert np.array_equal(b.get_state(0)["edges"], uniform)
    assert not np.array_equal(b.get_state(1)["edges"], uniform)
