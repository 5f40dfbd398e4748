"""Constants far from 1, FP64.  Breit-Wigner widths: products of widths, and of the
denominators (p - m)² + Γ² that divide them, beyond the range of a double where
their ratio is not; squares of widths that are subnormal or 0.

Uniform grids (every bin density is 1): the images of a narrow map's edges all
round to its mass, so which bin holds p is no longer defined.  Bars as for
every FP64 run.
"""
import os

import numpy as np
import pytest

from test_gpu_pass_shapes import BW, POW, problem

pytestmark = pytest.mark.gpu
NTHREADS = min(16, os.cpu_count() or 4)


@pytest.fixture(scope="module")
def V():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1811_09711_gb300 import vamp
    vamp.load()
    return vamp


@pytest.fixture(scope="module")
def O():
    from oracle import oracle as O
    O.build()
    return O


def check(V, O, pr, alpha=None, tol=1e-12):
    g, o = V.Vamp(pr, precision=V.PREC_FP64), O.Oracle(pr)
    if alpha is not None:
        g.set_state(alpha=alpha)
        o.set_state(alpha=alpha)
    rg, ro = g.sample_pass(20_000, 0), o.sample_pass(20_000, 0, combine=False, n_threads=NTHREADS)
    pg, po = g.get_pass(), o.get_pass()
    assert np.isfinite(ro.integral) and ro.integral != 0.0
    assert abs(rg.integral - ro.integral) <= tol * abs(ro.integral), (rg.integral, ro.integral)
    assert abs(rg.w_max - ro.w_max) <= tol * ro.w_max
    np.testing.assert_allclose(pg["Ic"], po["Ic"], rtol=tol, atol=0)
    np.testing.assert_allclose(pg["D"], po["D"], rtol=tol, atol=tol * po["D"].max())


@pytest.mark.parametrize("label,d,kinds,widths", [
    ("subnormal square", 2, [[BW], []], (1e-155, 2e-155)),
    ("square just normal", 2, [[BW], []], (2e-154, 3e-154)),
    ("two, matching", 3, [[BW, BW], []], (1e-70, 2e-70)),
    ("four, matching", 5, [[BW, BW, BW, BW], []], (1e-37, 2e-37)),
])
def test_matching_peaks(V, O, label, d, kinds, widths):
    check(V, O, problem(d, 8, 2, kinds, widths=widths))


@pytest.mark.parametrize("label,K,widths", [
    ("four wide, their own calls only", 1, (1e40, 2e40)),
    ("four wide", 2, (1e30, 2e30)),
    ("four narrow, their own calls only", 1, (1e-37, 2e-37)),
    ("four narrow: 1 / Γ^8 beyond a double", 2, (1e-41, 2e-41)),
])
def test_peaks_of_their_own(V, O, label, K, widths):
    pr = problem(5, 8, K, [[BW, BW, BW, BW], []], widths=widths)
    pr.peaks.b[:] = np.where(pr.peaks.kind == BW, 0.05, pr.peaks.b)
    check(V, O, pr)


def test_vanishing_square(V, O):
    """Γ² = 0: on its peak the weight is 0/0 or inf/inf and is reported; with
    the channel switched off its term elsewhere is an ordinary number."""
    pr = problem(2, 8, 2, [[BW], []], widths=(1e-200, 2e-200))
    with pytest.raises(V.VampError) as err:
        V.Vamp(pr, precision=V.PREC_FP64).sample_pass(20_000, 0)
    assert err.value.status == V.VAMP_ERR_NUMERIC
    check(V, O, pr, alpha=np.array([0.0, 1.0]))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("centre,kinds,apart", [
    (float("nan"), [[]], False),
    (float("nan"), [[BW], []], False),
    (-float("nan"), [[BW, POW]], False),
    (float("nan"), [[BW], []], True),
    (float("inf"), [[BW], [POW]], False),   # a mapped coordinate's exponent, inf - inf
])
def test_gaussian_centre_that_is_no_number(V, precision, centre, kinds, apart):
    """Accepted at creation; the weights are not finite, and that is reported."""
    pr = problem(3, 8, 2, kinds, peaks_apart=apart, gauss_centre=centre, gauss_norm=0)
    with pytest.raises(V.VampError) as err:
        V.Vamp(pr, precision=precision).sample_pass(20_000, 0)
    assert err.value.status == V.VAMP_ERR_NUMERIC
