"""The FP64 bin searches away from their usual start: maps whose FP32 inverse
knows the cell to several cells only (A small: widths above the range, masses
outside it), rows with most of their edges in a few cells.  Against the oracle,
bars as for every FP64 run."""
import os

import numpy as np
import pytest

from test_gpu_pass_shapes import BW, POW, check_runs, problem

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("n", [2, 5, 33, 256])
@pytest.mark.parametrize("widths", [(1.0, 5.0), (5.0, 50.0), (1e3, 1e4), (1e6, 1e7)])
def test_widths_above_the_range(V, O, n, widths):
    check_runs(V, O, problem(4, n, 4, [[BW, BW], [BW, POW], []], widths=widths), 2, 20_000)


@pytest.mark.parametrize("n", [33, 256])
def test_masses_outside(V, O, n):
    pr = problem(3, n, 4, [[BW, BW], []], widths=(0.05, 0.5))
    for ms in (pr.channels, pr.peaks):
        ms.a[:] = np.where(ms.kind == BW, np.where(ms.a < 0.5, ms.a - 2.0, ms.a + 1.2), ms.a)
    check_runs(V, O, pr, 2, 20_000)


@pytest.mark.parametrize("n,sigma", [(8, 0.002), (50, 0.01), (255, 0.02), (256, 0.002)])
def test_rows_with_most_edges_in_a_few_cells(V, O, n, sigma):
    check_runs(V, O, problem(2, n, 2, [[]], sigma=sigma), 4, 40_000)
