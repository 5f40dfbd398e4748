"""The in-bin fractions of pseudo-stratified calls, from one cell per axis to
2^20, odd and even: x and p of single calls against the oracle's, in FP64 and
FP32, and the bins of the channels that did not draw the call, which follow
from them.

The fraction (rest of an integer division over n_r 2^33) is within 2^-53 on
either side, an interpolated x rounds at 2^-53 twice more: bar 2^-51.  A mapped
p moves by dp/dx times that, and by the rounding of its own terms.  FP32
fractions keep 24 bits and edges too: bar 2^-22, and the bins are compared in
FP64 only.
"""
import numpy as np
import pytest

from test_gpu_kernel_ranges import random_edges
from test_gpu_pass_shapes import BW, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [1, 16, 255])
@pytest.mark.parametrize("d,calls", [(16, 40), (3, 32), (2, 98), (3, 40_000), (2, 4 * 641 * 641), (1, 800_004), (1, 179_999_998)])
def test_fractions(d, calls, n, precision):
    from oracle import oracle as O
    from paper_1811_09711_gb300 import vamp as V
    K = 2
    pr = problem(d, n, K, [[BW], []], widths=(0.1, 0.3), stratified=1)
    edges = random_edges(np.random.default_rng(n), K, d, n)
    o, g = O.Oracle(pr), V.Vamp(pr, precision=precision)
    o.set_state(edges)
    g.set_state(edges)
    total = o.allocate(calls)
    assert g.allocate(calls) == total
    m, G = pr.channels.a[0, 0], pr.channels.b[0, 0]
    A = np.arctan((1 - m) / G) + np.arctan(m / G)
    for c0 in sorted({0, total // 3, total // 2, max(0, total - 8)}):
        cnt = min(8, total - c0)
        r = g.eval_calls(0, 3, int(c0), cnt)
        for q in range(cnt):
            ref = o.eval_call(0, 3, int(c0) + q)
            assert r["channel"][q] == ref["channel"] and np.array_equal(r["jf"][q], ref["jf"])
            unit = 2.0 ** -51 if precision == 0 else 2.0 ** -22
            assert np.all(np.abs(r["x"][q] - ref["x"]) <= unit), c0 + q
            slope = np.ones(d)
            if ref["channel"] == 0:
                slope[0] += A * ((ref["p"][0] - m) ** 2 + G * G) / G
            assert np.all(np.abs(r["p"][q] - ref["p"]) <= 4 * unit * slope), c0 + q
            if precision == 0:
                assert np.array_equal(r["bins"][q], ref["bins"]), c0 + q
