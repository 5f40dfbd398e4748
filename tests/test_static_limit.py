"""The largest problems that the allocation-free pass takes.

Its arrays live in 8 MiB.  The channel counts below filled them when the limit
was set; growth of a channel's own records must not take them out again.  A
problem that fits is told apart on a machine without a GPU: it gets as far as
the missing device.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LARGEST = [(8, 50, 380), (14, 100, 114), (2, 4, 4741), (1, 1, 6474), (16, 256, 41), (4, 20, 1439)]

ASK = """
import numpy as np
from paper_1811_09711_gb300 import problems as P, vamp as V
for d, n, K in {cases}:
    for precision in (V.PREC_FP64, V.PREC_FP32_EVAL):
        ms = P.MapSet.identity(K)
        pr = P.Problem(name="limit", d=d, n_bins=n, channels=ms, peak_weight=np.full(K, 1.0 / K), peaks=ms.copy(),
                       gauss_sigma=0.2, gauss_centre=0.5, gauss_norm=P.GAUSS_NORM_UNIT, seed=1)
        try:
            V.sample_pass_static(pr, precision, 256, 256, 256, 1000, 0)
        except V.VampError as e:
            print(d, n, K, e.status, "static limit" in str(e))
"""


def ask(cases):
    # no device: nothing is launched, whatever the pointers
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="", PYTHONPATH=ROOT)
    out = subprocess.run([sys.executable, "-c", ASK.format(cases=cases)], env=env, check=True, capture_output=True, text=True)
    return [line.split()[3:] for line in out.stdout.splitlines()]


def test_largest_problems_fit():
    got = ask(LARGEST)
    assert got == [["3", "False"]] * (2 * len(LARGEST)), got  # VAMP_ERR_CUDA: no device


def test_larger_problems_do_not():
    got = ask([(d, n, K + K // 8) for d, n, K in LARGEST])
    assert got == [["1", "True"]] * (2 * len(LARGEST)), got  # VAMP_ERR_INVALID_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("d,n,K", [(8, 50, 380), (2, 4, 4741)])
def test_largest_problems_equal_a_context(d, n, K, precision):
    import torch
    from paper_1811_09711_gb300 import vamp as V
    from test_gpu_pass_shapes import BW, POW, problem
    pr = problem(d, n, K, [[BW], [POW], []])
    g = V.Vamp(pr, precision=precision)
    g.select_kernel(0)
    st = g.get_state()
    dev = {k: torch.tensor(st[k], dtype=torch.float64, device="cuda").contiguous() for k in ("edges", "alpha", "shift")}
    D = torch.empty((K, d, n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    r = V.sample_pass_static(pr, precision, dev["edges"].data_ptr(), dev["alpha"].data_ptr(), dev["shift"].data_ptr(),
                             100_000, 1, 0, D.data_ptr())
    c = g.sample_pass(100_000, 1)
    assert r.n_calls == c.n_calls
    assert abs(r.integral - c.integral) <= 1e-12 * abs(c.integral) and abs(r.w_max - c.w_max) <= 1e-12 * c.w_max
    Dc = g.get_pass()["D"]
    np.testing.assert_allclose(D.cpu().numpy(), Dc, rtol=1e-12, atol=1e-12 * Dc.max())
