"""A context keeps its generation workspace while its pass kernel changes.

A batch of calls is cut into chunks of 256 times the kernel's calls per
thread, each with a count and an offset of its own: a kernel with fewer calls
per thread has more of them for the same batch.  Whatever kernel generated
before, events equal those of a context that never ran another one (the same
kernel on the same state: bit by bit).
"""
import numpy as np
import pytest

from test_gpu_pass_shapes import BW, POW, problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1811_09711_gb300 import vamp
    vamp.load()
    return vamp


def events(g, state, w_max):
    g.set_state(state["edges"], state["alpha"], state["shift"], w_max)
    p, w, st = g.generate_torch(3000, gen_id=3)
    return p.tobytes(), w.tobytes(), st


@pytest.mark.parametrize("d,n,batch", [(8, 50, 1 << 16), (8, 50, 70_001), (6, 20, 1 << 16)])
def test_generate_after_a_kernel_of_more_calls_per_thread(V, d, n, batch):
    pr = problem(d, n, 6, [[BW, POW], [BW]]).replace(gen_batch=batch)
    ready = V.Vamp(pr, precision=V.PREC_FP32_EVAL)
    w_max = ready.sample_pass(50_000, 0).w_max
    state = ready.get_state()
    names = []
    for i in range(ready.kernel_candidates()):
        ready.select_kernel(i)
        names.append((ready.kernel_info()["calls_per_thread"], i, ready.kernel_name(1)))
    assert {c for c, _, _ in names} >= {1, 2} and any(s.startswith("k_union") for _, _, s in names)
    g = V.Vamp(pr, precision=V.PREC_FP32_EVAL)
    for _, i, name in sorted(names, reverse=True) + sorted(names):  # most calls per thread first, then back
        g.select_kernel(i)
        fresh = V.Vamp(pr, precision=V.PREC_FP32_EVAL)
        fresh.select_kernel(i)
        got, want = events(g, state, w_max), events(fresh, state, w_max)
        assert want[2]["n_written"] == 3000
        assert got == want, name


def test_generate_before_and_after_the_first_pass_picks_its_kernel(V):
    """Without pinning: a context that is given its state generates with the
    first candidate, and with the kernel that its first pass settles on after it."""
    pr = problem(6, 20, 20, [[BW], [POW], []])
    g = V.Vamp(pr, precision=V.PREC_FP32_EVAL)
    start = g.get_state()
    g.set_state(start["edges"], start["alpha"], start["shift"], 1.0)
    g.generate_torch(1000)
    w_max = g.sample_pass(200_000, 0).w_max
    state, name = g.get_state(), g.kernel_name(1)
    fresh = V.Vamp(pr, precision=V.PREC_FP32_EVAL)
    fresh.select_kernel(next(i for i in range(g.kernel_candidates()) if (fresh.select_kernel(i), fresh.kernel_name(1))[1] == name))
    assert events(g, state, w_max) == events(fresh, state, w_max)
