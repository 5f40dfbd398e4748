"""Sizes at which the library changes kernel, table or copy path.

A family's kernels (exact shape, range of d, any shape, and one or two calls
per thread) evaluate a call with the same FP32 factors: at most 2 d + 8 of
them per term, all terms positive, so two of them differ by at most
2 (2 d + 8) 2^-24 <= 4.8e-6 per weight at d = 16 if the compiler contracts
them differently, and by twice that in the squares of the d-values: bars
5e-6 and 1e-5.

Against the FP64 oracle an FP32 weight also changes where the rounding of p
moves a lookup across an edge: at most d n 2^-22 of a channel's lookups, each
by the ratio of neighbouring densities, here at most 10: bar
1e-5 + 10 d n 2^-22 on the pass integral.
"""
import os

import numpy as np
import pytest

from paper_1811_09711_gb300 import problems as P
from test_gpu_pass_shapes import BW, POW, check_runs, problem

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


def random_edges(rng, K, d, n, same=False):
    """Grids whose neighbouring widths differ by at most a factor 10."""
    w = rng.uniform(1.0, 10.0, (1 if same else K, d, n))
    w = np.repeat(w, K, axis=0) if same else w
    e = np.concatenate([np.zeros((K, d, 1)), np.cumsum(w, axis=2)], axis=2)
    e /= e[:, :, -1:]
    e[:, :, -1] = 1.0
    return e


@pytest.mark.parametrize("d,n,K", [(1, 5, 2), (4, 50, 3), (5, 50, 3), (8, 31, 6), (9, 20, 5), (12, 10, 7),
                                   (13, 10, 7), (16, 33, 4)])
def test_kernels_of_a_family_agree(V, d, n, K):
    pr = problem(d, n, K, [[BW, POW], [POW], []], sigma=0.3)
    rng = np.random.default_rng(d)
    edges = random_edges(rng, K, d, n)
    ref = {}
    ranged = set()
    for i in range(V.Vamp(pr, precision=V.PREC_FP32_EVAL).kernel_candidates()):
        g = V.Vamp(pr, precision=V.PREC_FP32_EVAL)
        g.select_kernel(i)
        name = g.kernel_name(0)
        fam = name.split("<")[0]
        if "-" in name:
            ranged.add(fam)
        g.set_state(edges)
        r = g.sample_pass(30_011, 1)
        ps = g.get_pass()
        r0, p0 = ref.setdefault(fam, (r, ps))
        assert np.array_equal(ps["Nc"], p0["Nc"]), name
        assert abs(r.integral - r0.integral) <= 5e-6 * abs(r0.integral), name
        assert abs(r.w_max - r0.w_max) <= 5e-6 * r0.w_max, name
        np.testing.assert_allclose(ps["D"], p0["D"], rtol=1e-5, atol=0, err_msg=name)
    assert set(ref) == {"k_pass", "k_union"}
    assert "k_pass" in ranged and ("k_union" in ranged) == (d <= 12)


@pytest.mark.parametrize("label,d,n,K,kinds,kw,same", [
    ("one row", 2, 100, 1, [[]], {}, False),
    ("odd number of rows", 3, 7, 5, [[BW], [], [POW]], {}, False),
    ("equal rows: every image many times", 2, 40, 64, [[]], {}, True),
    ("one bin", 2, 1, 33, [[BW], []], {}, False),
    ("most rows and edges", 1, 255, 64, [[BW], [], [POW]], {}, False),
    ("one row, most edges", 1, 256, 1, [[]], {}, False),
    ("all values in the first cells", 1, 100, 12, [[POW]], dict(deltas=(1e-9, 1e-8)), False),
    ("all values in a few cells", 2, 50, 3, [[BW], []], dict(widths=(1e-6, 1e-5)), False),
])
def test_union_tables_at_their_edges(V, O, label, d, n, K, kinds, kw, same):
    pr = problem(d, n, K, kinds, **kw)
    edges = random_edges(np.random.default_rng(3), K, d, n, same)
    o = O.Oracle(pr)
    o.set_state(edges)
    ro = o.sample_pass(60_000, 2, combine=False, n_threads=NTHREADS)
    g = V.Vamp(pr, precision=V.PREC_FP32_EVAL)
    assert g.select_family("k_union").startswith("k_union<")
    g.set_state(edges)
    rg = g.sample_pass(60_000, 2)
    assert np.array_equal(g.get_pass()["Nc"], o.get_pass()["Nc"])
    assert abs(rg.integral - ro.integral) <= (1e-5 + 10 * d * n * 2.0 ** -22) * abs(ro.integral)


@pytest.mark.parametrize("d,n,K", [(16, 127, 4), (16, 126, 4), (16, 128, 4), (1, 1, 1), (14, 100, 64)])
def test_state_round_trip_around_the_staging_size(V, d, n, K):
    """Grids up to 64 KB (8192 edges: the first case) travel in one staged copy
    with α and the shifts, larger ones by themselves; any part may be absent."""
    pr = problem(d, n, K, [[]])
    rng = np.random.default_rng(n)
    e, a, s = random_edges(rng, K, d, n), rng.dirichlet(np.ones(K)), rng.normal(size=K)
    for precision in (V.PREC_FP64, V.PREC_FP32_EVAL):
        g = V.Vamp(pr, precision=precision)
        want = g.get_state()
        for part in (dict(edges=e), dict(alpha=a), dict(shift=s), dict(alpha=a[::-1].copy(), shift=-s),
                     dict(edges=random_edges(rng, K, d, n), shift=s), {}):
            g.set_state(**part, w_max=0.25)
            want.update(part, w_max=0.25)
            got = g.get_state()
            for k in ("edges", "alpha", "shift"):
                assert np.array_equal(got[k], want[k]), (k, list(part))
            assert got["w_max"] == 0.25
        other = V.Vamp(pr, precision=precision)
        other.restore(g.checkpoint())
        back = other.get_state()
        assert all(np.array_equal(back[k], want[k]) for k in ("edges", "alpha", "shift"))


@pytest.mark.parametrize("d,calls", [(16, 40), (3, 16), (2, 98), (2, 2 * 641 * 641), (1, 400_002), (1, 89_999_999)])
def test_stratified_cells(V, O, d, calls):
    """Cell digits and fractions from one cell per axis to 2^20, odd and even,
    against the oracle's 64-bit integers, bit by bit."""
    pr = problem(d, 16, 1, [[]], stratified=1)
    o, g = O.Oracle(pr), V.Vamp(pr)
    n = o.allocate(calls)
    assert g.allocate(calls) == n
    for c0 in sorted({0, n // 3, n // 2, max(0, n - 8)}):
        cnt = min(8, n - c0)
        r = g.eval_calls(0, 3, int(c0), cnt)
        for q in range(cnt):
            ref = o.eval_call(0, 3, int(c0) + q)
            assert np.array_equal(r["jf"][q], ref["jf"]) and np.array_equal(r["bins"][q], ref["bins"]), c0 + q


@pytest.mark.parametrize("K", [33, 256, 257, 1000])
def test_many_channels(V, O, K):
    """The small kernels scan channels by warps of one block."""
    pr = problem(2, 4, K, [[], [BW]])
    check_runs(V, O, pr, 1, 40 * K + 7)
    g, o = V.Vamp(pr), O.Oracle(pr)
    g.sample_pass(40 * K + 7, 0)
    o.sample_pass(40 * K + 7, 0, combine=False, n_threads=NTHREADS)
    g.update_alpha()
    o.update_alpha()
    a, b = g.get_state(), o.get_state()
    # V_c within 1e-12 of the second moment about the shift (zero here), α' a root of it
    po = o.get_pass()
    assert po["Vc"].min() > 0
    tol = 1e-12 * (1 + np.max((po["Vc"] + po["Ic"] ** 2) / po["Vc"]))
    assert tol < 1e-6
    np.testing.assert_allclose(a["alpha"], b["alpha"], rtol=tol, atol=0)
    p, w, st = g.generate_torch(500, gen_id=1)
    assert st["n_written"] == 500 and np.all(np.isfinite(np.asarray(w)))
