"""Shapes at which the pass kernels change what they do, against the FP64 oracle.

The staged-tile pass keeps 1 to 32 copies of a segment's d-values in shared
memory (as many as fit 16 KB, fewer for a segment with under
four calls per bin and copy), cuts its calls into whole warps, and skips warps without
calls.  Sums of FP64 weights that agree with the oracle's to a few 1e-16 per
term, added in another order: bars 1e-12, as for every FP64 run.
"""
import os

import numpy as np
import pytest

from paper_1811_09711_gb300 import problems as P

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


def problem(d, n, K, kinds, seed=5, widths=(1e-3, 1e-2), sigma=0.2, deltas=(1e-4, 1e-2), peaks_apart=False, **kw):
    """K channels; kinds[c % len] lists the map kinds of channel c's coordinates 0.. (rotated by c)."""
    rng = np.random.default_rng(seed)
    ms = P.MapSet.identity(K)
    for c in range(K):
        ks = kinds[c % len(kinds)][:d]
        ms.n_mapped[c] = len(ks)
        for s, kind in enumerate(ks):
            ms.coord[c, s] = (c + s) % d
            ms.kind[c, s] = kind
            if kind == P.MAP_BW:
                ms.a[c, s] = rng.uniform(0.2, 0.8)
                ms.b[c, s] = np.exp(rng.uniform(*np.log(widths)))
            else:
                ms.b[c, s] = 0.0 if deltas[1] == 0.0 else np.exp(rng.uniform(*np.log(deltas)))
    w = rng.exponential(1.0, K)
    pk = ms.copy()
    if peaks_apart:
        pk.a[:] = np.where(pk.kind == P.MAP_BW, pk.a + 0.01, pk.a)
    args = dict(name="shapes", d=d, n_bins=n, channels=ms, peak_weight=w / w.sum(), peaks=pk, gauss_sigma=sigma,
                gauss_centre=0.5, gauss_norm=P.GAUSS_NORM_UNIT, seed=seed, iterations=2, calls=1000)
    args.update(kw)
    return P.Problem(**args)


def check_runs(V, O, pr, iters, calls, tol=1e-12):
    g, o = V.Vamp(pr, precision=V.PREC_FP64), O.Oracle(pr)
    for it in range(iters):
        shift = o.get_state()["shift"]
        rg = g.sample_pass(calls, it)
        ro = o.sample_pass(calls, it, combine=False, n_threads=NTHREADS)
        pg, po = g.get_pass(), o.get_pass()
        assert rg.n_calls == ro.n_calls and np.array_equal(pg["Nc"], po["Nc"])
        scale = np.sum(o.get_state()["alpha"] * np.abs(po["Ic"]))
        assert abs(rg.integral - ro.integral) <= tol * scale, (rg.integral, ro.integral)
        assert abs(rg.w_max - ro.w_max) <= tol * ro.w_max
        np.testing.assert_allclose(pg["D"], po["D"], rtol=tol, atol=tol * po["D"].max())
        m2 = po["Vc"] + (po["Ic"] - shift) ** 2
        assert np.all(np.abs(pg["Vc"] - po["Vc"]) <= tol * m2 + 1e-300)
        g.refine_grids()
        o.refine_grids()
        st = o.get_state()
        np.testing.assert_allclose(g.get_state()["edges"], st["edges"], rtol=0, atol=tol)
        g.set_state(st["edges"], st["alpha"], st["shift"], st["w_max"])  # the next pass starts from the same grids


BW, POW = P.MAP_BW, P.MAP_POW


@pytest.mark.parametrize("d,n,K,calls", [
    (4, 8, 1, 20_000),      # 32 copies (256 words each)
    (4, 256, 1, 40_000),    # 8 KB with one copy, two fit
    (2, 255, 1, 40_000),    # four copies, ragged
    (4, 20, 1, 1),          # N_min calls: one warp of one CTA
    (4, 20, 1, 9_728),      # 32 calls for each of 304 CTAs
    (4, 20, 1, 9_729),
    (4, 20, 1, 48_000),     # segments around one call per word: with and without copies
    (4, 20, 1, 49_000),
    (3, 10, 5, 30_011),     # segments that begin and end inside warps
])
def test_d_value_copies_and_warp_cuts(V, O, d, n, K, calls):
    check_runs(V, O, problem(d, n, K, [[], [BW]]), 2, calls)


@pytest.mark.parametrize("label,kw,iters,calls", [
    ("all power, delta 0", dict(d=4, n=33, K=4, kinds=[[POW, POW, POW, POW]], deltas=(0.0, 0.0)), 2, 20_000),
    ("four Breit-Wigners", dict(d=5, n=50, K=6, kinds=[[BW, BW, BW, BW], [BW]]), 2, 20_000),
    ("mixed slots, 64 channels", dict(d=7, n=100, K=64, kinds=[[BW, POW, BW], [POW], [], [BW, POW, POW, BW]]), 2, 40_000),
    ("peaks beside the channels", dict(d=6, n=31, K=9, kinds=[[BW, POW], [BW]], peaks_apart=True), 2, 20_000),
    ("narrow", dict(d=3, n=64, K=5, kinds=[[BW, POW], [BW]], widths=(1e-7, 1e-6), deltas=(1e-9, 1e-8)), 1, 20_000),
    ("no Gaussian", dict(d=3, n=20, K=3, kinds=[[BW], [POW]], sigma=0.0), 2, 20_000),
    ("exponents of 100", dict(d=9, n=20, K=3, kinds=[[BW], [POW]], sigma=0.04), 1, 20_000),
    ("exponents of 1800: summed", dict(d=4, n=20, K=3, kinds=[[BW], [POW]], sigma=0.01), 1, 20_000),
    ("largest", dict(d=16, n=256, K=3, kinds=[[BW, POW, BW, POW]]), 1, 5_003),
    ("one bin", dict(d=2, n=1, K=3, kinds=[[BW, POW], [POW]]), 1, 5_003),
])
def test_fp64_channel_products(V, O, label, kw, iters, calls):
    """The FP64 channel loop multiplies 64-bit mantissas and finds the bins of
    mapped coordinates from an FP32 inverse map: every pattern of slots, power
    laws down to p = tiny, Gaussian exponents beyond a packed number's."""
    check_runs(V, O, problem(**kw), iters, calls)


def test_fp64_map_far_outside(V, O):
    """Breit-Wigner maps whose mass lies far outside [0, 1] for their width
    (A below 0.3): the FP32 inverse map is no guide and the search starts at bin 0."""
    pr = problem(3, 40, 3, [[BW], []])
    for ms in (pr.channels, pr.peaks):
        ms.a[0, 0], ms.b[0, 0] = 1.8, 0.05
        ms.a[2, 0], ms.b[2, 0] = -3.0, 0.5
    check_runs(V, O, pr, 2, 20_000)
