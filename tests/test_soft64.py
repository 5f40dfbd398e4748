"""The 64-bit mantissa arithmetic of the FP64 kernels, on the host, against
arithmetic of 200 bits.

The header is one source for both sides; only the FP32 starting values (an
approximate instruction on the GPU, the C library here) and the widening
multiplication are spelled differently.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
mp.mp.prec = 200
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = tmp_path_factory.mktemp("soft64") / "soft64.so"
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", str(so), os.path.join(HERE, "soft64_host.cpp")],
                   check=True)
    return C.CDLL(str(so))


def call(lib, name, *ins, sign=False):
    """The function's results as exact numbers, and their mantissas."""
    n = len(ins[0])
    ins = [np.ascontiguousarray(x) for x in ins]
    m, e, s = np.zeros(n, np.uint64), np.zeros(n, np.int32), np.ones(n, np.int32)
    args = [*ins, m, e] + ([s] if sign else [])
    getattr(lib, name)(n, *[a.ctypes.data_as(C.c_void_p) for a in args])
    return [int(si) * mp.mpf(int(mi)) * mp.mpf(2) ** int(ei) for mi, ei, si in zip(m, e, s)], m


def worst(got, want):
    return max(float(abs(g / w - 1)) for g, w in zip(got, want))


def test_exp2(lib):
    """Ten products and sums of 2^-64 units at a value from 1 to 2, the last
    one doubled: 2^-59."""
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.uniform(-1100, 1100, 3000), rng.uniform(-1, 1, 3000), [0.0, -0.0, 1.0, -1.0, 0.25, 1e-300, -1e-300]])
    got, m = call(lib, "t_exp2", x)
    assert np.all(m >> np.uint64(63) == 1)
    # the argument's own place value: a fraction is cut at 2^-64
    assert worst(got, [mp.mpf(2) ** mp.mpf(float(v)) for v in x]) < 2.0 ** -59


def test_exp2_beyond(lib):
    """Infinities and large numbers leave the range of a double on their side, NaN above."""
    x = np.array([np.inf, 1e300, 2.0 ** 20, np.nan, -np.nan, -np.inf, -1e300])
    got, _ = call(lib, "t_exp2", x)
    assert all(g > mp.mpf(2) ** 1024 for g in got[:5]) and all(g < mp.mpf(2) ** -1100 for g in got[5:])


def test_log2(lib):
    """2^-60 absolute: the power's error, and 2^-63 of larger results."""
    rng = np.random.default_rng(2)
    x = np.concatenate([np.exp2(rng.uniform(-1000, 1000, 3000)), rng.uniform(0.5, 2, 3000), 1 + rng.normal(0, 1e-9, 500),
                        np.exp2(np.arange(-8.0, 9.0)), np.nextafter(np.exp2(np.arange(-8.0, 9.0)), 0)])
    got, _ = call(lib, "t_log2", x, sign=True)
    for v, g in zip(x, got):
        w = mp.log(mp.mpf(float(v)), 2)
        assert abs(g - w) < 2.0 ** -60 + 2.0 ** -62 * abs(w), v


@pytest.mark.parametrize("lo,hi,powers", [
    (1e-3, 1.0, (1.5,)),          # the measure of the rebinning, at its usual power
    (1e-3, 1.0, (0.3, 1.0, 3.0)),
    (1e-10, 1e10, (0.5, 0.25)),   # ω^β, at its usual powers
    (1e-30, 1e30, (0.5, 1.0, -0.5)),
    (1e-300, 1e300, (0.125,)),
])
def test_pow(lib, lo, hi, powers):
    """|y log2 x| 2^-62 of the products and the logarithm, 2^-58 of the
    power; a double's own rounding is 2^-53.  Below that, the result rounded to
    a double is as near as a library power's."""
    rng = np.random.default_rng(3)
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), 3000))
    for y in powers:
        got, m = call(lib, "t_pow", x, np.full_like(x, y))
        assert np.all(m >> np.uint64(63) == 1)
        bar = 2.0 ** -58 + abs(y) * max(abs(np.log2(lo)), abs(np.log2(hi))) * 2.0 ** -62
        assert bar < 2.0 ** -53
        assert worst(got, [mp.mpf(float(v)) ** mp.mpf(y) for v in x]) < bar


@pytest.mark.parametrize("top", [2.0, 1.01])
def test_eight_products(lib, top):
    """The k-th product has lost at most k leading bits and is short by three
    units at most: together less than 3 2^-63 (2 + 4 + ... + 2^8) < 2^-52.4."""
    rng = np.random.default_rng(4)
    x, y = rng.uniform(1, top, 4000), rng.uniform(1, top, 4000)
    got, m = call(lib, "t_products", x, y)
    assert np.all(m >> np.uint64(63) == 1)
    off = [float(g / (mp.mpf(float(a)) ** 4 * mp.mpf(float(b)) ** 4) - 1) for g, a, b in zip(got, x, y)]
    assert max(off) <= 0 and min(off) > -(2.0 ** -52.4)


def test_rcp(lib):
    """Eight units of 2^-63."""
    x = np.concatenate([np.exp(np.random.default_rng(5).uniform(-700, 700, 4000)), np.exp2(np.arange(-9.0, 9.0)),
                        np.nextafter(np.exp2(np.arange(-9.0, 9.0)), 0)])
    got, m = call(lib, "t_rcp", x)
    assert np.all(m >> np.uint64(63) == 1)
    assert worst(got, [1 / mp.mpf(float(v)) for v in x]) < 2.0 ** -60


def test_rcp_of_subnormal_numbers_and_zero(lib):
    x = np.concatenate([np.exp2(np.random.default_rng(6).uniform(-1074, -1021, 500)), [5e-324, 2.2250738585072014e-308, 1.0]])
    got, _ = call(lib, "t_any_rcp", x)
    assert worst(got, [1 / mp.mpf(float(v)) for v in x]) < 2.0 ** -60
    assert call(lib, "t_any_rcp", np.zeros(1))[0][0] > mp.mpf(2) ** 60000


def test_powm08(lib):
    """About 30 units of 2^-60: s^4 and its products are fixed-point numbers of 59 to 62 places."""
    rng = np.random.default_rng(7)
    x = np.concatenate([np.exp(rng.uniform(-20, 1, 3000)), np.exp(rng.uniform(-708, 0, 3000)), [2.2250738585072014e-308, 1.0]])
    got, m = call(lib, "t_powm08", x)
    assert np.all(m >> np.uint64(63) == 1)
    assert worst(got, [mp.mpf(float(v)) ** (mp.mpf(-4) / 5) for v in x]) < 2.0 ** -55


def doubles(lib, name, *ins):
    r = np.zeros(len(ins[0]))
    getattr(lib, name)(len(r), *[np.ascontiguousarray(a).ctypes.data_as(C.c_void_p) for a in ins],
                       r.ctypes.data_as(C.c_void_p))
    return [mp.mpf(float(v)) for v in r]


def test_tan(lib):
    """Half a unit of the result and 2^-58."""
    rng = np.random.default_rng(8)
    x = np.concatenate([rng.uniform(-np.pi / 2, np.pi / 2, 3000), np.pi / 2 - 10.0 ** rng.uniform(-15, 0, 3000),
                        10.0 ** rng.uniform(-300, 0, 500), [np.pi / 4, np.nextafter(np.pi / 4, 0), np.pi / 2]])
    assert worst(doubles(lib, "t_tan", x), [mp.tan(mp.mpf(float(v))) for v in x]) < 2.0 ** -53 + 2.0 ** -58
    assert doubles(lib, "t_tan", np.zeros(1)) == [0]


def test_div(lib):
    rng = np.random.default_rng(9)
    x, y = rng.normal(0, 1, 4000), np.exp(rng.uniform(-300, 300, 4000))
    assert worst(doubles(lib, "t_div", x, y), [mp.mpf(float(a)) / mp.mpf(float(b)) for a, b in zip(x, y)]) < 2.0 ** -53 + 2.0 ** -59
