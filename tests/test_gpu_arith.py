"""The arithmetic that the kernels use beside the FP64 pipe, at given points,
against numpy's FP64 and exact sums: the logarithm of temperatures, the rate
constants' exponentials, fixed-point sums, conversions between formats."""
import math

import numpy as np
import pytest

from paper_2108_07605_gb300 import lbm

pytestmark = pytest.mark.gpu
NAN, INF = float("nan"), float("inf")


def _rng():
    return np.random.Generator(np.random.Philox(key=21))


def test_log():
    """Temperatures: rounded once (0.63 ulp); numpy's own is within one.  Near 1,
    where the table's terms cancel, to 2^-56 of them instead."""
    x = np.concatenate([_rng().uniform(100.0, 20000.0, 100_000),
                        10.0 ** _rng().uniform(-300, 300, 50_000), 2.0 ** np.arange(-40, 60)])
    ref = np.log(x)
    assert np.all(np.abs(lbm.lbm_arith_check("log", x) - ref) <=
                  2.0 * np.spacing(np.maximum(np.abs(ref), 0.5)))
    x = 1.0 + np.arange(-50, 51) * 2.0 ** -45
    assert np.all(np.abs(lbm.lbm_arith_check("log", x) - np.log(x)) <= 2.0 ** -56)
    got = lbm.lbm_arith_check("log", np.array([0.0, -1.0, INF, NAN]))
    assert got[0] == -INF and np.isnan(got[1]) and got[2] == INF and np.isnan(got[3])


def test_exp2_significand():
    """2^-56 of the value, then one rounding; numpy's exp2 is within one ulp."""
    r = _rng()
    x = np.concatenate([r.uniform(-65408.0, 65408.0, 200_000), r.uniform(-1.0, 1.0, 50_000),
                        np.arange(-4000, 4000) * 0.5, np.arange(-900, 900) * 64.0,
                        np.arange(-100, 100) + 0.5 - 2.0 ** -40])
    x = np.round(x * 2.0 ** 40) / 2.0 ** 40              # x / 64 exact
    ref = np.exp2(x / 64.0)
    assert np.all(np.abs(lbm.lbm_arith_check("exp2", x) - ref) <= 2.0 * np.spacing(ref))
    got = lbm.lbm_arith_check("exp2", np.array([0.0, 64.0, 70000.0, -70000.0, INF, -INF, NAN]))
    assert list(got[:6]) == [1.0, 2.0, INF, 0.0, INF, 0.0] and np.isnan(got[6])


def test_exp2_pair():
    """48 bits, about ten operations (the bound of the other float-float
    functions), where FP32 holds both words."""
    x = np.round(_rng().uniform(-6400.0, 8000.0, 200_000) * 2.0 ** 30) / 2.0 ** 30
    ref = np.exp2(x / 64.0)
    assert np.all(np.abs(lbm.lbm_arith_check("exp2_pair", x) - ref) <= 2e-14 * ref)
    assert np.isnan(lbm.lbm_arith_check("exp2_pair", np.array([NAN]))[0])


def _sums(x):
    got = lbm.lbm_arith_check("sum", x).reshape(-1, 27)
    g = x.reshape(-1, 27)
    ref = np.array([[math.fsum(v), math.fsum(list(v[2::3]) + [-u for u in v[0::3]])] for v in g])
    return got[:, :2], ref, np.abs(g).max(axis=1)


@pytest.mark.parametrize("spread", [0, 3, 20, 200])
@pytest.mark.parametrize("signs", [False, True])
def test_fixed_point_sums(spread, signs):
    """Each term cut at 2^-63 of the largest's power of two, the sum at 2^-58,
    rounded once to FP64 (as the exact sum it is compared with)."""
    r = _rng()
    v = r.uniform(0.5, 1.0, (4000, 27)) * 10.0 ** -r.uniform(0, spread, (4000, 27))
    v *= 2.0 ** r.integers(-60, 60, (4000, 1))
    if signs:
        v *= r.choice([-1.0, 1.0], v.shape)
    got, ref, top = _sums(v.reshape(-1))
    cut = 2.0 ** -58 + 27 * 2.0 ** -63
    assert np.all(np.abs(got - ref) <= 2.0 ** -52 * np.abs(ref) + 2.0 * cut * top[:, None])


def test_fixed_point_sums_at_the_edges():
    v = np.zeros((6, 27))
    v[0] = 2.0 - 2.0 ** -52                     # the largest sum
    v[1] = -(2.0 - 2.0 ** -52)
    v[2, :3] = 1.0, -1.0, 2.0 ** -64            # far below the largest: nothing
    v[3, :2] = 2.0 ** -1000, 2.0 ** -1040
    v[4, 4] = 5e-324
    got, ref, _ = _sums(v.reshape(-1))
    assert got[0, 0] == ref[0, 0] and got[1, 0] == ref[1, 0] and got[2, 0] == 0.0
    assert got[3, 0] == 2.0 ** -1000 and got[4, 0] == 0.0 and got[5, 0] == 0.0
    for bad in (NAN, INF):
        w = np.ones(27)
        w[5] = bad
        assert np.all(np.isnan(lbm.lbm_arith_check("sum", w)[:2]))


def test_conversions():
    r = _rng()
    x = np.concatenate([r.standard_normal(100_000) * 10.0 ** r.uniform(-44, 38, 100_000),
                        2.0 ** np.arange(-149, 128), -(2.0 ** np.arange(-149, 128)),
                        np.nextafter(2.0 ** np.arange(-150, 129), 0.0),
                        np.float64(2.0 ** 24 + np.arange(64)) * 2.0 ** -24 + 2.0 ** -25])
    with np.errstate(over="ignore"):
        f32 = x.astype(np.float32).astype(np.float64)
    assert np.array_equal(lbm.lbm_arith_check("float", x), f32)
    special = np.array([0.0, -0.0, INF, -INF, 1e300, -1e300, 1e-300])
    with np.errstate(over="ignore"):
        assert np.array_equal(lbm.lbm_arith_check("float", special),
                              special.astype(np.float32).astype(np.float64))
    assert np.isnan(lbm.lbm_arith_check("float", np.array([NAN]))[0])
    # pairs: 2^-48 of the value (half a unit of the low word) where FP32 holds both words
    p = x[(np.abs(x) > 2.0 ** -74) & (np.abs(x) < 2.0 ** 127)]
    assert np.all(np.abs(lbm.lbm_arith_check("pair", p) - p) <= 2.0 ** -48 * np.abs(p))
    # with an exponent, and significands: FP64's range; significands exact
    w = np.concatenate([x, r.standard_normal(50_000) * 10.0 ** r.uniform(-300, 300, 50_000),
                        [0.0, 2.0 ** -1022, 1.7976931348623157e308]])
    assert np.array_equal(lbm.lbm_arith_check("sig", w), w)
    m = lbm.lbm_arith_check("mantissa", w)
    assert np.all(np.abs(m[:-1] - w[:-1]) <= 2.0 ** -48 * np.abs(w[:-1]))
    assert m[-1] == INF                    # the nearest pair to the largest double
    for op in ("sig", "mantissa"):
        assert lbm.lbm_arith_check(op, np.array([5e-324]))[0] == 0.0
        assert not np.isfinite(lbm.lbm_arith_check(op, np.array([NAN]))[0])


def test_bad_arguments():
    L = lbm.load_library()
    x = np.zeros(27)
    assert L.lbm_arith_check(0, None, 27, x.ctypes.data) == 1       # LBM_ERR_INVALID
    assert L.lbm_arith_check(8, x.ctypes.data, 27, x.ctypes.data) == 1
    assert L.lbm_arith_check(3, x.ctypes.data, 26, x.ctypes.data) == 1
    assert L.lbm_arith_check(0, x.ctypes.data, 1 << 25, x.ctypes.data) == 6      # LBM_ERR_RANGE
