"""The double-precision regressions' fixed-point moment sums on the CPU: the
header's own code (fixed_moments.cuh) on a warp of host coroutines, against exact
rational sums, over maturities, volatilities and distances of v0 from theta."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import fixed_moments_ref as R

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2206_03719_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fixed") / "fixed_moments_host.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I" + HERE, "-I" + CSRC, os.path.join(HERE, "fixed_moments_host.cpp"),
                    "-o", so], check=True)
    return ctypes.CDLL(so)


def _sums(lib, which, basis, per, e, v, y, xK, invTh, put):
    out = np.zeros(len(R.UNITS[basis]))
    ptr = lambda a: np.ascontiguousarray(a).ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    keep = [np.ascontiguousarray(a, dtype=float) for a in (e, v, y)]
    args = [ctypes.c_int(basis == "sv2"), ctypes.c_int(len(e)), ctypes.c_int(per)]
    args += [ptr(a) for a in keep] + [ctypes.c_double(xK), ctypes.c_double(invTh)]
    if which == "fixed":
        args.append(ctypes.c_int(put))
    getattr(lib, which + "_sums")(*args, ptr(out))
    return out


# type, deviation of log S, mean and deviation of w = v / theta - 1 (gamma
# variance, or normal where the deviation is marked by a minus sign)
SETTINGS = {
    "put, one year": ("put", 0.2, 0.0, 0.8),
    "call, one year": ("call", 0.2, 0.0, 0.8),
    "put, one week": ("put", 0.028, 0.0, 0.2),
    "put, one day": ("put", 0.0126, 0.0, 0.08),
    "call, one day, 5% volatility": ("call", 0.003, 0.0, 0.08),
    "put, one week, xi 0.01": ("put", 0.028, 0.0, -0.007),
    "put, one day, xi 0.005": ("put", 0.0126, 0.0, -0.0013),
    "call, one month, xi 0.001": ("call", 0.058, 0.0, -0.0014),
    "put, v0 = 1.5 theta": ("put", 0.1, 0.5, -0.02),
    "put, v0 = 21 theta": ("put", 0.1, 20.0, -0.5),
    "call deep in the money": ("call", 1.5, 0.0, 0.5),
}


def _paths(kind, n, seed, scale=1.0):
    """n in-the-money row values, variances and cash flows at strike 100 scale"""
    type_, sd, mean, dev = kind
    rng = np.random.default_rng(seed)
    K, theta = 100.0 * scale, 0.04
    z = rng.standard_normal(8 * n + 64)
    u = -0.7 * z + np.sqrt(0.51) * rng.standard_normal(len(z))
    S = K * np.exp(sd * z)
    if dev < 0:
        w = mean - dev * u
    else:  # gamma of mean 1 by ranks
        w = np.empty_like(u)
        w[np.argsort(u)] = np.sort(rng.gamma(1 / dev**2, dev**2, len(u))) - 1.0
    itm = np.flatnonzero(S < K if type_ == "put" else S > K)[:n]
    assert len(itm) == n
    e, v = S[itm], theta * (1.0 + w[itm])
    y = np.maximum(np.abs(e - K) + 0.2 * K * sd * rng.standard_normal(n), 0.0)
    return e, v, y, K, theta


def _fit_error(lib, basis, kind, n, seed, per):
    e, v, y, K, theta = _paths(kind, n, seed)
    s = _sums(lib, "fixed", basis, per, e, v, y, 1.0 / K, 1.0 / theta, kind[0] == "put")
    x, w = R.feature(e, 1.0 / K), R.feature(v, 1.0 / theta)
    m = R.moments(x, w, y, basis)
    got = {u: R.Fraction(float(t)) for u, t in zip(R.UNITS[basis], s)}
    got[0, 0, 0] = m[0, 0, 0]
    ref = R.solve(m, basis)
    bound, _ = R.error_bound(m, y, ref, basis)
    return R.scaled_error([float(b) for b in R.solve(got, basis)], ref, m, basis), bound


@pytest.mark.parametrize("basis", ["s2", "sv2"])
@pytest.mark.parametrize("name", list(SETTINGS))
def test_fits_within_the_error_of_double_precision(lib, name, basis):
    for n, per in ((40, 40), (700, 96)):
        err, bound = _fit_error(lib, basis, SETTINGS[name], n, n, per)
        assert err <= bound, (name, basis, n, err, bound)


@pytest.mark.parametrize("basis", ["s2", "sv2"])
@pytest.mark.parametrize("name", list(SETTINGS))
def test_sums_of_many_paths_have_no_bias(lib, name, basis):
    # a value is rounded to 2^-54 of twice the largest, a product of values a
    # few times: eight roundings of the sum of magnitudes, and of the largest
    # term growing like the root of the paths; a part left out of every path's
    # term would grow like their number
    n = 6000
    kind = SETTINGS[name]
    e, v, y, K, theta = _paths(kind, n, 17)
    s = _sums(lib, "fixed", basis, 1536, e, v, y, 1.0 / K, 1.0 / theta, kind[0] == "put")
    x, w = R.feature(e, 1.0 / K), R.feature(v, 1.0 / theta)
    m, a = R.moments(x, w, y, basis), R.moments(np.abs(x), np.abs(w), y, basis)
    for u, t in zip(R.UNITS[basis], s):
        largest = np.abs(x).max()**u[0] * np.abs(w).max()**u[1] * (y.max() if u[2] else 1.0)
        bound = 8 * R.EPS * (float(a[u]) + n**0.5 * largest)
        assert abs(float(R.Fraction(float(t)) - m[u])) <= bound, (u, bound / float(a[u]))


@pytest.mark.parametrize("basis", ["s2", "sv2"])
def test_fits_no_further_from_exact_than_double_sums(lib, basis):
    # geometric means over settings, sizes and seeds; 1.25 for the spread of a
    # mean over 66 errors that are each one draw
    logs = {"fixed": [], "double": []}
    for kind in SETTINGS.values():
        for n, per in ((40, 40), (400, 128), (2000, 384)):
            for seed in (1, 2):
                e, v, y, K, theta = _paths(kind, n, seed)
                x, w = R.feature(e, 1.0 / K), R.feature(v, 1.0 / theta)
                m = R.moments(x, w, y, basis)
                ref = R.solve(m, basis)
                for which in logs:
                    s = _sums(lib, which, basis, per, e, v, y, 1.0 / K, 1.0 / theta,
                              kind[0] == "put")
                    got = {u: R.Fraction(float(t)) for u, t in zip(R.UNITS[basis], s)}
                    got[0, 0, 0] = m[0, 0, 0]
                    err = R.scaled_error([float(b) for b in R.solve(got, basis)], ref, m, basis)
                    logs[which].append(np.log(err))
    assert np.mean(logs["fixed"]) <= np.mean(logs["double"]) + np.log(1.25)


@pytest.mark.parametrize("basis", ["s2", "sv2"])
def test_scales_follow_values_that_grow_and_any_units(lib, basis):
    # the smallest values first, so that the ranges grow many times; strikes
    # and cash flows from 2^-300 to 2^300: the same integers, shifted
    e, v, y, K, theta = _paths(("call", 0.8, 0.0, 0.8), 640, 5)
    grow = np.argsort(np.abs(e / K - 1.0) * np.abs(v / theta - 1.0) * (y + 1e-3))
    e, v, y = e[grow], v[grow], y[grow]
    x, w = R.feature(e, 1.0 / K), R.feature(v, 1.0 / theta)
    m = R.moments(x, w, y, basis)
    base = _sums(lib, "fixed", basis, 640, e, v, y, 1.0 / K, 1.0 / theta, False)
    a = R.moments(np.abs(x), np.abs(w), y, basis)
    for (u, t) in zip(R.UNITS[basis], base):
        # 54-bit values of at most twice the largest: an error of 2^-53 of the
        # largest a path and factor, growing like the root of the paths
        largest = np.abs(x).max()**u[0] * np.abs(w).max()**u[1] * (y.max() if u[2] else 1.0)
        bound = 16 * 2.0**-53 * (float(a[u]) + 26 * largest)
        assert abs(float(R.Fraction(float(t)) - m[u])) <= bound, (u, t)
    for k in (-300, 300):
        f = 2.0**k
        s = _sums(lib, "fixed", basis, 640, e * f, v, y * f, 1.0 / (K * f), 1.0 / theta, False)
        for u, t, b in zip(R.UNITS[basis], s, base):
            assert t == (b * f if u[2] else b), (u, k)


@pytest.mark.parametrize("basis", ["s2", "sv2"])
@pytest.mark.parametrize("n", [61 * 32, 125 * 32 + 1, 126 * 32])
def test_largest_sums(lib, basis, n):
    # as many paths as a lane may sum, each at the top of its range: no sum
    # overflows (with equal values the part left out of the squares is at most
    # 2^-58 of them, below the bound)
    K, theta = 100.0, 0.04
    e, v = np.full(n, K * 2.0**-50), np.full(n, theta * (9.0 - 2.0**-49))
    y = np.full(n, 128.0 * (1.0 - 2.0**-53))
    s = _sums(lib, "fixed", basis, n, e, v, y, 1.0 / K, 1.0 / theta, True)
    x, w = R.feature(e, 1.0 / K), R.feature(v, 1.0 / theta)
    assert 1 - 2.0**-40 < -x[0] < 1 and 8 - 2.0**-40 < w[0] < 8
    m, a = R.moments(x, w, y, basis), R.moments(np.abs(x), np.abs(w), y, basis)
    for u, t in zip(R.UNITS[basis], s):
        assert abs(float(R.Fraction(float(t)) - m[u])) <= 4 * R.EPS * float(a[u]), (u, t)


@pytest.mark.parametrize("basis", ["s2", "sv2"])
def test_zero_cash_flows_and_few_paths(lib, basis):
    for n in (1, 2, 31, 32, 33, 65):
        e, v, y, K, theta = _paths(SETTINGS["put, one day"], n, n)
        y[: n // 2] = 0.0
        s = _sums(lib, "fixed", basis, 640, e, v, y, 1.0 / K, 1.0 / theta, True)
        x, w = R.feature(e, 1.0 / K), R.feature(v, 1.0 / theta)
        m, a = R.moments(x, w, y, basis), R.moments(np.abs(x), np.abs(w), y, basis)
        for u, t in zip(R.UNITS[basis], s):
            largest = np.abs(x).max()**u[0] * np.abs(w).max()**u[1] * (y.max() if u[2] else 1.0)
            bound = 16 * 2.0**-53 * (float(a[u]) + n**0.5 * largest)
            assert abs(float(R.Fraction(float(t)) - m[u])) <= bound, (n, u)


def test_values_beyond_the_largest_range_are_summed_in_double(lib):
    # infinities and NaN in single lanes reach the sums they belong to and
    # leave the others as they were
    e, v, y, K, theta = _paths(SETTINGS["put, one year"], 100, 3)
    units = R.UNITS["sv2"]
    for bad, where in ((np.inf, "v"), (np.nan, "v"), (1e200, "y"), (np.inf, "y")):
        v2, y2 = v.copy(), y.copy()
        (v2 if where == "v" else y2)[57] = bad
        s = _sums(lib, "fixed", "sv2", 640, e, v2, y2, 1.0 / K, 1.0 / theta, True)
        ref = _sums(lib, "double", "sv2", 640, e, v2, y2, 1.0 / K, 1.0 / theta, True)
        for u, t, r in zip(units, s, ref):
            if np.isfinite(r):
                assert abs(t - r) <= 1e-13 * max(abs(r), 1.0), (bad, where, u, t, r)
            else:
                assert np.isnan(t) == np.isnan(r) and (np.isnan(r) or t == r), (bad, where, u, t, r)
