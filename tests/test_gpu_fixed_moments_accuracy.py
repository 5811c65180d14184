"""Regression coefficients of the double-precision backward pass against exact
rational fits of the same paths: short maturities, small volatilities of
variance, v0 away from theta, and dates whose distributions differ by orders of
magnitude; within the error that a double-precision fit may have
(fixed_moments_ref.error_bound)."""
import numpy as np
import pytest

import fixed_moments_ref as R
import oracle
from gpu_common import torch_cuda
from paper_2206_03719_gb300 import lsmc as L

pytestmark = pytest.mark.gpu
H = dict(S0=100.0, r=0.02, q=0.01, v0=0.04, kappa=1.5, theta=0.04, xi=0.3, rho=-0.7)
BASIS = {"s2": L.LSMC_BASIS_S2, "sv2": L.LSMC_BASIS_SV2}


@pytest.fixture(scope="module")
def torch():
    t = torch_cuda()
    from paper_2206_03719_gb300 import build
    build.build()
    L.load()
    return t


def _coefficients(torch, S, V, model, K, T, type_, basis):
    N, P = S.shape[0] - 1, S.shape[1]
    dS, dV = torch.from_numpy(S).cuda(), torch.from_numpy(V).cuda()
    out = torch.zeros(5, dtype=torch.float64, device="cuda")
    beta = torch.zeros((N, 6), dtype=torch.float64, device="cuda")
    ns = torch.zeros(1, dtype=torch.int32, device="cuda")
    L.lsmc_backward(dS.data_ptr(), dV.data_ptr(), P, N, L.LSMC_FP64, L.lsmc_heston(**model),
                    L.lsmc_contract(type_, L.LSMC_AMERICAN, K, T), BASIS[basis], out.data_ptr(),
                    beta.data_ptr(), ns.data_ptr())
    torch.cuda.synchronize()
    return beta.cpu().numpy()


def reference(S, V, model, K, T, put, basis):
    """Per date n = N - 1, ..., 1: (n, exact coefficients in units of the cash
    flow at t_n, moments, cash flows, closest decision to its threshold),
    decisions taken with the exact coefficients; coefficients None, and no
    exercise, where the regression is singular by the library's rule."""
    N = S.shape[0] - 1
    dt, r = T / N, model["r"]
    pay = lambda s: np.maximum(K - s, 0.0) if put else np.maximum(s - K, 0.0)  # noqa: E731
    Z = pay(S[N]) * np.exp(-r * N * dt)
    for n in range(N - 1, 0, -1):
        itm = np.flatnonzero(S[n] < K if put else S[n] > K)
        x, w = R.feature(S[n][itm], 1.0 / K), R.feature(V[n][itm], 1.0 / model["theta"])
        y = Z[itm] * np.exp(r * n * dt)
        m = R.moments(x, w, y, basis)
        pivot = R.smallest_pivot(m, basis)
        assert not 0.5e-13 < pivot < 2e-13, (n, pivot)
        if pivot < 1e-13:
            yield n, None, m, y, 1.0
            continue
        beta = R.solve(m, basis)
        b = [float(t) for t in beta]
        c = b[0] + b[1] * x + b[2] * x * x
        if basis == "sv2":
            c = c + b[3] * w + b[4] * x * w + b[5] * w * w
        h = pay(S[n][itm])
        near = np.min(np.abs(h - c) / np.maximum(np.abs(c), h))
        yield n, beta, m, y, near
        ex = itm[h > c]
        Z[ex] = pay(S[n][ex]) * np.exp(-r * n * dt)


def _check(torch, S, V, model, K, T, put, basis, what):
    got = _coefficients(torch, S, V, model, K, T, L.LSMC_PUT if put else L.LSMC_CALL, basis)
    for n, ref, m, y, near in reference(S, V, model, K, T, put, basis):
        if ref is None:
            assert np.isnan(got[n]).all(), (what, n, got[n])
            continue
        bound, cond = R.error_bound(m, y, ref, basis)
        err = R.scaled_error(got[n][: len(ref)], ref, m, basis)
        assert err <= bound, (what, n, err, bound, cond)
        assert near > 1e-9, (what, n, near)  # the next date's cash flows are certain


CASES = {  # T, changes of the model, put
    "one year": (1.0, {}, True),
    "one week": (1 / 52, {}, True),
    "one week, call": (1 / 52, {}, False),
    "one day": (1 / 252, {}, True),
    "one day, call at 5% volatility": (1 / 252, dict(v0=0.0025, theta=0.0025, xi=0.05), False),
    "one week, 2% volatility": (1 / 52, dict(v0=0.0004, theta=0.0004, xi=0.02), True),
    "one week, xi 0.02": (1 / 52, dict(xi=0.02), True),
    "one week, xi 0.005, call": (1 / 52, dict(xi=0.005), False),
    "one day, xi 0.005": (1 / 252, dict(xi=0.005), True),
    "one year, xi 0.001": (1.0, dict(xi=0.001), True),
    "one month, v0 = 1.5 theta": (1 / 12, dict(v0=0.06), True),
    "one month, v0 = 12 theta, call": (1 / 12, dict(v0=0.48), False),
}


@pytest.mark.parametrize("basis", ["s2", "sv2"])
@pytest.mark.parametrize("name", list(CASES))
def test_coefficients(torch, name, basis):
    T, change, put = CASES[name]
    model = dict(H, **change)
    S, V = oracle.paths(oracle.heston(**model), T, oracle.QE, 3001, 4, 7, 0)
    _check(torch, S, V, model, 100.0, T, put, basis, name)


@pytest.mark.parametrize("basis", ["s2", "sv2"])
@pytest.mark.parametrize("narrow_S, narrow_V", [(1e-3, 1e-2), (0.03, 0.02)])
def test_dates_of_very_different_spread(torch, basis, narrow_S, narrow_V):
    # the spread of S and v about the strike and theta changes by these factors
    # from date to date (with the first pair the narrow dates' regressions are
    # singular)
    S, V = oracle.paths(oracle.heston(**H), 1.0, oracle.QE, 3001, 6, 11, 0)
    for n in (2, 4, 5):
        S[n] = 100.0 + narrow_S * (S[n] - 100.0)
        V[n] = 0.04 + narrow_V * (V[n] - 0.04)
    _check(torch, S, V, H, 100.0, 1.0, True, basis, "spread")


@pytest.mark.parametrize("option", ["put", "call"])
@pytest.mark.parametrize("basis", ["s2", "sv2"])
def test_jobs_whose_sums_are_taken_out_more_than_once(torch, basis, option):
    # more paths a lane than its integers hold (beyond 31 sub-tiles of 4 paths,
    # 62 of 2), deep in the money so that every path is summed: the prices of
    # jobs of one sub-tile (no decision lies within 1e-12 of its threshold)
    from paper_2206_03719_gb300 import api, workloads
    K = 190.0 if option == "put" else 30.0
    wl = workloads.SMALL_FP64.replace(n_paths=40013, n_steps=5, basis=basis, option=option,
                                      greeks=("delta",), strikes=[K, 100.0],
                                      model=dict(H, q=0.04))
    rows = {}
    with api.Context(workspace_bytes=1 << 30) as ctx:
        for shape in ((1, 4), (15, 4), (16, 4), (31, 4), (32, 4), (63, 2), (64, 4)):
            ctx.set_backward_shape(*shape)
            rows[shape] = ctx.price(wl)
    for shape, got in rows.items():
        for g, r in zip(got, rows[1, 4]):
            for k in ("price", "price_se", "delta"):
                assert abs(g[k] - r[k]) <= 1e-12 * max(abs(r[k]), 1e-3), (shape, k, g[k], r[k])
            assert g["n_singular_solves"] == r["n_singular_solves"]


@pytest.mark.parametrize("basis", ["s2", "sv2"])
def test_call_deep_in_the_money(torch, basis):
    model = dict(H, S0=600.0, q=0.05)
    S, V = oracle.paths(oracle.heston(**model), 1.0, oracle.QE, 2001, 3, 13, 0)
    _check(torch, S, V, model, 100.0, 1.0, False, basis, "deep")
