"""The double-precision and float-pair steppers' tables and steps (forward_f64.h,
forward_df.h, Draw and qe_core): the quantile segments and the exponential's cubic against
40-digit values on the CPU; the draws and the paths of the GPU at the models
where the step changes form."""
import os
import re

import numpy as np
import pytest

import oracle

mp = pytest.importorskip("mpmath")
HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                      "paper_2206_03719_gb300", "csrc", "forward_f64.h")
OCT, SEG, DEG, EXPN = 10, 64, 6, 2048


def _tables():
    text = open(HEADER).read()
    const = {k: float(np.float32(v.rstrip("f"))) if v.endswith("f") else float(v)
             for k, v in re.findall(r"(kExp\w+) = ([-+.\de]+f?)[;,]", text)}
    body = text[text.index("kF64Tables = {"):]
    vals = [float(v) for v in re.findall(r"-?\d\.\d+e[+-]\d+", body)]
    n = OCT * SEG
    assert len(vals) == n + 3 * 2 * n + 3 * n + EXPN
    q0, rest = np.array(vals[:n]), np.array(vals[n:10 * n], dtype=np.float32).astype(float)
    qp = rest[:6 * n].reshape(3, n, 2).sum(-1)
    qf = rest[6 * n:].reshape(3, n)
    return const, np.concatenate([q0[None], qp, qf]), vals[10 * n:]


def _quantile(p):
    return -mp.sqrt(2) * mp.erfinv(1 - 2 * mp.mpf(p))


@pytest.mark.parametrize("octave", range(1, OCT + 1))
def test_quantile_segments_at_their_edges(octave):
    # the polynomials as stored, evaluated exactly: half a unit in the last
    # place of c_0 and 2^-48 of c_1 / 2 (at most 2^-54), 1.7e-16 together
    mp.mp.dps = 40
    _, qc, _ = _tables()
    for seg in (0, 1, 31, 62, 63):
        left = mp.mpf(2) ** -(octave + 1) * (1 + mp.mpf(seg) / SEG)
        width = mp.mpf(2) ** -(octave + 1) / SEG
        c = qc[:, (octave - 1) * SEG + seg]
        for t in (-0.5, 0.0, 0.5):
            v = mp.mpf(0)
            for x in c[::-1]:
                v = v * t + mp.mpf(float(x))
            z = _quantile(left + width * (mp.mpf(t) + mp.mpf(0.5)))
            assert abs(v - z) <= mp.mpf(1.7e-16) * max(1, abs(z))


def test_exponential_cubic_and_table():
    mp.mp.dps = 40
    const, _, e2 = _tables()
    for j in (0, 1, 1023, 2047):
        assert e2[j] == float(mp.mpf(2) ** (mp.mpf(j) / EXPN))
    for f in (-0.5, -0.3, 0.1, 0.5):
        g = mp.mpf(f) * 2 ** 22
        a1 = mp.mpf(const["kExpA1"]) + mp.mpf(const["kExpA1Lo"])
        a2 = mp.mpf(const["kExpA2"]) + mp.mpf(const["kExpA2Lo"])
        p = ((mp.mpf(const["kExpA3"]) * g + a2) * g + a1) * g
        assert abs(p - (mp.mpf(2) ** (mp.mpf(f) / EXPN) - 1)) < 2e-17
    unit = mp.mpf(const["kExpUnit"]) + mp.mpf(const["kExpUnitLo"])
    assert abs(unit * mp.log(2) / EXPN - 1) < 1e-30


@pytest.mark.gpu
def test_draws_within_one_rounding_of_the_segments():
    from gpu_common import torch_cuda
    from paper_2206_03719_gb300 import build
    from paper_2206_03719_gb300 import lsmc as L
    torch = torch_cuda()
    build.build()
    mp.mp.dps = 30
    n = 3000
    path = torch.arange(n, dtype=torch.int32, device="cuda")
    step = torch.full_like(path, 3)
    out = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    L.lsmc_draws(99, 1, path.data_ptr(), step.data_ptr(), n, L.LSMC_FP64, out.data_ptr())
    got = out.cpu().numpy()
    worst = 0.0
    for u, zv, _ in got:
        z = _quantile(mp.mpf(float(u)))
        # table 1.7e-16, the last sum half a unit in the last place (1.2e-16),
        # the pairs' product 2^-53 / 2; the tails use norm_quantile_f64 (6e-16)
        tail = min(u, 1.0 - u) < 2.0 ** -(OCT + 1)
        err = float(abs(mp.mpf(float(zv)) - z) / max(1, abs(z)))
        assert err <= (6e-16 if tail else 3.5e-16), (u, zv, err)
        worst = max(worst, err)
    print("draws: worst %.3g" % worst)


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [
    dict(xi=1e-9),                                 # psi -> 0: a is far below m
    dict(xi=2.5, kappa=0.3, theta=0.02),           # nearly always the exponential branch
    dict(v0=0.0),                                  # zero start
    dict(v0=1e-70, theta=1e-70, xi=1e-36),         # outside the range of the products
    dict(rho=1.0), dict(rho=-1.0),                 # K3 = 0
], ids=lambda k: ",".join("%s=%g" % i for i in k.items()))
def test_paths_where_the_step_changes_form_match_oracle(kw):
    from gpu_common import torch_cuda
    from paper_2206_03719_gb300 import build
    from paper_2206_03719_gb300 import lsmc as L
    torch = torch_cuda()
    build.build()
    model = dict(S0=100.0, r=0.02, q=0.0, v0=0.04, kappa=1.5, theta=0.04, xi=0.3, rho=-0.7)
    model.update(kw)
    P, N = 500, 30
    S = torch.empty((N + 1, P), dtype=torch.float64, device="cuda")
    V = torch.empty_like(S)
    L.lsmc_paths(L.lsmc_heston(**model), 0.5, L.LSMC_SCHEME_QE, L.LSMC_FP64, P, N, 5, 2,
                 S.data_ptr(), V.data_ptr())
    So, Vo = oracle.paths(oracle.heston(**model), 0.5, oracle.QE, P, N, 5, 2)
    # the stage tests' tolerances; log prices carry 1/xi of the variance's
    # rounding (K2 = rho / xi) at the smallest xi
    rtol_s = 1e-12 + 2e-16 * 100 * model["v0"] / model["xi"]
    assert np.allclose(S.cpu().numpy(), So, rtol=rtol_s, atol=0)
    # where the variance nearly vanishes (v1 = log(omp / U) / beta at omp ~ U) the
    # oracle's own rounding is amplified by the step: 1e-13 absolute
    assert np.allclose(V.cpu().numpy(), Vo, rtol=1e-11,
                       atol=1e-13 if model["theta"] > 1e-10 else 1e-84)


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [
    dict(xi=2.5, kappa=0.3, theta=0.02), dict(v0=0.0),
    dict(v0=1e-8, theta=1e-8, xi=1e-4),            # means outside the range of the products
    dict(rho=1.0), dict(rho=-1.0),
], ids=lambda k: ",".join("%s=%g" % i for i in k.items()))
def test_pair_paths_where_the_step_changes_form_match_oracle(kw):
    from gpu_common import torch_cuda
    from paper_2206_03719_gb300 import build
    from paper_2206_03719_gb300 import lsmc as L
    torch = torch_cuda()
    build.build()
    model = dict(S0=100.0, r=0.02, q=0.0, v0=0.04, kappa=1.5, theta=0.04, xi=0.3, rho=-0.7)
    model.update(kw)
    P, N = 500, 30
    S = torch.empty((N + 1, P, 2), dtype=torch.float32, device="cuda")
    V = torch.empty_like(S)
    L.lsmc_paths(L.lsmc_heston(**model), 0.5, L.LSMC_SCHEME_QE, L.LSMC_DF, P, N, 5, 2,
                 S.data_ptr(), V.data_ptr())
    So, Vo = oracle.paths(oracle.heston(**model), 0.5, oracle.QE, P, N, 5, 2)
    # the stage tests' tolerances for pairs; at xi = 2.5 the step amplifies a
    # rounding 2^-48 as it does 2^-53 in double (1e-13 there): 1e-11
    atol = 1e-11 if model["xi"] > 1 else 1e-14 * max(1.0, model["theta"] / 0.04)
    assert np.allclose(S.double().sum(-1).cpu().numpy(), So, rtol=1e-11, atol=0)
    assert np.allclose(V.double().sum(-1).cpu().numpy(), Vo, rtol=1e-10, atol=atol)


@pytest.mark.gpu
@pytest.mark.parametrize("A,P", [(1, 130), (2, 1), (3, 257), (5, 128)])
def test_reduction_in_pairs_of_assets_is_the_maximum_of_the_assets(A, P):
    # single precision and pairs: the maximum over separately reduced assets,
    # bit for bit (one asset per call cannot be: each draws by its index, so
    # the reduction over the first k assets grows with k); and pairs at an
    # address that is not a multiple of 8
    from gpu_common import torch_cuda
    from paper_2206_03719_gb300 import build, workloads
    from paper_2206_03719_gb300 import lsmc as L
    torch = torch_cuda()
    build.build()
    N = 7
    models = [L.lsmc_heston(**m) for m in workloads.stac_models(A)]

    def run(ms, prec, offset=0):
        n = (N + 1) * P * (2 if prec == L.LSMC_DF else 1)
        dt = torch.float64 if prec == L.LSMC_FP64 else torch.float32
        buf = torch.full((n + 1,), float("nan"), dtype=dt, device="cuda")
        M = buf[offset:offset + n]
        L.lsmc_multi_asset_max(ms, 0.5, L.LSMC_SCHEME_QE, prec, 0.0, P, N, 3, 1, M.data_ptr())
        torch.cuda.synchronize()
        return M.cpu().numpy().copy()

    for prec in (L.LSMC_FP64, L.LSMC_MIXED, L.LSMC_DF):
        got = run(models, prec)
        assert np.all(np.isfinite(got))
        if prec == L.LSMC_DF:
            assert np.array_equal(got, run(models, prec, 1))
            got = got.reshape(-1, 2).astype(np.float64).sum(-1)
        for k in range(1, A):
            part = run(models[:k], prec)
            if prec == L.LSMC_DF:
                part = part.reshape(-1, 2).astype(np.float64).sum(-1)
            assert np.all(got >= part)
        ref = oracle.multi_max([oracle.heston(**m) for m in workloads.stac_models(A)], 0.5,
                               oracle.QE, P, N, 3, 1,
                               grid=oracle.GRID_F32 if prec == L.LSMC_MIXED else oracle.GRID_F64)
        rtol = {L.LSMC_FP64: 1e-12, L.LSMC_DF: 1e-11, L.LSMC_MIXED: 1e-3}[prec]
        assert np.allclose(got.reshape(N + 1, P), ref, rtol=rtol, atol=0)
