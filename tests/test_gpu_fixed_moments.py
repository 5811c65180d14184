"""The double-precision regressions' fixed-point moment sums (fixed_moments.cuh)
where they can go wrong: remainders of a warp and of a tile, paths outside the
range taken from the previous date (summed in double), very small and very
large prices; against the oracle on the same paths at the parity bound."""
import numpy as np
import pytest

import oracle
from gpu_common import backward_parity, torch_cuda
from paper_2206_03719_gb300 import lsmc as L

pytestmark = pytest.mark.gpu
H = dict(S0=100.0, r=0.02, q=0.01, v0=0.04, kappa=1.5, theta=0.04, xi=0.3, rho=-0.7)


@pytest.fixture(scope="module")
def torch():
    t = torch_cuda()
    from paper_2206_03719_gb300 import build
    build.build()
    L.load()
    return t


def _run(torch, S, V, model, K, type_, basis):
    N, P = S.shape[0] - 1, S.shape[1]
    dS, dV = torch.from_numpy(S).cuda(), torch.from_numpy(V).cuda()
    out = torch.zeros(5, dtype=torch.float64, device="cuda")
    ns = torch.zeros(1, dtype=torch.int32, device="cuda")
    L.lsmc_backward(dS.data_ptr(), dV.data_ptr(), P, N, L.LSMC_FP64, L.lsmc_heston(**model),
                    L.lsmc_contract(type_, L.LSMC_AMERICAN, K, 1.0), basis, out.data_ptr(), None,
                    ns.data_ptr())
    return out.cpu().numpy(), int(ns.cpu().numpy()[0])


def _check(torch, S, V, model, K, type_, basis, what):
    got, ns = _run(torch, S, V, model, K, type_, basis)
    ref = backward_parity(got, S, V, model["S0"], K, 1.0, model["r"], model["theta"], type_=type_,
                          basis=basis, what=what)
    assert ns == ref["n_singular"], what


@pytest.mark.parametrize("basis", [L.LSMC_BASIS_S2, L.LSMC_BASIS_SV2])
@pytest.mark.parametrize("P", [1, 31, 33, 255, 257, 1025, 4111])
def test_remainders(torch, P, basis):
    S, V = oracle.paths(oracle.heston(**H), 1.0, oracle.QE, P, 12, 5, 0)
    _check(torch, S, V, H, 104.0, L.LSMC_PUT, basis, "remainders %d" % P)


@pytest.mark.parametrize("basis", [L.LSMC_BASIS_S2, L.LSMC_BASIS_SV2])
@pytest.mark.parametrize("type_", [L.LSMC_PUT, L.LSMC_CALL])
def test_paths_outside_the_range_of_the_previous_date(torch, type_, basis):
    # every third date a few paths (never the same) leave the others' range of
    # x or w by a factor of 20 or more
    P, N = 2500, 15
    S, V = oracle.paths(oracle.heston(**H), 1.0, oracle.QE, P, N, 9, 0)
    rng = np.random.default_rng(4)
    for n in range(2, N, 3):
        i = rng.choice(P, 40, replace=False)
        V[n, i[:20]] *= 30.0
        S[n, i[20:]] *= 12.0 if type_ == L.LSMC_CALL else 0.02
    _check(torch, S, V, H, 100.0, type_, basis, "outside the range")


@pytest.mark.parametrize("scale", [1e-7, 1e9])
def test_small_and_large_prices(torch, scale):
    model = dict(H, S0=100.0 * scale)
    S, V = oracle.paths(oracle.heston(**model), 1.0, oracle.QE, 2000, 10, 3, 0)
    _check(torch, S, V, model, 103.0 * scale, L.LSMC_PUT, L.LSMC_BASIS_SV2, "scale %g" % scale)
