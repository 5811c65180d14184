"""The single-precision multi-asset reduction where a CTA takes four assets
(2^19 paths and more): groups of assets that are not full, one group (plain
stores) and two (atomic maxima), a ragged last CTA; against the oracle on the
same streams, at the bounds of the reduction's other single-precision tests."""
import numpy as np
import pytest

import oracle
from gpu_common import torch_cuda
from paper_2206_03719_gb300 import lsmc as L
from paper_2206_03719_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho_assets", [0.0, 0.4])
@pytest.mark.parametrize("scheme", [L.LSMC_SCHEME_QE, L.LSMC_SCHEME_FT_EULER])
@pytest.mark.parametrize("A", [1, 3, 4, 5])
def test_four_assets_a_cta(A, scheme, rho_assets):
    torch = torch_cuda()
    from paper_2206_03719_gb300 import build
    build.build()
    P, N = (1 << 19) + 77, 3
    models = workloads.stac_models(A, seed=4)
    M = torch.full((N + 1, P), float("nan"), dtype=torch.float32, device="cuda")
    L.lsmc_multi_asset_max([L.lsmc_heston(**m) for m in models], 0.5, scheme, L.LSMC_MIXED,
                           rho_assets, P, N, 9, 2, M.data_ptr())
    torch.cuda.synchronize()
    got = M.cpu().numpy().astype(np.float64)
    ref = oracle.multi_max([oracle.heston(**m) for m in models], 0.5, scheme, P, N, 9, 2,
                           rho_assets=rho_assets, grid=oracle.GRID_F32)
    assert np.array_equal(got[0], np.full(P, np.float64(np.float32(ref[0, 0]))))
    rel = np.abs(got - ref) / ref
    assert np.quantile(rel, 0.999) < 2e-5 and rel.max() < 1e-3
