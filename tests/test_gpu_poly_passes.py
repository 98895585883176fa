"""The fused 2D complex64 passes of the polynomial smoother (a sweep, and the transfers beside
it, per launch) and its single-CTA coarse levels against the oracle: grids that end at, just
before and after the edge of a region's 24 (16-row regions: 8) own points, both region
heights, and every number of sweeps down and up.  Bound: that of the complex64 polynomial
V-cycle in test_gpu_parity.py (1e-4; the passes take the same steps in the same order)."""
import numpy as np
import pytest

import oracle as O
from paper_1012_5379_gb300 import inputs as I
from parity_check import assert_parity
from test_gpu_parity import poly_weights

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def helm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_5379_gb300 import build, helm as H
    build.build()
    H.load()
    return H


@pytest.mark.parametrize("dim,n,nu1,nu2", [(2, 31, 1, 1), (2, 39, 1, 1), (2, 47, 2, 2), (2, 71, 1, 0), (2, 95, 0, 1),
                                           (2, 143, 3, 1), (2, 319, 1, 1), (2, 383, 2, 1), (3, 7, 2, 2), (3, 15, 1, 1)])
def test_fused_poly_vcycle_matches_oracle(helm, dim, n, nu1, nu2):
    from oracle import polysmoother as PS
    k, tb, tg = 0.1 * (n + 1), np.radians(10.0), np.radians(30.0)
    levels = O.build_hierarchy(dim, n, tb, tg, I.ECS_FRAC, k=k)
    r = I.random_source(dim, n, 700 + n)
    want = PS.vcycle_poly(levels, poly_weights(helm, levels, k, tb, tg), r, nu1, nu2)
    h = helm.Handle(dim, n, tb, k=k, theta_gamma=tg, precision="c64", nu1=nu1, nu2=nu2, smoother="poly")
    rt = torch.from_numpy(r).cuda().to(torch.complex64)
    zt = torch.empty_like(rt)
    h.precond_apply(rt, zt)
    assert_parity(zt, want, 1e-4, "polynomial V-cycle")
