"""The fused passes of the complex64 2D V(1,1) cycle (sweep.cuh): restriction inside the coarser
level's sweep, coarse correction, residual and sweep of a level in one pass, the last update in
the output pass.  Sizes at the edges of their regions (own points 26, 24 and 8 to 26 rows of 32),
with and without a fused, a marching and a single-CTA level beside them, every sweep length."""
import numpy as np
import pytest

import oracle as O
from paper_1012_5379_gb300 import inputs as I
from parity_check import assert_parity

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


# against the oracle at the V-cycle's own tolerance (complex64: 5e-5, the bound every V-cycle test
# has; binary32 sums over nine levels)
@pytest.mark.parametrize("n,s,field", [(35, 3, False), (47, 1, True), (63, 4, False), (79, 2, False), (127, 3, True),
                                       (175, 4, True), (255, 3, False), (287, 2, True), (351, 1, False),
                                       (575, 3, False), (575, 4, True), (639, 3, True), (703, 2, False),
                                       (703, 4, False)])
def test_fused_vcycle(helm, n, s, field):
    k, tb = 0.15 * (n + 1), 0.3
    phi = (np.random.default_rng(n).uniform(0.8, 1.2, (n, n)) * k * k).astype(np.float32) if field else None
    r = I.random_source(2, n, 700 + n)
    h = helm.Handle(2, n, tb, k=None if field else k, phi=torch.from_numpy(phi).cuda() if field else None,
                    precision="c64", s=s, maxit=1)
    rt = torch.from_numpy(r).cuda().to(torch.complex64)
    z = torch.empty_like(rt)
    h.precond_apply(rt, z)
    first = z.clone()
    h.precond_apply(rt, z)
    assert torch.equal(first, z)
    levels = O.build_hierarchy(2, n, tb, k=None if field else k, phi=phi.astype(np.float64) if field else None)
    assert_parity(z, O.vcycle(levels, r, s=s), ("vcycle", "c64"), f"n={n} s={s}")


def test_mixed_batch_equals_alone_bitwise(helm):
    # finest levels in one CTA, fused, and marching, in one group
    hs, bs = [], []
    for i, n in enumerate((31, 63, 255, 1023, 127)):
        hs.append(helm.Handle(2, n, 0.35, k=0.03 * (n + 1), precision="c64", restart=20))
        bs.append(torch.from_numpy(I.random_source(2, n, i)).cuda())
    xs = [torch.zeros_like(b) for b in bs]
    infos = helm.batch_solve(hs, bs, xs, 1e-4)
    for h, b, x, inf in zip(hs, bs, xs, infos):
        solo = torch.zeros_like(b)
        sinfo = h.solve(b, solo, 1e-4)
        assert inf.iters == sinfo.iters and torch.equal(solo, x)
