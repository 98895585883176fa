"""Complex64 V-cycles at the size of their rounding errors.

The bounds of tests/parity_check.py (5e-5) hold for any field; on white noise, constant k and mild
fields the measured errors are 1 to 5e-7, and these bounds are two to three times that: a rim one
point short, a wrong edge coefficient or a sum in the wrong order of magnitude shows."""
import numpy as np
import pytest

import oracle as O
from oracle import polysmoother as PS
from paper_1012_5379_gb300 import inputs as I
from parity_check import assert_parity, errors
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


def apply(h, r, dtype=torch.complex64):
    rt = torch.from_numpy(r).cuda().to(dtype)
    z = torch.empty_like(rt)
    h.precond_apply(rt, z)
    return z


# region, fused, marching and single-CTA levels, with their edges (own points 26, 28, 30, 24 of 32)
@pytest.mark.parametrize("dim,n,s,nu1,nu2,field", [
    (2, 23, 3, 1, 1, False), (2, 39, 3, 1, 1, True), (2, 47, 4, 1, 1, False), (2, 55, 2, 1, 1, True),
    (2, 71, 1, 1, 1, False), (2, 87, 3, 2, 1, False), (2, 143, 3, 1, 1, True), (2, 223, 4, 1, 2, False),
    (2, 319, 3, 1, 1, False), (2, 575, 3, 1, 1, True), (2, 639, 3, 1, 0, False), (2, 703, 1, 1, 1, True),
    (2, 895, 3, 1, 1, False), (2, 1279, 2, 2, 1, False), (3, 9, 3, 1, 1, False), (3, 19, 3, 1, 1, True),
    (3, 23, 2, 1, 1, False), (3, 39, 1, 1, 1, True), (3, 47, 3, 1, 1, False), (3, 79, 3, 2, 1, True), (3, 95, 4, 1, 1, False)])
def test_gmres_cycles(helm, dim, n, s, nu1, nu2, field):
    k = 0.2 * (n + 1)
    phi = (np.random.default_rng(n).uniform(0.9, 1.1, (n,) * dim) * k * k).astype(np.float32) if field else None
    r = I.random_source(dim, n, 300 + n).astype(np.complex64)
    h = helm.Handle(dim, n, 0.3, k=None if field else k, phi=torch.from_numpy(phi).cuda() if field else None,
                    precision="c64", s=s, nu1=nu1, nu2=nu2, maxit=1)
    levels = O.build_hierarchy(dim, n, 0.3, k=None if field else k, phi=phi.astype(np.float64) if field else None)
    assert_parity(apply(h, r), O.vcycle(levels, r.astype(complex), nu1, nu2, s), 1.5e-6, f"n={n} s={s}")


@pytest.mark.parametrize("dim,n,nu1,nu2", [(2, 31, 1, 1), (2, 39, 1, 1), (2, 47, 2, 2), (2, 71, 1, 0), (2, 95, 0, 1),
                                           (2, 143, 3, 1), (2, 319, 1, 1), (2, 383, 2, 1), (3, 7, 2, 2), (3, 15, 1, 1)])
def test_polynomial_cycles(helm, dim, n, nu1, nu2):
    k, tb, tg = 0.1 * (n + 1), np.radians(10.0), np.radians(30.0)
    levels = O.build_hierarchy(dim, n, tb, tg, I.ECS_FRAC, k=k)
    r = I.random_source(dim, n, 700 + n).astype(np.complex64)
    want = PS.vcycle_poly(levels, poly_weights(helm, levels, k, tb, tg), r.astype(complex), nu1, nu2)
    h = helm.Handle(dim, n, tb, k=k, theta_gamma=tg, precision="c64", nu1=nu1, nu2=nu2, smoother="poly")
    assert_parity(apply(h, r), want, 7e-7, "polynomial V-cycle")


# errors of a pass per Richardson step that adds the diagonal's term last: 1.3e-7, 8.7e-7, 6.1e-6
# (the polynomial damps the coarsest levels' smooth waves badly: they carry the error); bound 1.5
# times that, for the scatter between right-hand sides
@pytest.mark.parametrize("n,tol", [(127, 2e-7), (1023, 1.3e-6), (2047, 9e-6)])
def test_polynomial_cycle_of_many_levels(helm, n, tol):
    """Against the complex128 cycle (held to the oracle elsewhere)."""
    tb, tg = np.radians(10.0), np.radians(30.0)
    hs = [helm.Handle(2, n, tb, k=0.1 * (n + 1), theta_gamma=tg, precision=p, smoother="poly", maxit=1)
          for p in ("c64", "c128")]
    es = []
    for seed in range(4):
        r = I.random_source(2, n, seed).astype(np.complex64)
        es.append(errors(apply(hs[0], r), apply(hs[1], r, torch.complex128))[0])
    assert np.mean(es) <= tol, es


@pytest.mark.parametrize("n,mean", [(255, 1.42e-7), (511, 1.50e-7)])
def test_polynomial_update_is_rounded_once(helm, n, mean):
    """x + w r with the small product rounded at its own size: the error of one Richardson step
    per pass over eight right-hand sides, whose mean scatters by 1.5%; both rounded at x's size
    cost 7%.  Bound 4%."""
    tb, tg = np.radians(10.0), np.radians(30.0)
    hs = [helm.Handle(2, n, tb, k=0.1 * (n + 1), theta_gamma=tg, precision=p, smoother="poly", maxit=1)
          for p in ("c64", "c128")]
    rs = [I.random_source(2, n, seed).astype(np.complex64) for seed in range(8)]
    es = [errors(apply(hs[0], r), apply(hs[1], r, torch.complex128))[0] for r in rs]
    assert np.mean(es) <= 1.04 * mean, es
