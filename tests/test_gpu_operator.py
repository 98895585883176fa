"""Operator products w = H v and w = M v (convert.cu) at the edges of their warps, marches and
axis cases: one partial warp, several warps with an absorbing layer's edge inside one, rows
that do not divide the march, real coefficients (M with beta = 0), one coefficient shared by
all axes (M with beta > 0), a field or a constant."""
import numpy as np
import pytest

import oracle as O
from paper_1012_5379_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TG, WF = I.THETA_GAMMA, I.ECS_FRAC


@pytest.fixture(scope="module")
def helm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_5379_gb300 import build, helm as H
    build.build()
    H.load()
    return H


# One product adds at most seven terms a point: the error of a sum stays below eight roundings
# (2^-53 or 2^-24) of its largest terms; v is random, so terms do not cancel and exceed the
# result by less than a factor two (complex64 rounds v and the coefficients as well).
@pytest.mark.parametrize("prec,tol", [("c128", 1e-13), ("c64", 1e-6)])
@pytest.mark.parametrize("dim,n,tb,field", [(2, 5, 0.35, False), (2, 39, 0.0, True), (2, 319, 0.35, False),
                                            (3, 7, 0.0, False), (3, 39, 0.35, True), (3, 47, 0.0, True),
                                            (3, 63, 0.35, False)])
def test_operator_cases(helm, dim, n, tb, field, prec, tol):
    k = 0.3 * (n + 1)
    phi = (np.random.default_rng(n).uniform(0.5, 1.5, (n,) * dim) * k * k).astype(np.float32) if field else None
    L = O.build_hierarchy(dim, n, tb, TG, WF, k=None if field else k,
                          phi=phi.astype(np.float64) if field else None)[0]
    h = helm.Handle(dim, n, tb, k=None if field else k,
                    phi=torch.from_numpy(phi).cuda() if field else None, precision=prec)
    v = I.random_source(dim, n, 3)
    dt = torch.complex128 if prec == "c128" else torch.complex64
    vt = torch.from_numpy(np.ascontiguousarray(v)).to("cuda", dt)
    for which, want in (("M", L.apply(v)), ("H", L.apply_h(v))):
        wt = torch.empty_like(vt)
        h.apply_operator(vt, wt, which)
        got = wt.cpu().numpy().astype(np.complex128)
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want), which


@pytest.mark.parametrize("prec,tol", [("c128", 1e-13), ("c64", 1e-6)])
@pytest.mark.parametrize("dim,n,tb,eps", [(2, 127, 0.0, 0.5), (2, 255, 0.0, 0.1), (2, 255, 0.3, 0.5), (3, 95, 0.0, 0.5),
                                          (3, 63, 0.25, 0.3)])
def test_complex_shift(helm, dim, n, tb, eps, prec, tol):
    """M with the complex shift in its diagonal (csl_eps), at sizes where whole warps lie between
    the absorbing layers and every off-diagonal there is real (theta_beta = 0): the worst point
    too, as a term lost in part of the grid is a step at the edge of that part."""
    k = 0.3 * (n + 1)
    L = O.build_hierarchy(dim, n, tb, TG, WF, k=k, csl_eps=eps)[0]
    h = helm.Handle(dim, n, tb, k=k, precision=prec, csl_eps=eps)
    v = I.random_source(dim, n, 5)
    vt = torch.from_numpy(np.ascontiguousarray(v)).to("cuda", torch.complex128 if prec == "c128" else torch.complex64)
    for which, want in (("M", L.apply(v)), ("H", L.apply_h(v))):
        wt = torch.empty_like(vt)
        h.apply_operator(vt, wt, which)
        got = wt.cpu().numpy().astype(np.complex128)
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want), which
        assert np.max(np.abs(got - want)) <= tol * np.max(np.abs(want)), which
