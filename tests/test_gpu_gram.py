"""The complex64 V-cycle's Gram sweeps (one pass per GMRES(s) sweep) against the oracle, at
the sizes where their launch shapes can go wrong: regions of 26 own points (and 28, 30, 24
for s = 2, 1, 4) that end exactly at, just before and just after a grid's edge, the smallest
and largest levels of every launch shape, a batch mixing constant and sampled wavenumbers,
and right-hand sides whose Krylov space is nearly or exactly degenerate.

The bound is that of every complex64 V-cycle (tests/parity_check.py): 5e-5, FP32 through the
levels; the Gram sums and their factorisation carry 47 bits and add nothing to it."""
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


def vcycle(helm, dim, n, r, tb=0.3, k=None, phi=None, **kw):
    h = helm.Handle(dim, n, tb, k=k, phi=None if phi is None else torch.from_numpy(phi).cuda(), precision="c64",
                    maxit=1, **kw)
    rt = torch.from_numpy(r).cuda().to(torch.complex64)
    zt = torch.empty_like(rt)
    h.precond_apply(rt, zt)
    return zt


@pytest.mark.parametrize("dim,n,s", [(2, 23, 3), (2, 27, 3), (2, 39, 3), (2, 47, 4), (2, 55, 2), (2, 71, 1), (2, 87, 3),
                                     (2, 143, 3), (2, 223, 4), (2, 319, 3), (2, 639, 3), (2, 703, 1), (2, 895, 3), (2, 1279, 2), (3, 9, 3), (3, 11, 4),
                                     (3, 19, 3), (3, 23, 2), (3, 39, 1), (3, 47, 4), (3, 79, 3), (3, 79, 2), (3, 95, 3),
                                     (3, 95, 4), (3, 159, 3)])
def test_sizes_at_region_edges(helm, dim, n, s):
    k = 0.2 * (n + 1)
    r = I.random_source(dim, n, 500 + n)
    got = vcycle(helm, dim, n, r, k=k, s=s)
    assert_parity(got, O.vcycle(O.build_hierarchy(dim, n, 0.3, k=k), r, 1, 1, s), ("vcycle", "c64"), f"n={n} s={s}")


@pytest.mark.parametrize("dim,n", [(2, 63), (2, 255), (3, 31), (3, 127)])
def test_batch_of_field_and_constant_problems_equals_alone_bitwise(helm, dim, n):
    """Problems with and without a wavenumber field share launches."""
    k, hs, bs = 0.15 * (n + 1), [], []
    for i in range(3):
        phi = torch.from_numpy(np.full((n,) * dim, (k * (1 + 0.05 * i)) ** 2, np.float32)).cuda() if i % 2 else None
        hs.append(helm.Handle(dim, n, 0.3, k=None if i % 2 else k, phi=phi, precision="c64", restart=20))
        bs.append(torch.from_numpy(I.random_source(dim, n, 60 + i)).cuda())
    xs = [torch.zeros_like(b) for b in bs]
    helm.batch_solve(hs, bs, xs, 1e-6)
    for h, b, x in zip(hs, bs, xs):
        solo = torch.zeros_like(b)
        h.solve(b, solo, 1e-6)
        assert torch.equal(solo, x)


def test_zero_and_degenerate_right_hand_sides(helm):
    """r = 0 gives z = 0; an exact eigenvector of M (no stretching, so every sweep's Krylov space
    has dimension one) is inverted as the oracle does; NaN does not stop the next call."""
    n, k = 63, 9.0
    r = np.zeros((n, n), complex)
    assert torch.count_nonzero(vcycle(helm, 2, n, r, k=k)) == 0
    x = np.arange(1, n + 1) / (n + 1)
    e = (np.sin(5 * np.pi * x)[:, None] * np.sin(3 * np.pi * x)[None, :]).astype(complex)
    levels = O.build_hierarchy(2, n, 0.0, 0.0, k=k)
    got = vcycle(helm, 2, n, e, tb=0.0, k=k, theta_gamma=0.0)
    assert_parity(got, O.vcycle(levels, e), ("vcycle", "c64"), "eigenvector")
    h = helm.Handle(2, n, 0.3, k=k, precision="c64", maxit=1)
    good = torch.from_numpy(I.random_source(2, n, 3)).cuda().to(torch.complex64)
    z0, z1, bad = torch.empty_like(good), torch.empty_like(good), good.clone()
    h.precond_apply(good, z0)
    bad[3, 5] = float("nan")
    h.precond_apply(bad, z1)
    h.precond_apply(good, z1)
    assert torch.equal(z0, z1)


@pytest.mark.parametrize("dim,n,prec,s", [(2, 19, "c128", 3), (2, 23, "c128", 4), (2, 27, "c128", 1), (2, 39, "c128", 2),
                                          (2, 95, "c128", 3), (2, 127, "c128", 4), (2, 639, "c128", 3),
                                          (2, 767, "c128", 3), (3, 9, "c128", 4), (3, 23, "c128", 3),
                                          (2, 111, "c64", 3), (2, 767, "c64", 3)])
def test_tile_sizes_and_complex128_sweeps(helm, dim, n, prec, s):
    """Both 2D tile sizes around their border (639 and 767), levels at the border of the
    coarse kernel (23), and every sweep length of the complex128 algebra: V-cycle bounds of
    tests/parity_check.py (c128 1e-11, c64 5e-5)."""
    k = 0.2 * (n + 1)
    r = I.random_source(dim, n, 900 + n)
    h = helm.Handle(dim, n, 0.3, k=k, precision=prec, s=s, maxit=1)
    rt = torch.from_numpy(r).cuda()
    if prec == "c64":
        rt = rt.to(torch.complex64)
    zt = torch.empty_like(rt)
    h.precond_apply(rt, zt)
    assert_parity(zt, O.vcycle(O.build_hierarchy(dim, n, 0.3, k=k), r, 1, 1, s), ("vcycle", prec), f"n={n} s={s}")


def test_complex128_breakdown(helm):
    """An exact eigenvector of M: the first Arnoldi step breaks down in binary64 too."""
    n, k = 63, 9.0
    x = np.arange(1, n + 1) / (n + 1)
    e = (np.sin(5 * np.pi * x)[:, None] * np.sin(3 * np.pi * x)[None, :]).astype(complex)
    h = helm.Handle(2, n, 0.0, k=k, theta_gamma=0.0, precision="c128", maxit=1)
    rt = torch.from_numpy(e).cuda()
    zt = torch.empty_like(rt)
    h.precond_apply(rt, zt)
    assert_parity(zt, O.vcycle(O.build_hierarchy(2, n, 0.0, 0.0, k=k), e), ("vcycle", "c128"), "eigenvector")


@pytest.mark.parametrize("n,nu1,nu2,field", [(39, 1, 1, True), (47, 1, 1, False), (47, 2, 1, True), (63, 1, 1, False),
                                             (79, 1, 1, True), (79, 1, 2, False), (95, 1, 0, False), (95, 1, 1, True)])
def test_four_step_march_3d(helm, n, nu1, nu2, field):
    """The marching sweep of four steps at the edges of its 24 own columns, from b and from a
    residual, with and without the last vector kept.  Bound 2e-6: five times the 2 to 4e-7 of a
    complex64 V-cycle on white noise, a tenth of what a rim one point short costs."""
    k = 0.2 * (n + 1)
    phi = (np.random.default_rng(n).uniform(0.8, 1.2, (n,) * 3) * k * k).astype(np.float32) if field else None
    r = I.random_source(3, n, 600 + n)
    got = vcycle(helm, 3, n, r, k=None if field else k, phi=phi, s=4, nu1=nu1, nu2=nu2)
    levels = O.build_hierarchy(3, n, 0.3, k=None if field else k, phi=phi.astype(np.float64) if field else None)
    assert_parity(got, O.vcycle(levels, r, nu1, nu2, 4), 2e-6, f"n={n}")
