"""Complex64 V-cycles with wavenumber fields of strong contrast against the oracle.

On the coarse levels such a field dominates the stencil and its values form separate clusters of
the spectrum: a sweep's Krylov vectors are then nearly dependent, and a basis or Gram matrix of
binary32 quality loses digits (up to five) that an orthogonalised basis keeps.  The bound of each
case is four times the error measured with sweeps orthogonalised step by step in binary32, in the
norm and at the worst point: the scatter between two roundings of one ill-conditioned cycle."""
import numpy as np
import pytest

import oracle as O
from paper_1012_5379_gb300 import inputs as I
from parity_check import errors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# kh on the finest grid; "disc 27" dominates the finest level too
FIELDS = {"layers 3": ("layers", 0.1, 0.3), "layers 5": ("layers", 0.12, 0.6), "layers 12": ("layers", 0.05, 0.6),
          "disc 6": ("disc", 0.1, 0.6), "disc 12": ("disc", 0.05, 0.6), "core 6": ("core", 0.1, 0.6),
          "disc 27": ("disc", 0.1, 2.7)}
# dim, n, field, source, s, errors of step-by-step orthogonalisation (norm, worst point)
CASES = [
    (2, 127, "layers 3", "white", 2, 3.9e-07, 4.9e-07), (2, 127, "layers 3", "white", 3, 2.7e-07, 3.4e-07),
    (2, 127, "layers 3", "white", 4, 3.5e-07, 4.3e-07), (2, 127, "layers 5", "white", 2, 3.8e-06, 3.3e-06),
    (2, 127, "layers 5", "white", 3, 3.9e-07, 4.4e-07), (2, 127, "layers 5", "white", 4, 7.5e-07, 9.3e-07),
    (2, 127, "layers 12", "white", 2, 1.2e-05, 1.1e-05), (2, 127, "layers 12", "white", 3, 1.9e-06, 1.6e-06),
    (2, 127, "layers 12", "white", 4, 2.8e-06, 3.0e-06), (2, 127, "disc 6", "white", 2, 9.7e-06, 1.0e-05),
    (2, 127, "disc 6", "white", 3, 6.0e-07, 6.8e-07), (2, 127, "disc 6", "white", 4, 9.5e-07, 1.0e-06),
    (2, 127, "disc 12", "white", 2, 2.9e-06, 3.3e-06), (2, 127, "disc 12", "white", 3, 5.3e-07, 6.7e-07),
    (2, 127, "disc 12", "white", 4, 1.9e-06, 1.6e-06), (2, 127, "core 6", "white", 2, 4.1e-06, 4.0e-06),
    (2, 127, "core 6", "white", 3, 6.0e-07, 6.2e-07), (2, 127, "core 6", "white", 4, 5.3e-07, 7.1e-07),
    (2, 127, "layers 12", "white", 1, 1.6e-07, 2.4e-07), (2, 255, "layers 5", "white", 2, 1.3e-06, 1.0e-06),
    (2, 255, "layers 5", "white", 3, 1.1e-06, 1.3e-06), (2, 255, "layers 5", "white", 4, 5.0e-07, 5.8e-07),
    (2, 255, "layers 12", "white", 2, 5.0e-05, 4.1e-05), (2, 255, "layers 12", "white", 3, 4.4e-06, 3.2e-06),
    (2, 255, "layers 12", "white", 4, 5.8e-05, 4.8e-05), (2, 255, "disc 12", "white", 2, 8.3e-06, 7.9e-06),
    (2, 255, "disc 12", "white", 3, 4.6e-06, 3.6e-06), (2, 255, "disc 12", "white", 4, 1.3e-05, 1.2e-05),
    (2, 639, "layers 12", "white", 3, 1.1e-05, 9.9e-06), (2, 639, "disc 6", "white", 3, 4.2e-06, 4.8e-06),
    (3, 63, "layers 5", "white", 2, 1.9e-07, 2.2e-07), (3, 63, "layers 5", "white", 3, 1.7e-07, 2.1e-07),
    (3, 63, "layers 5", "white", 4, 1.8e-07, 2.2e-07), (3, 63, "disc 6", "white", 2, 1.8e-07, 3.0e-07),
    (3, 63, "disc 6", "white", 3, 1.9e-07, 2.9e-07), (3, 63, "disc 6", "white", 4, 2.2e-07, 3.0e-07),
    (3, 95, "layers 12", "white", 3, 1.8e-07, 2.4e-07), (3, 95, "disc 6", "white", 4, 6.4e-07, 9.9e-07),
    (2, 639, "disc 27", "white", 2, 3.1e-04, 3.7e-04), (2, 639, "disc 27", "white", 4, 5.6e-03, 5.7e-03),
    (3, 47, "disc 27", "white", 3, 1.8e-06, 2.3e-06), (3, 79, "disc 27", "white", 2, 6.4e-05, 1.1e-04),
    (2, 127, "layers 12", "point", 3, 1.2e-06, 3.1e-07), (2, 127, "layers 12", "point", 4, 9.9e-07, 3.3e-07),
    (2, 127, "disc 6", "point", 3, 3.8e-07, 2.2e-07), (2, 127, "disc 6", "point", 4, 8.5e-07, 3.7e-07),
    (2, 127, "disc 12", "point", 3, 1.1e-06, 5.2e-07), (2, 127, "disc 12", "point", 4, 6.5e-07, 4.0e-07),
    (2, 255, "layers 12", "point", 3, 1.9e-05, 5.4e-06), (2, 255, "layers 12", "point", 4, 9.8e-05, 2.2e-05),
    (2, 255, "disc 6", "point", 3, 4.6e-07, 1.1e-07), (2, 255, "disc 6", "point", 4, 4.9e-07, 2.2e-07),
    (2, 255, "disc 12", "point", 3, 5.2e-06, 1.4e-06), (2, 255, "disc 12", "point", 4, 1.0e-05, 2.4e-06),
    (2, 127, "layers 3", "smooth", 3, 7.9e-06, 9.7e-06), (2, 127, "layers 3", "smooth", 4, 8.5e-06, 8.4e-06),
    (2, 127, "core 6", "smooth", 3, 7.4e-07, 1.0e-06), (3, 63, "layers 3", "point", 3, 1.1e-07, 3.9e-08),
    (3, 63, "disc 6", "point", 3, 2.4e-07, 3.2e-08),
]


@pytest.fixture(scope="module")
def helm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1012_5379_gb300 import build, helm as H
    build.build()
    H.load()
    return H


def field(name, dim, n):
    kind, lo, hi = FIELDS[name]
    x = np.arange(1, n + 1) / (n + 1)
    g = np.meshgrid(*([x] * dim), indexing="ij")
    r2 = sum((a - 0.5) ** 2 for a in g)
    kh = {"layers": np.where(np.floor(5 * g[0]).astype(int) % 2 == 0, lo, hi), "disc": np.where(r2 < 0.09, lo, hi),
          "core": np.where(r2 < 0.02, hi, lo)}[kind]
    return ((kh * (n + 1)) ** 2).astype(np.float32)


def source(kind, dim, n):
    if kind == "white":
        r = I.random_source(dim, n, 800 + n)
    elif kind == "point":
        r = np.zeros((n,) * dim, complex)
        r[(n // 2,) * dim] = 1.0
    else:
        x = np.arange(1, n + 1) / (n + 1)
        r = np.sin(3 * np.pi * x)
        for _ in range(dim - 1):
            r = r[..., None] * np.sin(2 * np.pi * x)
    return r.astype(np.complex64)


@pytest.mark.parametrize("dim,n,name,src,s,e_norm,e_point", CASES)
def test_contrast(helm, dim, n, name, src, s, e_norm, e_point):
    phi, r = field(name, dim, n), source(src, dim, n)
    h = helm.Handle(dim, n, 0.3, phi=torch.from_numpy(phi).cuda(), precision="c64", s=s, maxit=1)
    rt = torch.from_numpy(r).cuda()
    z = torch.empty_like(rt)
    h.precond_apply(rt, z)
    want = O.vcycle(O.build_hierarchy(dim, n, 0.3, phi=phi.astype(np.float64)), r.astype(complex), 1, 1, s)
    got_norm, got_point = errors(z, want)
    assert got_norm <= 4 * e_norm and got_point <= 4 * e_point, (got_norm, got_point)


@pytest.mark.parametrize("dim,n,s", [(2, 255, 3), (2, 639, 3), (2, 639, 4), (3, 31, 2), (3, 47, 3), (3, 79, 3)])
def test_batch_of_wide_and_ordinary_levels_equals_alone_bitwise(helm, dim, n, s):
    """Levels a field dominates take kernels of their own, beside those of the batch's others."""
    hs, bs = [], []
    for i, name in enumerate(("disc 27", None, "disc 6", "layers 3", "disc 27")):
        kw = {"k": 0.2 * (n + 1)} if name is None else {"phi": torch.from_numpy(field(name, dim, n)).cuda()}
        hs.append(helm.Handle(dim, n, 0.3, precision="c64", s=s, restart=4, maxit=5, **kw))
        bs.append(torch.from_numpy(I.random_source(dim, n, 40 + i)).cuda())
    xs = [torch.zeros_like(b) for b in bs]
    helm.batch_solve(hs, bs, xs, 1e-9)
    for h, b, x in zip(hs, bs, xs):
        solo = torch.zeros_like(b)
        h.solve(b, solo, 1e-9)
        assert torch.equal(solo, x) and torch.isfinite(torch.view_as_real(x)).all()


@pytest.mark.parametrize("dim,n,kh,s,width,e_norm", [(2, 127, 0.16, 3, 0.07, 6.9e-4), (2, 127, 0.16, 4, 0.07, 2.4e-3),
                                                     (2, 127, 0.16, 4, 0.025, 7.8e-7), (2, 255, 0.16, 4, 0.025, 7.8e-4),
                                                     (2, 255, 0.3, 4, 0.07, 3.5e-5), (3, 127, 0.16, 3, 0.07, 3.7e-3),
                                                     (3, 127, 0.16, 4, 0.07, 1.4e-3)])
def test_smooth_source(helm, dim, n, kh, s, width, e_norm):
    """Gaussian sources: M k_0 and M^2 k_0 are small beside the diagonal, and a shifted basis of
    them nearly dependent.  Against the complex128 V-cycle (which other tests hold to the oracle
    at 1e-11); the bound as above, four times the step-by-step error."""
    x = np.arange(1, n + 1) / (n + 1)
    q = np.exp(-((x - 0.4) / width) ** 2)
    r = q
    for _ in range(dim - 1):
        r = r[..., None] * q
    z = {}
    for prec, dt in (("c64", torch.complex64), ("c128", torch.complex128)):
        h = helm.Handle(dim, n, 0.3, k=kh * (n + 1), precision=prec, s=s, maxit=1)
        rt = torch.from_numpy(r.astype(np.complex64)).cuda().to(dt)
        z[prec] = torch.empty_like(rt)
        h.precond_apply(rt, z[prec])
    assert errors(z["c64"], z["c128"])[0] <= 4 * e_norm


@pytest.mark.parametrize("n,kh,e_norm", [(127, 0.16, 3.0e-7), (127, 0.3, 2.6e-7)])
def test_point_source_of_four_steps_3d(helm, n, kh, e_norm):
    """s = 4 on a marching level, where a few planes hold all of a vector: against the complex128
    V-cycle, four times the step-by-step error."""
    z = {}
    for prec, dt in (("c64", torch.complex64), ("c128", torch.complex128)):
        h = helm.Handle(3, n, 0.3, k=kh * (n + 1), precision=prec, s=4, maxit=1)
        r = torch.zeros((n,) * 3, dtype=dt, device="cuda")
        r[(n // 2,) * 3] = 1.0
        z[prec] = torch.empty_like(r)
        h.precond_apply(r, z[prec])
    assert errors(z["c64"], z["c128"])[0] <= 4 * e_norm
