"""The coarsest solve of a nearly singular operator (a Dirichlet grid with k^2 next to an
eigenvalue, without layers or stretching) against exact rational elimination.  A handle whose
only level is the coarsest applies nothing else."""
from fractions import Fraction

import numpy as np
import pytest

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


def exact_solve(A, b):
    """A x = b for real A and complex b, in rational arithmetic."""
    m = len(b)
    M = [[Fraction(float(v)) for v in row] + [Fraction(float(b[i].real)), Fraction(float(b[i].imag))]
         for i, row in enumerate(A)]
    for k in range(m):
        p = next(i for i in range(k, m) if M[i][k] != 0)
        M[k], M[p] = M[p], M[k]
        for i in range(k + 1, m):
            f = M[i][k] / M[k][k]
            if f:
                M[i] = [x - f * y for x, y in zip(M[i], M[k])]
    x = [None] * m
    for k in range(m - 1, -1, -1):
        x[k] = [(M[k][m + c] - sum(M[k][q] * x[q][c] for q in range(k + 1, m))) / M[k][k] for c in (0, 1)]
    return np.array([float(re) + 1j * float(im) for re, im in x])


# The inverse's entries are correct to a rounding and a row adds at most 27 products: an error of
# 30 roundings (binary64) of |A^-1| |b|, which a random b's solution reaches within a factor of
# ten; complex64 rounds the solution.
@pytest.mark.parametrize("prec,tol", [("c128", 3e-14), ("c64", 2e-7)])
@pytest.mark.parametrize("dim,n,delta", [(2, 3, 1e-3), (2, 3, 1e-8), (2, 3, 1e-11), (2, 4, 1e-9), (3, 3, 1e-3), (3, 3, 1e-10)])
def test_nearly_singular_coarsest(helm, dim, n, delta, prec, tol):
    a, d, c = [v.real for v in helm.axis_coefficients(n, 0.125, 0.0, 0.0)]
    mu = np.sort(np.linalg.eigvals(np.diag(d) + np.diag(a[1:], -1) + np.diag(c[:-1], 1)).real)
    k = np.sqrt((mu[0] + (dim - 1) * mu[1]) * (1 + delta))
    m = n ** dim
    A = np.zeros((m, m))
    for r in range(m):
        x, y, z = r % n, r // n % n, r // (n * n)
        diag = d[x] + d[y]
        if dim == 3:
            diag = diag + d[z]
        A[r, r] = diag - k * k
        for i, st in ((x, 1), (y, n), (z, n * n))[:dim]:
            if i > 0:
                A[r, r - st] = a[i]
            if i < n - 1:
                A[r, r + st] = c[i]
    g = np.random.default_rng(3)
    b = (g.standard_normal(m) + 1j * g.standard_normal(m)).astype(np.complex64)
    want = exact_solve(A, b)
    h = helm.Handle(dim, n, 0.0, k=float(k), theta_gamma=0.0, precision=prec, maxit=1)
    assert h.levels() == [n]
    rt = torch.from_numpy(b.reshape((n,) * dim)).cuda().to(torch.complex128 if prec == "c128" else torch.complex64)
    zt = torch.empty_like(rt)
    h.precond_apply(rt, zt)
    got = zt.cpu().numpy().astype(np.complex128).ravel()
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
