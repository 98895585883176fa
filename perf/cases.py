"""What a user of the solver has it do, as measurable cases.

A user builds a ``helm.Handle`` once (grid, wavenumber, angles, hierarchy, workspace)
and then calls it with one right-hand side after another:

  * ``precond_apply``: one V(nu1, nu2) cycle as the preconditioner of the user's own Krylov
    method, in complex64 or complex128, with the GMRES(s) or the polynomial smoother;
  * ``solve`` / ``solve_host`` / ``batch_solve``: whole FGMRES solves of one or several
    problems, from device or host arrays;
  * ``apply_operator``: H v or M v (residuals, the user's own Krylov method).

Sizes, wavenumbers (kh in 0.1 .. 0.31), angles and layers are those of
``paper_1012_5379_gb300/inputs.py``, of the tests and of ``bench.py``.  Handles are part of
the state (a user keeps them); right-hand sides and fields come from the seed.
"""
import math

import numpy as np
import torch

from paper_1012_5379_gb300 import helm

THETA_GAMMA = 0.5     # layer angle of the constant-k and bump-field workloads
ECS_FRAC = 0.125      # layer width of those workloads
GAUSS_DOMAIN = 50.0   # physical box of the Gaussian model
GAUSS_BETA = math.radians(10.3132)
GAUSS_GAMMA = math.pi / 6
DTYPE = {"c64": torch.complex64, "c128": torch.complex128}


def _vcycle(name, dim, n, prec, medium="const", kh=0.16, beta=0.3, nu1=1, nu2=1, s=3, smoother="gmres"):
    return {"name": name, "call": "vcycle", "dim": dim, "n": n, "prec": prec, "medium": medium, "kh": kh,
            "beta": beta, "nu1": nu1, "nu2": nu2, "s": s, "smoother": smoother}


def _solve(name, call, dim, n, prec, medium="const", kh=0.16, beta=0.3, restart=0, maxit=400, tol=1e-8, count=1):
    return {"name": name, "call": call, "dim": dim, "n": n, "prec": prec, "medium": medium, "kh": kh,
            "beta": beta, "restart": restart, "maxit": maxit, "tol": tol, "count": count}


def listed():
    return [
        # the smallest preconditioner call: the 127^2 grid of the served requests, every level
        # in cache and each pass a few microseconds, so launches and latency are all of it
        _vcycle("vcycle 2D 127 c64", 2, 127, "c64"),
        # the 64^2 column of the Gaussian model: a grid whose pitch is no power of two, one-sided
        # layers, a wavenumber field, in complex128 (the automatic precision of small grids)
        _vcycle("vcycle 2D 79 c128 gauss", 2, 79, "c128", medium="gauss", kh=0.31, beta=GAUSS_BETA),
        # the ordinary 2D call: the grid of the theta_beta sweep
        _vcycle("vcycle 2D 1023 c64", 2, 1023, "c64"),
        # the 512^2 column of the Gaussian model: a ragged 639^2 grid with a wavenumber field
        _vcycle("vcycle 2D 639 c64 gauss", 2, 639, "c64", medium="gauss", kh=0.34, beta=GAUSS_BETA),
        # a large 2D grid, streaming from HBM
        _vcycle("vcycle 2D 4095 c64", 2, 4095, "c64"),
        # the polynomial smoother (Sec. 4) on the ordinary 2D grid
        _vcycle("vcycle 2D 1023 c64 poly", 2, 1023, "c64", kh=0.1, beta=0.4, smoother="poly"),
        # the ordinary 3D call (a served shape), constant wavenumber
        _vcycle("vcycle 3D 127 c64", 3, 127, "c64"),
        # the benchmark's preconditioner: 255^3 with the heterogeneous wavenumber field
        _vcycle("vcycle 3D 255 c64 bumps", 3, 255, "c64", medium="bumps", kh=0.3125, beta=0.4),
        # the operator on the benchmark's grid, for a user's own residual
        {"name": "operator H 3D 255 c128", "call": "operator", "dim": 3, "n": 255, "prec": "c128",
         "medium": "bumps", "kh": 0.3125, "beta": 0.4, "which": "H"},
        # a whole small solve from host arrays: 127^2, k = 20, complex128, 1e-8
        _solve("solve_host 2D 127 c128", "solve_host", 2, 127, "c128", kh=20.0 / 128, beta=0.4),
        # eight independent 2D problems solved together ({255, 511, 1023}^2, restart 40)
        _solve("batch 2D 8 problems c64", "batch", 2, 1023, "c64", restart=40, count=8),
        # the benchmark's solve: 255^3, heterogeneous field, FGMRES(40)
        _solve("solve 3D 255 c64 bumps", "solve", 3, 255, "c64", medium="bumps", kh=0.3125, beta=0.4, restart=40),
    ]


def _grid(rng, lo, hi, odd, dim=2):
    """A size whose grid coarsens: n + 1 = q 2^j in [lo + 1, hi + 1], log-uniform; q = 4 (a
    power of two) or, for ragged grids, 5, 6 or (2D) 7."""
    want = math.exp(rng.uniform(math.log(lo + 1), math.log(hi + 1)))
    best = None
    for q in ((5, 6, 7)[: 5 - dim] if odd else (4,)):
        p = q
        while p <= hi + 1:
            if p >= lo + 1 and (best is None or abs(math.log(p / want)) < abs(math.log(best / want))):
                best = p
            p *= 2
    return best - 1


def draw(rng):
    kind = rng.choices(["vc2", "vc2s", "vc3", "poly", "op", "solve2", "solve3", "batch"],
                       [3, 2, 3, 1, 1, 1, 1, 1])[0]
    kh = round(rng.uniform(0.1, 0.3), 4)
    beta = round(rng.uniform(0.2, 0.4), 3)
    odd = rng.random() < 0.4
    if kind == "vc2":
        n = _grid(rng, 127, 4095, odd)
        nu1, nu2, s = rng.choice([(1, 1, 3), (1, 1, 3), (1, 0, 3), (2, 1, 2)])
        c = _vcycle("", 2, n, "c64", medium=rng.choice(["const", "const", "gauss"]), kh=kh, beta=beta, nu1=nu1,
                    nu2=nu2, s=s)
    elif kind == "vc2s":
        c = _vcycle("", 2, _grid(rng, 63, 255, odd), "c128", kh=kh, beta=beta)
    elif kind == "vc3":
        n = _grid(rng, 31, 255, odd, 3)
        c = _vcycle("", 3, n, "c64", medium=rng.choice(["const", "bumps"]), kh=kh, beta=beta)
    elif kind == "poly":
        c = _vcycle("", 2, _grid(rng, 127, 2047, False), "c64", kh=round(rng.uniform(0.08, 0.12), 4), beta=0.4,
                    smoother="poly")
    elif kind == "op":
        dim = rng.choice([2, 3])
        c = {"call": "operator", "dim": dim, "n": _grid(rng, 127, 2047 if dim == 2 else 255, odd, dim),
             "prec": rng.choice(["c64", "c128"]), "medium": rng.choice(["const", "bumps"]) if dim == 3 else "const",
             "kh": kh, "beta": beta, "which": rng.choice(["H", "M"])}
    elif kind == "solve2":
        c = _solve("", rng.choice(["solve", "solve_host"]), 2, _grid(rng, 63, 127, odd), "c128", kh=kh, beta=beta)
    elif kind == "solve3":
        c = _solve("", "solve", 3, _grid(rng, 63, 191, odd, 3), "c64", kh=kh, beta=beta, restart=40)
    else:
        c = _solve("", "batch", 2, rng.choice([255, 511, 1023]), "c64", kh=kh, beta=0.3, restart=40,
                   count=rng.randint(2, 8))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)


def _complex_normal(shape, prec, g):
    """Unit-variance complex normal right-hand side, layers included."""
    return torch.randn(shape, dtype=DTYPE[prec], device="cuda", generator=g)


def _bumps(dim, n, k0, seed):
    """k(x)^2 with k = k0 (1 + 0.3 g), g a clipped sum of eight Gaussian bumps (float32)."""
    r = np.random.default_rng(seed)
    x = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") / (n + 1)
    f = torch.zeros((n,) * dim, dtype=torch.float64, device="cuda")
    for _ in range(8):
        c, a = r.uniform(0.0, 1.0, dim), r.uniform(-1.0, 1.0)
        t = torch.full((), float(a), dtype=torch.float64, device="cuda")
        for ax in range(dim):
            e = torch.exp(-((x - float(c[ax])) ** 2) / (2 * 0.1 ** 2))
            t = t[..., None] * e
        f += t
    k = k0 * (1.0 + 0.3 * f.clamp_(-1.0, 1.0))
    return (k * k).to(torch.float32).contiguous()


def _gauss(n, kh):
    """The Gaussian model's field on the unit box: Lam^2 (nu (e^{-x^2} + e^{-y^2}) + k^2) on a box of
    length Lam = 62.5 whose far fifth is the layer, nu = 7 (float32)."""
    lam = 1.25 * GAUSS_DOMAIN
    x = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") * (lam / (n + 1))
    e = torch.exp(-x * x)
    k = kh * (n + 1) / lam
    return (lam * lam * (7.0 * (e[None, :] + e[:, None]) + k * k)).to(torch.float32).contiguous()


def _geometry(case):
    """theta_gamma, layer width and layer sides of a case's grid."""
    if case["medium"] == "gauss":
        return GAUSS_GAMMA, 0.2, "high"
    return THETA_GAMMA, ECS_FRAC, "both"


def _medium(case, seed):
    dim, n, kh = case["dim"], case["n"], case["kh"]
    if case["medium"] == "bumps":
        return None, _bumps(dim, n, kh * (n + 1), seed)
    if case["medium"] == "gauss":
        return None, _gauss(n, kh)
    return kh * (n + 1), None


def _handle(case, n, k, phi, **kw):
    gamma, frac, sides = _geometry(case)
    return helm.Handle(case["dim"], n, case["beta"], k=k, phi=phi, theta_gamma=gamma, ecs_frac=frac,
                       ecs_sides=sides, precision=case["prec"], **kw)


def _members(case):
    """Sizes and wavenumbers of a batch: up to the case's n, mixed as the batched workload is."""
    sizes = [n for n in (255, 511, 1023) if n <= case["n"]]
    r = np.random.default_rng(case["count"] * 1009 + round(case["kh"] * 1e4))  # the mix belongs to the case
    out = []
    for i in range(case["count"]):
        n = sizes[(len(sizes) - 1 + i) % len(sizes)]
        out.append((n, float(r.uniform(0.1, 0.3)) * (n + 1)))
    return out


def prepare(case, seed):
    g, call, dim, n = _gen(seed), case["call"], case["dim"], case["n"]
    shape = (n,) * dim
    if call == "vcycle":
        k, phi = _medium(case, seed)
        h = _handle(case, n, k, phi, nu1=case["nu1"], nu2=case["nu2"], s=case["s"], smoother=case["smoother"],
                    restart=1, maxit=1)
        r = _complex_normal(shape, case["prec"], g)
        return {"call": call, "h": h, "r": r, "z": torch.empty_like(r), "phi": phi}
    if call == "operator":
        k, phi = _medium(case, seed)
        h = _handle(case, n, k, phi, restart=1, maxit=1)
        v = _complex_normal(shape, case["prec"], g)
        return {"call": call, "h": h, "v": v, "w": torch.empty_like(v), "which": case["which"], "phi": phi}
    kw = {"restart": case["restart"], "maxit": case["maxit"]}
    if call == "batch":
        hs, bs = [], []
        for (m, k) in _members(case):
            hs.append(_handle(case, m, k, None, **kw))
            bs.append(_complex_normal((m, m), "c128", g))
        return {"call": call, "hs": hs, "bs": bs, "xs": [torch.zeros_like(b) for b in bs], "tol": case["tol"]}
    k, phi = _medium(case, seed)
    h = _handle(case, n, k, phi, **kw)
    b = _complex_normal(shape, "c128", g)
    if call == "solve_host":
        hb = torch.empty(shape, dtype=torch.complex128, pin_memory=True)
        hb.copy_(b)
        return {"call": call, "h": h, "b": hb, "x": torch.empty_like(hb, pin_memory=True), "tol": case["tol"]}
    return {"call": call, "h": h, "b": b, "x": torch.zeros_like(b), "tol": case["tol"], "phi": phi}


def run(state):
    call = state["call"]
    if call == "vcycle":
        return state["h"].precond_apply(state["r"], state["z"])
    if call == "operator":
        return state["h"].apply_operator(state["v"], state["w"], state["which"])
    if call == "solve_host":
        state["h"].solve_host(state["b"], state["x"], state["tol"])
        return state["x"]
    if call == "batch":
        for x in state["xs"]:
            x.zero_()
        helm.batch_solve(state["hs"], state["bs"], state["xs"], state["tol"])
        return list(state["xs"])
    state["x"].zero_()
    state["h"].solve(state["b"], state["x"], state["tol"])
    return state["x"]


def work(case):
    """The call's inputs read once and its outputs written once.  Operations: one operator
    application costs 8 (2 dim + 1) per point, a GMRES(s) sweep s applications and about 16 s (s + 3)
    / 2 in inner products and updates; a cycle 1 / (1 - 2^-dim) times its finest level.  A solve is
    counted with one cycle, one H application and its residual only (the number of iterations is not
    known beforehand)."""
    dim = case["dim"]
    if case["call"] == "batch":
        pts = float(sum(m ** dim for m, _ in _members(case)))
    else:
        pts = float(case["n"] ** dim)
    op = 8.0 * (2 * dim + 1)
    elem = 8.0 if case["prec"] == "c64" else 16.0
    field = 4.0 if case["medium"] != "const" else 0.0
    if case["call"] == "operator":
        return {"bytes": pts * (2 * elem + field), "flops": pts * op}
    nu1, nu2, s = case.get("nu1", 1), case.get("nu2", 1), case.get("s", 3)
    cycle = ((nu1 + nu2) * (s * op + 8.0 * s * (s + 3)) + 2 * op + 16.0) / (1.0 - 0.5 ** dim)
    if case["call"] == "vcycle":
        return {"bytes": pts * (2 * elem + field), "flops": pts * cycle}
    return {"bytes": pts * (32.0 + field), "flops": pts * (cycle + 2 * op)}


# ------------------------------------------------------------------------------ 64 bits
# The same calls in plain complex128 torch: complex-stretched spacings, the three-point
# scheme, full weighting and (bi/tri)linear interpolation, GMRES(s) smoothing, FGMRES(40).
def _spacings(n, gamma, frac, sides, beta):
    h = 1.0 / (n + 1)

    def z(x):
        lo = min(x, frac) if sides == "both" else 0.0
        hi = max(0.0, x - (1.0 - frac))
        return (lo + hi) * np.exp(1j * gamma) + (x - lo - hi) * np.exp(1j * beta)

    return np.diff(np.array([z(i * h) for i in range(n + 2)]))


def _coefs(n, gamma, frac, sides, beta):
    sp = _spacings(n, gamma, frac, sides, beta)
    l, r = sp[:-1], sp[1:]
    return [torch.from_numpy(v).cuda() for v in (-2.0 / ((l + r) * l), 2.0 / (l * r), -2.0 / ((l + r) * r))]


class _Level:
    def __init__(self, dim, n, coef, phi):
        self.dim, self.n, self.phi = dim, n, phi
        self.a, self.d, self.c = coef

    def apply(self, u):
        out = -self.phi * u
        for ax in range(self.dim):
            sh = [1] * self.dim
            sh[ax] = -1
            m = self.n - 1
            out += self.d.view(sh) * u
            out.narrow(ax, 1, m).add_(self.a[1:].view(sh) * u.narrow(ax, 0, m))
            out.narrow(ax, 0, m).add_(self.c[:m].view(sh) * u.narrow(ax, 1, m))
        return out


def _levels(dim, n, gamma, frac, sides, beta, phi):
    out = []
    while True:
        out.append(_Level(dim, n, _coefs(n, gamma, frac, sides, beta), phi))
        if n <= 3 or (n + 1) % 2:
            return out
        n = (n + 1) // 2 - 1
        if torch.is_tensor(phi):
            phi = phi[(slice(1, None, 2),) * dim].contiguous()


def _dense_solve(lev, b):
    m = lev.n ** lev.dim
    eye = torch.eye(m, dtype=torch.complex128, device="cuda")
    mat = torch.stack([lev.apply(e.view((lev.n,) * lev.dim)).reshape(-1) for e in eye], 1)
    return torch.linalg.solve(mat, b.reshape(-1)).view(b.shape)


def _restrict(r):
    for ax in range(r.dim()):
        m = (r.shape[ax] + 1) // 2 - 1
        at = [r.narrow(ax, o, 2 * m - 1)[(slice(None),) * ax + (slice(None, None, 2),)] for o in (0, 1, 2)]
        r = 0.25 * at[0] + 0.5 * at[1] + 0.25 * at[2]
    return r


def _prolong(e, n):
    for ax in range(e.dim()):
        shape = list(e.shape)
        shape[ax] = n
        out = torch.zeros(shape, dtype=e.dtype, device=e.device)
        m = e.shape[ax]
        pre = (slice(None),) * ax
        out[pre + (slice(1, 2 * m, 2),)] = e
        out[pre + (slice(0, 2 * m - 1, 2),)] += 0.5 * e
        out[pre + (slice(2, 2 * m + 1, 2),)] += 0.5 * e
        e = out
    return e


def _gmres_sweep(lev, b, x, s):
    r = b if x is None else b - lev.apply(x)
    beta = float(torch.linalg.vector_norm(r))
    if beta == 0.0:
        return torch.zeros_like(b) if x is None else x
    basis, hess, m = [r / beta], np.zeros((s + 1, s), complex), s
    for j in range(s):
        w = lev.apply(basis[j])
        for i in range(j + 1):
            hess[i, j] = complex(torch.vdot(basis[i].reshape(-1), w.reshape(-1)))
            w = w - hess[i, j] * basis[i]
        hess[j + 1, j] = float(torch.linalg.vector_norm(w))
        if abs(hess[j + 1, j]) <= 1e-14 * beta:
            m = j + 1
            break
        basis.append(w / hess[j + 1, j])
    rhs = np.zeros(m + 1, complex)
    rhs[0] = beta
    y = np.linalg.lstsq(hess[: m + 1, :m], rhs, rcond=None)[0]
    out = torch.zeros_like(b) if x is None else x.clone()
    for j in range(m):
        out += complex(y[j]) * basis[j]
    return out


def _cycle(levels, b, nu1, nu2, s, l=0):
    lev = levels[l]
    if l == len(levels) - 1:
        return _dense_solve(lev, b)
    x = None
    for _ in range(nu1):
        x = _gmres_sweep(lev, b, x, s)
    r = b if x is None else b - lev.apply(x)
    e = _prolong(_cycle(levels, _restrict(r), nu1, nu2, s, l + 1), lev.n)
    x = e if x is None else x + e
    for _ in range(nu2):
        x = _gmres_sweep(lev, b, x, s)
    return x


def _fgmres(hop, levels, b, tol):
    x, r, bn = torch.zeros_like(b), b.clone(), float(torch.linalg.vector_norm(b))
    for _ in range(12):
        beta = float(torch.linalg.vector_norm(r))
        if beta <= tol * bn:
            break
        v, z, hess = [r / beta], [], np.zeros((41, 40), complex)
        for j in range(40):
            z.append(_cycle(levels, v[j], 1, 1, 3))
            w = hop.apply(z[j])
            for i in range(j + 1):
                hess[i, j] = complex(torch.vdot(v[i].reshape(-1), w.reshape(-1)))
                w = w - hess[i, j] * v[i]
            hess[j + 1, j] = float(torch.linalg.vector_norm(w))
            v.append(w / hess[j + 1, j])
            rhs = np.zeros(j + 2, complex)
            rhs[0] = beta
            y = np.linalg.lstsq(hess[: j + 2, : j + 1], rhs, rcond=None)[0]
            if np.linalg.norm(rhs - hess[: j + 2, : j + 1] @ y) <= 0.3 * tol * bn:
                break
        for yi, zi in zip(y, z):
            x += complex(yi) * zi
        r = b - hop.apply(x)
    return x


def exact(case, seed):
    g, call, dim, n = _gen(seed), case["call"], case["dim"], case["n"]
    gamma, frac, sides = _geometry(case)
    if case.get("smoother") == "poly":
        return None  # its weights follow from a choice (Sec. 4) that is the library's own
    if call in ("vcycle", "operator"):
        k, phi = _medium(case, seed)
        f = k * k if phi is None else phi.double()
        v = _complex_normal((n,) * dim, case["prec"], g).to(torch.complex128)
        if call == "operator":
            beta = 0.0 if case["which"] == "H" else case["beta"]
            return _Level(dim, n, _coefs(n, gamma, frac, sides, beta), f).apply(v)
        levels = _levels(dim, n, gamma, frac, sides, case["beta"], f)
        return _cycle(levels, v, case["nu1"], case["nu2"], case["s"])
    if call == "batch" or n ** dim > 300000:
        return None  # the solution itself, converged in 64 bits, would take too long
    k, phi = _medium(case, seed)
    f = k * k if phi is None else phi.double()
    b = _complex_normal((n,) * dim, "c128", g)
    hop = _Level(dim, n, _coefs(n, gamma, frac, sides, 0.0), f)
    x = _fgmres(hop, _levels(dim, n, gamma, frac, sides, case["beta"], f), b, 1e-12)
    return x.cpu() if call == "solve_host" else x
