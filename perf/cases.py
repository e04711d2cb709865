"""Workloads of the RS-S library as a user's program calls it, for timing and for checking results.

Two kinds of pass.  A "step" builds a factorization and solves with it (``rss_factor`` then
``rss_solve``, or ``rss_solve_iterative`` for the paper's scattering problem): what a program does for
each new operator.  A "solve" applies a factorization that the program holds to new right-hand sides:
what a serving loop does for each request or panel.  Points are the cell centres of a uniform
side x side grid, side = sqrt(leaf) 2^m, and the diagonal is 1 as in the repository's workloads
(Lippmann-Schwinger: the paper's self-cell quadrature).  Right-hand sides are N(0, 1).
"""
import math

import numpy as np
import torch

import paper_2310_15458_gb300 as P

KIND = {"laplace": P.LAPLACE, "helmholtz": P.HELMHOLTZ, "lippmann_schwinger": P.HELMHOLTZ_LS}


def _case(name, pass_, kernel, side, leaf, eps, kappa, nrhs, shuffle=False):
    return {"name": name, "pass": pass_, "kernel": kernel, "side": side, "leaf": leaf, "eps": eps,
            "kappa": kappa, "nrhs": nrhs, "shuffle": shuffle}


def listed():
    return [
        # the smallest named workload: few boxes, every launch and every serial chain counts
        _case("step_laplace_64", "step", "laplace", 64, 64, 1e-8, 0.0, 1),
        # an ordinary problem, too small to fill the chip at any level but the finest
        _case("step_laplace_256", "step", "laplace", 256, 64, 1e-6, 0.0, 1),
        # leaf boxes of 7 x 7 points in no particular order: sizes off every tile boundary
        _case("step_laplace_448_leaf49", "step", "laplace", 448, 49, 1e-7, 0.0, 3, True),
        # the benchmark's workload, a million unknowns
        _case("step_laplace_1024", "step", "laplace", 1024, 64, 1e-6, 0.0, 1),
        # complex, several right-hand sides at once
        _case("step_helmholtz_256", "step", "helmholtz", 256, 64, 1e-6, 25.0, 16),
        # the paper's scattering problem: factor, then GMRES to 1e-12 with the factor as preconditioner
        _case("refine_lippmann_512", "refine", "lippmann_schwinger", 512, 64, 1e-6, 25.0, 1),
        # the smallest call: one right-hand side on a small resident factor
        _case("solve_laplace_64", "solve", "laplace", 64, 64, 1e-8, 0.0, 1),
        # one right-hand side on the largest resident factor
        _case("solve_laplace_1024", "solve", "laplace", 1024, 64, 1e-6, 0.0, 1),
        # a request of the serving mix
        _case("solve_laplace_256_rhs16", "solve", "laplace", 256, 64, 1e-6, 0.0, 16),
        # a full panel of the serving mix, real and complex
        _case("solve_laplace_512_rhs64", "solve", "laplace", 512, 64, 1e-6, 0.0, 64),
        _case("solve_helmholtz_256", "solve", "helmholtz", 256, 64, 1e-6, 25.0, 1),
        _case("solve_helmholtz_256_rhs64", "solve", "helmholtz", 256, 64, 1e-6, 25.0, 64),
    ]


def draw(rng):
    """A pass, a kernel, a leaf of 4 x 4 to 10 x 10 points, a grid, a tolerance and a number of columns."""
    pass_ = rng.choice(["step", "solve"])
    kernel = rng.choice(["laplace", "laplace", "helmholtz", "lippmann_schwinger"])
    if kernel == "lippmann_schwinger" and pass_ == "step":
        pass_ = "refine"
    ls = rng.choice([4, 5, 6, 7, 8, 8, 9, 10])
    most = 900 if kernel == "laplace" else 320   # no more work than the largest listed case
    grids = [ls << m for m in range(3, 9) if 48 <= ls << m <= most]
    side = rng.choice(grids)
    eps = 10.0 ** rng.uniform(-9.0 if kernel == "laplace" else -7.0, -4.0)
    kappa = 0.0 if kernel == "laplace" else rng.uniform(8.0, 50.0 if kernel == "helmholtz" else 30.0)
    nrhs = 1 if pass_ == "refine" else int(round(math.exp(rng.uniform(0.0, math.log(64.0)))))
    c = _case("", pass_, kernel, side, ls * ls, eps, kappa, nrhs, rng.random() < 0.3)
    del c["name"]
    return c


def _points(case, seed):
    s = case["side"]
    g = (np.arange(s) + 0.5) / s
    pts = np.empty((s, s, 2))
    pts[:, :, 0] = g[None, :]
    pts[:, :, 1] = g[:, None]
    pts = pts.reshape(-1, 2)
    if case["shuffle"]:
        pts = pts[np.random.default_rng(seed).permutation(s * s)]
    return pts


def _rhs(case, seed):
    n, k = case["side"] ** 2, case["nrhs"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float64 if case["kernel"] == "laplace" else torch.complex128
    if dt == torch.complex128:
        b = torch.view_as_complex(torch.randn(k, n, 2, generator=g, device="cuda", dtype=torch.float64))
    else:
        b = torch.randn(k, n, generator=g, device="cuda", dtype=dt)
    return b[0] if case["pass"] == "refine" else b.T   # column-major n x nrhs


def _factor(case, tree):
    ls = case["kernel"] == "lippmann_schwinger"
    return P.rss_factor(tree, kind=KIND[case["kernel"]], eps=case["eps"], h=1.0 / case["side"],
                        kappa=case["kappa"], diag_rule=1 if ls else 0,
                        proxy_radius_over_side=2.5 if ls else 1.25)


def prepare(case, seed):
    state = {"case": case, "tree": P.rss_build_tree(_points(case, seed), case["leaf"]), "b": _rhs(case, seed)}
    if case["pass"] == "solve":
        state["factor"] = _factor(case, state["tree"])
    return state


def run(state):
    case = state["case"]
    f = state["factor"] if case["pass"] == "solve" else _factor(case, state["tree"])
    if case["pass"] == "refine":
        return P.rss_solve_iterative(f, state["b"], tol=1e-12)[0]
    return P.rss_solve(f, state["b"].clone())   # the solve overwrites its argument; the program keeps b


def work(case):
    """One pass's unavoidable work.  Per grid point a real factorization at eps = 1e-6 holds about 900
    entries, about in proportion to the digits asked for; a solve reads each once (16 bytes complex) and
    does a multiply-add with it per column; a factorization takes about 3.6e5 operations per point
    (compression, elimination and Schur updates; complex products count four times) and writes them."""
    n, k = case["side"] ** 2, case["nrhs"]
    cplx = case["kernel"] != "laplace"
    size, ops = (16, 4) if cplx else (8, 1)
    digits = -math.log10(case["eps"]) / 6.0
    entries = 900.0 * digits * n
    flops = 2.0 * ops * entries * k
    if case["pass"] != "solve":
        flops += 3.6e5 * ops * digits * n
    return {"bytes": size * (entries + 2.0 * n * k), "flops": flops}


# ------------------------------------------------------------------ A^{-1} b in plain torch, 64 bits

EULER = 0.5772156649015329


def _j0_y0(z):
    """J0 and Y0 to rounding: power series below 5, above it Miller's backward recurrence with Neumann's
    series for Y0 (arguments up to about 75)."""
    small = z < 5.0
    a, q = torch.where(small, z, 1.0), torch.where(small, z * z / 4, 0.25)
    term, harm, j, y = torch.ones_like(z), 0.0, torch.ones_like(z), torch.zeros_like(z)
    for k in range(1, 31):
        term = term * -q / (k * k)
        harm += 1.0 / k
        j = j + term
        y = y - harm * term
    y = (2 / math.pi) * ((torch.log(a / 2) + EULER) * j + y)
    b = torch.where(small, 5.0, z)
    hi, lo = torch.zeros_like(z), torch.full_like(z, 1e-300)   # J_{n+1}, J_n up to a factor, n = 170
    norm, neumann = 2 * lo, torch.zeros_like(z)
    for n in range(170, 0, -1):
        hi, lo = lo, (2 * n / b) * lo - hi                      # now lo = J_{n-1}
        if n % 2 == 1 and n > 1:
            norm = norm + 2 * lo
            neumann = neumann + (-1) ** ((n - 1) // 2) * lo / ((n - 1) // 2)
    norm = norm + lo
    jb = lo / norm
    yb = (2 / math.pi) * (torch.log(b / 2) + EULER) * jb - (4 / math.pi) * neumann / norm
    return torch.where(small, j, jb), torch.where(small, y, yb)


def _self_cell(h, kappa):
    """Integral of (i/4) H0(kappa |x|) over an h x h cell, by its symmetry one integral over an angle of
    rho H1(kappa rho) / kappa + 2i / (pi kappa^2), rho = h / (2 cos theta); H1 by its power series."""
    t, w = np.polynomial.legendre.leggauss(48)
    rho = 0.5 * h / np.cos((t + 1) * (math.pi / 8))
    z = kappa * rho
    j, y, psi = 0.0, 0.0, 1 - 2 * EULER   # psi: digamma(k + 1) + digamma(k + 2)
    for k in range(16):
        term = (-1) ** k * (z / 2) ** (2 * k + 1) / (math.factorial(k) * math.factorial(k + 1))
        j, y = j + term, y - psi * term / math.pi
        psi += 1.0 / (k + 1) + 1.0 / (k + 2)
    y = y + (2 / math.pi) * np.log(z / 2) * j     # Y1 + 2 / (pi z)
    return complex(2j * np.sum(w * (math.pi / 8) * (rho / kappa) * (j + 1j * y)))


def _operator(case, pts):
    """x -> A x for rows of x, by a circulant embedding of the grid's displacement kernel."""
    s, h, kappa = case["side"], 1.0 / case["side"], case["kappa"]
    d = torch.arange(2 * s, device="cuda", dtype=torch.float64)
    d = torch.where(d < s, d, d - 2 * s) * h
    r = torch.sqrt(d[:, None] ** 2 + d[None, :] ** 2)
    r[0, 0] = 1.0
    if case["kernel"] == "laplace":
        k = torch.log(r) * (-h * h / (2 * math.pi)) + 0j
    else:
        j, y = _j0_y0(kappa * r)
        k = torch.complex(-y, j) * (0.25 * h * h)
    k[0, 0] = 0.0
    spec = torch.fft.fft2(k)
    p = torch.from_numpy(pts).cuda()
    at = torch.round(p[:, 1] / h - 0.5).long() * s + torch.round(p[:, 0] / h - 0.5).long()
    weight, diag = 1.0, 1.0
    if case["kernel"] == "lippmann_schwinger":
        weight = kappa * torch.exp(-16.0 * ((p - 0.5) ** 2).sum(1))
        diag = 1.0 + weight ** 2 * _self_cell(h, kappa)

    def apply(x):
        grid = torch.zeros(x.shape[0], s * s, dtype=torch.complex128, device="cuda")
        grid[:, at] = (weight * x).to(torch.complex128)
        y = torch.fft.ifft2(torch.fft.fft2(grid.view(-1, s, s), s=(2 * s, 2 * s)) * spec)[:, :s, :s]
        y = diag * x + weight * y.reshape(-1, s * s)[:, at]
        return y if x.is_complex() else y.real

    return apply


def _gmres(apply, b, steps, cycles=6):
    """Restarted GMRES on each row of b (the operators are identity plus compact)."""
    x = torch.zeros_like(b)
    for _ in range(cycles):
        r = b - apply(x)
        beta = torch.linalg.vector_norm(r, dim=1, keepdim=True)
        if float((beta / torch.linalg.vector_norm(b, dim=1, keepdim=True)).max()) < 2e-16:
            break
        v = [r / beta.clamp_min(1e-300)]
        hess = torch.zeros(b.shape[0], steps + 1, steps, dtype=b.dtype, device="cuda")
        for j in range(steps):
            w = apply(v[j])
            for _ in range(2):
                for i in range(j + 1):
                    c = (v[i].conj() * w).sum(1)
                    hess[:, i, j] += c
                    w = w - c[:, None] * v[i]
            nw = torch.linalg.vector_norm(w, dim=1)
            hess[:, j + 1, j] = nw
            v.append(w / nw.clamp_min(1e-300)[:, None])
        e = torch.zeros(b.shape[0], steps + 1, 1, dtype=b.dtype, device="cuda")
        e[:, 0, 0] = beta[:, 0]
        q, t = torch.linalg.qr(hess)
        y = torch.linalg.solve_triangular(t, q.mH @ e, upper=True)[:, :, 0]
        if not bool(torch.isfinite(torch.view_as_real(y) if y.is_complex() else y).all()):
            break   # an exact breakdown: x is the solution already
        for j in range(steps):
            x = x + y[:, j:j + 1] * v[j]
    return x


def exact(case, seed):
    b = _rhs(case, seed)
    apply = _operator(case, _points(case, seed))
    steps = {"laplace": 20, "helmholtz": 40, "lippmann_schwinger": 150}[case["kernel"]]
    if b.dim() == 1:
        return _gmres(apply, b[None], steps)[0]
    cols = [_gmres(apply, c, steps) for c in b.T.contiguous().split(8)]
    return torch.cat(cols).T
