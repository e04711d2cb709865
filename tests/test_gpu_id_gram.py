"""The ID from the exact Gram matrix against the oracle's Householder QR.

Ranks, index sets (in pivot order) and LU pivots must be identical; T agrees in
norm within (1 + depth) max(1e-10, 1e-14 / eps) (the rounding of R11^{-1},
cond(R11) ~ 1 / eps, once per compressed level below); the solution agrees with
the oracle's to 1e-9.  The sizes cover one column block and several (n_B below
and above 32, 64 and 96, not multiples of them), stacks of one and of several
512-row parts, a part that ends inside a 32-row block, proxy counts off the block
size, and complex stacks.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W
from oracle import rss as orss
from oracle.rss import KernelSpec

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

CASES = [   # kind, side, leaf, eps, kappa, proxy_n
    ("laplace", 32, 1, 1e-6, 0.0, 7),
    ("laplace", 32, 4, 1e-9, 0.0, 64),
    ("laplace", 40, 25, 1e-5, 0.0, 33),
    ("laplace", 56, 49, 1e-7, 0.0, 64),
    ("laplace", 64, 64, 1e-8, 0.0, 64),
    ("laplace", 72, 81, 1e-9, 0.0, 100),
    ("laplace", 80, 100, 1e-4, 0.0, 64),
    ("laplace", 64, 256, 1e-6, 0.0, 64),   # G too large for one CTA: the reflectors
    ("helmholtz", 40, 25, 1e-6, 25.0, 64),
    ("helmholtz", 64, 64, 1e-9, 40.0, 65),
    ("ls", 64, 64, 1e-6, 30.0, 64),
    ("ls", 72, 81, 1e-4, 12.0, 31),
]


@pytest.mark.parametrize("kind,side,leaf,eps,kappa,proxy_n", CASES)
def test_gram_id_matches_oracle(kind, side, leaf, eps, kappa, proxy_n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    pk = {"laplace": P.LAPLACE, "helmholtz": P.HELMHOLTZ, "ls": P.HELMHOLTZ_LS}[kind]
    ls, pts = kind == "ls", W.grid_points(side)
    f = P.rss_factor(P.rss_build_tree(pts, leaf), kind=pk, eps=eps, h=1.0 / side, kappa=kappa,
                     proxy_n=proxy_n, diag_rule=1 if ls else 0)
    diag = P.rss_self_integral(pk, 1.0 / side, kappa) if ls else 1.0
    fac = orss.factor(pts, KernelSpec(kind, h=1.0 / side, kappa=kappa, diag=diag), eps, leaf=leaf, nproxy=proxy_n)
    sides = sorted({rec.side for rec in fac.records}, reverse=True)
    for rec in fac.records:
        got = P.rss_box_record(f, rec.side, rec.box)
        for name, want in (("S", rec.S), ("R", rec.R), ("C", rec.C), ("piv", rec.piv)):
            assert np.array_equal(got[name], want), (rec.side, rec.box, name)
        if rec.T.size:
            tol = (1 + sides.index(rec.side)) * max(1e-10, 1e-14 / eps)
            assert np.linalg.norm(got["T"] - rec.T) < tol * np.linalg.norm(rec.T), (rec.side, rec.box)
    b = W.gaussian_rhs(side * side, 2, kind != "laplace", 9)
    x = torch.from_numpy(np.ascontiguousarray(b.T)).cuda().T
    P.rss_solve(f, x)
    xo = orss.solve(fac, b)
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-9 * np.linalg.norm(xo)
