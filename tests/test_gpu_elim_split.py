"""Sparsification, LU and inverses of a box (Eqs. 7, 8), with and without row exchanges.

Box sizes lie below, at and above the 16-row blocks and column groups of the
kernels, with few boxes per colour class (narrow groups) and many (wide groups).

* Exactly low-rank far field, small diagonal: the factorization is exact, so the
  solution equals the dense solve to rounding, 1e-12 max(1, cond(A)).
* Zero diagonal (Helmholtz) or a small negative one (Laplace): the LU of X_RR
  exchanges rows (on all but the smallest grid).  Near-ties may be resolved differently, so what is compared with
  the oracle does not depend on the exchanges: X_RR = P^T L U to the tolerance of a
  record, t = (1 + depth) max(1e-10, 1e-14 / eps), and E F = X_CR X_RR^{-1} X_RC to
  t cond(X_RR).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W
from oracle import rss as orss
from oracle.dense import dense_matrix
from oracle.rss import KernelSpec

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    return P


@pytest.mark.parametrize("kind", ["rpoly", "poly"])
@pytest.mark.parametrize("side,leaf", [(16, 4), (24, 9), (32, 16), (40, 25), (64, 4), (64, 64), (40, 100)])
def test_small_diagonal_matches_dense_solve(P, kind, side, leaf):
    cplx = kind == "poly"
    coef = (0.3, 0.5 - 0.2j, 0.7, 0.1 + 0.4j) if cplx else (0.3, 0.5, -0.7, 0.4)
    spec = KernelSpec(kind, h=1.0 / side, coef=coef, scale=0.02, diag=2e-3, phase=(3.0, -2.0) if cplx else (0.0, 0.0))
    pts = W.grid_points(side)
    f = P.rss_factor(P.rss_build_tree(pts, leaf), kind=P.TEST_POLY if cplx else P.TEST_RPOLY, eps=1e-13, h=spec.h,
                     diag=spec.diag, coef=coef, scale=spec.scale, phase=spec.phase)
    A = dense_matrix(pts, spec)
    b = W.gaussian_rhs(side * side, 2, cplx, 5)
    x = torch.from_numpy(np.ascontiguousarray(b.T)).cuda().T
    P.rss_solve(f, x)
    xd = np.linalg.solve(A, b)
    assert np.linalg.norm(x.cpu().numpy() - xd) <= 1e-12 * max(1.0, np.linalg.cond(A)) * np.linalg.norm(xd)


def unpivoted(LU, piv):
    X = (np.tril(LU, -1) + np.eye(len(piv))) @ np.triu(LU)
    for j in range(len(piv) - 1, -1, -1):
        X[[j, piv[j]]] = X[[piv[j], j]]
    return X


@pytest.mark.parametrize("kind,side,leaf,eps", [
    ("laplace", 16, 4, 1e-6), ("laplace", 32, 16, 1e-6), ("laplace", 40, 25, 1e-4), ("laplace", 64, 64, 1e-6),
    ("helmholtz", 24, 9, 1e-6), ("helmholtz", 32, 16, 1e-6), ("helmholtz", 56, 49, 1e-4)])
def test_row_exchanges_match_oracle(P, kind, side, leaf, eps):
    cplx = kind == "helmholtz"
    spec = KernelSpec(kind, h=1.0 / side, kappa=25.0 if cplx else 0.0, diag=0.0 if cplx else -1e-4)
    pts = W.grid_points(side)
    f = P.rss_factor(P.rss_build_tree(pts, leaf), kind=P.HELMHOLTZ if cplx else P.LAPLACE, eps=eps, h=spec.h,
                     kappa=spec.kappa, diag=spec.diag)
    fac = orss.factor(pts, spec, eps, leaf=leaf)
    sides = sorted({rec.side for rec in fac.records}, reverse=True)
    assert side == 16 or any((rec.piv != np.arange(rec.piv.size)).any() for rec in fac.records)
    for rec in fac.records:
        got = P.rss_box_record(f, rec.side, rec.box)
        tol = (1 + sides.index(rec.side)) * max(1e-10, 1e-14 / eps)
        X, Xg = unpivoted(rec.LU, rec.piv), unpivoted(got["LU"], got["piv"])
        assert np.linalg.norm(Xg - X) <= tol * np.linalg.norm(X), (rec.side, rec.box)
        S, Sg = rec.E @ rec.F, got["E"] @ got["F"]
        assert np.linalg.norm(Sg - S) <= tol * np.linalg.cond(X) * max(np.linalg.norm(S), 1e-300), (rec.side, rec.box)
