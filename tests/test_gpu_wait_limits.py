"""Bounded device waits that run out, kernel by kernel.

wait_polls = -1 makes every wait it governs give up without polling.  The kernels then
let what they issued finish, free their tensor memory and return, so the call reports the
timeout (rss_factor: RSS_ETIMEOUT; a solve: NaN in every entry) and the process goes on:
the same call with the default limits must succeed afterwards.  No GPU is hung or faulted.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    return P


def problem(P, kind, side, leaf, **kw):
    cplx = kind == "helmholtz"
    arg = dict(kind=P.HELMHOLTZ if cplx else P.LAPLACE, eps=1e-6, h=1.0 / side, kappa=25.0 if cplx else 0.0, **kw)
    return cplx, P.rss_build_tree(W.grid_points(side), leaf), arg


@pytest.mark.parametrize("kind,side,leaf", [("laplace", 64, 64), ("laplace", 128, 16), ("laplace", 256, 64),
                                            ("helmholtz", 64, 64), ("helmholtz", 96, 36)])
def test_tensor_core_sweeps(P, kind, side, leaf):
    """The products of the sweeps (digits kept by the factor, and cut on the fly) with 40
    columns; schur_mma_sync keeps the factorization off the waits that wait_polls governs."""
    cplx, tree, arg = problem(P, kind, side, leaf, schur_mma_sync=True)
    bad, good = P.rss_factor(tree, wait_polls=-1, **arg), P.rss_factor(tree, **arg)
    b = torch.from_numpy(np.ascontiguousarray(W.gaussian_rhs(tree.n, 40, cplx, 5).T)).cuda()
    if b.numel() * b.element_size() <= 8 << 20:
        x = b.clone()
        P.rss_solve_noalloc(bad, x.T)
        assert bool(torch.isnan(x).all())
    for _ in range(3):
        x = b.clone()
        P.rss_solve(bad, x.T)
        assert bool(torch.isnan(x).all())
    x, one = b.clone(), b[3].clone()
    P.rss_solve(good, x.T)
    P.rss_solve(bad, one)   # (one column: no bounded wait)
    assert float(torch.linalg.vector_norm(x[3] - one) / torch.linalg.vector_norm(one)) <= 1e-12


@pytest.mark.parametrize("kind,side,leaf,id_cluster", [
    ("laplace", 64, 64, 0), ("helmholtz", 64, 64, 0), ("laplace", 256, 16, 0),    # the ID's products, first
    ("laplace", 64, 64, 1), ("laplace", 128, 16, 1), ("laplace", 96, 36, 1),      # reflectors: panels, then Schur
    ("helmholtz", 64, 64, 1), ("helmholtz", 128, 16, 1), ("helmholtz", 96, 144, 1),
    ("laplace", 96, 144, 1), ("laplace", 64, 256, 1)])                            # FP64 panels: Schur alone
def test_factorization(P, kind, side, leaf, id_cluster):
    cplx, tree, arg = problem(P, kind, side, leaf, id_cluster=id_cluster)
    for _ in range(2):
        with pytest.raises(P.RSSError, match="ETIMEOUT") as ei:
            P.rss_factor(tree, wait_polls=-1, **arg)
        assert ei.value.status == 5
    b = torch.from_numpy(W.gaussian_rhs(tree.n, 1, cplx, 6)[:, 0].copy()).cuda()
    f = P.rss_factor(tree, **arg)
    r = P.rss_matvec(f, P.rss_solve(f, b.clone())) - b
    assert float(torch.linalg.vector_norm(r) / torch.linalg.vector_norm(b)) <= 1e-5
