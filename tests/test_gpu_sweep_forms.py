"""The FP64 sweeps by launch form, cluster size and column count: the same bits.

A column's sums have a fixed order whatever shares the launch: solving a panel must
give, column by column, the bits of one-column solves, for classes that take a
cluster of CTAs per box and for classes that fill the GPU (with more columns the
same class moves from one to the other), and the persistent form the bits of the
launches per class.  And A^{-1} must invert A: the residual by FFT stays below 10 eps.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,side,leaf,eps", [("laplace", 32, 1, 1e-6), ("laplace", 72, 81, 1e-6),
                                                ("laplace", 256, 64, 1e-6), ("laplace", 512, 64, 1e-4),
                                                ("helmholtz", 64, 64, 1e-6), ("helmholtz", 160, 25, 1e-5)])
def test_panels_and_forms_give_the_bits_of_single_columns(kind, side, leaf, eps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    cplx = kind == "helmholtz"
    tree = P.rss_build_tree(W.grid_points(side), leaf)
    arg = dict(kind=P.HELMHOLTZ if cplx else P.LAPLACE, eps=eps, h=1.0 / side, kappa=25.0 if cplx else 0.0)
    f = P.rss_factor(tree, **arg)
    b = W.gaussian_rhs(side * side, 15, cplx, 21)
    bt = torch.from_numpy(np.ascontiguousarray(b.T)).cuda().T
    one = {}
    for j in (0, 2, 4, 8, 14):
        one[j] = P.rss_solve(f, bt[:, j].clone())
    r = P.rss_matvec(f, one[0]) - bt[:, 0]
    assert float(torch.linalg.vector_norm(r) / torch.linalg.vector_norm(bt[:, 0])) <= 10 * eps
    for nrhs in (3, 5, 9, 15):
        x = P.rss_solve(f, bt[:, :nrhs].T.clone().T)   # (the solve overwrites its argument)
        for j in one:
            if j < nrhs:
                assert torch.equal(x[:, j], one[j]), (nrhs, j)
    q = P.rss_factor(tree, tune_table={"launch": "persistent", "spread": 1, "ctas_per_sm": 1}, **arg)
    assert torch.equal(P.rss_solve(q, bt[:, 0].clone()), one[0])
