"""The tensor-core sweeps at the edges of what a colour class may hold."""
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


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("side,leaf", [(32, 16), (64, 64), (128, 4)])
@pytest.mark.parametrize("nrhs", [16, 40])
def test_classes_without_neighbours_left(P, cplx, side, leaf, nrhs):
    """A = 2 I: every box has rank 0, and the last colour classes have c = 0, so their
    product with E has no row.  Solves of several panels in a row, one stream: x = b / 2
    (products rounded at 2^-53 of a column's largest entry)."""
    f = P.rss_factor(P.rss_build_tree(W.grid_points(side), leaf), kind=P.TEST_POLY if cplx else P.TEST_RPOLY, eps=1e-6,
                     h=1.0 / side, coef=(), diag=2.0)
    b = [torch.from_numpy(np.ascontiguousarray(W.gaussian_rhs(side * side, nrhs, cplx, s).T)).cuda() for s in range(8)]
    x = [P.rss_solve(f, v.clone().T) for v in b]
    for v, w in zip(b, x):
        assert float(torch.linalg.vector_norm(w.T - v / 2) / torch.linalg.vector_norm(v)) < 1e-15
