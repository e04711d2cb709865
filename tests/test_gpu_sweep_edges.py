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


@pytest.mark.parametrize("kind,side,leaf,eps,nrhs", [
    ("laplace", 48, 144, 1e-6, 32), ("laplace", 96, 144, 1e-9, 65), ("laplace", 64, 256, 1e-6, 33),
    ("laplace", 128, 256, 1e-10, 40), ("laplace", 80, 100, 1e-11, 64), ("laplace", 192, 144, 1e-6, 17),
    ("helmholtz", 48, 144, 1e-6, 16), ("helmholtz", 96, 144, 1e-9, 33), ("helmholtz", 64, 256, 1e-6, 17),
    ("helmholtz", 80, 100, 1e-10, 40)])
def test_boxes_of_more_than_one_row_tile(P, kind, side, leaf, eps, nrhs):
    """Boxes of 129 to about 400 points: the row tiles of one box read what the others
    write.  Against one-column solves, as in the panels of smaller boxes: at most four
    products of 6000 2^-53 for each class, below 1e-12 of the solution; repeated solves
    and any split into panels give the same bits."""
    cplx = kind == "helmholtz"
    f = P.rss_factor(P.rss_build_tree(W.grid_points(side), leaf), kind=P.HELMHOLTZ if cplx else P.LAPLACE, eps=eps,
                     h=1.0 / side, kappa=25.0 if cplx else 0.0)
    assert max(L["k_max"] for L in P.rss_info(f)["levels"]) * 4 > 128 or leaf > 128
    b = torch.from_numpy(np.ascontiguousarray(W.gaussian_rhs(side * side, nrhs, cplx, 5).T)).cuda()
    fly = b.clone()
    if b.numel() * b.element_size() <= 8 << 20:
        P.rss_solve_noalloc(f, fly.T)   # real: no digits kept yet, cut on the fly
    else:
        fly = None
    x = P.rss_solve(f, b.clone().T).T
    for _ in range(4):
        assert torch.equal(x, P.rss_solve(f, b.clone().T).T)
    for j in (0, 7, nrhs - 1):
        one = P.rss_solve(f, b[j].clone())
        assert float(torch.linalg.vector_norm(x[j] - one) / torch.linalg.vector_norm(one)) <= 1e-12, j
    if fly is not None:
        assert float(torch.linalg.vector_norm(fly - x) / torch.linalg.vector_norm(x)) <= 1e-12


def test_panel_without_memory_for_the_digits(P):
    """A real panel of 64 columns on a device whose memory is nearly all taken: the digits
    that the factor would keep do not fit, so they are cut per call (under the scales of a
    CTA's share of a long sum, so not to the same bits); with memory again, the same solve
    keeps them.  Both against one-column solves, as above."""
    side = 256
    f = P.rss_factor(P.rss_build_tree(W.grid_points(side), 64), eps=1e-6, h=1.0 / side)
    b = torch.from_numpy(np.ascontiguousarray(W.gaussian_rhs(side * side, 64, False, 4).T)).cuda()
    P.rss_solve(f, b[:15].clone().T)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    P.rss_trim_memory(0)
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(max(0, free - (600 << 20)), dtype=torch.uint8, device="cuda")
    x = P.rss_solve(f, b.clone().T).clone()
    torch.cuda.synchronize()
    del hold
    torch.cuda.empty_cache()
    P.rss_trim_memory(0)
    free = torch.cuda.mem_get_info()[0]
    y = P.rss_solve(f, b.clone().T)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] > 600 << 20   # (the digits, now)
    for j in (0, 31, 63):
        one = P.rss_solve(f, b[j].clone())
        for z in (x.T, y.T):
            assert float(torch.linalg.vector_norm(z[j] - one) / torch.linalg.vector_norm(one)) <= 1e-12, j
