"""The sweeps of 16 and more right-hand sides on the tensor cores, against one-column solves.

The slice products lose nothing that FP64 keeps: cutting at 55 bits of a row's and a
column's largest entry costs at most 6000 * 2^-53 per product, of which a solve has
four per class of at most 9 * 6 classes; one-column FP64 solves differ from exact ones by
as much.  Both together stay below 1e-12 of the solution's norm at the small condition
numbers of these factors' blocks.  The edges: rows and columns that are no multiple of
8, 32 or 64, boxes of fewer than 32 and of nearly 128 points, boxes of more (those
classes take the FP64 sweeps), inner dimensions past one exact stretch, one column
group's remainder of a single column, the digits cached by the factor and cut on the fly.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,side,leaf,eps,nrhs", [
    ("laplace", 32, 4, 1e-6, 32), ("laplace", 72, 81, 1e-7, 65), ("laplace", 96, 144, 1e-4, 33),
    ("laplace", 88, 121, 1e-6, 64), ("laplace", 160, 25, 1e-5, 130), ("laplace", 256, 64, 1e-6, 40), ("laplace", 128, 64, 1e-6, 16), ("laplace", 96, 36, 1e-5, 31),
    ("helmholtz", 32, 16, 1e-6, 16), ("helmholtz", 48, 36, 1e-6, 17), ("helmholtz", 72, 81, 1e-7, 33), ("helmholtz", 96, 144, 1e-4, 64),
    ("helmholtz", 128, 64, 1e-6, 65)])
def test_panel_on_tensor_cores_equals_fp64_columns(kind, side, leaf, eps, nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    cplx = kind == "helmholtz"
    tree = P.rss_build_tree(W.grid_points(side), leaf)
    arg = dict(kind=P.HELMHOLTZ if cplx else P.LAPLACE, eps=eps, h=1.0 / side, kappa=25.0 if cplx else 0.0)
    f = P.rss_factor(tree, **arg)
    b = torch.from_numpy(np.ascontiguousarray(W.gaussian_rhs(side * side, nrhs, cplx, 5).T)).cuda().T
    fly = b.T.clone().T
    if side * side * nrhs <= 1 << 18:
        P.rss_solve_noalloc(f, fly)          # no digits yet: cut on the fly
    else:
        fly = None
    x = P.rss_solve(f, b.T.clone().T)
    y = P.rss_solve(f, b.T.clone().T)
    assert torch.equal(x, y)
    for j in sorted({0, 1, 15, nrhs - 1}):
        one = P.rss_solve(f, b[:, j].clone())
        rel = float(torch.linalg.vector_norm(x[:, j] - one) / torch.linalg.vector_norm(one))
        assert rel <= 1e-12, (j, rel)
    if fly is not None:
        assert float(torch.linalg.vector_norm(fly - x) / torch.linalg.vector_norm(x)) <= 1e-12


def test_small_requests_keep_their_bits_in_a_wide_complex_panel():
    """Requests of fewer than 16 columns take the FP64 sweeps alone, so also in a panel
    of 16 and more: the same bits."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    f = P.rss_factor(P.rss_build_tree(W.grid_points(32), 16), kind=P.HELMHOLTZ, eps=1e-6, h=1.0 / 32, kappa=25.0)
    srv = P.rss_server_create(1 << 30, 64)
    fid = P.rss_server_add(srv, f)
    bs = [W.gaussian_rhs(32 * 32, 1 + q % 15, True, 70 + q) for q in range(24)]
    tickets = [P.rss_server_submit(srv, fid, b) for b in bs]
    for b, t in zip(bs, tickets):
        x, _ = P.rss_server_wait(srv, t, timeout=60.0)
        solo = np.asfortranarray(b.copy())
        P.rss_solve(f, solo)
        assert np.array_equal(x, solo)
