"""rss_solve_iterative does not read scratch that it never wrote.

The library's pool hands freed blocks to the next call, so the Krylov vectors
may start as any bits, NaN among them.  A solve of NaN right-hand sides leaves
its working copy (all NaN) in the pool; the iterative solve that follows must
give the same bits as one that ran before.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["laplace", "helmholtz"])
def test_iterative_solve_after_nan_scratch(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    side, cplx = 64, kind == "helmholtz"
    tree = P.rss_build_tree(W.grid_points(side), 64)
    f = P.rss_factor(tree, kind=P.HELMHOLTZ if cplx else P.LAPLACE, eps=1e-4, h=1.0 / side,
                     kappa=25.0 if cplx else 0.0)
    dt = torch.complex128 if cplx else torch.float64
    b = torch.from_numpy(W.gaussian_rhs(side * side, 1, cplx, 3)[:, 0].copy()).cuda()
    x0, it0, _ = P.rss_solve_iterative(f, b, tol=1e-13)
    assert it0 > 0
    for nrhs in (24, 30, 64):
        bad = torch.full((nrhs, side * side), float("nan"), dtype=dt, device="cuda").T
        P.rss_solve(f, bad)
        torch.cuda.synchronize()
        x, it, _ = P.rss_solve_iterative(f, b, tol=1e-13)
        assert it == it0
        assert np.array_equal(x.cpu().numpy(), x0.cpu().numpy())
