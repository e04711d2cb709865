"""Small complex requests packed into wide panels: the large colour classes take the
tensor-core products, the others the FP64 sweeps.  Every result equals the request's own
solve to rounding (1e-12, as for real factors), in panels of a few columns exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,leaf,columns,packed", [(256, 16, 1, 64), (192, 36, 5, 64), (256, 64, 3, 128), (256, 16, 1, 20)])
def test_small_complex_requests_in_panels(side, leaf, columns, packed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    f = P.rss_factor(P.rss_build_tree(W.grid_points(side), leaf), kind=P.HELMHOLTZ, eps=1e-6, h=1.0 / side, kappa=25.0)
    srv = P.rss_server_create(4 << 30, packed)
    fid = P.rss_server_add(srv, f)
    bs = [W.gaussian_rhs(side * side, columns, True, 40 + q) for q in range(2 * packed // columns)]
    tickets = [P.rss_server_submit(srv, fid, b) for b in bs]
    worst = 0.0
    for q, (b, t) in enumerate(zip(bs, tickets)):
        x, _ = P.rss_server_wait(srv, t, timeout=120.0)
        if q % 8 == 0 or q == len(bs) - 1:
            solo = np.asfortranarray(b.copy())
            P.rss_solve(f, solo)
            worst = max(worst, np.linalg.norm(x - solo) / np.linalg.norm(solo))
    assert worst <= (1e-12 if packed >= 32 else 0.0)
    assert P.rss_server_stats(srv)["max_requests_per_batch"] > 1
