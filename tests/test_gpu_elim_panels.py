"""E and F of Eqs. 7, 8 as digit products (tcgen05) against the FP64 panels.

Box sizes at the edges of the products: n below one stage of K, at most and above
three stages (tiles of 128 and of 96 rows), above 64 for complex boxes (several
stretches of K), r with a last group of at most and of more than 16 columns, one box
per colour class (passes shared by CTAs) and many.  Where the pivots agree, E and F
agree to the tolerance of a record, t = (1 + depth) max(1e-10, 1e-14 / eps) (depth:
levels eliminated before).  The blocks of later classes and levels hold the Schur
updates of earlier ones, so those (complex: r up to 32, 48, 192 and above; real: tiles and
row blocks, one triangle formed and mirrored; boxes of
one class with more and fewer stages) are compared with the FP64 ones as well.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,side,leaf,eps", [
    ("laplace", 32, 16, 1e-6), ("laplace", 64, 4, 1e-8), ("laplace", 72, 81, 1e-6), ("laplace", 88, 121, 1e-6),
    ("laplace", 128, 64, 1e-4), ("laplace", 160, 100, 1e-6), ("helmholtz", 32, 16, 1e-6), ("helmholtz", 32, 4, 1e-8),
    ("helmholtz", 96, 144, 1e-6), ("helmholtz", 80, 100, 1e-4), ("helmholtz", 128, 64, 1e-6),
    ("helmholtz", 64, 256, 1e-4), ("laplace", 256, 64, 1e-6), ("laplace", 256, 16, 1e-4)])
def test_panels_on_tensor_cores_match_fp64(kind, side, leaf, eps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    cplx = kind == "helmholtz"
    tree = P.rss_build_tree(W.grid_points(side), leaf)
    arg = dict(kind=P.HELMHOLTZ if cplx else P.LAPLACE, eps=eps, h=1.0 / side, kappa=25.0 if cplx else 0.0)
    f = P.rss_factor(tree, **arg)
    q = P.rss_factor(tree, schur_fp64=True, **arg)
    g = side // int(round(leaf ** 0.5))
    depth, compared = 0, 0
    while g >= 4:
        for box in range(g * g):
            try:
                a, b = P.rss_box_record(f, g, box), P.rss_box_record(q, g, box)
            except P.RSSError:   # (a box that eliminates nothing has no record)
                continue
            if not (np.array_equal(a["S"], b["S"]) and np.array_equal(a["R"], b["R"]) and np.array_equal(a["piv"], b["piv"])):
                continue
            assert np.array_equal(a["C"], b["C"])
            for key in ("E", "F"):
                if b[key].size:
                    e = np.linalg.norm(a[key] - b[key]) / np.linalg.norm(b[key])
                    assert e < (1 + depth) * max(1e-10, 1e-14 / eps), (g, box, key, e)
            compared += 1
        g //= 2
        depth += 1
    assert compared >= 16   # (boxes of 4 points eliminate nothing)
