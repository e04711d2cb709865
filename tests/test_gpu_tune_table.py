"""rss_tune_solve times every launch form once: candidates that differ only in "spread",
which no form uses, are the same launches and carry the same time."""
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,nrhs", [("laplace", 1), ("helmholtz", 5)])
def test_candidates_of_one_form_share_their_time(kind, nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_15458_gb300 as P
    f = P.rss_factor(P.rss_build_tree(W.grid_points(64), 16), kind=P.HELMHOLTZ if kind == "helmholtz" else P.LAPLACE,
                     eps=1e-6, h=1.0 / 64, kappa=25.0 if kind == "helmholtz" else 0.0)
    table = P.rss_tune_solve(f, nrhs)
    forms = {}
    for c in table["candidates"]:
        forms.setdefault((c["launch"], c.get("ctas_per_sm"), c.get("tail_boxes")), set()).add(c["ms"])
    assert len(table["candidates"]) == 11 and len(forms) == 6
    assert all(len(ms) == 1 for ms in forms.values())
    assert table["ms"] == min(min(ms) for ms in forms.values())
