"""Calls from several host threads at once, each on its own stream and its own factor.

The factors' boxes differ in size, so the same kernels are launched with different
amounts of shared memory at the same time.  Every call must succeed and give the bits
that it gives alone.
"""
import threading

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


def in_threads(jobs):
    """Run the jobs in threads that start together; the first exception is raised here."""
    gate, errors = threading.Barrier(len(jobs)), []

    def body(job):
        try:
            gate.wait()
            job()
        except Exception as e:
            errors.append(e)

    ts = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def sizes(P, kind):
    cplx = kind == "helmholtz"
    arg = dict(kind=P.HELMHOLTZ if cplx else P.LAPLACE, eps=1e-6, kappa=25.0 if cplx else 0.0)
    return cplx, [(P.rss_build_tree(W.grid_points(side), leaf), dict(h=1.0 / side, **arg))
                  for side, leaf in ((32, 16), (88, 121), (64, 64))]


@pytest.mark.parametrize("kind", ["laplace", "helmholtz"])
@pytest.mark.parametrize("nrhs,form", [(32, "per_class"), (16, "per_class"), (2, "persistent")])
def test_solves_of_different_factors_in_threads(P, kind, nrhs, form):
    cplx, trees = sizes(P, kind)
    jobs = []
    for tree, arg in trees:
        f = P.rss_factor(tree, tune_table={"launch": form, "spread": 1, "ctas_per_sm": 1}, **arg)
        b = torch.from_numpy(np.ascontiguousarray(W.gaussian_rhs(tree.n, nrhs, cplx, 5).T)).cuda()
        want = P.rss_solve(f, b.clone().T).clone()

        def job(f=f, b=b, want=want):
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                for _ in range(150):
                    x = P.rss_solve(f, b.clone().T, stream=st)
                assert torch.equal(x, want)
            st.synchronize()

        jobs.append(job)
    torch.cuda.synchronize()
    in_threads(jobs)


@pytest.mark.parametrize("kind", ["laplace", "helmholtz"])
@pytest.mark.parametrize("id_cluster", [0, 2])
def test_factorizations_in_threads(P, kind, id_cluster):
    cplx, trees = sizes(P, kind)
    jobs = []
    for tree, arg in trees:
        b = torch.from_numpy(W.gaussian_rhs(tree.n, 1, cplx, 6)[:, 0].copy()).cuda()
        want = P.rss_solve(P.rss_factor(tree, id_cluster=id_cluster, **arg), b.clone()).clone()

        def job(tree=tree, arg=arg, b=b, want=want):
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                for _ in range(8):
                    x = P.rss_solve(P.rss_factor(tree, id_cluster=id_cluster, stream=st, **arg), b.clone(), stream=st)
                    assert torch.equal(x, want)
            st.synchronize()

        jobs.append(job)
    torch.cuda.synchronize()
    in_threads(jobs)
