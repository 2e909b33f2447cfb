"""A step gives the same bits whichever way it is asked for: with the strips on a stream of their own or not
(sbp_set_tuning, sbp_autotune), from a graph, while the kernels are timed (sbp_profile); and the launches counted for a
graph are those counted for plain steps.  Single blocks and blocks without interfaces, where a step is one launch, with
strip tiles of 8 and 32 nodes, and larger ones, where it is several."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _problem(order, n, two):
    P = W.random_problem(kinds=("robin", "displacement", "displacement", "robin"), n=n, order=order, two_blocks=two)
    P.sources = [W.PointSource(0, x, (0.6, -0.8), 1.0, 3.0, 0.1) for x in ((0.5, 0.5), (0.0, 0.3))]
    return P


def _run(P, prec, how):
    from paper_2003_12811_gb300 import Solver
    S = Solver(P, prec)
    u, v = W.smooth_state(P), W.smooth_state(P, seed=5)
    dt = S.suggest_dt(0.25)
    S.set_state([a - dt * b for a, b in zip(u, v)], u, 0.05)
    if how == "overlap":
        S.sbp_set_tuning(0, 1)
    elif how == "autotuned":
        S.sbp_autotune()
    S.sbp_profile(how in ("profiled", "profiled graph"))
    if how != "profiled" and how != "profiled graph":
        S.sbp_profile(True)
        S.sbp_profile(False)                                # only the counters
    (S.sbp_step_graph if "graph" in how else S.step)(10, dt)
    out = S.state()
    n = S.sbp_profile_read()[1] if "profiled" not in how else None
    S.close()
    return out[0] + out[1], n


@pytest.mark.parametrize("prec,order,n,two", [("fp32", 6, (150, 141), False), ("fp32", 6, (27, 1300), False), ("fp32", 4, (700, 690), False),
                                              ("fp32", 6, (1300, 40), False), ("fp32", 6, (150, 90), True), ("fp64", 6, (61, 57), False),
                                              ("fp64", 4, (90, 61), True), ("fp64", 6, (331, 290), False), ("fp64", 2, (30, 29), False)])
def test_the_way_of_asking_does_not_change_results(prec, order, n, two):
    P = _problem(order, n, two)
    ref, launches = _run(P, prec, "plain")
    assert max(np.abs(a).max() for a in ref) > 0
    for how in ("overlap", "graph", "profiled", "profiled graph", "autotuned"):
        got, k = _run(P, prec, how)
        assert all(np.array_equal(a, b) for a, b in zip(got, ref)), how
        if how == "graph":
            assert list(k)[:2] + list(k)[3:4] == list(launches)[:2] + list(launches)[3:4]
