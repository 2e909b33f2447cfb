"""Steps in one launch (strip and interior tiles side by side, sources and interface traces inside), against
the FP64 oracle and against the separate launches, over the grids at which its tables differ: short and long strip
tiles, interfaces aligned and reversed, sources on strips, off them and on both sides of a tile's edge, more blocks than
one launch takes.  Bars as in test_gpu_parity (FP64 1e-12, FP32 1e-4 relative L2 of stepped smooth fields)."""
import math

import numpy as np
import pytest

import workloads as W
from oracle.scheme import Oracle

pytestmark = pytest.mark.gpu

KINDS = ("robin", "displacement", "displacement", "robin")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _problem(order, n, two, rev):
    P = W.random_problem(kinds=KINDS, n=n, order=order, two_blocks=two, reversed_interface=rev)
    P.sources = [W.PointSource(0, x, (0.6, -0.8), 1.0, 3.0, 0.1) for x in ((0.5, 0.5), (0.0, 0.3), (0.47, 0.98))]
    return P


def _run(P, prec, steps, dt, overlap=False, graph=False):
    from paper_2003_12811_gb300 import Solver
    S = Solver(P, prec)
    u, v = W.smooth_state(P), W.smooth_state(P, seed=5)
    if overlap:
        S.sbp_set_tuning(0, 1)
    S.set_state([a - dt * b for a, b in zip(u, v)], u, 0.05)
    (S.sbp_step_graph if graph else S.step)(steps, dt)
    out = S.state()
    S.close()
    return out


@pytest.mark.parametrize("order,n,two,rev", [(2, (9, 7), False, False), (4, (40, 33), True, False), (6, (45, 37), True, True),
                                             (6, (150, 141), False, False), (6, (301, 63), True, False), (6, (27, 700), False, False),
                                             (6, (331, 290), False, False)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_steps(order, n, two, rev, prec):
    P = _problem(order, n, two, rev)
    O = Oracle(P)
    dt = O.suggest_dt(0.25)
    u, v = W.smooth_state(P), W.smooth_state(P, seed=5)
    _, ref, _ = O.leapfrog(O.pack([a - dt * b for a, b in zip(u, v)]), O.pack(u), 0.05, dt, 12)
    ref = O.unpack(ref)
    _, got = _run(P, prec, 12, dt)
    if prec == "fp64":
        assert max(np.abs(a - b).max() for a, b in zip(got, ref)) <= 1e-12 * max(np.abs(b).max() for b in ref)
    else:
        err = math.sqrt(sum(np.sum((a - b) ** 2) for a, b in zip(got, ref)) / sum(np.sum(b ** 2) for b in ref))
        assert err <= 1e-4, err
    # replayed from a graph: the same launches
    _, again = _run(P, prec, 12, dt, graph=True)
    assert all(np.array_equal(a, b) for a, b in zip(got, again))
    # the strips in a launch of their own: the same arithmetic but for the traces' rounding
    _, apart = _run(P, prec, 12, dt, overlap=True)
    tol = 1e-13 if prec == "fp64" else 2e-6
    assert max(np.abs(a - b).max() for a, b in zip(got, apart)) <= tol * max(np.abs(b).max() for b in ref)


def test_more_blocks_than_one_launch_takes():
    P = W.config2(n=28, nbx=3, nby=3)
    O = Oracle(P)
    dt = O.suggest_dt(0.25)
    u, v = W.smooth_state(P), W.smooth_state(P, seed=5)
    _, ref, _ = O.leapfrog(O.pack([a - dt * b for a, b in zip(u, v)]), O.pack(u), 0.05, dt, 8)
    _, got = _run(P, "fp64", 8, dt)
    ref = O.unpack(ref)
    assert max(np.abs(a - b).max() for a, b in zip(got, ref)) <= 1e-12 * max(np.abs(b).max() for b in ref)
